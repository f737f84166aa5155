// Batched forward pass of assembled substrate networks: every non-input node takes
// the sigmoid of the weighted sum of its sources' previous values, all nodes at
// once (synchronous update), for a fixed number of steps; input nodes hold the
// pattern. Patterns share the pass: node values are [node][pattern] in shared
// memory, two buffers.
//
// Networks are very unequal (most of a population's are empty, the largest hold
// nearly all connections), so what bounds the call is the largest network: its
// connections, 8 bytes each, are read from L2 once a step, and each reads its
// source's values from shared memory. A network above kAnnClusterConns connections
// therefore takes a cluster of 8 CTAs, its nodes divided by connections; every CTA
// keeps a copy of all values and writes its nodes' new values into the 8 copies
// (distributed shared memory), one cluster barrier a step. Smaller networks take a
// CTA each, in a second launch that overlaps the first. Within a CTA a group of
// lanes takes a node and strides over its connections (coalesced loads, ascending
// sources, so that the value reads rarely conflict), summed by shuffles; the group is
// a warp, or 8 lanes where a network's nodes have few connections (in a CTA of its own:
// 4 lanes where it has many nodes).
//
// Measured with 4 patterns and 3 steps, against a thread per (node, pattern) in one
// CTA per network: 1000 networks, the largest of hundreds of thousands of connections,
// 658, 528 and 1054 -> 73, 50 and 74 us. The largest alone takes 14 us a step (clusters of 16: 10 us,
// but the networks beside it then share its SMs: 85 us for the 1000).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "../../include/emr.h"

namespace {

namespace cg = cooperative_groups;

constexpr int kAnnCluster = 8;               // CTAs of a large network (the portable cluster size)
constexpr int kAnnThreads = 512;             // threads of each
constexpr int kAnnSmallThreads = 256;        // threads of a CTA with a network of its own
constexpr int kAnnAhead = 4;                 // connections a lane has in flight
// Connections above which a network takes a cluster (a cluster's barrier and copies cost a small
// network more than the other SMs save), with 2048, 4096, 8192, 16384: 1000 networks, the largest of
// hundreds of thousands, 78, 79, 73, 72 us; 29 networks, the largest of 10.7 K, 21, 20, 21, 29.
constexpr int64_t kAnnClusterConns = 8192;
// Connections that the nodes of a network can have, up to which no network takes one and the first
// launch, 8 us of the call when it finds none, is left out (952 networks of up to 4.7 K: 30.5 -> 22.5 us, 19 with the sigmoids over the lanes).
constexpr int64_t kAnnNoClusters = 2 * kAnnClusterConns;
constexpr int kAnnWideDegree = 16;           // connections a node from which a whole warp takes a node

struct AnnArgs {
  int32_t P, n_in, n_out, K, steps;
  const int64_t *node_off, *conn_off;
  const int32_t *conn_src, *conn_dst;
  const float *conn_w, *patterns;
  float* out;
  int64_t cluster_conns;  // connections above which a network is ann_large_kernel's
};

// V values at p (V * 4 byte aligned for V > 1)
template <int V>
__device__ __forceinline__ void load_values(const float* p, float (&v)[V]) {
  if constexpr (V == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else if constexpr (V == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = p[0];
  }
}

// First connection in [lo, hi) whose destination is at least n, by a whole warp (32-ary search).
__device__ __forceinline__ int64_t first_of(const int32_t* __restrict__ dst, int64_t lo, int64_t hi, int32_t n) {
  const int lane = threadIdx.x & 31;
  while (hi > lo) {
    const int64_t step = (hi - lo + 31) / 32, at = lo + step * (lane + 1) - 1;
    const unsigned below = __ballot_sync(0xffffffffu, at < hi && dst[at] < n);  // a prefix of the probes
    lo += step * __popc(below);
    hi = min(hi, lo + step - 1);
  }
  return lo;
}

// One step of the CTA's nodes [n_lo, n_hi), G lanes a node.
template <int V, int KC, int G, int NT, bool CLUSTER>
__device__ __forceinline__ void ann_step(const AnnArgs& A, const cg::cluster_group& cl, const float* cur, float* nxt,
                                         const int32_t* in_beg, int32_t n_lo, int32_t n_hi,
                                         const int32_t* __restrict__ src, const float* __restrict__ w) {
  const int gl = threadIdx.x % G, K = A.K;
  for (int32_t b = n_lo + int(threadIdx.x & ~31u) / G; b < n_hi; b += NT / G) {  // warp-uniform
    const int32_t n = b + int(threadIdx.x & 31u) / G;
    const bool valid = n < n_hi;
    const int32_t e0 = valid ? in_beg[n - n_lo] : 0, e1 = valid ? in_beg[n - n_lo + 1] : 0;
    for (int k0 = 0; k0 < K; k0 += KC) {
      float z[KC];
#pragma unroll
      for (int j = 0; j < KC; j++) z[j] = 0.f;
      auto add = [&](int32_t s, float we) {
#pragma unroll
        for (int j = 0; j < KC; j += V) {
          if (V == 1 && k0 + j >= K) break;
          float v[V];
          load_values<V>(cur + size_t(s) * K + k0 + j, v);
#pragma unroll
          for (int i = 0; i < V; i++) z[j + i] = fmaf(we, v[i], z[j + i]);
        }
      };
      int32_t e = e0 + gl;
      for (; e < e1; e += kAnnAhead * G) {  // kAnnAhead connections in flight
        int32_t s[kAnnAhead];
        float we[kAnnAhead];
#pragma unroll
        for (int i = 0; i < kAnnAhead; i++)
          if (e + i * G < e1) { s[i] = src[e + i * G]; we[i] = w[e + i * G]; }
#pragma unroll
        for (int i = 0; i < kAnnAhead; i++)
          if (e + i * G < e1) add(s[i], we[i]);
      }
      __syncwarp();
#pragma unroll
      for (int o = G / 2; o; o >>= 1) {
#pragma unroll
        for (int j = 0; j < KC; j++) z[j] += __shfl_xor_sync(0xffffffffu, z[j], o);
      }
      float* to = nxt + size_t(n) * K + k0;
      if constexpr (CLUSTER) {
        if (valid && gl < kAnnCluster) {  // lane l writes copy l
          to = cl.map_shared_rank(to, gl);
#pragma unroll
          for (int j = 0; j < KC; j++)
            if (k0 + j < K) to[j] = 1.f / (1.f + expf(-z[j]));
        }
      } else {  // every lane has every pattern's sum: lane l takes patterns l, l + G, ...
#pragma unroll
        for (int j0 = 0; j0 < KC; j0 += G) {
          float zl = z[j0];
#pragma unroll
          for (int i = 1; i < G && j0 + i < KC; i++) zl = gl == i ? z[j0 + i] : zl;
          const int j = j0 + gl;
          if (valid && j < KC && k0 + j < K) to[j] = 1.f / (1.f + expf(-zl));
        }
      }
    }
  }
}

// Network g by one CTA, or (CLUSTER) by the cluster, whose CTAs all call this. MID: a CTA's network
// may have more than kAnnClusterConns connections.
template <int V, int KC, int NT, bool CLUSTER, bool MID>
__device__ __forceinline__ void ann_network(const AnnArgs& A, const cg::cluster_group& cl, int64_t g, float* sm) {
  const int tid = threadIdx.x, K = A.K;
  const int32_t N = A.n_in + A.n_out + int32_t(A.node_off[g + 1] - A.node_off[g]);
  const int64_t c0 = A.conn_off[g], C = A.conn_off[g + 1] - c0;
  const int32_t* dst = A.conn_dst + c0;
  float* cur = sm;
  float* nxt = sm + size_t(N) * K;
  int32_t* in_beg = reinterpret_cast<int32_t*>(sm + 2 * size_t(N) * K);  // connections into the CTA's nodes
  const int rank = CLUSTER ? int(cl.block_rank()) : 0, ranks = CLUSTER ? kAnnCluster : 1;
  if (tid < 64) {  // the CTA's nodes, so that each takes about C / ranks connections, and their connections
    const int q = rank + (tid >> 5);
    int32_t n = q == 0 ? A.n_in : q == ranks ? N : dst[C * q / ranks];
    n = min(max(n, A.n_in), N);
    const int64_t e = q == ranks ? C : first_of(dst, 0, C, n);
    if ((tid & 31) == 0) {  // (in the values' place: N >= 2)
      reinterpret_cast<int32_t*>(sm)[tid >> 5] = n;
      reinterpret_cast<int32_t*>(sm)[2 + (tid >> 5)] = int32_t(e);
    }
  }
  __syncthreads();
  const int32_t* range = reinterpret_cast<const int32_t*>(sm);
  const int32_t n_lo = range[0], n_hi = max(range[1], n_lo), e_lo = range[2], e_hi = max(range[3], e_lo);
  __syncthreads();
  for (int32_t t = tid; t < N * K; t += NT) {
    const int32_t n = t / K, k = t - n * K;
    const float v = n < A.n_in ? A.patterns[size_t(k) * A.n_in + n] : 0.f;
    cur[t] = v;
    nxt[t] = v;
  }
  // connections are sorted by destination: node n's are [in_beg[n - n_lo], in_beg[n - n_lo + 1])
  for (int32_t e0 = e_lo + tid; e0 <= e_hi; e0 += kAnnAhead * NT) {
    int32_t a[kAnnAhead], b[kAnnAhead];
#pragma unroll
    for (int i = 0; i < kAnnAhead; i++) {
      const int32_t e = e0 + i * NT;
      a[i] = e > e_lo && e <= e_hi ? dst[e - 1] : n_lo - 1;
      b[i] = e < e_hi ? dst[e] : n_hi;
    }
#pragma unroll
    for (int i = 0; i < kAnnAhead; i++) {
      const int32_t e = e0 + i * NT;
      if (e <= e_hi)
        for (int32_t n = max(a[i] + 1, n_lo); n <= min(b[i], n_hi); n++) in_beg[n - n_lo] = e;
    }
  }
  if constexpr (CLUSTER) cl.sync(); else __syncthreads();
  const int32_t* src = A.conn_src + c0;
  const float* w = A.conn_w + c0;
  // Lanes a node. A large network: by its nodes' connections. A small one: as many as give every node
  // its lanes at once, 4 at least, since a pass over the nodes costs more in latency than connections
  // (952 networks of up to 95 nodes and 4.7 K connections, 4 patterns, 5 steps: 67 us with a warp a node from 16
  // connections a node on, 8 lanes below; 35 so, before the larger of them left the clusters).
  // The lanes set the order of a node's sum, so they follow from the network alone: its bits are the
  // same in every call. Up to kAnnNoClusters connections, where the call's other networks decide between
  // a CTA and a cluster, 8 in both (30 batches of 200 networks, the largest of 110 to 700 hidden nodes, 1 to 16
  // patterns, 4 steps: 35.9 us in the mean, 36.8 with each kernel's own rule there).
  const int32_t nodes = n_hi - n_lo;
  const int32_t degree = C > kAnnNoClusters ? kAnnWideDegree : int32_t(kAnnNoClusters) + 1;  // (no node has as many)
  const bool eight = MID && C > kAnnClusterConns;
  const bool wide = CLUSTER ? e_hi - e_lo >= degree * nodes : !eight && nodes <= NT / 32;
  const bool narrow = !CLUSTER && !eight && nodes > NT / 8;
  for (int32_t step = 0; step < A.steps; step++) {
    if (wide)
      ann_step<V, KC, 32, NT, CLUSTER>(A, cl, cur, nxt, in_beg, n_lo, n_hi, src, w);
    else if (CLUSTER || !narrow)
      ann_step<V, KC, 8, NT, CLUSTER>(A, cl, cur, nxt, in_beg, n_lo, n_hi, src, w);
    else
      ann_step<V, KC, 4, NT, CLUSTER>(A, cl, cur, nxt, in_beg, n_lo, n_hi, src, w);
    if constexpr (CLUSTER) cl.sync(); else __syncthreads();
    float* tmp = cur;
    cur = nxt;
    nxt = tmp;
  }
  if (rank == 0)
    for (int32_t t = tid; t < K * A.n_out; t += NT) {
      const int32_t k = t / A.n_out, o = t - k * A.n_out;
      A.out[(size_t(g) * K + k) * A.n_out + o] = cur[size_t(A.n_in + o) * K + k];
    }
  __syncthreads();  // the buffers are free
}

// V: values a load (K a multiple of it), KC: patterns a pass over the connections.
//
// The large networks, dealt to the clusters in turn (every warp finds the same ones).
template <int V, int KC>
__global__ void __launch_bounds__(kAnnThreads, 1024 / kAnnThreads) ann_large_kernel(const AnnArgs A) {
  extern __shared__ __align__(16) float sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // the small networks fill the SMs left free
  const cg::cluster_group cl = cg::this_cluster();
  const int lane = threadIdx.x & 31;
  const int64_t n_cl = gridDim.x / kAnnCluster, my = blockIdx.x / kAnnCluster;
  constexpr int kRounds = 8;  // 32 networks each, loaded together
  int64_t n_big = 0;
  for (int64_t g0 = 0; g0 < A.P; g0 += 32 * kRounds) {
    unsigned big[kRounds];
#pragma unroll
    for (int k = 0; k < kRounds; k++) {
      const int64_t g = g0 + 32 * k + lane;
      big[k] = g < A.P && A.conn_off[g + 1] - A.conn_off[g] > A.cluster_conns;
    }
#pragma unroll
    for (int k = 0; k < kRounds; k++) big[k] = __ballot_sync(0xffffffffu, big[k]);
#pragma unroll 1
    for (int k = 0; k < kRounds; k++) {
      unsigned b = 0;
#pragma unroll
      for (int i = 0; i < kRounds; i++) b = i == k ? big[i] : b;
      for (; b; b &= b - 1, n_big++)
        if (n_big % n_cl == my) ann_network<V, KC, kAnnThreads, true, false>(A, cl, g0 + 32 * k + __ffs(b) - 1, sm);
    }
  }
}

// The other networks, a CTA each. Launched to overlap ann_large_kernel (they share no output);
// the last CTA waits for it as it exits, so that this launch completes after it.
template <int V, int KC, bool MID>
__global__ void __launch_bounds__(kAnnSmallThreads, 1024 / kAnnSmallThreads) ann_small_kernel(const AnnArgs A) {
  extern __shared__ __align__(16) float sm[];
  const int64_t g = blockIdx.x;
  const cg::cluster_group cl = cg::this_cluster();
  if (A.conn_off[g + 1] - A.conn_off[g] <= A.cluster_conns)
    ann_network<V, KC, kAnnSmallThreads, false, MID>(A, cl, g, sm);
  if (g == A.P - 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <int V, int KC>
cudaError_t launch_ann(AnnArgs A, int64_t max_conns, size_t smem, int sms, cudaStream_t st) {
  cudaError_t e;
  // (the variant for networks that stay off the clusters despite their connections: its rule, taken by
  // all, made the others' steps slower, 21.5 -> 24.3 us for 200 networks and one pattern)
  const auto small = max_conns > kAnnClusterConns && max_conns <= kAnnNoClusters ? ann_small_kernel<V, KC, true>
                                                                                : ann_small_kernel<V, KC, false>;
  if (smem > 48 * 1024) {
    if ((e = cudaFuncSetAttribute(ann_large_kernel<V, KC>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) !=
            cudaSuccess ||
        (e = cudaFuncSetAttribute(small, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) != cudaSuccess)
      return e;
  }
  const int64_t clusters = std::max<int64_t>(1, std::min<int64_t>(A.P, 2 * sms / kAnnCluster));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(clusters * kAnnCluster));
  cfg.blockDim = dim3(kAnnThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kAnnCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (max_conns <= kAnnNoClusters) {
    A.cluster_conns = INT64_MAX;
    cfg.numAttrs = 0;
  } else if ((e = cudaLaunchKernelEx(&cfg, ann_large_kernel<V, KC>, A)) != cudaSuccess) {
    return e;
  }
  cfg.gridDim = dim3(unsigned(A.P));
  cfg.blockDim = dim3(kAnnSmallThreads);
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  return cudaLaunchKernelEx(&cfg, small, A);
}

}  // namespace

extern "C" emr_status emr_ann_forward(int32_t P, int32_t n_in, int32_t n_out, int32_t max_hidden,
                                      const int64_t* node_off, const int64_t* conn_off, const int32_t* conn_src,
                                      const int32_t* conn_dst, const float* conn_w, int32_t K, const float* patterns,
                                      int32_t steps, float* out, void* stream) {
  if (P <= 0 || n_in <= 0 || n_out <= 0 || max_hidden < 0 || K <= 0 || steps < 0 || !node_off || !conn_off ||
      !patterns || !out)
    return EMR_ERR_ARG;
  const size_t N = size_t(n_in) + size_t(n_out) + size_t(max_hidden);
  const size_t smem = 2 * N * size_t(K) * 4 + (N + 1) * 4;
  int dev = 0, limit = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return EMR_ERR_CUDA;
  if (smem > size_t(limit)) return EMR_ERR_RANGE;
  const AnnArgs A{P, n_in, n_out, K, steps, node_off, conn_off, conn_src, conn_dst, conn_w, patterns, out,
                  kAnnClusterConns};
  // a pair of nodes is connected at most once (were it more, every network would take a CTA: slower, not wrong)
  const int64_t max_conns = int64_t(N) * int64_t(N - size_t(n_in));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  if (K % 8 == 0) e = launch_ann<4, 8>(A, max_conns, smem, sms, st);
  else if (K % 4 == 0) e = launch_ann<4, 4>(A, max_conns, smem, sms, st);
  else if (K == 2) e = launch_ann<2, 2>(A, max_conns, smem, sms, st);
  else if (K == 1) e = launch_ann<1, 1>(A, max_conns, smem, sms, st);
  else if (K == 3) e = launch_ann<1, 4>(A, max_conns, smem, sms, st);
  else e = launch_ann<1, 8>(A, max_conns, smem, sms, st);
  if (e != cudaSuccess) return EMR_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? EMR_OK : EMR_ERR_CUDA;
}
