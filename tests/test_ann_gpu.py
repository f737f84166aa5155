"""The forward pass at the edges of its work split: networks on both sides of the size that takes a
cluster of CTAs, node degrees on both sides of a warp per node, empty networks, every pattern count's
load width, and zero steps, against a float64 pass over dense matrices."""
import numpy as np
import pytest
import torch

from paper_2608_27612_gb300 import emr


def _networks(sizes, density, n_in, n_out, seed, acyclic=False):
    rng = np.random.default_rng(seed)
    src, dst, n_conn = [], [], []
    for H in sizes:
        N = n_in + n_out + H
        m = rng.random((N, N)) < density
        m[:n_in] = False
        if acyclic:
            m &= np.tri(N, N, -1, dtype=bool)
        d, s = np.nonzero(m)
        src.append(s), dst.append(d)
        n_conn.append(len(s))
    off = lambda v: np.concatenate([[0], np.cumsum(v)]).astype(np.int64)
    cat = lambda v: np.concatenate(v).astype(np.int32)
    w = rng.normal(0, 1, sum(n_conn)).astype(np.float32)
    return emr.Networks(n_in, n_out, off(sizes), np.zeros(sum(sizes), np.int32), off(n_conn), cat(src), cat(dst), w,
                        np.zeros(len(w), np.uint8))


def _reference(nets, pat, steps):
    """Outputs in float64, and a bound of a float32 pass's error: the terms of a sum of k values are
    rounded at most k + 1 times, an error e of a source gives |w| e, and the sigmoid (slope 1/4, value
    below 1) adds a few roundings of its own."""
    out, err = [], []
    n_in, n_out = nets.n_in, nets.n_out
    eps = 2.0 ** -24
    for g in range(nets.P):
        N = n_in + n_out + int(nets.node_off[g + 1] - nets.node_off[g])
        _, s, d, w, _ = nets.genome(g)
        m = np.zeros((N, N))
        m[d, s] = w
        v, e = np.zeros((N, len(pat))), np.zeros((N, len(pat)))
        v[:n_in] = np.asarray(pat, np.float64).T
        k = np.count_nonzero(m, axis=1)[:, None] + 1
        for _ in range(steps):
            z, ez = m @ v, np.abs(m) @ e + eps * k * (np.abs(m) @ np.abs(v))
            v, e = v.copy(), e.copy()
            v[n_in:] = 1 / (1 + np.exp(-z[n_in:]))
            e[n_in:] = ez[n_in:] / 4 + 8 * eps
        out.append(v[n_in:n_in + n_out].T)
        err.append(e[n_in:n_in + n_out].T)
    return np.stack(out), np.stack(err)


@pytest.mark.gpu
@pytest.mark.parametrize("K,steps", [(1, 3), (2, 2), (3, 1), (4, 3), (5, 2), (8, 4), (12, 1), (27, 3), (4, 0)])
@pytest.mark.parametrize("density", [0.02, 0.5])
def test_forward_equals_float64(K, steps, density):
    # sizes around 2048 connections at density 0.5; 200 hidden nodes and more take a cluster there, none at 0.02
    sizes = [0, 1, 7, 58, 60, 61, 62, 63, 64, 66, 0, 200, 333, 2] + [3] * 40 + [400, 0]
    nets = _networks(sizes, density, 3, 2, seed=K + 10 * steps)
    pat = np.random.default_rng(K).normal(0, 1, (K, 3)).astype(np.float32)
    got = emr.ann_forward(nets, pat, steps).cpu().numpy()
    ref, err = _reference(nets, pat, steps)
    assert np.all(np.abs(got - ref) <= err + 1e-30)


@pytest.mark.gpu
def test_more_networks_than_resident_ctas():
    nets = _networks([5] * 1500 + [100] + [5] * 900, 0.5, 2, 1, seed=3, acyclic=True)
    pat = np.array([[0, 0], [0, 1], [1, 0], [1, 1]], np.float32)
    got = emr.ann_forward(nets, pat, 3).cpu().numpy()
    ref, err = _reference(nets, pat, 3)
    assert np.all(np.abs(got - ref) <= err + 1e-30)


@pytest.mark.gpu
def test_shared_memory_limit():
    """The largest value buffers the call accepts, and one node more refused."""
    limit = torch.cuda.get_device_properties(0).shared_memory_per_block_optin
    K = 4
    H = (limit - 4) // (8 * K + 4) - 3
    pat = np.ones((K, 2), np.float32)
    nets = _networks([H, 4], 0.002, 2, 1, seed=5)
    got = emr.ann_forward(nets, pat, 2).cpu().numpy()
    ref, err = _reference(nets, pat, 2)
    assert np.all(np.abs(got - ref) <= err + 1e-30)
    with pytest.raises(emr.EmrError):
        emr.ann_forward(_networks([H + 1], 0.002, 2, 1, seed=5), pat, 2)


@pytest.mark.gpu
@pytest.mark.parametrize("sizes,density", [
    ([120, 122, 124, 126, 128, 130, 132, 0, 300, 8, 9, 33], 0.5),   # the split of 8192 connections lies near 125 hidden nodes
    ([4, 5, 6, 27, 28, 29, 30, 116, 122, 0, 60], 0.9),              # at most 16384 connections by the nodes: no cluster launch
    ([123, 6, 0, 128], 0.97),                                       # the first past it
])
def test_lanes_and_clusters_at_their_lines(sizes, density):
    """Lane counts change at 8 and 32 computed nodes (n_out + hidden), clusters at 8192 connections."""
    for K in (1, 4, 8):
        nets = _networks(sizes, density, 3, 2, seed=K)
        pat = np.random.default_rng(K).normal(0, 1, (K, 3)).astype(np.float32)
        got = emr.ann_forward(nets, pat, 3).cpu().numpy()
        ref, err = _reference(nets, pat, 3)
        assert np.all(np.abs(got - ref) <= err + 1e-30)


def _one(nets, g):
    h, src, dst, w, t = nets.genome(g)
    return emr.Networks(nets.n_in, nets.n_out, np.array([0, len(h)], np.int64), h, np.array([0, len(w)], np.int64), src,
                        dst, w, t)


def _joined(a, b):
    cat = lambda f: np.concatenate([getattr(a, f), getattr(b, f)])
    off = lambda f: np.concatenate([getattr(a, f), getattr(a, f)[-1] + getattr(b, f)[1:]])
    return emr.Networks(a.n_in, a.n_out, off("node_off"), cat("hidden"), off("conn_off"), cat("src"), cat("dst"),
                        cat("w"), cat("type"))


@pytest.mark.gpu
@pytest.mark.parametrize("K", [1, 4, 6])
def test_a_network_gives_the_same_bits_in_any_batch(K):
    """Each network alone, beside its neighbours, and beside one that sizes the call's buffers far above it:
    connection counts on both sides of the one that takes a cluster, nodes on both sides of a lane count's."""
    sizes = [6, 30, 60, 88, 92, 96, 100, 104, 112, 120, 126, 140]
    nets = _networks(sizes, 0.95, 3, 2, seed=K)
    pat = np.random.default_rng(K).normal(0, 1, (K, 3)).astype(np.float32)
    every = emr.ann_forward(nets, pat, 3)
    large = emr.ann_forward(_joined(nets, _networks([700], 0.1, 3, 2, seed=7)), pat, 3)
    for g in range(len(sizes)):
        alone = emr.ann_forward(_one(nets, g), pat, 3)[0]
        assert torch.equal(alone, every[g]), sizes[g]
        assert torch.equal(alone, large[g]), sizes[g]
    for k in range(K):
        assert torch.equal(emr.ann_forward(nets, pat[k:k + 1], 3)[:, 0], every[:, k]), k
