"""emr_eval_filter_tiles + emr_select (combine, compaction and kept weights over
the tiles whose flag shows band bits) give exactly the lists of emr_eval_filter +
emr_mask_combine(_types) + emr_compact_records, and the flags are exactly the
tiles holding band bits."""
import numpy as np
import pytest
import torch

from paper_2608_27612_gb300 import emr
from paper_2608_27612_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def tile_word_ranges(g):
    D = g.D
    wo = list(g.word_off)
    ranges = [(0, wo[min(D, 4) + 1])]
    for k in range(emr.dense_tiles(D) - 1):
        b = wo[5] + 128 * k
        ranges.append((b, b + 128))
    return ranges


def compare(w, mode=emr.EMR_EAGER, types=emr.CONN_ALL):
    dsc = emr.Discovery(w.pop, w.sources, w.D, w.theta, w.band, w.w_min, mode, types=types)
    dsc.run_fused()
    torch.cuda.synchronize()
    ref = dsc.lists()
    ref_counts = dsc.counts.cpu().numpy().copy()
    band_ref = dsc.band_bits.cpu().numpy().copy()
    dsc.idx.zero_(); dsc.w.zero_(); dsc.counts.zero_(); dsc.offsets.zero_()
    dsc.run_select()
    torch.cuda.synchronize()
    got = dsc.lists()
    assert np.array_equal(dsc.counts.cpu().numpy(), ref_counts)
    for (ri, rw), (gi, gw) in zip(ref, got):
        assert np.array_equal(ri, gi) and np.array_equal(rw.view(np.uint32), gw.view(np.uint32))
    band = dsc.band_bits.cpu().numpy()
    assert np.array_equal(band, band_ref)  # same fused evaluation
    # the one-call path gives the same lists
    dsc.idx.zero_(); dsc.w.zero_(); dsc.counts.zero_(); dsc.offsets.zero_()
    dsc.run_discover()
    torch.cuda.synchronize()
    one = dsc.lists()
    for (ri, rw), (gi, gw) in zip(ref, one):
        assert np.array_equal(ri, gi) and np.array_equal(rw.view(np.uint32), gw.view(np.uint32))
    flags = dsc.tile_flags.cpu().numpy()
    want = np.stack([band[:, b:e].any(axis=1) for b, e in tile_word_ranges(dsc.grid)], axis=1)
    assert np.array_equal(flags.astype(bool), want)
    return sum(len(i) for i, _ in ref), flags.mean()


@pytest.mark.parametrize("D", [0, 1, 2, 3, 4, 5, 6])
def test_select_small_depths(D):
    w = W.c2(D=D, P=60)
    compare(w)


def test_select_c2_depth7_modes_and_types():
    w = W.c2(D=7, P=80)
    kept, frac = compare(w)
    assert kept > 0 and frac < 0.5
    compare(w, emr.EMR_GATED)
    compare(w, emr.EMR_EAGER, emr.CONN_F | emr.CONN_L)


def test_select_interpreter_class_and_sharp_genomes():
    big = W.random_population(6, seed=31, h_lo=14, h_hi=30, e_max=120)
    rest = W.c5(D=7).pop
    pop = W.population_from_lists([big.genome(k) for k in range(6)] + [rest.genome(k) for k in range(10)])
    w = W.Workload("mixed_d7", pop, W.c5().sources, 7, 0.03, 0.3)
    compare(w)
    compare(w, emr.EMR_GATED)


def test_select_weight_filter_and_c1():
    w = W.c2(D=6, P=50)
    compare(W.Workload("c2_wmin", w.pop, w.sources, 6, w.theta, w.band, 0.1))
    compare(W.c1())


def test_select_per_genome_slots():
    w = W.c4_round2_random(D=6, P=20, S=32)
    compare(w)
    compare(w, emr.EMR_EAGER, emr.CONN_F | emr.CONN_B)


def test_copy_async_round_trip():
    """emr_copy_async moves bytes host -> device -> host (pinned buffers) on a stream."""
    src = torch.arange(1 << 16, dtype=torch.int32).pin_memory()
    dev = torch.empty_like(src, device="cuda")
    back = torch.zeros_like(src).pin_memory()
    stream = torch.cuda.Stream()
    emr.copy_async(dev, src, src.numel() * 4, stream)
    emr.copy_async(back, dev, src.numel() * 4, stream)
    stream.synchronize()
    assert torch.equal(back, src)
    emr.copy_async(back, dev, 0, stream)  # nothing to copy


def test_select_several_segments_per_pair():
    """Depth 8: 86 tiles, two whole segments of 32 and a part; steep genomes flag many tiles of each."""
    rest = W.c5(D=8).pop
    pop = W.population_from_lists([rest.genome(k) for k in range(10)])
    w = W.Workload("segments_d8", pop, W.c5().sources, 8, 0.02, 0.1)
    kept, frac = compare(w)
    assert kept > 0 and frac > 0
    compare(w, emr.EMR_GATED, emr.CONN_F | emr.CONN_S)


@pytest.mark.parametrize("P", [1, 255, 257, 2047, 2049, 5000])
def test_offsets_are_the_scanned_counts(P):
    """4 pairs up to 20000 (four slots a genome): one CTA of the scan (4096 counts) and several."""
    w = W.c2(D=2, P=P)
    dsc = emr.Discovery(w.pop, w.sources, w.D, w.theta, 0.1)
    dsc.run_discover()
    c, o = dsc.counts.cpu().numpy(), dsc.offsets.cpu().numpy()
    assert c.sum() > 0 or P == 1
    assert np.array_equal(o, np.concatenate([[0], np.cumsum(c)]))


@pytest.mark.parametrize("D", [0, 1, 3, 4])
def test_select_of_a_few_pairs(D):
    """Up to four pairs on a grid of one tile: the one-CTA selection, its lists cut at the capacity."""
    rest = W.c5(D=D).pop
    kept = 0
    for k in range(8):
        pop = W.population_from_lists([rest.genome(k)])
        for src in (W.c5().sources, W.shared_sources([(0.1, -1.0, W.SIDE_OUT)])):
            w = W.Workload("few_d%d" % D, pop, src, D, 0.02, 0.05)
            n, _ = compare(w)
            compare(w, emr.EMR_GATED, emr.CONN_F | emr.CONN_L)
            kept += n
            if n > 1:  # a list that does not fit: the first cap entries, the true counts
                d = emr.Discovery(w.pop, w.sources, D, w.theta, w.band)
                d.run_discover()
                c = emr.Discovery(w.pop, w.sources, D, w.theta, w.band, cap=n - 1)
                c.run_discover()
                assert torch.equal(c.offsets, d.offsets) and torch.equal(c.counts, d.counts)
                assert torch.equal(c.idx, d.idx[:n - 1]) and torch.equal(c.w, d.w[:n - 1])
    assert kept > 0


@pytest.mark.parametrize("P", [32, 33, 1024, 1025, 1030])
def test_every_pair_is_scheduled_once(P):
    """Four slots a genome: around a pair a thread (128) and the line from which bins are counted by the pairs'
    warps (4096). A pair left out or taken twice would leave its list empty or another's."""
    w = W.c2(D=4, P=P)
    d = emr.Discovery(w.pop, w.sources, w.D, w.theta, w.band)
    d.run_discover()
    lists = d.lists()
    for g0 in range(0, P, 30):  # the same genomes in populations of at most 30
        part = emr.Discovery(W.population_from_lists([w.pop.genome(g) for g in range(g0, min(P, g0 + 30))]), w.sources,
                             w.D, w.theta, w.band)
        part.run_discover()
        for (i, v), (j, u) in zip(part.lists(), lists[4 * g0:]):
            assert np.array_equal(i, j) and np.array_equal(v.view(np.uint32), u.view(np.uint32))


@pytest.mark.parametrize("n", [4095, 4096, 4097, 3 * 4096 + 5, 524288, 524289, 1 << 20, 1300001])
def test_compaction_of_many_pairs(n):
    """Pairs on both sides of one CTA of the offsets' scan (4096 counts) and of 128 CTAs, from where each scans
    several times 4096: four positions a pair, kept at random."""
    g = emr.grid_build(0)
    gen = torch.Generator().manual_seed(n)
    mask = torch.randint(0, 16, (n, 1), generator=gen, dtype=torch.int32) * (torch.rand(n, 1, generator=gen) < 0.3)
    out = torch.arange(4 * n, dtype=torch.float32).view(n, 4)
    kept = ((mask >> torch.arange(4)) & 1).bool()  # [n, 4]
    total = int(kept.sum())
    i64 = lambda k: torch.full((k,), -1, dtype=torch.int64, device="cuda")
    counts, offsets = i64(n), i64(n + 1)
    idx = torch.full((total,), -1, dtype=torch.int32, device="cuda")
    w = torch.full((total,), -1.0, device="cuda")
    ws = torch.empty(emr.compact_workspace_size(g, n), dtype=torch.uint8, device="cuda")
    emr.compact(mask.cuda(), out.cuda(), g, n, idx, w, total, counts, offsets, ws)
    c = kept.sum(1)
    assert torch.equal(counts.cpu(), c)
    assert torch.equal(offsets.cpu(), torch.cat([torch.zeros(1, dtype=torch.int64), c.cumsum(0)]))
    pair, pos = kept.nonzero(as_tuple=True)
    assert torch.equal(idx.cpu(), pos.int()) and torch.equal(w.cpu(), out[pair, pos])


def test_segments_over_several_scan_ctas():
    """1400 pairs of three segments: more segment counts than one CTA of the scan takes."""
    kept, _ = compare(W.c2(D=8, P=350))
    assert kept > 0
