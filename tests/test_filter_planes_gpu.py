"""emr_variance_filter writes every word of its three planes, and every variance, over whatever the caller's
buffers held: split words of depth D are 0, and no stale bit or value stays."""
import numpy as np
import pytest
import torch

from paper_2608_27612_gb300 import emr
from parity_util import unpack_planes


def _filter(g, out, halo, n, mode, fill, var_offset=0):
    planes = [torch.full((n, g.n_words), fill, dtype=torch.int32, device="cuda") for _ in range(3)]
    mask, split, band = planes
    var = torch.full((var_offset + n * g.n_total,), float("nan"), device="cuda")[var_offset:]
    emr.variance_filter(out, halo, g, n, 1, 0.3, 0.5, 0.0, mode, mask, split, band, var)
    return planes, var.view(n, g.n_total)


def _inputs(D, n):
    gen = torch.Generator().manual_seed(D)
    g = emr.grid_build(D)
    scale = torch.rand(n, 1, generator=gen)  # some pairs split everywhere, some nowhere
    return g, torch.randn(n, g.n_total, generator=gen) * scale, torch.randn(n, g.n_halo, generator=gen) * scale


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [emr.EMR_EAGER, emr.EMR_GATED])
@pytest.mark.parametrize("D", [0, 1, 2, 3, 4, 5, 7])
def test_every_word_is_written(D, mode):
    n = 9
    g, out, halo = _inputs(D, n)
    dev = out.cuda(), halo.cuda()
    clean, var = _filter(g, *dev, n, mode, 0)
    dirty, var2 = _filter(g, *dev, n, mode, -1)
    for name, a, b in zip(("mask", "split", "band_bits"), clean, dirty):
        assert torch.equal(a, b), name
    assert torch.equal(var, var2)  # (NaN where not written)
    lo = g.level_off[D]
    assert not dirty[1][:, g.word_off[D]:].any() and not var[:, lo:].any()
    # against float64: a variance of values up to m is a sum of at most six squares up to 4 m^2, each rounded
    # twice, and eight additions
    v = np.zeros((n, g.n_total))
    v[:, :lo] = out.double().numpy()[:, 4:].reshape(n, lo, 4).var(axis=2)
    tol = 16 * 2.0 ** -24 * 4 * float(out.abs().max()) ** 2
    assert np.abs(var.cpu().numpy() - v).max() <= tol
    bits = unpack_planes(dirty[1].cpu().numpy(), g)
    clear = np.abs(v - 0.3) > tol
    assert np.array_equal(bits[clear], (v > 0.3)[clear])


@pytest.mark.gpu
@pytest.mark.parametrize("D", [0, 4, 5, 6])
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_variances_at_any_float(D, offset):
    """var_dbg may be a view that begins at any float of a larger buffer."""
    n = 3
    g, out, halo = _inputs(D, n)
    dev = out.cuda(), halo.cuda()
    _, want = _filter(g, *dev, n, emr.EMR_EAGER, 0)
    _, got = _filter(g, *dev, n, emr.EMR_EAGER, 0, offset)
    assert got.data_ptr() % 16 == 4 * offset
    assert torch.equal(got, want)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["x", "y", "diagonal"])
def test_variance_of_two_values_is_rounded_once(kind):
    """Cells whose children hold two values, two of each: V = (a - b)^2 / 4 from the fp32 difference, the square
    rounded once and scaled by a power of two, at every depth."""
    D, n = 6, 5
    g = emr.grid_build(D)
    gen = torch.Generator().manual_seed(3)
    ab = torch.randn(n, g.n_total // 4, 2, generator=gen)
    out = ab[..., {"x": [0, 1, 0, 1], "y": [0, 0, 1, 1], "diagonal": [0, 1, 1, 0]}[kind]].reshape(n, g.n_total)
    _, var = _filter(g, out.cuda(), torch.zeros(n, g.n_halo, device="cuda"), n, emr.EMR_EAGER, 0)
    t = ab[..., 0] - ab[..., 1]
    lo = g.level_off[D]
    assert torch.equal(var.cpu()[:, :lo], (0.25 * (t * t))[:, 1:])
