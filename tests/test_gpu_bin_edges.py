"""Rays on, next to and far from the bins' edges, and values FP32 cannot hold: every ray
in the bin that FP64 arithmetic chooses."""
import numpy as np
import pytest
import torch

from paper_2309_08655_gb300 import inputs as I
from paper_2309_08655_gb300 import rt
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def rays(n, nth, nph, nnu, nu_hi, v0, seed, scale_k, offset):
    """End points whose direction and frequency lie ``offset`` (relative) from an edge for
    a third of the rays each, at the poles for a few."""
    rng = np.random.default_rng(seed)
    th = np.arccos(rng.uniform(-1, 1, n))
    ph = rng.uniform(0, 2 * np.pi, n)
    y = rng.uniform(-0.05 * nu_hi, 1.05 * nu_hi, n)
    a, b, c = np.arange(n) % 3 == 0, np.arange(n) % 3 == 1, np.arange(n) % 3 == 2
    sgn = rng.choice([-1.0, 1.0], n)
    th[a] = np.clip(np.round(th[a] / (np.pi / nth)) * (np.pi / nth) + sgn[a] * offset, 0, np.pi)
    ph[b] = np.round(ph[b] / (2 * np.pi / nph)) * (2 * np.pi / nph) + sgn[b] * offset
    y[c] = np.round(y[c] / (nu_hi / nnu)) * (nu_hi / nnu) * (1 + sgn[c] * offset)
    poles = np.array([0.0, np.pi, 1e-9, 1e-4, np.pi - 1e-9, np.pi - 1e-4])[:n]
    th[:poles.size], ph[:poles.size] = poles, 1.0
    d = np.array([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)])
    x = rng.standard_normal((3, n))
    st = np.zeros((8, n))
    st[:3] = 1e4 * x / np.linalg.norm(x, axis=0)
    st[3:6] = d * scale_k * 10.0 ** rng.uniform(-1, 1, n)
    st[6] = y * 0.5 * v0 * v0
    w = np.exp(rng.normal(0, 3, n))
    w[7:8] = 0.0
    s = rng.choice([0, 1, 1, 1, 2, 3], n).astype(np.uint8)
    return st, w, s


@pytest.mark.parametrize("n,nth,nph,nnu", [(1, 1, 1, 1), (4097, 64, 32, 128), (20000, 7, 5, 1),
                                           (5000, 180, 360, 3), (3000, 1, 1, 2000)])
@pytest.mark.parametrize("scale_k,offset", [(1e-9, 0.0), (1e-9, 1e-15), (1e3, 1e-9),
                                            (1e-60, 3e-7), (1e-9, 1e-5), (1e45, 1e-4)])
def test_bins_are_those_of_fp64(oracle, n, nth, nph, nnu, scale_k, offset):
    kw = dict(I.star_config0(), M_sun=0.0)      # direction = that of k, no rounding of its own
    v0 = 200.0 / 299792.458
    st, w, s = rays(n, nth, nph, nnu, 9.0, v0, n + nnu, scale_k, offset)
    star = rt.Star(rt.make_params(**kw))
    t = [torch.from_numpy(v).to(G.dev()) for v in (st, w, s)]
    h, sky, spec, oor = G.gpu_bin(star, *t, nth=nth, nph=nph, nnu=nnu)
    h_o, oor_o = oracle.bin_rays(oracle.star_vector(**kw), st, w, s, nth, nph, nnu, 0.0, 9.0)
    # weights are exact multiples of the fixed point's unit to 2^-60 of the total; a ray on
    # an edge to rounding may fall either side in the oracle, whose functions are the host's
    tol = 1e-12 * max(w.sum(), 1e-300)
    if offset > 1e-12:
        assert np.abs(h - h_o).max() <= tol and abs(oor - oor_o) <= tol
    assert abs(h.sum() + oor - h_o.sum() - oor_o) <= tol
    assert np.abs(sky - h.sum(2)).max() <= tol and np.abs(spec - h.sum((0, 1))).max() <= tol
    # the sharded entry points add the same integers, marginals included
    acc = torch.zeros(rt.bin_acc_entries(nth, nph, nnu), dtype=torch.int64, device=G.dev())
    rt.rt_bin_part_max(n, t[1], t[2], nth, nph, nnu, acc)
    rt.rt_bin_part_accumulate(star, n, n, *t, nth, nph, nnu, 0.0, 9.0, acc)
    nh = nth * nph * nnu
    cube = acc[2:2 + nh].reshape(nth * nph, nnu)
    assert torch.equal(acc[2 + nh:2 + nh + nth * nph], cube.sum(1))
    assert torch.equal(acc[2 + nh + nth * nph:], cube.sum(0))
    out = [torch.empty(k, dtype=G.F64, device=G.dev()) for k in (nh, nth * nph, nnu, 1)]
    rt.rt_bin_part_finalize(nth, nph, nnu, n, acc, *out)
    assert np.array_equal(out[0].cpu().numpy(), h.reshape(-1))
    assert np.array_equal(out[1].cpu().numpy(), sky.reshape(-1))
    assert np.array_equal(out[2].cpu().numpy(), spec) and float(out[3][0]) == oor
