"""The sampling kernel where its paths meet: the cells and ends of the speed table,
conversion next to the surface, and batches of more stars than one launch takes."""
import numpy as np
import pytest
import torch

from paper_2309_08655_gb300 import inputs as I
from paper_2309_08655_gb300 import maxwell, rt
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def edge_uniforms():
    """u at, just below and just above every 31st cell border, the ends of the table and
    the median, and far into both tails."""
    special = pytest.importorskip("scipy.special")
    x = [maxwell.centre(c) for c in range(0, maxwell.CELLS, 31)]
    lo = [2.0 ** (np.floor(np.log2(v)) - 8) for v in x]          # half a cell below
    edges = np.array([v - h for v, h in zip(x, lo)] + [maxwell.X_LO, maxwell.X_MID, 3.9999, 4.0,
                                                       maxwell.MEDIAN])
    u = special.gammainc(1.5, edges * edges)
    u = np.concatenate([u, u * (1 - 1e-7), u * (1 + 1e-7),
                        [2.0 ** -54, 1e-12, 1e-6, 0.5, 1 - 1e-9, 1 - 2.0 ** -52]])
    return np.clip(u, 2.0 ** -54, 1 - 2.0 ** -53)


@pytest.mark.parametrize("plasma,m_a", [(0, 1.094e-6), (5, 4e-5)])
def test_speed_table_edges(oracle, plasma, m_a):
    kw = dict(I.star_config0(), plasma=plasma, plasma_a=4.0, m_a_eV=m_a)
    ue = edge_uniforms()
    u = I.sample_uniforms(11, ue.size)
    u[4] = ue
    _, st, w, s, _ = G.gpu_sample(kw, u)
    st_o, w_o, s_o = oracle.sample(oracle.star_vector(**kw), u)
    st, w, s = G.to_np(st, w, s)
    assert np.array_equal(s, s_o)
    # the energy's relative error is twice the speed's; below the median the oracle's
    # distribution cancels to eps erf(x) / (x^3), at most 1e-13 in the table's range
    tab = (ue > 3e-5) & (ue < 1 - 1e-6)
    assert np.abs(st[6, tab] / st_o[6, tab] - 1).max() < 1e-12
    ok = (s_o == oracle.RAY_READY) & tab
    assert ok.sum() > 20
    assert G.rel_state_diff(st[:, ok], st_o[:, ok]).max() < 1e-12
    assert np.abs(w[ok] / w_o[ok] - 1).max() < 1e-11


@pytest.mark.parametrize("nstars", [1, 32, 33, 70])
def test_batch_sampling_is_that_of_single_calls(nstars):
    """Ragged counts (some empty), a star without a surface: bitwise the single calls."""
    rng = np.random.default_rng(nstars)
    counts = [int(c) for c in rng.integers(0, 200, nstars)]
    counts[-1] = 129
    kws = [dict(I.stars_config1()[0], m_a_eV=float(m), phase_mode=i % 2)
           for i, m in enumerate(np.geomspace(1e-6, 2e-4, nstars))]
    stars = [rt.Star(rt.make_params(**k)) for k in kws]
    batch = rt.Batch(stars, counts)
    N = batch.N
    u = torch.from_numpy(I.sample_uniforms(7, N)).to(G.dev())
    st = torch.empty((8, N), dtype=G.F64, device=G.dev())
    w = torch.empty(N, dtype=G.F64, device=G.dev())
    s = torch.empty(N, dtype=torch.uint8, device=G.dev())
    norm = [max(c, 1) + 5 for c in counts]
    rt.rt_batch_set_norm(batch, norm)
    rt.rt_sample_batch(batch, u, st, w, s)
    off = 0
    for star, c, nn in zip(stars, counts, norm):
        if c:
            uc = u[:, off:off + c].contiguous()
            a = torch.empty((8, c), dtype=G.F64, device=G.dev())
            b = torch.empty(c, dtype=G.F64, device=G.dev())
            d = torch.empty(c, dtype=torch.uint8, device=G.dev())
            rt.rt_sample_conversion_surface_part(star, c, nn, uc, a, b, d)
            assert torch.equal(a, st[:, off:off + c])
            assert torch.equal(b, w[off:off + c]) and torch.equal(d, s[off:off + c])
        off += c


@pytest.mark.parametrize("scale", [1 + 1e-12, 1 + 1e-7, 1.001])
def test_conversion_next_to_the_surface(oracle, scale):
    """A spherical profile whose resonance lies at or just above r = R."""
    kw = dict(I.star_config0(), plasma=4, plasma_a=scale, dispersion=1)
    u = I.sample_uniforms(3, 257)
    _, st, w, s, _ = G.gpu_sample(kw, u)
    st_o, w_o, s_o = oracle.sample(oracle.star_vector(**kw), u)
    st, w, s = G.to_np(st, w, s)
    assert np.array_equal(s, s_o) and (s == oracle.RAY_READY).all()
    assert G.rel_state_diff(st, st_o).max() < 1e-12
    assert np.abs(w / w_o - 1).max() < 1e-11


@pytest.mark.parametrize("n,theta", [(1, 0.0), (130, 0.0), (1000, 0.0), (70001, 0.5)])
def test_samples_next_to_the_null_cone(oracle, n, theta):
    """Every sample within 1e-2 rad of the cone: the blocks' lists fill and flush, the
    last one partly filled; and an inclined star, whose lists gather a few of many."""
    kw = dict(I.star_config0(), theta_m=theta, psi=0.0, phase_mode=0)
    u = I.sample_uniforms(5, n)
    if theta == 0.0:                     # the cone of the aligned star: cos^2 = 1/3
        u[0] = 0.5 * (1 - np.cos(np.arccos(1 / np.sqrt(3)) + 5e-3 * (2 * u[0] - 1)))
    _, st, w, s, _ = G.gpu_sample(kw, u)
    st_o, w_o, s_o = oracle.sample(oracle.star_vector(**kw), u)
    st, w, s = G.to_np(st, w, s)
    assert np.array_equal(s, s_o)
    ok = s_o == oracle.RAY_READY
    assert G.rel_state_diff(st[:, ok], st_o[:, ok]).max(initial=0.0) < 1e-12
    assert np.abs(w[ok] / w_o[ok] - 1).max(initial=0.0) < 1e-11
