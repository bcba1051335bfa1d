"""Histograms of few sky cells and many frequencies: rows in segments, over the sizes
where a row is cut (below, at and above 256 bins, the last segment short), with and
without the marginals, from one call and from the sharded entry points."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2309_08655_gb300 import inputs as I  # noqa: E402
from paper_2309_08655_gb300 import rt  # noqa: E402

from . import gpu_util as G  # noqa: E402


@pytest.mark.parametrize("nth,nph,nnu", [(1, 1, 255), (1, 1, 256), (1, 1, 257), (1, 1, 70001),
                                         (3, 5, 4097), (100, 90, 513), (110, 100, 300),
                                         (1, 1, 3000017)])
def test_rows_in_segments(nth, nph, nnu):
    n = 4000
    dev = G.dev()
    rng = np.random.default_rng(nnu)
    v0 = 200.0 / 299792.458
    st = np.zeros((8, n))
    x = rng.standard_normal((3, n))
    st[:3] = 1e4 * x / np.linalg.norm(x, axis=0)
    st[3:6] = 1e-9 * rng.standard_normal((3, n))
    st[6] = rng.uniform(0.0, 9.2, n) * 0.5 * v0 * v0
    w = np.exp(rng.normal(0, 3, n))
    s = np.full(n, rt.RAY_ESCAPED, dtype=np.uint8)
    star = rt.Star(rt.make_params(**I.star_config0()))
    t = [torch.from_numpy(v).to(dev) for v in (st, w, s)]
    bins = (nth, nph, nnu, 0.0, 9.0)
    nh = nth * nph * nnu
    # the integer sums, marginals included
    acc = torch.zeros(rt.bin_acc_entries(nth, nph, nnu), dtype=torch.int64, device=dev)
    rt.rt_bin_part_max(n, t[1], t[2], nth, nph, nnu, acc)
    rt.rt_bin_part_accumulate(star, n, n, *t, *bins, acc)
    keep = acc.clone()
    out = [torch.full((k,), -1.0, dtype=G.F64, device=dev) for k in (nh, nth * nph, nnu, 1)]
    rt.rt_bin_part_finalize(nth, nph, nnu, n, acc, *out)
    assert torch.equal(acc, keep)        # read only
    unit = out[0].sum() / acc[2:2 + nh].sum()      # a power of two, to rounding
    unit = 2.0 ** torch.round(torch.log2(unit))
    assert torch.equal(out[0], acc[2:2 + nh] * unit)
    assert torch.equal(out[1], acc[2 + nh:2 + nh + nth * nph] * unit)
    assert torch.equal(out[2], acc[2 + nh + nth * nph:] * unit)
    # one call, with and without the marginals, twice (the sums start at zero each time)
    for _ in range(2):
        h, sky, spec, oor = G.gpu_bin(star, *t, nth=nth, nph=nph, nnu=nnu)
        assert np.array_equal(h.reshape(-1), out[0].cpu().numpy())
        assert np.array_equal(sky.reshape(-1), out[1].cpu().numpy())
        assert np.array_equal(spec, out[2].cpu().numpy()) and oor == float(out[3][0])
    hist = torch.full((nh,), -1.0, dtype=G.F64, device=dev)
    o = torch.empty(1, dtype=G.F64, device=dev)
    rt.rt_bin_spectrum(star, n, *t, *bins, hist, None, None, o)
    assert torch.equal(hist, out[0])
