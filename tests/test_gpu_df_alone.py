"""A double-float ray's result is a function of the ray alone: not of the rays beside it,
the launch's shape, the claim order, the handle (star, batch, captured graph) or the run
-- for rays guided along the null cone, too, however many there are.

The rays that start within 1e-3 rad of the cone are traced in FP64 (six lanes per ray),
the others in double-float; which of the two may depend on nothing but the start."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2309_08655_gb300 import inputs as I  # noqa: E402
from paper_2309_08655_gb300 import rt  # noqa: E402

from . import gpu_util as G  # noqa: E402

KW = dict(I.star_config0(), phase_mode=0, psi=0.0)
OPTS = dict(rtol=1e-8, precision=rt.PREC_DF, max_steps=400)


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2309_08655_gb300.build import build
    build()
    assert torch.cuda.is_available()


def _near(n, width):
    """Samples of the aligned star within ``width`` rad of its null cone."""
    u = I.sample_uniforms(9, n)
    u[0] = 0.5 * (1 - np.cos(np.arccos(1 / np.sqrt(3)) + width * (2 * u[0] - 1)))
    return G.gpu_sample(KW, u)


def _run(star, st0, s0, **opts):
    st, s = st0.clone(), s0.clone()
    rt.rt_trace_forward(star, st.shape[1], st, s, opts=rt.make_opts(**dict(OPTS, **opts)))
    assert not ((s == rt.RAY_READY) | (s >= rt.RAY_NSTATUS)).any()
    return st, s


def _same(a, b):
    return torch.equal(a[0].view(torch.int64), b[0].view(torch.int64)) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("n,width", [(1, 1e-4), (33, 9e-4), (700, 2e-2), (6000, 9e-4),
                                     (9000, 1.2e-3)])
def test_launch_shape_order_and_run_do_not_matter(n, width):
    star, st0, w, s0, _ = _near(n, width)
    ref = _run(star, st0, s0)
    for opts in (dict(), dict(block=32, blocks_per_sm=1), dict(block=256, blocks_per_sm=1),
                 dict(block=64, blocks_per_sm=2, claim_order=rt.CLAIM_COST, rays_per_claim=5)):
        assert _same(_run(star, st0, s0, **opts), ref), opts


@pytest.mark.parametrize("n", [40, 700])
def test_neighbours_do_not_matter(n):
    star, st0, w, s0, _ = _near(n, 1.2e-3)
    ref = _run(star, st0, s0)
    _, far, _, fs, _ = G.gpu_sample(KW, I.sample_uniforms(3, 500))
    _, more, _, ms, _ = _near(5000, 9e-4)
    for a, b in ((far, fs), (more, ms)):
        st, s = _run(star, torch.cat([a, st0], 1).contiguous(), torch.cat([b, s0]).contiguous())
        assert _same((st[:, -n:].contiguous(), s[-n:]), ref)
    for k in (0, n // 2, n - 1):         # alone
        one = _run(star, st0[:, k:k + 1].contiguous(), s0[k:k + 1].contiguous())
        assert _same(one, (ref[0][:, k:k + 1].contiguous(), ref[1][k:k + 1]))


def test_batch_and_captured_graph_agree_with_single_calls():
    n = 900
    u = I.sample_uniforms(9, n)
    u[0] = 0.5 * (1 - np.cos(np.arccos(1 / np.sqrt(3)) + 2e-3 * (2 * u[0] - 1)))
    stars = [rt.Star(rt.make_params(**KW)) for _ in range(2)]
    ud = torch.from_numpy(np.concatenate([u, u], 1)).to(G.dev())
    opts = rt.make_opts(**OPTS)

    def buffers():
        return (torch.empty((8, 2 * n), dtype=G.F64, device=G.dev()),
                torch.empty(2 * n, dtype=G.F64, device=G.dev()),
                torch.empty(2 * n, dtype=torch.uint8, device=G.dev()))
    # a graph of a batch that has traced nothing yet
    batch = rt.Batch(stars, [n, n])
    st, w, s = buffers()
    ctr = torch.zeros(8, dtype=torch.int64, device=G.dev())
    hist = torch.empty((2, 8, 4, 16), dtype=G.F64, device=G.dev())
    oor = torch.empty(2, dtype=G.F64, device=G.dev())
    g = rt.Graph(batch, ud, st, w, s, ctr, opts, 8, 4, 16, 0.0, 9.0, hist, oor)
    g.launch()
    torch.cuda.synchronize()
    # the direct calls on another fresh batch, and one star at a time
    direct = rt.Batch(stars, [n, n])
    st2, w2, s2 = buffers()
    rt.rt_sample_batch(direct, ud, st2, w2, s2)
    st0, s0 = st2[:, :n].clone(), s2[:n].clone()
    rt.rt_trace_batch(direct, st2, s2, opts=opts)
    assert _same((st, s), (st2, s2))
    one = _run(stars[0], st0, s0)
    assert _same((st2[:, :n].contiguous(), s2[:n]), one)
    assert _same((st2[:, n:].contiguous(), s2[n:]), one)
    g.close()


def test_guided_rays_agree_with_fp64(oracle):
    """End points of rays guided along the cone against the oracle, where the oracle's end
    point does not depend on rounding."""
    n = 600
    star, st0, w, s0, _ = _near(n, 9e-4)
    a, b = G.to_np(st0, s0)
    end, status, good, _ = G.well_conditioned(oracle, oracle.star_vector(**KW), a, b, 1e-10)
    good &= b == rt.RAY_READY
    st, s = _run(star, st0, s0, rtol=1e-10, max_steps=100000)
    st, s = G.to_np(st, s)
    assert good.sum() > 20
    assert np.array_equal(s[good], status[good])
    assert G.rel_state_diff(st[:, good], end[:, good]).max() < 1e-10
