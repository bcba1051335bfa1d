"""Tail mode empties the queue: every ray of a launch is traced once, whatever the
grid, the claim size and the number of rays.

A warp that parks its rays for the six-lane groups must know that the queue is empty,
not only that some of its lanes take no rays (short launches use part of each warp),
and the rest of a parked lane's chunk of claimed entries still has to be traced."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2309_08655_gb300 import inputs as I  # noqa: E402
from paper_2309_08655_gb300 import rt  # noqa: E402

from . import gpu_util as G  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2309_08655_gb300.build import build
    build()
    assert torch.cuda.is_available()


SHAPES = [(0, 0), (32, 1), (32, 3), (64, 1), (96, 1), (128, 2)]


@pytest.mark.parametrize("n", [1, 37, 3000, 9001, 30000])
@pytest.mark.parametrize("precision", [rt.PREC_FP64, rt.PREC_MIXED])
def test_every_ray_is_traced_once(n, precision):
    kw = dict(I.stars_config1()[0], m_a_eV=1e-5)
    star, st0, w, s0, _ = G.gpu_sample(kw, I.sample_uniforms(31, n))
    ready = int((s0 == rt.RAY_READY).sum())
    assert ready > 0.5 * n
    for block, bps in SHAPES:
        for claim in (1, 3, 64):
            for order in (rt.CLAIM_INDEX, rt.CLAIM_COST):
                st, s = st0.clone(), s0.clone()
                nacc, nrej, ctr = G.gpu_trace(star, st, s, rtol=1e-6, max_steps=120, block=block,
                                              blocks_per_sm=bps, rays_per_claim=claim,
                                              claim_order=order, precision=precision)
                left = int(((s == rt.RAY_READY) | (s >= rt.RAY_NSTATUS)).sum())
                assert left == 0, (block, bps, claim, order, left)
                c = ctr.cpu().numpy()
                assert c[2] == ready, (block, bps, claim, order, c)
                assert c[0] == int(nacc.sum()) and c[1] == int(nrej.sum())


def test_every_ray_of_a_batch_is_traced_once():
    kws = [I.stars_config1()[j] for j in (0, 2, 5)]
    stars = [rt.Star(rt.make_params(**k)) for k in kws]
    batch = rt.Batch(stars, [2500, 0, 1501])
    N = batch.N
    u = torch.from_numpy(I.sample_uniforms(5, N)).to(G.dev())
    st = torch.empty((8, N), dtype=G.F64, device=G.dev())
    w = torch.empty(N, dtype=G.F64, device=G.dev())
    s = torch.empty(N, dtype=torch.uint8, device=G.dev())
    for block, bps in SHAPES:
        for claim in (1, 4):
            rt.rt_sample_batch(batch, u, st, w, s)
            ready = int((s == rt.RAY_READY).sum())
            ctr = torch.zeros(8, dtype=torch.int64, device=G.dev())
            rt.rt_trace_batch(batch, st, s, counters=ctr, opts=rt.make_opts(
                rtol=1e-6, max_steps=120, block=block, blocks_per_sm=bps, rays_per_claim=claim))
            assert not ((s == rt.RAY_READY) | (s >= rt.RAY_NSTATUS)).any(), (block, bps, claim)
            assert int(ctr[2]) == ready
