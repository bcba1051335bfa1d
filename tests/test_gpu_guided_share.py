"""Guided rays in warps of their own: bitwise the results of the plain queue for the
mixed and rotating paths, whatever the launch -- few rays, every ray next to the null
cone, and more of them than the launch's warps take at once."""
import numpy as np
import pytest
import torch

from paper_2309_08655_gb300 import inputs as I
from paper_2309_08655_gb300 import rt
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _near(n, width):
    """Samples of the aligned star within ``width`` rad of its null cone."""
    u = I.sample_uniforms(9, n)
    u[0] = 0.5 * (1 - np.cos(np.arccos(1 / np.sqrt(3)) + width * (2 * u[0] - 1)))
    return G.gpu_sample(dict(I.star_config0(), phase_mode=0, psi=0.0), u)


@pytest.mark.parametrize("n,width", [(1, 1e-4), (40, 9e-4), (700, 2e-2), (6000, 9e-4)])
@pytest.mark.parametrize("block,bps", [(32, 1), (0, 0)])
def test_mixed_shares_are_the_plain_queue(n, width, block, bps):
    star, st0, _, s0, _ = _near(n, width)
    far = G.gpu_sample(dict(I.star_config0(), phase_mode=0, psi=0.0), I.sample_uniforms(3, 64))
    out = []
    for tail_rays in (0, 64):            # alone, and among rays that are not guided
        st = torch.cat([st0, far[1][:, :tail_rays]], 1).contiguous()
        s = torch.cat([s0, far[3][:tail_rays]]).contiguous()
        opts = rt.make_opts(rtol=1e-6, precision=rt.PREC_MIXED, tail=1, block=block,
                            blocks_per_sm=bps, max_steps=400)
        rt.rt_trace_forward(star, st.shape[1], st, s, opts=opts)
        assert not (s == 9).any() and not (s == 0).any()   # none left in a share or the queue
        out.append((st[:, :n].clone(), s[:n].clone()))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
