"""Guided rays in warps of their own: bitwise the results of the plain queue for the
rotating magnetosphere, whatever the launch -- few rays, every ray next to the null
cone, more of them than the launch's warps take at once; and in double-float, where
FP64 groups take them, every ray ends once."""
import numpy as np
import pytest
import torch

from paper_2309_08655_gb300 import inputs as I
from paper_2309_08655_gb300 import rt
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _near(n, width, rotation):
    """Samples of the aligned star within ``width`` rad of its null cone, and others."""
    kw = dict(I.star_config0(), phase_mode=0, psi=0.0, rotation=rotation)
    u = I.sample_uniforms(9, n)
    u[0] = 0.5 * (1 - np.cos(np.arccos(1 / np.sqrt(3)) + width * (2 * u[0] - 1)))
    return G.gpu_sample(kw, u), G.gpu_sample(kw, I.sample_uniforms(3, 64))


@pytest.mark.parametrize("n,width", [(1, 1e-4), (40, 9e-4), (700, 2e-2), (6000, 9e-4)])
@pytest.mark.parametrize("block,bps", [(32, 1), (0, 0)])
@pytest.mark.parametrize("precision", [rt.PREC_FP64, rt.PREC_DF])
def test_shares(n, width, block, bps, precision):
    rotation = int(precision == rt.PREC_FP64)
    near, far = _near(n, width, rotation)
    out = []
    for others in (0, 64):               # alone, and among rays that are not guided
        st = torch.cat([near[1], far[1][:, :others]], 1).contiguous()
        s = torch.cat([near[3], far[3][:others]]).contiguous()
        opts = rt.make_opts(rtol=1e-6, precision=precision, block=block, blocks_per_sm=bps,
                            max_steps=300)
        rt.rt_trace_forward(near[0], st.shape[1], st, s, opts=opts)
        # none left in a share (the internal status 9) or in the queue
        assert not (s == 9).any() and not (s == rt.RAY_READY).any()
        out.append((st[:, :n].clone(), s[:n].clone()))
    if rotation:
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
