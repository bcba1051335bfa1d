"""The six-lane groups of the FP64 tail mode against one lane per ray and against
the oracle, over the media and dispersions: the pass table of the Goldreich-Julian
anisotropic medium, the whole right-hand side on every lane for the others.

Both integrate the same equations with sums in another order, so on the rays whose
end point is insensitive to rounding (spread between the oracle's strict and
contracted builds at most 1e-12) they agree as the lane-per-ray path does with the
oracle: 1e-10."""
import numpy as np
import pytest
import torch

from paper_2309_08655_gb300 import inputs as I
from paper_2309_08655_gb300 import rt
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 300])
@pytest.mark.parametrize("plasma,dispersion,m_a", [
    (rt.PLASMA_GJ, 0, 1e-5), (rt.PLASMA_GJ, 1, 1e-5), (rt.PLASMA_TWISTED, 0, 1e-4),
    (rt.PLASMA_TWISTED, 1, 1e-4)])
def test_groups_against_lanes(oracle, n, plasma, dispersion, m_a):
    kw = dict(I.stars_config1()[0], m_a_eV=m_a, plasma=plasma, plasma_a=4.0,
              dispersion=dispersion)
    star, st0, w, s0, _ = G.gpu_sample(kw, I.sample_uniforms(21, n))
    a, b = G.to_np(st0, s0)
    end, status, good, _ = G.well_conditioned(oracle, oracle.star_vector(**kw), a, b, 1e-10)
    good &= b == rt.RAY_READY
    for tail in (1, 31, 0):              # lanes; parked at once; parked at five
        st, s = st0.clone(), s0.clone()
        na = torch.zeros(n, dtype=torch.int32, device=G.dev())
        nr = torch.zeros_like(na)
        rt.rt_trace_forward(star, n, st, s, na, nr, opts=rt.make_opts(tail=tail))
        st, s = G.to_np(st, s)
        assert np.array_equal(s[good], status[good])
        if good.any():
            assert G.rel_state_diff(st[:, good], end[:, good]).max() < 1e-10
