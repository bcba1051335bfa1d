"""The gradient's replay starts where the forward trace starts, bit for bit, for the
samples next to the null cone, too (the sampling kernel iterates those to the last bit,
and rays guided along the cone carry a last-bit change of the start to other steps)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2309_08655_gb300 import build as B  # noqa: E402
from paper_2309_08655_gb300 import inputs as I  # noqa: E402
from paper_2309_08655_gb300 import rt  # noqa: E402

from . import gpu_util as G  # noqa: E402

# the replay's set-up of a ray, called for every sample
SRC = r"""
#include "rt_adjoint.cu"
namespace rtk {
namespace {
__global__ void starts(AdjParams P, double* y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < P.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    SampOut<Dual<NSAMP_TANGENTS>> so;
    Lane L;
    double w, cps, sps;
    const bool ok = begin_ray(P, i, so, w, L, cps, sps);
    for (int j = 0; j < 6; ++j) y[j * P.n + i] = ok ? L.y[j] : 0.0;
    y[6 * P.n + i] = ok ? w : 0.0;
  }
}
}  // namespace
}  // namespace rtk
extern "C" int run(const rt_star* star, long n, const double* u, const double* state,
                   const double* weight, unsigned char* status, double* y, double* F_ray,
                   double* G_ray, int* flags) {
  const rtk::StarDev h = rtk::star_host_desc(star);
  rtk::AdjParams P;
  typedef rtk::Dual<rtk::NSAMP_TANGENTS> D;
  auto& d = P.sc;
  d.rs = D(h.rs); d.cp = D(h.cp); d.sin_tm = D(h.sin_tm); d.cos_tm = D(h.cos_tm);
  d.B0_eV2 = D(h.B0_eV2); d.R_eV = D(h.R_eV); d.n_inf = D(h.n_inf); d.ma_eV = D(h.ma_eV);
  d.v0 = h.v0; d.psi_fixed = h.psi_fixed; d.plasma_a = h.plasma_a; d.g_eV = h.g_eV;
  d.w_unit = h.w_unit; d.rlc = h.rlc; d.per_cm3 = rtk::PER_CM3_EV3; d.disp = h.dispersion;
  d.plasma = h.plasma; d.fa_model = h.fa_model; d.phase_mode = h.phase_mode;
  d.weight_mode = h.weight_mode;
  P.R_km = h.R_km; P.ma_eV = h.ma_eV; P.rs_prop = h.rs_prop; P.cp = h.cp;
  P.plasma_a = h.plasma_a; P.cos_tm = h.cos_tm; P.sin_tm = h.sin_tm;
  P.dispersion = h.dispersion; P.plasma = h.plasma;
  P.rtol = P.atol = 1e-10;
  P.n = n; P.u = u; P.state = state; P.weight = weight; P.status = status;
  P.F_ray = F_ray; P.G_ray = G_ray; P.flags = flags;
  rtk::starts<<<64, 128>>>(P, y);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def starts(tmp_path_factory):
    B.build()
    assert torch.cuda.is_available()
    d = tmp_path_factory.mktemp("starts")
    src, so = os.path.join(d, "starts.cu"), os.path.join(d, "starts.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-I", B.INCLUDE, "-I", B.CSRC, "-I", B.BUILD, src, B.LIB,
                    "-o", so], check=True, capture_output=True)
    rt.lib()
    L = ctypes.CDLL(so)

    def call(star, u, st, w, s):
        n = u.shape[1]
        t = [torch.from_numpy(np.ascontiguousarray(u)).to(G.dev()), st, w, s.clone()]
        t += [torch.zeros((k, n), dtype=G.F64, device=G.dev()) for k in (7, 1, 6)]
        t += [torch.zeros(n, dtype=torch.int32, device=G.dev())]
        assert L.run(star.handle, ctypes.c_long(n), *(ctypes.c_void_p(x.data_ptr()) for x in t)) == 0
        return t[4]
    return call


@pytest.mark.parametrize("n,width,theta,phase,seed", [
    (1, 9e-3, 0.0, 0, 4), (3000, 9e-3, 0.0, 0, 5), (3000, 9e-3, 1e-3, 0, 6),
    (600, 9e-4, 0.0, 1, 7), (20000, None, 0.5, 1, 8)])
def test_replay_starts_at_the_samples(starts, n, width, theta, phase, seed):
    kw = dict(I.star_config0(), phase_mode=phase, psi=0.3, theta_m=theta)
    u = I.sample_uniforms(seed, n)
    if width:                            # the cone of the aligned star: cos^2 = 1/3
        u[0] = 0.5 * (1 - np.cos(np.arccos(1 / np.sqrt(3)) + width * (2 * u[0] - 1)))
    star, st, w, s, _ = G.gpu_sample(kw, u)
    ready = s == rt.RAY_READY
    assert ready.sum() > 0.5 * n
    y = starts(star, u, st, w, s)
    scale = torch.tensor([1.0 / kw["R_km"]] * 3 + [1.0 / kw["m_a_eV"]] * 3, dtype=G.F64,
                         device=G.dev())[:, None]
    assert torch.equal(y[:6, ready], (st[:6] * scale)[:, ready])
    assert torch.equal(y[6, ready], w[ready])
    assert not y[:, ~ready].any()


def test_no_guided_ray_is_left_out():
    """The replays of rays next to the cone against the forward run with one lane per ray:
    the same rays escape and none is left out."""
    n = 1500
    kw = dict(I.star_config0(), phase_mode=0, psi=0.0, theta_m=0.0)
    u = I.sample_uniforms(5, n)
    u[0] = 0.5 * (1 - np.cos(np.arccos(1 / np.sqrt(3)) + 9e-3 * (2 * u[0] - 1)))
    star, st, w, s, _ = G.gpu_sample(kw, u)
    nacc, nrej, ctr = G.gpu_trace(star, st, s, rtol=1e-6, tail=1)
    grad = torch.empty(6, dtype=G.F64, device=G.dev())
    F = torch.empty(1, dtype=G.F64, device=G.dev())
    s2 = torch.empty_like(s)
    c2 = torch.zeros(8, dtype=torch.int64, device=G.dev())
    rt.rt_flux_gradient(star, n, torch.from_numpy(u).to(G.dev()), nacc, 1.1, 4.0, grad, F, status=s2,
                        counters=c2, opts=rt.make_opts(rtol=1e-6))
    assert int(c2[4]) == 0
    assert torch.equal(s2, s)
    assert np.isfinite(grad.cpu().numpy()).all()
