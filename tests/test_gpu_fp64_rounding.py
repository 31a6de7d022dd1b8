"""Rounding of the FP64 temperature update T' = (T + dt (g T_gamma + hh)) / (1 + dt (2 H + g)) against
extended precision, with the library's own substep coefficients (a host program over csrc/rec_cosmo.cu
prints them).  Cold, weakly ionised gas at low redshift, where T' stays of the order of T and no operand
hides the others: evaluated as it is defined the rms error is 0.83 units of 2^-53, over one common
denominator 0.95 without and 0.99 with heating (from the same formulas in host arithmetic with fused
multiply-adds); the bound lies between."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_11448_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "rec_cosmo.cu"
int main(int, char** v) {
  rec_params p;
  std::memset(&p, 0, sizeof p);
  p.h = 0.67; p.omega_b_h2 = 0.0224; p.omega_c_h2 = 0.12; p.Y_p = 0.24; p.T_cmb0 = 2.7255; p.N_eff = 3.046;
  p.L_box_kpc = 24; p.fudge = 1.14; p.f_alpha = 1; p.n_sub = 1; p.mixing = REC_MIX_FULL; p.heating = std::atof(v[3]);
  const rec::Cosmo c = rec::make_cosmo(p);
  const rec::StepCoef k = rec::step_coef(c, p, std::atof(v[1]), std::atof(v[2]), 1);
  std::printf("%a %a %a %a %a %a\\n", k.dt, k.H, k.Tg, k.kc, k.hq, k.fHe);
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
@pytest.mark.parametrize("heating", [0.0, 1e-16])
def test_temperature_update(tmp_path, heating):
    from paper_2312_11448_gb300 import rec
    src, exe = tmp_path / "coef.cu", tmp_path / "coef"
    src.write_text(PROGRAM)
    subprocess.run([NVCC, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    n, L = 20, np.longdouble
    rng = np.random.default_rng(3)
    d = rng.lognormal(0.0, 0.8, n ** 3)
    d /= d.mean()
    box = rec.Box(n, d, np.zeros((n ** 3, 3)), 64, precision="fp64", mixing="full", heating=heating)
    import torch
    sq = []
    for z in np.linspace(150.0, 400.0, 12):
        z = float(z)
        z1 = float(math.expm1(math.log1p(z) - 0.00274))
        dt, H, Tg, kc, hq, fHe = (L(float.fromhex(v)) for v in subprocess.run(
            [str(exe), repr(z), repr(z1), repr(heating)], check=True, capture_output=True, text=True).stdout.split())
        x = rng.uniform(1e-3, 2e-2, n ** 3)
        T = 2.7255 * (1.0 + z) * rng.uniform(0.2, 0.7, n ** 3)
        box.x.copy_(torch.as_tensor(x))
        box.T.copy_(torch.as_tensor(T))
        box.refresh(z)
        box.step(0, z, z1)
        box.sync()
        xl, Tl, dl = x.astype(L), T.astype(L), box.host("delta").astype(L)
        opx = 1 + fHe + xl
        g, hh = kc * xl / opx, hq / (dl * opx)
        want = (Tl + dt * (g * Tg + hh)) / (1 + dt * (2 * H + g))
        sq.append(np.mean(((box.host("T").astype(L) - want) / want) ** 2))
    box.close()
    assert float(np.sqrt(np.mean(sq))) * 2.0 ** 53 < 0.90
