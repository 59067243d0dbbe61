"""The FP64 energy pass in two kernels (one per Heun stage) at the edges of its 32 x 8 tiles, against
the FP64 CPU oracle: widths and heights at, below and above multiples of the tile, an odd width (a node
pair past the edge), open and periodic in x, with and without staging.

Tolerance: the FP64 parity bar, 1e-12 of a field's maximum (velocities: of the largest speed); 20 steps
of a few hundred rounded operations each keep far below it.
"""
import numpy as np
import pytest

import synthetic_inputs as si
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    from oracle import build as ob
    from paper_1912_02018_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()
    ob.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("nx,ny,D,periodic_x,tma", [(64, 32, 9.0, 0, "1"), (65, 33, 9.0, 0, "1"), (63, 31, 9.0, 1, "1"),
                                                    (100, 40, 12.0, 0, "0"), (37, 17, 6.0, 0, "1"),
                                                    (129, 72, 20.0, 1, "1")])
def test_two_stage_energy_pass_matches_oracle(monkeypatch, nx, ny, D, periodic_x, tma):
    from paper_1912_02018_gb300 import Sim

    monkeypatch.setenv("LBM_TMA", tma)
    case = si.Case(nx=nx, ny=ny, D=D, xc=nx / 2.0 - 0.3, yc=ny / 2.0 + 0.2, Re=40.0, superheat_Tc=0.08, nu_ratio=1.5,
                   periodic_x=periodic_x, seed=nx)
    drho = case.drho()
    sim = Sim.from_case(case, f64=True, init={"drho": drho}).step(20)
    ref = Oracle(case, drho=drho).step(20)
    fluid = ref.field("solid") == 0
    speed = np.hypot(ref.field("ux"), ref.field("uy"))[fluid].max()
    got = sim.fields()
    for k in ("rho", "ux", "uy", "T", "psi"):
        scale = speed if k in ("ux", "uy") else np.abs(ref.field(k)[fluid]).max()
        assert np.abs(got[k] - ref.field(k))[fluid].max() <= 1e-12 * scale, k
    hg, hr = sim.heat_flux(), ref.heat_flux()
    assert hg["count"] == hr["count"] and abs(hg["q_mean"] - hr["q_mean"]) <= 1e-12 * abs(hr["q_mean"])
