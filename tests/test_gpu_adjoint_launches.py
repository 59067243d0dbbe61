"""kernel_launches of lbm_info counts what an adjoint window launches: its forward steps (a step's launches as
lbm_step counts them, the psi pass of the first one where there is one), the same steps recomputed from the
checkpoints, and five reverse kernels a step."""
import pytest

import synthetic_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    from paper_1912_02018_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("f64,nx,ny", [(True, 48, 24), (False, 48, 24), (False, 160, 96)])
def test_window_launches_are_counted(f64, nx, ny):
    from paper_1912_02018_gb300 import Sim

    case = si.cylinder_case(nx, ny, 8.0, Re=300.0, superheat_Tc=0.05)
    sim = Sim.from_case(case, f64=f64)
    n0 = sim.info()["kernel_launches"]
    sim.step(1)
    first = sim.info()["kernel_launches"] - n0
    sim.step(1)
    later = sim.info()["kernel_launches"] - n0 - first
    n1 = sim.info()["kernel_launches"]
    sim.adjoint_window(24, ckpt_every=10)  # segments of 10, 10 and 4 steps
    forward = first + 23 * later
    recompute = 3 * first + 21 * later
    assert sim.info()["kernel_launches"] - n1 == forward + recompute + 24 * 5
    sim.close()
