"""The force planes of lbm_fields in the FP32 build are, bit for bit, the force that the collision of that
population storage applies: its stencil and force evaluated here in numpy, operation by operation (a
product of two FP32 numbers is exact in FP64, so an FMA is a product and a sum there, rounded once)."""
import numpy as np
import pytest

import synthetic_inputs as si

pytestmark = pytest.mark.gpu

F = np.float32
ISO = {1: 4.0 / 21.0, 2: 4.0 / 45.0, 4: 1.0 / 60.0, 5: 2.0 / 315.0, 8: 1.0 / 5040.0}
# Eq. (interForce): the pairs (e, -e) in the order in which the FP16-storage collision adds them
PAIRS = [(1, 0), (2, 0), (-2, 1), (-1, 1), (0, 1), (1, 1), (2, 1), (-2, 2), (-1, 2), (0, 2), (1, 2), (2, 2)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    from paper_1912_02018_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build()
    torch.cuda.set_device(0)


def _fma(a, b, c):
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(F)


def _shifted(psi, periodic_x):
    ny, nx = psi.shape
    x = np.arange(nx)

    def at(dx, dy):
        col = (x + dx) % nx if periodic_x else np.clip(x + dx, 0, nx - 1)
        return np.roll(psi, -dy, 0)[:, col]
    return at


def _pairs_gradient(at):
    """Pair by pair (FP16 populations)."""
    sx, sy = np.zeros_like(at(0, 0)), np.zeros_like(at(0, 0))
    for ex, ey in PAIRS:
        w, d = ISO[ex * ex + ey * ey], at(ex, ey) - at(-ex, -ey)
        if ex:
            sx = _fma(F(w * ex), d, sx)
        if ey:
            sy = _fma(F(w * ey), d, sy)
    return sx, sy


def _rows_gradient(at):
    """Row by row, the outer ones first (FP32 and FP64 populations)."""
    w = {(k, c): F(ISO.get(k * k + c * c, 0.0)) for k in range(3) for c in range(3)}
    gx, gy = np.zeros_like(at(0, 0)), np.zeros_like(at(0, 0))
    for k in (2, 1, 0):
        for y in ((-k, k) if k else (0,)):
            X1, X2 = at(1, y) - at(-1, y), at(2, y) - at(-2, y)
            gx = _fma(w[k, 1], X1, _fma(F(2) * w[k, 2], X2, gx))
        if k:
            s = [at(0, k) - at(0, -k)] + [(at(c, k) + at(-c, k)) - (at(c, -k) + at(-c, -k)) for c in (1, 2)]
            gy = _fma(F(k) * w[k, 0], s[0], _fma(F(k) * w[k, 1], s[1], _fma(F(k) * w[k, 2], s[2], gy)))
    return gx, gy


@pytest.mark.parametrize("storage,psi_mode", [("f32", 0), ("f32", 1), ("f32", 2), ("f64", 0), ("f16s", 0)])
@pytest.mark.parametrize("nx,ny,periodic_x", [(131, 97, 0), (128, 100, 1), (61, 45, 0)])
def test_force_planes_are_the_collisions_own(nx, ny, periodic_x, storage, psi_mode):
    from paper_1912_02018_gb300 import Sim

    case = si.Case(nx=nx, ny=ny, D=14.0, xc=nx / 3.0, yc=ny / 2.0, Re=40.0, superheat_Tc=0.08, periodic_x=periodic_x,
                   seed=nx)
    sim = Sim.from_case(case, f64=False, storage=storage, psi_mode=psi_mode).step(7)
    got, info = sim.fields(("rho", "psi", "Fx", "Fy", "solid")), sim.info()
    sim.close()
    psi, rho = got["psi"].astype(F), got["rho"].astype(F)
    assert np.array_equal(psi, got["psi"])
    drho, g = rho - F(info["rho_l"]), F(info["g"])
    if storage == "f16s":
        sx, sy = _pairs_gradient(_shifted(psi, periodic_x))
        a = F(F(-case.G) * F(1.0 / 3.0)) * psi
        fx, fy = a * sx - drho * g, a * sy
    else:
        sx, sy = _rows_gradient(_shifted(psi, periodic_x))
        a = F(-case.G / 3.0) * psi
        fx, fy = _fma(-g, drho, a * sx), a * sy
    fluid = got["solid"] == 0
    for k, want in (("Fx", fx), ("Fy", fy)):
        assert want.dtype == F
        assert np.array_equal(got[k][fluid], want[fluid].astype(np.float64)), k
