"""The FP32 step at the edges of its tiles, against the FP64 CPU oracle: collision tiles of 60 x 12
(psi in the tile), 60 x 4 (psi read) and 64 x 8 nodes (single phase), energy tiles of 60 x 4 and
60 x 16 nodes.  Widths and heights at, below and above multiples of the tile, odd ones, lattices
smaller than a tile, open and periodic in x, both sides of the rules that choose the tile (12000
nodes; 152 energy tiles); staged by TMA and by plain loads, which must agree in every bit.

Tolerance: the FP32 parity bars of 200 steps: 1e-5 of a field's maximum for rho, T and psi, 1e-3 of
the largest speed for the velocities, 1e-3 for the mean heat flux.  Ten steps stay below them.
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


@pytest.mark.parametrize("nx,ny,D,periodic_x,G,storage", [
    (60, 48, 9.0, 0, -2.0, "f32"), (61, 33, 9.0, 0, -2.0, "f32"), (59, 31, 9.0, 1, -2.0, "f32"),
    (37, 17, 6.0, 0, -2.0, "f32"), (121, 99, 20.0, 1, -2.0, "f32"),       # psi from the energy pass
    (120, 100, 20.0, 0, -2.0, "f32"), (181, 73, 20.0, 0, -2.0, "f32"), (243, 61, 20.0, 1, -2.0, "f32"),
    (1200, 11, 5.0, 0, -2.0, "f32"),                                       # psi in the collision's tiles
    (541, 245, 40.0, 0, -2.0, "f32"), (600, 257, 40.0, 1, -2.0, "f32"),    # 16-row energy tiles
    (243, 61, 20.0, 0, -2.0, "f64"),                                       # FP64 populations
    (65, 41, 9.0, 0, 0.0, "f32"), (127, 39, 9.0, 1, 0.0, "f32"), (128, 40, 9.0, 0, 0.0, "f32"),  # no force
])
def test_fp32_step_at_tile_edges(monkeypatch, nx, ny, D, periodic_x, G, storage):
    from paper_1912_02018_gb300 import Sim

    case = si.Case(nx=nx, ny=ny, D=D, xc=nx / 3.0 - 0.3, yc=ny / 2.0 + 0.2, Re=40.0, superheat_Tc=0.08, nu_ratio=1.5,
                   periodic_x=periodic_x, G=G, seed=nx)
    drho = case.drho()
    runs = []
    for tma in ("1", "0"):
        monkeypatch.setenv("LBM_TMA", tma)
        runs.append(Sim.from_case(case, f64=False, storage=storage, init={"drho": drho}).step(10))
    names = ("rho", "ux", "uy", "T", "psi") if G else ("rho", "ux", "uy", "T")
    got, plain = runs[0].fields(names), runs[1].fields(names)
    ref = Oracle(case, drho=drho).step(10)
    fluid = ref.field("solid") == 0
    speed = np.hypot(ref.field("ux"), ref.field("uy"))[fluid].max()
    for k in names:
        assert np.array_equal(got[k], plain[k]), k
        err = np.abs(got[k] - ref.field(k))[fluid].max()
        if k in ("ux", "uy"):
            assert err <= 1e-3 * speed, (k, err)
        else:
            assert err <= 1e-5 * np.abs(ref.field(k)[fluid]).max(), (k, err)
    hg, hr = runs[0].heat_flux(), ref.heat_flux()
    assert hg["count"] == hr["count"] and abs(hg["q_mean"] - hr["q_mean"]) <= 1e-3 * abs(hr["q_mean"])


@pytest.mark.parametrize("f64", [True, False])
def test_hot_vapour_at_the_outlet_is_no_fault(f64):
    # Vapour at 2.3 T_c in the last columns has a psi (p < rho / 3); liquid at that temperature has none.  The
    # last tile reaches past the outlet (64 columns in tiles of 60), where nothing may be evaluated from a
    # density that is not there.
    from paper_1912_02018_gb300 import Sim

    case = si.Case(nx=64, ny=200, D=10.0, xc=16.0, yc=100.0, Re=30.0, superheat_Tc=0.05, noise_amp=0.0)
    probe = Sim.from_case(case, f64=True)
    info = probe.info()
    probe.close()
    x = np.arange(case.nx)
    T = info["T_sat"] + (2.3 * info["Tc"] - info["T_sat"]) * np.clip((x - 40) / 20.0, 0.0, 1.0)
    shape = (case.ny, case.nx)
    sim = Sim.from_case(case, f64=f64, init={"rho": np.full(shape, info["rho_v"]), "T": np.tile(T, (case.ny, 1))})
    sim.step(2).sync()
    sim.close()


@pytest.mark.parametrize("nx,ny,D,periodic_x,storage,psi_mode,collision", [
    # psi evaluated as IEEE FP64 (by the energy pass, for the collision to read) and as FP32 (in the collision's
    # tiles), below and above 12000 nodes and 152 energy tiles
    (61, 33, 9.0, 0, "f32", 1, 0), (243, 61, 20.0, 1, "f32", 1, 0), (541, 245, 40.0, 0, "f32", 1, 0),
    (600, 257, 40.0, 1, "f32", 1, 0),
    (61, 33, 9.0, 0, "f32", 2, 0), (243, 61, 20.0, 1, "f32", 2, 0), (541, 245, 40.0, 0, "f32", 2, 0),
    (600, 257, 40.0, 1, "f32", 2, 0),
    # FP64 populations: psi from the energy pass's second pull, in 4- and 16-row tiles
    (61, 33, 9.0, 1, "f64", 0, 0), (541, 245, 40.0, 0, "f64", 0, 0), (600, 257, 40.0, 1, "f64", 0, 0),
    (541, 245, 40.0, 1, "f64", 1, 0), (243, 61, 20.0, 0, "f64", 2, 0), (600, 257, 40.0, 0, "f64", 2, 0),
    # the BGK operator over both ways to psi
    (61, 33, 9.0, 0, "f32", 0, 1), (243, 61, 20.0, 0, "f32", 0, 1), (243, 61, 20.0, 1, "f64", 0, 1),
])
def test_fp32_psi_routes_and_restart(nx, ny, D, periodic_x, storage, psi_mode, collision):
    # against the oracle with the tolerance of the test above, and bit for bit against a run restored midway,
    # whose first psi comes from k_rho_psi where the other run's comes from the energy pass or the tile
    from paper_1912_02018_gb300 import Sim

    case = si.Case(nx=nx, ny=ny, D=D, xc=nx / 3.0 - 0.3, yc=ny / 2.0 + 0.2, Re=40.0, superheat_Tc=0.08, nu_ratio=1.5,
                   periodic_x=periodic_x, seed=nx + psi_mode, collision=collision)
    drho = case.drho()
    kw = dict(f64=False, storage=storage, psi_mode=psi_mode)
    sim = Sim.from_case(case, init={"drho": drho}, **kw).step(5)
    state = sim.get_state_native()
    sim.step(5)
    again = Sim.from_case(case, **kw)
    again.set_state_native(*state)
    again.step(5)
    names = ("rho", "ux", "uy", "T", "psi", "Fx", "Fy")
    got, restored = sim.fields(names), again.fields(names)
    for k in names:
        assert np.array_equal(got[k], restored[k]), k
    for a, b in zip(sim.get_state_native(), again.get_state_native()):
        assert np.array_equal(a, b)
    ref = Oracle(case, drho=drho).step(10)
    fluid = ref.field("solid") == 0
    speed = np.hypot(ref.field("ux"), ref.field("uy"))[fluid].max()
    for k in ("rho", "ux", "uy", "T", "psi"):
        err = np.abs(got[k] - ref.field(k))[fluid].max()
        if k in ("ux", "uy"):
            assert err <= 1e-3 * speed, (k, err)
        else:
            assert err <= 1e-5 * np.abs(ref.field(k)[fluid]).max(), (k, err)
    sim.close()
    again.close()



def test_single_phase_domain_of_a_batch():
    # a batch collides every FP32 domain in the tiles with psi, a context of its own without psi one node per
    # lane: the same bits
    from paper_1912_02018_gb300 import Batch, Sim

    cases = [si.Case(nx=nx, ny=ny, D=9.0, xc=nx / 3.0, yc=ny / 2.0, Re=40.0, superheat_Tc=0.05, G=G, seed=nx)
             for nx, ny, G in ((127, 41, 0.0), (131, 97, -2.0), (64, 33, 0.0))]
    batch = Batch(cases).step(12)
    for i, case in enumerate(cases):
        one = Sim.from_case(case).step(12)
        names = ("rho", "ux", "uy", "T") + (("psi",) if case.G else ())
        got, want = batch.domain(i).fields(names), one.fields(names)
        for k in names:
            assert np.array_equal(got[k], want[k]), (i, k)
        one.close()
