"""Which path a gradient takes (sim_info.adj_path), so that the comparisons of
test_gpu_resident_gradient.py and test_gpu_corner_receivers.py compare what
they mean to: their cases run resident unless GSIM_RESIDENT is 0, where they
run launches per step."""
import numpy as np
import pytest

import synth
import test_gpu_corner_receivers
import test_gpu_resident_gradient

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

STEPS, RESIDENT, VOLUME = 1, 2, 3


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2605_30541_gb300 as p
    p.abi.load()
    return p


def path(pkg, cfg, shots, rec, fp16=0, budget=0):
    shape = (cfg["nz"], cfg["nx"]) if cfg["ndim"] == 2 else (cfg["nz"], cfg["ny"], cfg["nx"])
    sim = pkg.Simulator(cfg, np.full(shape, 2000.0, np.float32), max_shots=shots, max_rec=len(rec), adj_budget=budget)
    assert pkg.sim_get_info(sim.handle).adj_path == 0
    src = np.tile([5.0 * (n - 1) for n in shape[::-1]], (shots, 1))
    w = torch.as_tensor(synth.ricker(15.0, 0.02, 1e-3, cfg["nt"]), dtype=torch.float32, device="cuda")
    d = torch.zeros((shots, cfg["nt"], len(rec)), device="cuda")
    pkg.sim_adjoint(sim.handle, shots, w, src, len(rec), rec, d, None, None, fp16, torch.zeros(shape, device="cuda"))
    sim.sync()
    p = pkg.sim_get_info(sim.handle).adj_path
    sim.close()
    return p


@pytest.mark.parametrize("nz,nx,nb,bc,fs,nt,shots,vertical,fp16,two", test_gpu_resident_gradient.CASES)
def test_resident_gradient_cases(pkg, monkeypatch, nz, nx, nb, bc, fs, nt, shots, vertical, fp16, two):
    cfg = dict(ndim=2, nz=nz, ny=1, nx=nx, h=10.0, dt=1e-3, nt=nt, bc=bc, nb=nb, free_surface=fs, R=1e-3, f_ref=15.0)
    zm, xm, t = (nz - 1) * 10.0, (nx - 1) * 10.0, np.linspace(0.0, 1.0, 41)
    rec = np.stack([np.full(41, 0.37 * xm), t * zm] if vertical else [t * xm, np.full(41, 10.0)], axis=1)
    budget = 55 * 4 * 400 * (nz + 60) if two else 0
    for half in range(fp16 + 1):
        monkeypatch.setenv("GSIM_RESIDENT", "1")
        assert path(pkg, cfg, shots, rec, half, budget) == RESIDENT
        monkeypatch.setenv("GSIM_RESIDENT", "0")
        assert path(pkg, cfg, shots, rec, half, budget) == STEPS


@pytest.mark.parametrize("nz,nx,nb,bc,fs,shots", test_gpu_corner_receivers.CASES)
def test_corner_cases(pkg, monkeypatch, nz, nx, nb, bc, fs, shots):
    cfg, _, _, _, rec = test_gpu_corner_receivers.case(nz, nx, nb, bc, fs, shots)
    for half in (0, 1):
        monkeypatch.setenv("GSIM_RESIDENT", "1")
        assert path(pkg, cfg, shots, rec, half) == RESIDENT
        monkeypatch.setenv("GSIM_RESIDENT", "0")
        assert path(pkg, cfg, shots, rec, half) == STEPS


def test_volume(pkg):
    cfg = dict(ndim=3, nz=20, ny=18, nx=22, h=10.0, dt=8e-4, nt=20, bc="sponge", nb=[4] * 6, free_surface=0, R=1e-3, f_ref=15.0)
    assert path(pkg, cfg, 1, np.array([[50.0, 60.0, 70.0], [110.0, 90.0, 100.0]])) == VOLUME
