"""Receivers off the grid in both coordinates whose four cells lie in four
subdomains of the resident kernel: one per row astride the edge between cell
columns 127 and 128 (and 255 and 256) of the padded grid, on grids whose
subdomains end at the same row on both sides and on grids where they do not.
Forward and gradient against the per-step kernels: with CPML the forward has
their roundings but for contractions and with the sponge its own weights, so
each trace agrees within 1e-5 of its norm (the bar of test_gpu_resident.py),
or within the smallest normal number: below it FP32 has no relative precision;
the gradient's forward has the same roundings, so its gather is equal bit for
bit, and the gradient agrees within 2e-5 (the bar of
test_gpu_resident_gradient.py)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2605_30541_gb300 as p
    p.abi.load()
    return p


CASES = [
    # nz, nx, nb, bc, fs, shots
    (40, 200, [0, 0, 0, 0, 0, 0], "none", 0, 1),
    (61, 240, [0, 12, 0, 0, 12, 12], "cpml", 1, 2),
    (90, 330, [9, 9, 0, 0, 9, 9], "cpml", 0, 1),
    (90, 330, [15, 15, 0, 0, 15, 15], "sponge", 0, 3),
    (150, 150, [0, 20, 0, 0, 20, 20], "sponge", 1, 9),
    (201, 201, [20, 20, 0, 0, 20, 20], "cpml", 0, 16),
]


def case(nz, nx, nb, bc, fs, shots, nt=151):
    cfg = dict(ndim=2, nz=nz, ny=1, nx=nx, h=10.0, dt=1e-3, nt=nt, bc=bc, nb=nb, free_surface=fs, R=1e-3, f_ref=15.0)
    v = synth.smooth(synth.procedural_2d(nz, nx, 10.0, 4007), 5.0).astype(np.float32)
    w = synth.ricker(25.0, 0.03, 1e-3, nt).astype(np.float32)
    xs = [128 * k - 1 - nb[4] for k in (1, 2) if 128 * k - nb[4] < nx]  # interior column of padded column 128 k - 1
    rec = np.array([((x + 0.37) * 10.0, (z + 0.61) * 10.0) for x in xs for z in range(nz - 1)])
    src = np.stack([np.linspace(xs[0] * 10.0 - 40.0, xs[-1] * 10.0 + 55.0, shots), np.linspace(40.0, 8.0 * nz, shots)],
                   axis=1)
    return cfg, v, w, src, rec


@pytest.mark.parametrize("nz,nx,nb,bc,fs,shots", CASES)
def test_forward(pkg, monkeypatch, nz, nx, nb, bc, fs, shots):
    cfg, v, w, src, rec = case(nz, nx, nb, bc, fs, shots)
    out = {}
    for on in ("0", "1"):
        monkeypatch.setenv("GSIM_RESIDENT", on)
        monkeypatch.setenv("GSIM_MARCH", "0")
        sim = pkg.Simulator(cfg, v, max_shots=shots, max_rec=len(rec))
        out[on] = sim.forward(w, src, rec)["gather"].cpu().numpy().astype(np.float64)
        sim.sync()
        assert (pkg.sim_get_info(sim.handle).last_path == 2) == (on == "1")
        sim.close()
    e = np.linalg.norm(out["1"] - out["0"], axis=1)
    assert (e <= 1e-5 * np.linalg.norm(out["0"], axis=1) + np.finfo(np.float32).tiny).all()


@pytest.mark.parametrize("nz,nx,nb,bc,fs,shots", CASES)
@pytest.mark.parametrize("fp16", [0, 1])
def test_gradient(pkg, monkeypatch, nz, nx, nb, bc, fs, shots, fp16):
    cfg, v, w, src, rec = case(nz, nx, nb, bc, fs, shots)
    d = torch.zeros((shots, cfg["nt"], len(rec)), device="cuda")
    out = {}
    for on in ("0", "1"):
        monkeypatch.setenv("GSIM_RESIDENT", on)
        sim = pkg.Simulator(cfg, v, max_shots=shots, max_rec=len(rec))
        grad, gather, mis = torch.zeros((nz, nx), device="cuda"), torch.zeros_like(d), np.zeros(1)
        pkg.sim_adjoint(sim.handle, shots, torch.as_tensor(w, device="cuda"), src, len(rec), rec, d, gather, mis, fp16, grad)
        sim.sync()
        out[on] = gather.cpu().numpy(), grad.cpu().numpy().astype(np.float64)
        sim.close()
    (h0, g0), (h1, g1) = out["0"], out["1"]
    assert np.array_equal(h0, h1)
    if not fp16:
        assert np.linalg.norm(g1 - g0) <= 2e-5 * np.linalg.norm(g0)
