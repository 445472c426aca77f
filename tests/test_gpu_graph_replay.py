"""A handle's captured time loops are replayed for the call they were captured
for only: gradients of changing shot counts on one handle (a survey taken in
mini-batches) against a fresh handle for each. The launches and their order are
the same, so gather, misfit and gradient are equal bit for bit. On a GPU of 152
SMs the counts of the first three cases run as 14 and 2 x 15 shots, 18 and
2 x 17, 2 x 8 and 3 x 11 (shots XOR 16 times the launch's shots agrees), the
larger count first or second; the last case runs the per-step kernels."""
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


@pytest.mark.parametrize("nz,nx,nb,bc,fs,counts,fp16,resident", [
    (201, 201, [20, 20, 0, 0, 20, 20], "cpml", 0, (14, 30, 14), 1, "1"),
    (201, 201, [20, 20, 0, 0, 20, 20], "cpml", 0, (34, 18, 34), 0, "1"),
    (150, 300, [0, 30, 0, 0, 30, 30], "cpml", 1, (32, 16), 1, "1"),
    (151, 301, [40, 40, 0, 0, 40, 40], "sponge", 0, (14, 30), 0, "1"),
    (60, 90, [12, 12, 0, 0, 12, 12], "cpml", 0, (3, 5, 3), 0, "0"),
])
def test_shot_counts_on_one_handle(pkg, monkeypatch, nz, nx, nb, bc, fs, counts, fp16, resident):
    nt, nrec = 60, 23
    monkeypatch.setenv("GSIM_RESIDENT", resident)
    cfg = dict(ndim=2, nz=nz, ny=1, nx=nx, h=10.0, dt=1e-3, nt=nt, bc=bc, nb=nb, free_surface=fs, R=1e-3, f_ref=15.0)
    v = synth.smooth(synth.procedural_2d(nz, nx, 10.0, 4003), 5.0).astype(np.float32)
    w = torch.as_tensor(synth.ricker(25.0, 0.02, 1e-3, nt), dtype=torch.float32, device="cuda")
    xm = (nx - 1) * 10.0
    most = max(counts)
    src = np.stack([np.linspace(0.05 * xm, 0.95 * xm, most), np.linspace(20.0, 60.0, most)], axis=1)
    rec = np.stack([np.linspace(0.0, xm, nrec), np.full(nrec, 30.0)], axis=1)
    d = torch.as_tensor(1e-3 * np.random.default_rng(nx).standard_normal((most, nt, nrec)), dtype=torch.float32,
                        device="cuda")

    def gradient(sim, shots):
        grad, gather, mis = torch.zeros((nz, nx), device="cuda"), torch.zeros((shots, nt, nrec), device="cuda"), np.zeros(1)
        pkg.sim_adjoint(sim.handle, shots, w, src[:shots].copy(), nrec, rec, d[:shots].contiguous(), gather, mis, fp16, grad)
        sim.sync()
        return grad.cpu().numpy(), gather.cpu().numpy(), float(mis[0])

    one = pkg.Simulator(cfg, v, max_shots=most, max_rec=nrec)
    got = [gradient(one, shots) for shots in counts]
    one.close()
    for shots, (g, h, m) in zip(counts, got):
        fresh = pkg.Simulator(cfg, v, max_shots=most, max_rec=nrec)
        g0, h0, m0 = gradient(fresh, shots)
        fresh.close()
        assert np.isfinite(g0).all() and np.linalg.norm(g0) > 0 and all(np.any(h0[k]) for k in range(shots))
        assert np.array_equal(h, h0) and m == m0 and np.array_equal(g, g0)
