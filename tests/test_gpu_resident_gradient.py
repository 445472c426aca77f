"""The gradient's resident path (runs of steps between checkpoints in one
cooperative launch each) against the per-step kernels on the same inputs: the
forward and recorded states have the same roundings, so the gather is equal
bit for bit; the adjoint sweep sums the same terms in another order, so with
FP32 storage the gradient agrees within 2e-5. FP16 imaging terms are scaled
per warp instead of per tile, which moves their error and not their size:
the distance to the FP32-storage gradient may be 1.5 times that of the
per-step kernels plus 2e-5 of its norm. Cases: subdomain edges in both axes
(several columns, a last subdomain of few rows), both boundaries, free
surface, vertical receivers (a residual in every row), two checkpoint levels,
several launches per run of steps, segments of odd length."""
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
    # nz, nx, nb, bc, fs, nt, shots, vertical receivers, fp16, two levels
    (48, 70, [12, 12, 0, 0, 12, 12], "cpml", 0, 101, 2, False, 0, False),
    (48, 70, [0, 12, 0, 0, 12, 12], "cpml", 1, 101, 2, False, 1, False),
    (48, 70, [12, 12, 0, 0, 12, 12], "sponge", 0, 101, 2, False, 1, False),
    (151, 201, [0, 20, 0, 0, 20, 33], "sponge", 1, 90, 3, True, 0, False),
    (151, 301, [7, 20, 0, 0, 20, 3], "cpml", 0, 90, 2, True, 0, False),
    (119, 246, [5, 5, 0, 0, 5, 5], "cpml", 0, 83, 1, False, 0, True),
    (201, 201, [20, 20, 0, 0, 20, 20], "cpml", 0, 50, 16, False, 1, False),
    (130, 230, [0, 20, 0, 0, 20, 20], "cpml", 1, 50, 37, False, 1, False),
    (40, 40, [0, 0, 0, 0, 0, 0], "cpml", 0, 4, 1, False, 0, False),
]


@pytest.mark.parametrize("nz,nx,nb,bc,fs,nt,shots,vertical,fp16,two", CASES)
def test_matches_per_step_kernels(pkg, monkeypatch, nz, nx, nb, bc, fs, nt, shots, vertical, fp16, two):
    cfg = dict(ndim=2, nz=nz, ny=1, nx=nx, h=10.0, dt=1e-3, nt=nt, bc=bc, nb=nb, free_surface=fs, R=1e-3, f_ref=15.0)
    v = synth.smooth(synth.procedural_2d(nz, nx, 10.0, 4001), 5.0).astype(np.float32)
    w = torch.as_tensor(synth.ricker(15.0, 0.02, 1e-3, nt), dtype=torch.float32, device="cuda")
    zm, xm = (nz - 1) * 10.0, (nx - 1) * 10.0
    src = np.stack([np.linspace(0.1 * xm, 0.9 * xm, shots), np.linspace(0.2 * zm, 0.6 * zm, shots)], axis=1)
    t = np.linspace(0.0, 1.0, 41)
    rec = np.stack([np.full(41, 0.37 * xm), t * zm] if vertical else [t * xm, np.full(41, 10.0)], axis=1)
    d = torch.as_tensor(1e-3 * np.random.default_rng(nx).standard_normal((shots, nt, 41)), dtype=torch.float32,
                        device="cuda")
    out = {}
    for on, half in [("0", 0), ("1", 0)] + ([("0", 1), ("1", 1)] if fp16 else []):
        monkeypatch.setenv("GSIM_RESIDENT", on)
        # room for two checkpoint levels only, or as much as there is
        budget = 55 * 4 * 400 * (nz + 60) if two else 0
        sim = pkg.Simulator(cfg, v, max_shots=shots, max_rec=41, adj_budget=budget)
        grad, gather, mis = torch.zeros((nz, nx), device="cuda"), torch.zeros((shots, nt, 41), device="cuda"), np.zeros(1)
        for _ in range(2):  # a captured run, then its replay
            grad.zero_()
            pkg.sim_adjoint(sim.handle, shots, w, src, 41, rec, d, gather, mis, half, grad)
        sim.sync()
        out[on, half] = gather.cpu().numpy(), grad.cpu().numpy().astype(np.float64), float(mis[0])
        sim.close()
    (h0, g0, m0), (h1, g1, m1) = out["0", 0], out["1", 0]
    assert np.array_equal(h0, h1)
    assert abs(m1 - m0) <= 2e-5 * m0
    assert np.isfinite(g1).all() and np.linalg.norm(g1 - g0) <= 2e-5 * np.linalg.norm(g0)
    if fp16:
        assert np.array_equal(out["0", 1][0], out["1", 1][0])
        e0, e1 = (np.linalg.norm(out[on, 1][1] - g0) for on in ("0", "1"))
        assert e1 <= 1.5 * e0 + 2e-5 * np.linalg.norm(g0)
