"""The FP64 fold of the imaging sums onto the interior cells (csrc/adjoint.cu)
where its work is split by size: blocks of absorbing cells above and below
the width one warp takes (512 cells), absorbing layers on some faces only,
one-cell extents and several shots, by the FP64 gradient against the oracle
(relative L2 <= 1e-10, the bar of the FP64 gradient tests)."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("nz,nx,nb,shots", [
    (24, 31, [24, 23, 0, 0, 22, 25], 2),   # corner blocks of 528 .. 650 cells
    (24, 31, [21, 21, 0, 0, 21, 22], 1),   # 484 and 506
    (19, 40, [0, 30, 0, 0, 0, 20], 2),     # two faces, one corner
    (19, 40, [0, 0, 0, 0, 17, 0], 1),      # one face
    (1, 40, [12, 13, 0, 0, 10, 0], 1),     # one row gathers both z faces
    (17, 23, [0, 0, 0, 0, 0, 0], 1),       # nothing to fold
])
def test_fold_matches_oracle(pkg, nz, nx, nb, shots):
    cfg = dict(ndim=2, nz=nz, ny=1, nx=nx, h=10.0, dt=1e-3, nt=60, bc="sponge", nb=nb, free_surface=0, R=1e-3,
               f_ref=15.0)
    v = np.linspace(1600.0, 2600.0, nz * nx).reshape(nz, nx)
    w = synth.ricker(15.0, 0.02, 1e-3, 60).astype(np.float64)
    zm, xm = (nz - 1) * 10.0, (nx - 1) * 10.0
    src = np.array([[0.3 * xm, 0.4 * zm], [0.8 * xm, 0.7 * zm]])[:shots]
    rec = np.stack([np.linspace(0.0, xm, 9), np.linspace(0.0, zm, 9)], axis=1)
    d = 0.01 * np.random.default_rng(nx + nb[5]).standard_normal((shots, 60, 9))
    ref = sum(oracle.gradient(cfg, v, w, s, rec, d[k])["grad"] for k, s in enumerate(src))
    sim = pkg.Simulator(cfg, v, max_shots=shots, max_rec=9, precision=pkg.SIM_FP64)
    grad = torch.zeros((nz, nx), dtype=torch.float64, device="cuda")
    pkg.sim_adjoint(sim.handle, shots, torch.as_tensor(w, device="cuda"), src, 9, rec, torch.as_tensor(d, device="cuda"),
                    None, np.zeros(1), 0, grad)
    sim.sync()
    g = grad.cpu().numpy()
    sim.close()
    assert np.linalg.norm(g - ref) <= 1e-10 * np.linalg.norm(ref)
