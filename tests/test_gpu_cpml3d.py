"""The 3D CPML launch (csrc/cpml3d.cu) and the z-march that adds its terms, at
the edges of what they take: widened strips of exactly 72 rows (z, y) or 12
float4s (x) and one more (the general kernels run instead), strips that meet
when widened, strips on one face only or one cell wide, and grids narrower than
a tile. Gather and FP32-storage gradient against the FP64 oracle, relative L2
<= 1e-4 as in the other 3D tests."""
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


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.mark.parametrize("nz,ny,nx,nb,fs", [
    (16, 14, 18, [68, 4, 6, 6, 5, 5], 0),    # 72 rows along z
    (16, 14, 18, [69, 4, 6, 6, 5, 5], 0),    # 73
    (14, 16, 18, [5, 5, 4, 69, 5, 5], 0),    # 73 along y
    (14, 16, 18, [0, 5, 5, 5, 44, 3], 1),    # 12 float4s along x
    (14, 16, 18, [5, 5, 5, 5, 3, 49], 0),    # 14
    (6, 5, 7, [9, 9, 8, 10, 7, 9], 0),       # strips that meet on every axis
    (13, 15, 61, [0, 6, 5, 0, 0, 7], 1),     # one face of each axis
    (15, 13, 40, [1, 1, 1, 1, 1, 1], 0),     # one cell
])
def test_matches_oracle(pkg, nz, ny, nx, nb, fs):
    nt = 110
    cfg = dict(ndim=3, nz=nz, ny=ny, nx=nx, h=10.0, dt=8e-4, nt=nt, bc="cpml", nb=nb, free_surface=fs, R=1e-3, f_ref=15.0)
    v = np.linspace(1700.0, 2500.0, nz * ny * nx).reshape(nz, ny, nx).astype(np.float32)
    w = synth.ricker(20.0, 0.03, 8e-4, nt)
    ext = 10.0 * (np.array([nx, ny, nz]) - 1)
    src = np.array([0.45, 0.55, 0.5]) * ext
    rec = np.random.default_rng(nz + nb[0]).uniform(0.1, 0.9, (12, 3)) * ext
    v64, w64 = v.astype(np.float64), w.astype(np.float64)
    d = 0.5 * oracle.forward(cfg, v64, w64, src=src, rec=rec)["gather"]
    o = oracle.gradient(cfg, v64, w64, src, rec, d)
    sim = pkg.Simulator(cfg, v, max_shots=1, max_rec=12)
    grad, gather = torch.zeros((nz, ny, nx), device="cuda"), torch.zeros((1, nt, 12), device="cuda")
    mis = np.zeros(1)
    pkg.sim_adjoint(sim.handle, 1, torch.as_tensor(w, dtype=torch.float32, device="cuda"), src[None].copy(), 12, rec,
                    torch.as_tensor(d[None], dtype=torch.float32, device="cuda"), gather, mis, 0, grad)
    sim.sync()
    g, h = grad.cpu().numpy(), gather.cpu().numpy()[0]
    sim.close()
    assert rel(h, 2.0 * d) <= 1e-4
    assert abs(float(mis[0]) - o["misfit"]) <= 1e-4 * o["misfit"]
    assert rel(g, o["grad"]) <= 1e-4
