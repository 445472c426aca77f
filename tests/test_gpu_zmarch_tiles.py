"""The tiles of the 3D z-march by name (64 x 16 and 32 x 32 columns staged by
bulk tensor copies, 128 x 8 by per-thread copies): every tile and z chunk gives
the same bits, forward with FP32 and FP16 snapshots, and gradient (record and
adjoint modes). Extents end inside a tile, at its edge and one past it in x and
y; sources and receivers lie on and astride tile and chunk edges."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TILES = ("async", "tma-64", "tma-32")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2605_30541_gb300 as p
    p.abi.load()
    return p


CASES = [
    # nz, ny, nx, nb (all faces; 0 at the top with a free surface), bc, fs
    (21, 20, 52, 6, "cpml", 1),    # padded 64 x 32: tile edges
    (17, 21, 53, 6, "cpml", 0),    # one past
    (30, 17, 31, 5, "sponge", 0),
    (9, 70, 121, 4, "cpml", 0),    # several tiles
    (25, 33, 33, 0, "none", 1),
]


def case(nz, ny, nx, nb, bc, fs, nt):
    cfg = dict(ndim=3, nz=nz, ny=ny, nx=nx, h=10.0, dt=8e-4, nt=nt, bc=bc, nb=[0 if fs else nb] + [nb] * 5, free_surface=fs,
               R=1e-3, f_ref=15.0, snap_every=7, snap_begin=2, snap_end=nt)
    v = synth.procedural_3d(nz, ny, nx, 10.0, 67).astype(np.float32)
    w = synth.ricker(25.0, 0.02, 8e-4, nt).astype(np.float32)
    zm, ym, xm = ((n - 1) * 10.0 for n in (nz, ny, nx))
    edge = lambda k, n: min(max(0.0, (k - nb - 0.5) * 10.0), n)  # noqa: E731 (between padded cells k - 1 and k)
    src = np.array([[edge(32, xm), edge(16, ym), 0.4 * zm], [0.3 * xm, 0.6 * ym, min(zm, 73.0)]])
    rec = np.array([[edge(a, xm), edge(b, ym), c * zm] for a in (32, 64) for b in (16, 32) for c in (0.2, 0.55)] +
                   [[0.5 * xm, 0.5 * ym, 10.0]])
    return cfg, v, w, src, rec


@pytest.mark.parametrize("nz,ny,nx,nb,bc,fs", CASES)
@pytest.mark.parametrize("fp16", [False, True])
def test_forward(pkg, monkeypatch, nz, ny, nx, nb, bc, fs, fp16):
    cfg, v, w, src, rec = case(nz, ny, nx, nb, bc, fs, 61)
    first = None
    for tile in TILES:
        for chunk in (500, 8, 5):
            monkeypatch.setenv("GSIM_ZMARCH", tile)
            monkeypatch.setenv("GSIM_ZCHUNK", str(chunk))
            sim = pkg.Simulator(cfg, v, max_shots=2, max_rec=len(rec), snap_fp16=fp16)
            out = sim.forward(w, src, rec, snapshots=True)
            sim.sync()
            got = out["gather"].cpu().numpy(), out["snaps"].cpu().numpy()
            sim.close()
            assert np.isfinite(got[0]).all() and np.abs(got[0]).max() > 0
            if first is None:
                first = got
            assert np.array_equal(got[0], first[0]) and np.array_equal(got[1], first[1]), (tile, chunk)


@pytest.mark.parametrize("nz,ny,nx,nb,bc,fs", CASES)
@pytest.mark.parametrize("fp16", [0, 1])
def test_gradient(pkg, monkeypatch, nz, ny, nx, nb, bc, fs, fp16):
    cfg, v, w, src, rec = case(nz, ny, nx, nb, bc, fs, 53)
    cfg.update(snap_every=0, snap_begin=0, snap_end=0)
    d = torch.zeros((2, cfg["nt"], len(rec)), device="cuda")
    first = None
    for tile in TILES:
        for chunk in (500, 7):
            monkeypatch.setenv("GSIM_ZMARCH", tile)
            monkeypatch.setenv("GSIM_ZCHUNK", str(chunk))
            sim = pkg.Simulator(cfg, v, max_shots=2, max_rec=len(rec))
            grad, gather, mis = torch.zeros(v.shape, device="cuda"), torch.zeros_like(d), np.zeros(1)
            pkg.sim_adjoint(sim.handle, 2, torch.as_tensor(w, device="cuda"), src, len(rec), rec, d, gather, mis, fp16, grad)
            sim.sync()
            got = gather.cpu().numpy(), grad.cpu().numpy()
            sim.close()
            assert np.isfinite(got[1]).all() and np.abs(got[1]).max() > 0
            if first is None:
                first = got
            assert np.array_equal(got[0], first[0]) and np.array_equal(got[1], first[1]), (tile, chunk)
