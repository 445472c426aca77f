"""The fault warp's segment test and its own FP64 functions (csrc/model.cu) at
the sizes and angles where they can go wrong, against the oracle with the bar
of tests/test_gpu_model.py (2e-6 of the velocity range, labels bit for bit):
rows that end inside a 32-voxel segment and a 128-voxel tile, widths that are
no multiple of 4, depths that are no multiple of 8, die-off regions narrower
than a segment and wider than the grid, an axis inside the grid (every
quadrant of the angle, offset zero from the axis), a slip of more than a
quarter radian, a radius of 1e7 cells, and no labels."""
import numpy as np
import pytest

import synth
from oracle import model as om

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def model():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2605_30541_gb300 import model as m
    return m


def params(**kw):
    p = dict(cz=20.0, cy=0.0, cx=60.0, azimuth=np.pi / 2, dip=np.deg2rad(60.0), radius=500.0, slip=6.0, direction=1,
             d_die=20.0, d_perp=1e9, theta_die=np.deg2rad(40.0))
    p.update(kw)
    return p


CASES = [
    ((33, 1, 128), params(d_die=5.0)),
    ((9, 1, 129), params(cz=4.0, direction=-1)),
    ((41, 1, 517), params(cx=300.0, d_die=600.0)),
    ((30, 1, 95), params(cx=45.0, radius=9.0, dip=np.deg2rad(30.0), slip=4.0, d_die=30.0, theta_die=np.pi)),
    # the axis on a voxel: centre (20, 40), offset zero from it
    ((40, 1, 80), params(cz=20.0 + 12.0, cx=40.0, dip=np.pi / 2, radius=12.0, slip=2.0, d_die=15.0, theta_die=np.pi)),
    ((30, 1, 100), params(radius=1e7, slip=3.0, cx=50.0, theta_die=1e-3)),
    ((17, 6, 70), params(cz=8.0, cy=3.0, cx=35.0, azimuth=0.7, radius=60.0, slip=-5.0, d_perp=12.0)),
    ((12, 5, 33), params(cz=6.0, cy=2.0, cx=16.0, azimuth=-2.4, radius=40.0, slip=15.0, d_perp=4.0)),
]


@pytest.mark.parametrize("k", range(len(CASES)))
@pytest.mark.parametrize("labels", [True, False])
def test_fault_matches_oracle(model, k, labels):
    shape, p = CASES[k]
    nz, ny, nx = shape
    rng = np.random.default_rng(100 + k)
    v = synth.smooth(rng.uniform(1500.0, 4500.0, shape).astype(np.float32), 1.5).astype(np.float32)
    lab = rng.integers(0, 12, shape).astype(np.int32)
    vo, lo = om.fault(v, lab, p, 1234.0, -1)
    vg, lg = model.fault(torch.as_tensor(v, device="cuda"), torch.as_tensor(lab, device="cuda") if labels else None,
                         fill=1234.0, fill_label=-1, **p)
    assert np.abs(vg.cpu().numpy() - vo).max() <= 2e-6 * max(float(np.ptp(vo)), float(np.abs(vo).max()))
    if labels:
        assert np.array_equal(lg.cpu().numpy(), lo)
    else:
        assert lg is None
    assert (vo != v).any()
