"""Interpolation weights of the model warps next to a sample (csrc/model.cu):
displacements and source positions a hair above a whole cell, down to the
smallest subnormal, against the oracle with the bar of tests/test_gpu_model.py
(2e-6 of the velocity range, labels bit for bit)."""
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


def field(shape, seed):
    rng = np.random.default_rng(seed)
    v = synth.smooth(rng.uniform(1500.0, 4500.0, shape).astype(np.float32), 1.5).astype(np.float32)
    return v, rng.integers(0, 12, shape).astype(np.int32)


def check(vg, lg, vo, lo):
    assert np.abs(vg.cpu().numpy() - vo).max() <= 2e-6 * max(float(np.ptp(vo)), float(np.abs(vo).max()))
    assert np.array_equal(lg.cpu().numpy(), lo)


TINY = [1e-45, 1e-38, 1e-30, 1e-25, 1e-20, 5e-20, 6e-20, 1e-18, 1e-12, 9e-13, 1e-10, 1e-7, 1.2e-7, 1e-5, 1e-3]


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_squish_by_a_hair(model, sign):
    v, lab = field((23, 2, 2 * len(TINY)), 51)
    dz = np.zeros((2, v.shape[2]), np.float32)
    dz[0, :len(TINY)] = dz[1, len(TINY):] = sign * np.array(TINY)
    vg, lg = model.squish(torch.as_tensor(v, device="cuda"), torch.as_tensor(lab, device="cuda"), dz, 1234.0, -1)
    check(vg, lg, *om.squish(v, lab, dz.astype(np.float64), 1234.0, -1))


def test_squish_by_a_bump_with_tails(model):
    v, lab = field((31, 1, 1000), 52)
    x = np.arange(1000, dtype=np.float32)
    dz = (12.0 * np.exp(-((x - 500.0) / 30.0) ** 2 / 2.0)).astype(np.float32)[None]
    assert ((dz > 0) & (dz < 5.4e-20)).sum() > 200
    vg, lg = model.squish(torch.as_tensor(v, device="cuda"), torch.as_tensor(lab, device="cuda"), dz, 1234.0, -1)
    check(vg, lg, *om.squish(v, lab, dz.astype(np.float64), 1234.0, -1))


@pytest.mark.parametrize("azimuth", [np.pi / 2, -np.pi / 2, 0.0, np.pi])
@pytest.mark.parametrize("direction", [1, -1])
def test_fault_along_an_axis(model, azimuth, direction):
    """cos(pi / 2) = 6e-17 in FP64: positions along the other axis are whole
    cells but for that times the slip, on plane or column 0 a few 1e-17 and less."""
    v, lab = field((24, 25, 26), 54)
    p = dict(cz=12.0, cy=12.0, cx=12.0, azimuth=azimuth, dip=np.deg2rad(55.0), radius=70.0, slip=2.0,
             direction=direction, d_die=11.0, d_perp=14.0, theta_die=np.deg2rad(12.0))
    vg, lg = model.fault(torch.as_tensor(v, device="cuda"), torch.as_tensor(lab, device="cuda"), fill=999.0,
                         fill_label=-2, **p)
    check(vg, lg, *om.fault(v, lab, p, 999.0, -2))
