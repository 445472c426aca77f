"""Model warps with positions far outside the grid or no numbers
(csrc/model.cu): a displacement or offset of any size reads the edge or is
filled, as the rule for positions beyond the grid says, and one that is no
number gives no velocity or the fill; every index stays within the grid."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def model():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2605_30541_gb300 import model as m
    return m


def test_squish(model):
    far = np.array([np.nan, np.inf, -np.inf, 1e30, -1e30, 3e9, -3e9, 2147483648.0, -2147483648.0, 2147483520.0, 1e5, -1e5],
                   np.float32)
    rng = np.random.default_rng(3)
    v = rng.uniform(1500.0, 4500.0, (40, 2, 16)).astype(np.float32)
    lab = rng.integers(0, 12, v.shape).astype(np.int32)
    dz = np.zeros((2, 16), np.float32)
    dz[1, :len(far)] = far
    vg, lg = model.squish(torch.as_tensor(v, device="cuda"), torch.as_tensor(lab, device="cuda"), dz, 1234.0, -1)
    vg, lg = vg.cpu().numpy(), lg.cpu().numpy()
    moved = dz != 0
    assert np.array_equal(vg[:, ~moved], v[:, ~moved]) and np.array_equal(lg[:, ~moved], lab[:, ~moved])
    out, num = vg[:, moved], ~np.isnan(dz[moved])
    assert np.all(out[:, num] == 1234.0) and np.all(lg[:, moved][:, num] == -1)
    assert np.all(np.isnan(out[:, ~num]) | (out[:, ~num] == 1234.0))


@pytest.mark.parametrize("off", [2147483647, -2147483648, 39, -39])
def test_deposit_offsets(model, off):
    nz, nx, t = 30, 20, 12
    eta = torch.arange(10.0, device="cuda")[:, None].expand(10, nx).contiguous()
    v = torch.full((nz, nx), 2000.0, device="cuda")
    vg, _ = model.deposit(v, None, t, None, [2500.0], a_eta=1.0, eta=eta, offsets=[off])
    assert torch.equal(vg[:t], torch.full((t, nx), 2500.0 + (9.0 if off > 0 else 0.0), device="cuda"))
