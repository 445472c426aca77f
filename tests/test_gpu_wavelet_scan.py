"""The chunked scan of the band-pass recursion (csrc/wavelet.cu) at the sizes
where it can go wrong: records shorter than one sample per thread, chunk
lengths of exactly one and one plus a remainder, a last chunk of one sample,
the other orders (their own instance), and a record too long for shared
memory (the workspace in global memory).

Tolerance: 1e-9 of the peak, the bar of the production bands; a host model
of the scan against extended precision has 2e-13 up to order 8 and 1.2e-11
at order 16, the oracle's own rounding is below 4e-13."""
import numpy as np
import pytest

from oracle import wavelet as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2605_30541_gb300 as p
    p.abi.load()
    return p


# order 4 pads 27 samples at each end: nt + 54 samples in 1024 chunks (970 and 8138: full chunks)
@pytest.mark.parametrize("order,nt", [(4, 28), (4, 201), (4, 969), (4, 970), (4, 971), (4, 8138), (4, 8139), (1, 1001), (2, 900),
                                      (3, 1501), (5, 1200), (8, 1501), (16, 1501)])
def test_scan_matches_the_definition(pkg, order, nt):
    lo, hi, f0 = W.BANDS[2]
    ref = W.bandpass_ricker(f0, lo, hi, 1e-3, nt, order=order)
    g = pkg.bandpass_ricker(nt, 1e-3, f0, lo, hi, order=order, dtype="float64").cpu().numpy()
    assert np.max(np.abs(g - ref)) <= 1e-9 * np.abs(ref).max()


def test_record_beyond_shared_memory(pkg):
    lo, hi, f0 = W.BANDS[4]
    nt = 230001
    ref = W.bandpass_ricker(f0, lo, hi, 1e-3, nt)
    g = pkg.bandpass_ricker(nt, 1e-3, f0, lo, hi, dtype="float64").cpu().numpy()
    assert np.max(np.abs(g - ref)) <= 1e-9 * np.abs(ref).max()
