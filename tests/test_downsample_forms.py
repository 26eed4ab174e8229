"""Every form of the downsampling kernel: 16, 4 and 1 channels per load of
time-major blocks, words and bytes of channel-major rows, blocks that start at any
byte, rows of 16-bit lane sums at their largest (factor 256, all samples 255) and the
byte form beyond. Bytes equal the oracle's."""
import numpy as np
import pytest

from oracle import plans as PL
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FACTORS = (1, 2, 4, 16, 128, 256, 512, 1024)


def _check(tx, X, layout, f, shift):  # noqa: F811
    nchan, n = X.shape
    buf = torch.empty(nchan * n + shift, dtype=torch.uint8, device="cuda")   # 256-byte aligned
    src = buf[shift:]
    src.copy_(torch.from_numpy(np.ascontiguousarray(X.T if layout == "tf" else X)).cuda().reshape(-1))
    got = tx.downsample(src, layout, nchan, n, f).cpu().numpy()
    got = got.reshape(n // f, nchan).T if layout == "tf" else got.reshape(nchan, n // f)
    assert np.array_equal(got, PL.downsample(X, f)), (f, shift)


@pytest.mark.parametrize("layout", ["tf", "ft"])
@pytest.mark.parametrize("nchan", [16, 20, 68, 80, 7])
def test_forms(tx, layout, nchan):  # noqa: F811
    X = np.random.default_rng(nchan).integers(0, 256, size=(nchan, 2048), dtype=np.uint8)
    for f in FACTORS:
        for shift in (0, 1, 4, 8):
            _check(tx, X, layout, f, shift)


@pytest.mark.parametrize("layout", ["tf", "ft"])
@pytest.mark.parametrize("nchan", [32, 12, 5])
def test_largest_sums(tx, layout, nchan):  # noqa: F811
    for f in FACTORS:
        _check(tx, np.full((nchan, 1024), 255, dtype=np.uint8), layout, f, 0)


# channel-major rows whose length is no multiple of four: rows start at any byte
@pytest.mark.parametrize("n,f", [(1002, 2), (1001, 1), (6, 2), (2, 2), (1004, 4)])
def test_odd_rows(tx, n, f):  # noqa: F811
    X = np.random.default_rng(n).integers(0, 256, size=(13, n), dtype=np.uint8)
    for layout in ("ft", "tf"):
        for shift in (0, 1, 4):
            _check(tx, X, layout, f, shift)
