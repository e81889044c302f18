"""Single kernels at the sizes where their vector paths, tiles and splits meet
their edges, against exact integers or the oracle."""
import numpy as np
import pytest

import oracle
from paper_2101_01025_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2101_01025_gb300 as aat
    return aat


@pytest.mark.parametrize("off", [0, 1, 2, 3])
@pytest.mark.parametrize("n,pad", [(1, 0), (2, 1), (3, 0), (4, 4), (5, 2), (33, 3), (64, 0), (257, 1)])
def test_zero_upper_clears_the_strict_upper_triangle_only(lib, n, pad, off):
    """Rows that start at every offset modulo 16 bytes; entries outside the
    n x n result and the lower triangle keep their values."""
    import torch
    p, k = 65521, 7
    A = synth.residues(11 + n, (n, k), p)
    ldc = n + pad
    buf = torch.full((off + n * ldc + 5,), -7, dtype=torch.int32, device="cuda")
    C = torch.as_strided(buf, (n, n), (ldc, 1), off)
    lib.aat_modp(torch.from_numpy(A).cuda(), p, C=C, flags=lib.AAT_ZERO_UPPER, levels=0)
    want = np.full(buf.shape, -7, dtype=np.int32)
    ref = oracle.aat_modp_low(A, p).astype(np.int64)
    for r in range(n):
        want[off + r * ldc:off + r * ldc + n] = 0
        want[off + r * ldc:off + r * ldc + r + 1] = ref[r, :r + 1]
    assert np.array_equal(buf.cpu().numpy(), want)
