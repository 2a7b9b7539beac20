"""Split-precision operand packs and GEMM epilogue where r is odd or even but no multiple of four, on the GPU.

Operand rows are written in groups of four K positions that cross the ends of the rows, slabs and packed pairs they come
from; GEMM rows that start on no 16-byte boundary, or end within 32 columns, leave the CTA-pair kernel through shared
memory.  The one-SM kernel stores such rows directly, so both must give the same bits; the operands are checked
against the oracle, with the tolerances of the mixed-precision residual test.
"""
import numpy as np
import pytest

from tests.gpu_helpers import maxrel, oracle_residual_blocks
from tests.test_gpu_mixed import TOL
from tests.test_gpu_pair import _problem, _residual

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def acse():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02550_gb300 import api
    return api


@pytest.mark.parametrize("prec", ["bf16x3", "tf32", "tf32x3"])
@pytest.mark.parametrize("r", [18, 19, 22])
def test_ragged_sizes(acse, prec, r):
    p = _problem(r, r // 2, r // 3, 400 + r)
    A2, n2 = _residual(acse, p, prec, 2)
    A1, n1 = _residual(acse, p, prec, 1)
    assert all(np.array_equal(a, b) for a, b in zip(A2, A1)) and n2 == n1
    want, _ = oracle_residual_blocks(p, (p.Daa, p.Dab, p.Dbb))
    assert maxrel(A2, want) < TOL[prec]


def test_ragged_odd_large(acse):
    p = _problem(31, 9, 8, 431)   # several K blocks of packed pairs; the last slabs of a block row are fewer
    A2, n2 = _residual(acse, p, "bf16x3", 2)
    A1, n1 = _residual(acse, p, "bf16x3", 1)
    assert all(np.array_equal(a, b) for a, b in zip(A2, A1)) and n2 == n1
    want, _ = oracle_residual_blocks(p, (p.Daa, p.Dab, p.Dbb))
    assert maxrel(A2, want) < TOL["bf16x3"]
