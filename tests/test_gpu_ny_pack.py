"""The packing and assembly of the NY operands at sizes between their cases, on the GPU.

The pack kernel takes whole r x r slabs, several a block, in groups of four columns where r^2 (or, for one order of the
indices, r) allows it: r = 9, 11 and 17 leave single elements, 10 groups that cross a row; 9, 11 and 17 leave slabs for a
last block that is not full, 17 takes fewer slabs a block than the smaller sizes.  Against the oracle, with the
tolerances of the residual parity test.
"""
import pytest

from tests.gpu_helpers import maxrel, to_np
from tests.test_gpu_ny import TOL, _oracle_residual, _problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def acse():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02550_gb300 import api
    return api


@pytest.mark.parametrize("r,precs", [(9, ("fp64", "bf16x3", "tf32x3")), (10, ("fp64", "bf16x3", "tf32x3")),
                                     (11, ("fp64", "bf16x3", "tf32x3")), (12, ("fp64", "bf16x3", "tf32x3")),
                                     (17, ("fp64", "bf16x3"))])
def test_ny_pack_against_oracle(acse, r, precs):
    p = _problem(r, r // 2, r // 3, 80 + r, "pair")
    want, _ = _oracle_residual(p)
    for prec in precs:
        ctx = acse.ACSE(r, p.n_alpha, p.n_beta, p.h, p.V, prec, recon="NY")
        A, _ = ctx.residual(ctx.to_blocks((p.Daa, p.Dab, p.Dbb)))
        assert maxrel(to_np(A), want) < TOL[prec], prec
