"""The reverse sweep is linear in its weights at any scale: the gradient at (c wE, c wN), c a power of two, is c times
the gradient at (wE, wN), bit for bit (FP64 sums and fixed point below per-row powers of two both scale exactly),
for FP64 and Ozaki contexts, with the digit kernel (8 slices) and without it (10), ragged and whole r."""
import pytest

import acse_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,slices", [("fp64", 0), ("ozaki", 8), ("ozaki", 10)])
@pytest.mark.parametrize("r", [5, 16, 21])
def test_gradient_scales_with_its_weights(r, prec, slices):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02550_gb300 import api
    h, V = I.make_integrals(r, 40 + r)
    D0 = I.random_pair_tensor_blocks(r, 41 + r, hermitian=1, scale=0.02)
    ctx = api.ACSE(r, 3, 2, h, V, prec, oz_slices=slices)
    ck = [ctx.to_blocks(D0)]

    def grad(c):
        dh, dV, dD = ctx.backward(ck, 1, 1e-3, wE=c, wN=0.5 * c)
        torch.cuda.synchronize()
        return (dh, dV, *dD)

    one = grad(1.0)
    for c in (2.0 ** -80, 2.0 ** -200, 2.0 ** 150):
        for g, g1 in zip(grad(c), one):
            assert torch.equal(g, c * g1)
    ctx.close()
