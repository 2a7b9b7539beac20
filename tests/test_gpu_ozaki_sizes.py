"""Ozaki contexts over slices and sizes against an FP64 context on the same inputs: every number of digits of the
O(r^5) kernel (3 to 6), each of its padded widths at an r that does not fill it, the double-float kernels (9 and 10
slices), and two K chunks of the GEMMs (r = 64), in a residual, a step and a gradient.

Tolerance: the operands keep 6 S bits, so the error goes as 2^-6S (2.9, 4.4 and 3.8 2^-6S of max |A| measured at r = 9 for
S = 4, 5 and 6, about ten times that at r = 48): 64 2^-6S, and 1e-12 as everywhere from 8 slices on.  Gradients go
through some ten passes: ten times that."""
import pytest

import acse_inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _tol(slices):
    return max(1e-12, 64.0 * 2.0 ** (-6 * slices))


def _rel(got, want):
    return max(float((g - w).abs().max()) for g, w in zip(got, want)) / max(float(w.abs().max()) for w in want)


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02550_gb300 import api as a
    return a


def _contexts(api, r, slices):
    h, V = I.make_integrals(r, 60 + r)
    D = I.random_pair_tensor_blocks(r, 61 + r, hermitian=1, scale=0.02)
    oz, ref = (api.ACSE(r, 4, 3, h, V, p, oz_slices=s) for p, s in (("ozaki", slices), ("fp64", 0)))
    return oz, ref, oz.to_blocks(D)


@pytest.mark.parametrize("r,slices", [(18, 4), (63, 4), (45, 5), (37, 6), (19, 7), (32, 7), (37, 8), (45, 8), (50, 8), (63, 8),
                                      (15, 9), (21, 9), (24, 9), (18, 10), (32, 10), (45, 10), (64, 10)])
def test_residual_and_step(api, r, slices):
    oz, ref, D = _contexts(api, r, slices)
    A, n2 = oz.residual(D)
    Aw, n2w = ref.residual(D)
    d, dw = (tuple(x.clone() for x in D) for _ in range(2))
    oz.step(d, 1.0)
    ref.step(dw, 1.0)
    assert _rel(A, Aw) <= _tol(slices)
    assert float(n2) == pytest.approx(float(n2w), rel=_tol(slices))
    assert _rel([a - b for a, b in zip(d, D)], [a - b for a, b in zip(dw, D)]) <= _tol(slices)
    oz.close()
    ref.close()


@pytest.mark.parametrize("r,slices,n", [(18, 8, 1), (27, 8, 1), (21, 7, 1), (18, 5, 1), (18, 10, 1), (32, 9, 1), (64, 8, 0)])
def test_gradient(api, r, slices, n):
    oz, ref, D = _contexts(api, r, slices)
    got, want = [], []
    for ctx, out in ((oz, got), (ref, want)):
        dh, dV, dD = ctx.backward([D], n, 1e-4, wE=1.0, wN=0.5)
        out.extend(([dh], [dV], dD))
    for g, w in zip(got, want):
        assert _rel(g, w) <= 10.0 * _tol(slices)
    oz.close()
    ref.close()
