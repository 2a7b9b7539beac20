"""FP64 and Ozaki contexts on a D that is not pair-Hermitian: it is contracted as given, as the split precisions do, in
the form of Appendix B that has used the Hermiticity of K (`_G` below: the terms with the indices of K exchanged are
the transposes of the others).  Residual and step against that form from the oracle's parts (1e-12 normwise, as for
these paths everywhere); the asymmetry from large to small; the decision is made on the device for every D, also in a
replayed step."""
import numpy as np
import pytest

import acse_inputs as I
from oracle import acse_oracle as O
from tests.gpu_helpers import maxrel, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02550_gb300 import api as a
    return a


def _problem(r, na, nb, seed, asym=1.0):
    h, V = I.make_integrals(r, seed)
    D = I.random_pair_tensor_blocks(r, seed + 1, hermitian=1, scale=0.05)
    X = I.random_pair_tensor_blocks(r, seed + 2, hermitian=-1, scale=0.05 * asym)
    return I.Problem(f"asym_r{r}", r, na, nb, h, V, *(np.ascontiguousarray(d + x) for d, x in zip(D, X)))


def _G(W, D, N, s):
    """4 (Y - s Y^T) - 12 (B - B_{k<->l}) + 12 s (B^T - B^T_{i<->j}) in spin orbitals."""
    g = O.gamma(D, N)
    M, _ = O.cumulant_M(D, g)
    Y = np.einsum("ijpq,klpq->ijkl", D, W, optimize=True)
    B = O._three_body_V(W, M, g)
    X = B - B.transpose(0, 1, 3, 2)
    return 4.0 * (Y - s * Y.transpose(2, 3, 0, 1)) - 12.0 * X + 12.0 * s * X.transpose(2, 3, 0, 1)


def _want(p, D, eps):
    """A, ||A||^2 and D + eps U as blocks."""
    Ds = O.so_from_blocks(*D)
    A = _G(0.5 * O.reduced_hamiltonian(p.h, p.V, p.N), Ds, p.N, 1.0)
    U = 0.5 * _G(A, Ds, p.N, -1.0)
    return O.blocks_from_so(A), O.norm2(A), O.blocks_from_so(Ds + eps * U)


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
@pytest.mark.parametrize("r,na,nb", [(2, 1, 1), (7, 3, 2), (16, 5, 4), (21, 6, 5)])
def test_residual_and_step(api, prec, r, na, nb):
    p = _problem(r, na, nb, 800 + r)
    ctx = api.ACSE(r, na, nb, p.h, p.V, prec)
    D = ctx.to_blocks((p.Daa, p.Dab, p.Dbb))
    A, n2 = ctx.residual(D)
    want, n2w, Dw = _want(p, (p.Daa, p.Dab, p.Dbb), 1e-3)
    assert maxrel(to_np(A), want) <= 1e-12
    assert float(n2) == pytest.approx(n2w, rel=1e-12)
    ctx.step(D, 1e-3)
    assert maxrel(to_np(D), Dw) <= 1e-12
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
def test_small_asymmetry_is_contracted(api, prec):
    """The change of A with an asymmetry of 1e-9 of D is A's own: the difference of the two residuals, of relative
    size 1e-9, against the oracle's to 1e-3 of it (both carry 1e-13 of A or less)."""
    r, na, nb = 9, 3, 3
    p0, p1 = _problem(r, na, nb, 900, 0.0), _problem(r, na, nb, 900, 1e-9)
    ctx = api.ACSE(r, na, nb, p0.h, p0.V, prec)
    got, want = [], []
    for p in (p0, p1):
        D = (p.Daa, p.Dab, p.Dbb)
        got.append(to_np(ctx.residual(ctx.to_blocks(D))[0]))
        want.append(_want(p, D, 0.0)[0])
    dg, dw = [b - a for a, b in zip(*got)], [b - a for a, b in zip(*want)]
    assert maxrel(dg, dw) <= 1e-3
    ctx.close()


def test_replayed_step_decides_for_every_D(api):
    """Steps on the same buffers (captured on the second call, replayed from then on), the D in them Hermitian, not,
    Hermitian again: each equals the step of a fresh context bit by bit."""
    r, na, nb = 6, 3, 2
    sym, gen = _problem(r, na, nb, 950, 0.0), _problem(r, na, nb, 950, 1.0)
    stream = torch.cuda.Stream()
    from paper_2604_02550_gb300 import _lib
    with torch.cuda.stream(stream):
        ctx = api.ACSE(r, na, nb, sym.h, sym.V, "fp64", stream=stream)
        buf = ctx.zeros_blocks()
        s = torch.empty(3, dtype=torch.float64, device="cuda")
        for p in (sym, sym, sym, gen, sym, gen):
            D = ctx.to_blocks((p.Daa, p.Dab, p.Dbb))
            for dst, src in zip(buf, D):
                dst.copy_(src)
            _lib.acse_step(ctx.ctx, *buf, 1e-3, s[0:1], s[1:2], s[2:3])
            one = api.ACSE(r, na, nb, p.h, p.V, "fp64", stream=stream)
            one.step(D, 1e-3)
            stream.synchronize()
            for a, b in zip(buf, D):
                assert torch.equal(a, b)
            one.close()
        ctx.close()


def test_batch_fp64(api):
    """FP64 batch instances with and without a Hermitian D in one grouped launch."""
    from paper_2604_02550_gb300 import _lib
    probs = [_problem(5, 2, 2, 970, 0.0), _problem(6, 3, 2, 971, 1.0), _problem(4, 2, 1, 972, 1.0)]
    b = _lib.acse_batch_create(probs, "fp64")
    Ds = [tuple(torch.as_tensor(x, device="cuda") for x in (p.Daa, p.Dab, p.Dbb)) for p in probs]
    for i, D in enumerate(Ds):
        _lib.acse_batch_set_D(b, i, *D, 1e-3)
    _lib.acse_batch_run(b, len(probs), 1, stop_rule=False)
    for i, p in enumerate(probs):
        out = tuple(torch.empty_like(x) for x in Ds[i])
        _lib.acse_batch_get_D(b, i, *out)
        Dw = _want(p, (p.Daa, p.Dab, p.Dbb), 1e-3)[2]
        assert maxrel(to_np(out), Dw) <= 1e-12
    _lib.acse_batch_destroy(b)
