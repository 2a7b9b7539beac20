"""The particle-hole products on symmetrised pairs and the packed same-spin pairs of the FP64 and Ozaki paths
against the oracle, at the sizes where tiles and pair numberings can go wrong: r = 2 (one pair a < b), odd r,
r = 16 (the tensor-core transformation by 1D; whole 256-wide Ozaki tiles for r^2 but not for r(r+1)), and r = 27
(the 32 x 32 tiles of the FP64 GEMM).  Residual (s = +1) and step (s = -1): 1e-12 normwise, as for these
paths everywhere; gradients against complex-step derivatives of the oracle: 1e-9."""
import numpy as np
import pytest

import acse_inputs as I
from oracle import acse_oracle as O
from tests.gpu_helpers import maxrel, oracle_residual_blocks, oracle_step_blocks, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_02550_gb300 import api as a
    return a


def _problem(r, na, nb, seed):
    h, V = I.make_integrals(r, seed)
    D = I.random_pair_tensor_blocks(r, seed + 1, hermitian=1, scale=0.05)
    return I.Problem(f"rand_r{r}", r, na, nb, h, V, *D)


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
@pytest.mark.parametrize("r,na,nb", [(2, 1, 1), (7, 3, 2), (16, 5, 4), (21, 6, 5), (27, 7, 6)])
def test_residual_and_step(api, prec, r, na, nb):
    p = _problem(r, na, nb, 500 + r)
    ctx = api.ACSE(r, na, nb, p.h, p.V, prec)
    D = ctx.to_blocks((p.Daa, p.Dab, p.Dbb))
    A, n2 = ctx.residual(D)
    want, n2w = oracle_residual_blocks(p, (p.Daa, p.Dab, p.Dbb))
    assert maxrel(to_np(A), want) <= 1e-12
    assert float(n2) == pytest.approx(n2w, rel=1e-12)
    if r <= 21:
        E, _, _ = ctx.step(D, 1e-3)
        Dw, Ew, _ = oracle_step_blocks(p, (p.Daa, p.Dab, p.Dbb), 1e-3)
        assert maxrel(to_np(D), Dw) <= 1e-12
        assert float(E) == pytest.approx(Ew, abs=1e-10 * max(1.0, abs(Ew)))
    ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "ozaki"])
@pytest.mark.parametrize("r", [2, 5, 16])
def test_gradient(api, prec, r):
    na, nb = (1, 1) if r == 2 else (3, 2)
    h, V = I.make_integrals(r, 600 + r)
    D0 = I.random_pair_tensor_blocks(r, 601 + r, hermitian=1, scale=0.02)
    eps, n, wE, wN = 1e-4, 1, 1.0, 0.5
    ctx = api.ACSE(r, na, nb, h, V, prec)
    dh, dV, dD = ctx.backward([ctx.to_blocks(D0)], n, eps, wE, wN)
    dh, dV, dD = dh.cpu().numpy(), dV.cpu().numpy(), to_np(dD)
    ctx.close()
    rng = np.random.default_rng(r)
    for k in range(2):
        eh = rng.normal(size=(r, r))
        eh = eh + eh.T
        eV = rng.normal(size=(r,) * 4)
        for perm in ((1, 0, 2, 3), (0, 1, 3, 2), (2, 3, 0, 1)):
            eV = eV + eV.transpose(perm)
        eD = I.random_pair_tensor_blocks(r, 700 + k, hermitian=1, scale=1.0)
        want = O.complex_step_dir(h, V, na + nb, O.so_from_blocks(*D0), eps, n, eh, eV, O.so_from_blocks(*eD), wE, wN)
        got = np.sum(dh * eh) + np.sum(dV * eV) + sum(np.sum(a * b) for a, b in zip(dD, eD))
        assert got == pytest.approx(want, rel=1e-9, abs=1e-9 * abs(want))
