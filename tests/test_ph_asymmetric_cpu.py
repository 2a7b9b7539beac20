"""The particle-hole products on symmetrised pairs for a D that is not pair-Hermitian (csrc/acse_ph.cu), emulated in
numpy, no device needed: M+ gets 2P more rows antisymmetric in (i,l), M- 2S more symmetric ones, and the second flip
is a product of its own on the first flip of W with both index pairs of M exchanged.  V5 and both flips must equal the
full products.  Tolerance as in test_ph_pairs_cpu.py."""
import numpy as np
import pytest

import acse_inputs as I
from tests.test_ph_pairs_cpu import _close, _flip, _pack, _ph, _pk, _ps


def _pack_general(T, r):
    """(plus, minus) of k_ph_pack for M: 2S rows even in (i,l) then 2P odd ones; 2P odd rows then 2S even ones."""
    x = _ph(T).reshape(2, r, r, 2, r, r)
    S, P = r * (r + 1) // 2, r * (r - 1) // 2
    plus, minus = np.zeros((2 * r * r, 2 * S)), np.zeros((2 * r * r, 2 * P))
    for K in range(2):
        for Q in range(2):
            for k in range(r):
                for q in range(k, r):
                    for p in range(r):
                        for t in range(p, r):
                            a, b = x[K, k, q, Q, p, t], x[K, k, q, Q, t, p]
                            a2, b2 = x[K, q, k, Q, p, t], x[K, q, k, Q, t, p]
                            e, ep, o, op = 0.5 * (a + a2), 0.5 * (b + b2), 0.5 * (a - a2), 0.5 * (b - b2)
                            cs = Q * S + _ps(r, p, t)
                            plus[K * S + _ps(r, k, q), cs] = e + ep if p < t else e
                            if k < q:
                                plus[2 * S + K * P + _pk(r, k, q), cs] = o + op if p < t else o
                            if p < t:
                                ca = Q * P + _pk(r, p, t)
                                minus[2 * P + K * S + _ps(r, k, q), ca] = e - ep
                                if k < q:
                                    minus[K * P + _pk(r, k, q), ca] = o - op
    return plus, minus


def _expand_general(V1, V2, r, s):
    S, P = r * (r + 1) // 2, r * (r - 1) // 2
    out = np.zeros((2, r, r, 2, r, r))
    for K in range(2):
        for k in range(r):
            for q in range(k, r):
                rowS, rowA = K * S + _ps(r, k, q), (K * P + _pk(r, k, q)) if k < q else -1
                r1, r2 = (rowS, rowA) if s > 0 else (rowA, rowS)
                for Ib in range(2):
                    for i in range(r):
                        for l in range(r):
                            lo, hi, sg = min(i, l), max(i, l), (i < l) - (i > l)
                            xx = yy = 0.0
                            if r1 >= 0:
                                xx = V1[r1, Ib * S + _ps(r, lo, hi)]
                                if sg:
                                    xx += sg * V1[r1, 2 * S + Ib * P + _pk(r, lo, hi)]
                            if r2 >= 0:
                                yy = V2[r2, 2 * P + Ib * S + _ps(r, lo, hi)]
                                if sg:
                                    yy += sg * V2[r2, Ib * P + _pk(r, lo, hi)]
                            out[K, k, q, Ib, i, l] = xx + yy
                            if k < q:
                                out[K, q, k, Ib, i, l] = xx - yy if s > 0 else yy - xx
    return out.reshape(2 * r * r, 2 * r * r)


@pytest.mark.parametrize("hermitian", [0, 1])
@pytest.mark.parametrize("s", [1, -1])
@pytest.mark.parametrize("r", [2, 3, 5, 6])
def test_products_of_a_general_M(r, s, hermitian):
    M = I.random_pair_tensor_blocks(r, 110 + r, hermitian=hermitian)
    W = I.random_pair_tensor_blocks(r, 120 + r, hermitian=s)
    Mp, Mm = _pack_general(M, r)
    Wp, Wm = _pack(W, r, 0.5, s > 0)
    _close(_expand_general(Wp @ Mp.T, Wm @ Mm.T, r, s), _ph(W) @ _ph(M).T)
    R2 = r * r
    Wf2 = W[1].transpose(1, 2, 0, 3).reshape(R2, R2)
    Mf2 = M[1].transpose(1, 2, 0, 3).reshape(R2, R2)
    flip2 = M[1].transpose(2, 1, 3, 0).reshape(R2, R2)   # [(k,q)][(p,t)] = M_ab[t][q][k][p]
    U = _flip(W) @ flip2.T
    _close(s * U.reshape((r,) * 4).transpose(1, 0, 3, 2).reshape(R2, R2), Wf2 @ Mf2.T)
    if hermitian:
        _close(flip2, _flip(M))
