"""The identities behind the particle-hole product on symmetrised pairs (csrc/acse_ph.cu) and its reversal
(csrc/acse_adjoint.cu), emulated in numpy on random tensors of the right symmetries, no device needed:

* V5[(k,q)][(i,l)] = sum W^{kp}_{qt} M^{ip}_{lt} over both spins of (p,t) equals V1 + V2 from the products over
  p <= t and p < t, for a pair-Hermitian and a pair-anti-Hermitian W, and the second flip is the image of the first;
* transforming V5 by 1D equals the product of the transformed W with M;
* the cotangent of M_ph from v1, v2 equals the direct one projected onto M's symmetry class.
Tolerance: the sums have at most 2 r^2 + r terms of order one, rounding stays below 1e-13 of the largest entry."""
import numpy as np
import pytest

import acse_inputs as I

TOL = 1e-13


def _ps(r, a, b):
    return a * r - a * (a - 1) // 2 + (b - a)


def _pk(r, a, b):
    return a * r - a * (a + 1) // 2 + (b - a - 1)


def _ph(T):
    """T[(K,k,q)][(P,p,t)] of a pair tensor's blocks (aa, ab, bb)."""
    aa, ab, bb = T
    r = aa.shape[0]
    R2 = r * r
    out = np.empty((2, R2, 2, R2))
    out[0, :, 0] = aa.transpose(0, 2, 1, 3).reshape(R2, R2)
    out[0, :, 1] = ab.transpose(0, 2, 1, 3).reshape(R2, R2)
    out[1, :, 0] = ab.transpose(1, 3, 0, 2).reshape(R2, R2)
    out[1, :, 1] = bb.transpose(0, 2, 1, 3).reshape(R2, R2)
    return out.reshape(2 * R2, 2 * R2)


def _flip(T):
    r = T[1].shape[0]
    return T[1].transpose(0, 3, 1, 2).reshape(r * r, r * r)


def _pack(T, r, f, plus_s):
    """(plus, minus) of k_ph_pack: rows over k <= q (plus_s) or k < q, the other way round for minus."""
    x = _ph(T).reshape(2, r, r, 2, r, r)
    S, P = r * (r + 1) // 2, r * (r - 1) // 2
    plus = np.zeros((2, S if plus_s else P, 2, S))
    minus = np.zeros((2, P if plus_s else S, 2, P))
    for k in range(r):
        for q in range(k, r):
            for p in range(r):
                for t in range(p, r):
                    a, b = x[:, k, q, :, p, t], x[:, k, q, :, t, p]
                    if plus_s or k < q:
                        plus[:, _ps(r, k, q) if plus_s else _pk(r, k, q), :, _ps(r, p, t)] = f * (a + b) if p < t else a
                    if p < t and (k < q or not plus_s):
                        minus[:, _pk(r, k, q) if plus_s else _ps(r, k, q), :, _pk(r, p, t)] = f * (a - b)
    return plus.reshape(plus.shape[0] * plus.shape[1], -1), minus.reshape(minus.shape[0] * minus.shape[1], -1)


def _expand(V1, V2, r, s):
    S, P = r * (r + 1) // 2, r * (r - 1) // 2
    V1, V2 = V1.reshape(2, -1, 2, S), V2.reshape(2, -1, 2, P)
    out = np.zeros((2, r, r, 2, r, r))
    for k in range(r):
        for q in range(r):
            lo, hi = min(k, q), max(k, q)
            sw = 1 if k < q else -1 if k > q else 0
            for i in range(r):
                for l in range(r):
                    sg = 1 if i < l else -1 if i > l else 0
                    v = 0.0
                    if s > 0:
                        v = v + V1[:, _ps(r, lo, hi), :, _ps(r, min(i, l), max(i, l))]
                        if sw and sg:
                            v = v + sw * sg * V2[:, _pk(r, lo, hi), :, _pk(r, min(i, l), max(i, l))]
                    else:
                        if sw:
                            v = v + sw * V1[:, _pk(r, lo, hi), :, _ps(r, min(i, l), max(i, l))]
                        if sg:
                            v = v + sg * V2[:, _ps(r, lo, hi), :, _pk(r, min(i, l), max(i, l))]
                    out[:, k, q, :, i, l] = v
    return out.reshape(2 * r * r, 2 * r * r)


def _close(a, b):
    assert np.abs(a - b).max() <= TOL * max(1.0, np.abs(b).max())


@pytest.mark.parametrize("s", [1, -1])
@pytest.mark.parametrize("r", [2, 3, 5, 6])
def test_products_on_pairs(r, s):
    M = I.random_pair_tensor_blocks(r, 10 + r, hermitian=1)
    W = I.random_pair_tensor_blocks(r, 20 + r, hermitian=s)
    want = _ph(W) @ _ph(M).T
    Mp, Mm = _pack(M, r, 1.0, True)
    Wp, Wm = _pack(W, r, 0.5, s > 0)
    got = _expand(Wp @ Mp.T, Wm @ Mm.T, r, s)
    _close(got, want)
    # the flips: V5f2 = s V5f1 with both index pairs exchanged
    f1 = _flip(W) @ _flip(M).T
    Wf2 = W[1].transpose(1, 2, 0, 3).reshape(r * r, r * r)   # [(k,q)][(p,t)] = W_ab[p][k][q][t]
    Mf2 = M[1].transpose(1, 2, 0, 3).reshape(r * r, r * r)
    f2 = Wf2 @ Mf2.T
    _close(s * f1.reshape((r,) * 4).transpose(1, 0, 3, 2).reshape(r * r, r * r), f2)
    # 1D after the product or before it
    g = np.random.default_rng(r).normal(size=(r, r))
    after = np.einsum("jq,kqx->kjx", g, want[:r * r].reshape(r, r, -1)).reshape(r * r, -1)
    Z = np.einsum("jq,kqx->kjx", g, _ph(W)[:r * r].reshape(r, r, -1)).reshape(r * r, -1)
    _close(after, Z @ _ph(M).T)


@pytest.mark.parametrize("s", [1, -1])
@pytest.mark.parametrize("r", [2, 3, 5])
def test_reversed_products_on_pairs(r, s):
    W = I.random_pair_tensor_blocks(r, 30 + r, hermitian=s)
    S, P, R2 = r * (r + 1) // 2, r * (r - 1) // 2, r * r
    V = np.random.default_rng(40 + r).normal(size=(2 * R2, 2 * R2))
    Mb = (V.T @ _ph(W)).reshape(2, r, r, 2, r, r)                       # cotangent of M_ph[(I,i,l)][(P,p,t)]
    want = 0.5 * (Mb + Mb.transpose(0, 2, 1, 3, 5, 4))                  # its part invariant under both exchanges
    x = V.reshape(2, r, r, 2, r, r)
    Wp, Wm = _pack(W, r, 0.5, s > 0)
    n1, n2 = (S, P) if s > 0 else (P, S)
    v1, v2 = np.zeros((2, S, 2, n1)), np.zeros((2, P, 2, n2))
    for k in range(r):
        for q in range(k, r):
            for i in range(r):
                for l in range(i, r):
                    a, b, c, d = x[:, k, q, :, i, l], x[:, k, q, :, l, i], x[:, q, k, :, i, l], x[:, q, k, :, l, i]
                    if k == q:
                        c = d = 0.0 * a
                    if s > 0 or k < q:
                        v1[:, _ps(r, i, l), :, _ps(r, k, q) if s > 0 else _pk(r, k, q)] = 0.5 * (a + b + s * (c + d)).T
                    if i < l and (s < 0 or k < q):
                        v2[:, _pk(r, i, l), :, _pk(r, k, q) if s > 0 else _ps(r, k, q)] = 0.5 * (a - b - s * (c - d)).T
    v1, v2 = v1.reshape(2 * S, -1), v2.reshape(2 * P, -1)
    B1, B2 = (Wp, Wm) if s > 0 else (Wm, Wp)                            # K-major: W+ and W- transposed
    mp, mm = (v1 @ B1.T).reshape(2, S, 2, S), (v2 @ B2.T).reshape(2, P, 2, P)
    got = np.zeros_like(want)
    for i in range(r):
        for l in range(r):
            for p in range(r):
                for t in range(r):
                    v = mp[:, _ps(r, min(i, l), max(i, l)), :, _ps(r, min(p, t), max(p, t))].copy()
                    if i != l and p != t:
                        sg = 1 if (i < l) == (p < t) else -1
                        v += sg * mm[:, _pk(r, min(i, l), max(i, l)), :, _pk(r, min(p, t), max(p, t))]
                    got[:, i, l, :, p, t] = v
    _close(got, want)
