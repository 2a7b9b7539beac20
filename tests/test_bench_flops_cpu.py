"""The operation counts that bench.py reports rates against are those of the products the library multiplies (no device
needed): the lists of a residual and of an update pass (acse_gemm_list_f64), written out."""
import pytest

import bench


@pytest.mark.parametrize("r", [2, 3, 8, 31, 48, 64])
def test_symmetrised_pass(r):
    S, A, R2, P = r * (r + 1), r * (r - 1), r * r, r * (r - 1) // 2
    common = [(R2, R2, R2)] * 3 + [(P, P, P)] * 4            # flip, X_ab, Y_ab; X and Y of aa and bb
    residual = [(S, S, S), (A, A, A)] + common
    update = [(A, S, S), (S, A, A)] + common
    want = sum(2 * m * n * k for m, n, k in residual + update)
    assert 2 * bench.flops_per_pass(r, symmetrised=True) == want
    assert bench.flops_per_pass(r, packed=True, symmetrised=True) == bench.flops_per_pass(r, symmetrised=True)
    assert bench.flops_per_pass(r, symmetrised=True) <= bench.flops_per_pass(r, packed=True)


def test_moduli_of_the_default_workload():
    assert bench.oz_moduli_count(8, 48 * 49) == 17
    assert bench.flops_per_pass(48) == 32 * 48 ** 6
