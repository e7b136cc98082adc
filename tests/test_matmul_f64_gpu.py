"""The FP64 products of the dense algebra in both forms (FP64 units; tensor cores with operands cut into seven
8-bit digits) against sums in 80/128-bit floating point.

Bound of the tensor-core form.  A row is rounded to 55 fractional bits below the power of two 2^E above its largest
entry, so an operand is off by at most 2^(E-56) <= 2^-55 max|a|; the left-out digit pairs i + j >= 7 are at most
sum over groups g >= 7 of (13 - g) 2^14 256^(12-g) / 2^110 < 2^-53.3 of 2^(EA+EB) <= 4 max|a| max|b| per real
product.  With four real products per complex one an entry is off by less than K 2^-48 max|a| max|b| (rows of the
left, columns of the right operand) and one rounding of the result.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.init()
    from paper_2111_11058_gb300 import build as B
    B.build()
    import paper_2111_11058_gb300 as pkg
    return pkg


def _op(X, op):
    return X if op == 0 else X.T if op == 1 else X.conj().T if op == 2 else X.conj()


def _longdot(A, B):
    """A B with long double sums (64 or 113 bits of mantissa, by machine)."""
    r = lambda x: x.astype(np.longdouble)  # noqa: E731
    ar, ai, br, bi = r(A.real), r(A.imag), r(B.real), r(B.imag)
    return ar @ br - ai @ bi, ar @ bi + ai @ br


def _err(C, ref):
    return np.maximum(np.abs(C.real - ref[0]), np.abs(C.imag - ref[1])).astype(np.float64)


def _mats(rng, M, N, K, opA, opB, grade):
    A = rng.standard_normal((M, K)) + 1j * rng.standard_normal((M, K))
    B = rng.standard_normal((K, N)) + 1j * rng.standard_normal((K, N))
    if grade:   # rows and columns of very different size, and entries below each row's last digit
        A *= 2.0 ** rng.integers(-40, 40, (M, 1)) * 2.0 ** rng.integers(-70, 1, (M, K))
        B *= 2.0 ** rng.integers(-40, 40, (1, N))
    inv = {0: lambda X: X, 1: lambda X: X.T, 2: lambda X: X.conj().T, 3: lambda X: X.conj()}
    return A, B, np.ascontiguousarray(inv[opA](A)), np.ascontiguousarray(inv[opB](B))


# tile edges (128 left rows, 32 right columns, 16 of K per stage, 64 of K per drain), both orientations, one and
# several CTAs per tile, every storage order and conjugation the solver uses
@pytest.mark.parametrize("M,N,K,opA,opB,grade", [
    (1, 1, 1, 0, 0, False), (5, 3, 7, 2, 0, False), (128, 32, 16, 0, 0, False), (129, 33, 17, 0, 2, False),
    (32, 128, 65, 0, 0, True), (127, 31, 63, 3, 1, False), (128, 128, 914, 3, 1, False), (45, 686, 640, 0, 2, True),
    (300, 100, 1100, 1, 0, False), (7, 686, 700, 0, 2, False), (257, 130, 128, 2, 3, True), (96, 1000, 2500, 0, 0, False),
])
def test_tensor_core_form(P, M, N, K, opA, opB, grade):
    rng = np.random.default_rng(M * 7919 + N * 104729 + K)
    A, B, sA, sB = _mats(rng, M, N, K, opA, opB, grade)
    ref = _longdot(A, B)
    C = P.matmul_f64(sA, sB, opA, opB, unit=2)
    mag = np.abs(A).max(1)[:, None] * np.abs(B).max(0)[None, :]
    e = _err(C, ref)
    assert (e <= K * 2.0 ** -48 * mag + 2.0 ** -52 * np.abs(C)).all()
    # no larger than the FP64 units' error, both relative to the 2-norms of the rows and columns
    # (at small K both are a few roundings of the result)
    nrm = np.linalg.norm(A, axis=1)[:, None] * np.linalg.norm(B, axis=0)[None, :]
    e1 = _err(P.matmul_f64(sA, sB, opA, opB, unit=1), ref)
    assert np.sqrt(np.mean((e / nrm) ** 2)) <= max(1.0 * np.sqrt(np.mean((e1 / nrm) ** 2)), 2.0 ** -53)


def test_accumulate_and_same_bits(P):
    rng = np.random.default_rng(5)
    A, B, _, _ = _mats(rng, 200, 90, 500, 0, 0, False)
    C0 = rng.standard_normal((200, 90)) + 1j * rng.standard_normal((200, 90))
    C = P.matmul_f64(A, B, unit=2)
    assert np.array_equal(P.matmul_f64(A, B, unit=2, C=C0), C0 + C)
    assert np.array_equal(P.matmul_f64(A, B, unit=2), C)
    # entries at the accumulators' limit: every digit at +-128
    x = np.full((128, 256), 1.0 - 2.0 ** -53)
    y = np.full((256, 64), -(1.0 - 2.0 ** -53)) * (1 + 1j)
    assert np.abs(P.matmul_f64(x, y, unit=2) - x @ y).max() <= 256 * 2.0 ** -48


def test_special_values(P):
    rng = np.random.default_rng(6)
    A, B, _, _ = _mats(rng, 40, 40, 40, 0, 0, False)
    A[3, 5] = np.nan
    B[7, 9] = np.inf
    A[10] = 0.0
    A[11] *= 1e-300
    B[:, 2] *= 1e-15
    C = P.matmul_f64(A, B, unit=2)
    assert np.isnan(C[3]).all() and np.isnan(C[:, 9].real).all()
    ok = np.ones((40, 40), bool)
    ok[3] = False
    ok[:, 9] = False
    assert np.isfinite(C[ok]).all() and (C[10][ok[10]] == 0).all()
    B[:, 9] = 0
    A[3] = 0
    e = _err(C, _longdot(A, B))
    assert e[ok].max() <= 1e-12
    assert e[11, 2] <= 1e-300 * 1e-15 * 1e-10 + 2.0 ** -1074   # a result below the smallest normal number


# the small kernels: entries few and many, k short and long, every storage order the solver uses (FP64 sums: the
# usual bound K u |a| |b| with u = 2^-53, four real products)
@pytest.mark.parametrize("M,N,K,opA,opB", [
    (7, 7, 686, 3, 1), (7, 300, 686, 0, 2), (7, 686, 300, 0, 0), (300, 7, 330, 2, 0), (300, 7, 290, 0, 0),
    (7, 7, 300, 2, 0), (300, 7, 7, 0, 0), (1, 1, 1, 0, 0), (45, 45, 31, 0, 1), (45, 47, 64, 1, 3), (2, 1025, 97, 0, 0),
    (129, 17, 63, 1, 0),
])
def test_small_products(P, M, N, K, opA, opB):
    rng = np.random.default_rng(M + 31 * N + 1009 * K)
    A, B, sA, sB = _mats(rng, M, N, K, opA, opB, False)
    C0 = rng.standard_normal((M, N)) + 1j * rng.standard_normal((M, N))
    ref = _longdot(A, B)
    C = P.matmul_f64(sA, sB, opA, opB, C=C0)
    mag = np.abs(A) @ np.abs(B) + np.abs(C0)
    assert (_err(C, (ref[0] + C0.real, ref[1] + C0.imag)) <= (2 * K + 8) * 2.0 ** -53 * mag).all()
