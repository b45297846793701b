"""The last level's triangular sweeps (vbarms_apply with no reduction level) at
the sizes where they change path: block rows of 1-8, 9-16, 17-32 and more
scalars, rows of more than 32 and of more than 64 blocks, rows whose values do
not fit on chip, dependencies of more than 8 columns; FP64 and mixed factors,
the fixed-scratch solve beside the plain one, and non-finite input."""
import numpy as np
import pytest

import oracle
from gpu_helpers import cuda_ok, torch, vb

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

# (block sizes from, to, block rows, couplings on each side of a row)
CASES = {
    "small": (1, 8, 70, 9),
    "mid": (7, 16, 40, 6),
    "large": (12, 32, 24, 5),
    "huge": (30, 40, 9, 3),
    "many_blocks": (1, 3, 160, 75),
    "off_chip": (8, 16, 36, 18),
    "mixed": (1, 34, 40, 8),
}


def _matrix(lo, hi, nb, band, seed, halves=False):
    rng = np.random.default_rng(seed)
    bsz = rng.integers(lo, hi + 1, nb).astype(np.int32)
    bptr, bcol, voff, val = [0], [], [0], []
    for i in range(nb):
        for j in range(max(0, i - band), min(nb, i + band + 1)):
            if halves and (i < nb // 2) != (j < nb // 2):
                continue
            b = rng.standard_normal((bsz[i], bsz[j])) * 0.1
            if i == j:  # dominant by rows, interchanges in some blocks
                b = b + np.eye(bsz[i]) * (0.2 * bsz.max() * (2 * band + 1))
                if i % 3 == 0:
                    b = b[::-1]
            bcol.append(j)
            val.append(np.ascontiguousarray(b).ravel())
            voff.append(voff[-1] + b.size)
        bptr.append(len(bcol))
    return (bsz, np.array(bptr, np.int64), np.array(bcol, np.int32), np.array(voff, np.int64), np.concatenate(val))


def _apply(V, P, x):
    xd = torch.from_numpy(x).cuda()
    y, ys = torch.zeros_like(xd), torch.zeros_like(xd)
    V.vbarms_apply(P, xd, y)
    V.vbarms_apply_static(P, xd, ys)
    y, ys = y.cpu().numpy(), ys.cpu().numpy()
    assert np.array_equal(y, ys, equal_nan=True), "the fixed-scratch solve differs"
    return y


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name", CASES)
def test_sweeps_match_oracle(name, precision):
    V = vb()
    m = _matrix(*CASES[name], seed=sorted(CASES).index(name))
    n = int(m[0].sum())
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision=precision)
    Po = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 0, 0.0, -1)
    x = np.random.default_rng(7).standard_normal(n)
    y, yo = _apply(V, P, x), Po.apply(x)
    # FP64: the solve's parity bound.  FP32 factor and solve: 3 n u |L||U| each
    # way, |A^-1||L||U| <= 3 on these dominant matrices, u = 2^-24
    tol = 1e-12 if precision == "fp64" else 9 * n * 2.0 ** -24
    assert np.linalg.norm(y - yo) <= tol * np.linalg.norm(yo)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bits", [0xFFFFFFFFFFFFFFFF, 0x7FF0000000000000])
def test_sweeps_non_finite(precision, bits):
    """A NaN of all ones (the word that marks an unpublished unknown) and an
    infinity reach what depends on them and nothing else, and nothing waits."""
    V = vb()
    m = _matrix(1, 20, 40, 6, seed=3, halves=True)
    n = int(m[0].sum())
    half = int(m[0][:20].sum())
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision=precision, wait_limit=2_000_000_000)
    x = np.random.default_rng(8).standard_normal(n)
    clean = _apply(V, P, x)
    x[half // 2] = np.array([bits], np.uint64).view(np.float64)[0]
    y = _apply(V, P, x)
    assert np.array_equal(y[half:], clean[half:])
    assert not np.isfinite(y[:half]).all()
    # the next application of the same handle starts clean
    x[half // 2] = 0.0
    assert np.isfinite(_apply(V, P, x)).all()


def test_sweeps_zero_and_tiny_right_hand_sides():
    """Right-hand sides outside the range of the reciprocal divisions and the
    FP32 subtraction take the general operations: scaling x by a power of two
    scales every unknown of the FP64 solve exactly."""
    V = vb()
    m = _matrix(1, 18, 50, 7, seed=5)
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision="fp64")
    P32 = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1, precision="fp32")
    x = np.random.default_rng(9).standard_normal(int(m[0].sum()))
    y, y32 = _apply(V, P, x), _apply(V, P32, x)
    for e in (-400, 400):
        assert np.array_equal(_apply(V, P, np.ldexp(x, e)), np.ldexp(y, e))
    for e in (-60, 60):
        assert np.array_equal(_apply(V, P32, np.ldexp(x, e)), np.ldexp(y32, e))
    assert not _apply(V, P, 0.0 * x).any() and not _apply(V, P32, 0.0 * x).any()


@pytest.mark.parametrize("nb", [1, 2, 31, 32, 33, 64, 257])
def test_level_orders_of_few_rows(nb):
    """The order that the sweeps take their rows in is computed 32 rows to a
    warp: whole and partial groups, chains inside one group."""
    V = vb()
    m = _matrix(1, 3, nb, 2, seed=nb)
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 0, 0.0, -1)
    x = np.random.default_rng(nb).standard_normal(int(m[0].sum()))
    yo = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 0, 0.0, -1).apply(x)
    assert np.linalg.norm(_apply(V, P, x) - yo) <= 1e-12 * np.linalg.norm(yo)


@pytest.mark.parametrize("name", CASES)
def test_one_reduction_level_matches_oracle(name):
    """The reduction level's pivot solves (a thread or a warp per block, by size)
    and the products with G and W."""
    V = vb()
    m = _matrix(*CASES[name], seed=20 + sorted(CASES).index(name))
    x = np.random.default_rng(11).standard_normal(int(m[0].sum()))
    P = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 1, 0.0, -1)
    yo = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 1, 0.0, -1).apply(x)
    assert np.linalg.norm(_apply(V, P, x) - yo) <= 1e-12 * np.linalg.norm(yo)
    P32 = V.vbarms_factor(V.vbarms_vbsr_from_blocks(*m), 1, 0.0, -1, precision="fp32")
    assert np.linalg.norm(_apply(V, P32, x) - yo) <= 9 * len(x) * 2.0 ** -24 * np.linalg.norm(yo)
