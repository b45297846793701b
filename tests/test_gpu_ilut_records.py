"""The last-level block ILUT's stage buffers: records of every size beside one
another, and fill between a column whose record was fetched ahead and the current
one whose record is larger than both buffers together."""
import numpy as np
import pytest

import oracle
from gpu_helpers import compare_factor, cuda_ok, vb

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not cuda_ok(), reason="needs a CUDA GPU")]

STAGE_SMALL = 4096   # a record that fits in one buffer of every workspace shape
STAGE_LARGE = 12288  # a record that fits in no two


def _sparse(nb, deg, share, seed):
    """Random pattern, a share of the block rows with 26 to 32 scalars, the others
    with 1 to 3; dominant by rows."""
    rng = np.random.default_rng(seed)
    bsz = np.where(rng.random(nb) < share, rng.integers(26, 33, nb), rng.integers(1, 4, nb)).astype(np.int32)
    pat = np.eye(nb, dtype=bool)
    for i in range(nb):
        pat[i, rng.choice(nb, deg, replace=False)] = True
    pat |= pat.T
    bptr, bcol, voff, val = [0], [], [0], []
    for i in range(nb):
        for j in np.flatnonzero(pat[i]):
            b = rng.standard_normal((bsz[i], bsz[j])) * 0.1
            if i == j:
                b += np.eye(bsz[i]) * 0.2 * bsz[pat[i]].sum()
            bcol.append(j)
            val.append(b.ravel())
            voff.append(voff[-1] + b.size)
        bptr.append(len(bcol))
    return (bsz, np.array(bptr, np.int64), np.array(bcol, np.int32), np.array(voff, np.int64), np.concatenate(val)), pat


def _overtaken(bsz, pat, size):
    """Steps in which a column A may be fetched ahead, after which two columns B < D
    < A that the step's fill brought are eliminated: B's record read in place, D's
    brought into a buffer."""
    nb, n, u = len(bsz), bsz.astype(np.int64), []

    def record(k):
        nk, ucnt = n[k], len(u[k])
        return 64 + nk * 4 + nk * max(nk, 8) * size + 2 * nk * size + 12 * ucnt + nk * n[u[k]].sum() * size

    found = 0
    for i in range(nb):
        row = set(np.flatnonzero(pat[i]))
        todo, prev = sorted(j for j in row if j < i), []
        while todo:
            k = todo.pop(0)
            ahead = todo[0] if todo else None
            new = [j for j in u[k] if j not in row]
            row.update(new)
            todo = sorted(todo + [j for j in new if j < i])
            prev.append((k, ahead))
            if len(prev) >= 3:
                (_, a), (b, _), (d, _) = prev[-3:]
                if a is not None and d < a and record(b) > STAGE_LARGE and max(record(a), record(d)) <= STAGE_SMALL:
                    found += 1
        u.append(np.array(sorted(j for j in row if j > i), np.int64))
    return found


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_records_read_in_place_between_records_fetched_ahead(seed):
    m, pat = _sparse(160, 2, 0.15, seed)
    assert _overtaken(m[0], pat, 8) > 0 and _overtaken(m[0], pat, 4) > 0
    V = vb()
    A = V.vbarms_vbsr_from_blocks(*m)
    Po = oracle.Prec(oracle.VBMat(m[0], m[0], *m[1:]), 0, 0.0, -1)
    compare_factor(V.vbarms_factor(A, 0, 0.0, -1), Po)
    P = V.vbarms_factor(A, 0, 0.0, -1, precision="fp32")
    n = int(m[0].sum())
    # u = 2^-24: the no-drop factors of a dominant matrix, |dLU| <= 3 n u |L||U|
    for w in ("L", "U", "D"):
        g, o = P.export(0, w), Po.mat(0, w)
        assert np.array_equal(g["bcol"], o.bcol) and np.array_equal(g["voff"], o.voff)
        assert np.linalg.norm(g["val"] - o.val) <= 3 * n * 2.0 ** -24 * np.linalg.norm(o.val), w
    assert np.array_equal(P.vector(0, "piv"), Po.vec(0, "piv"))
