"""Rows of the compressed cores are orthonormal to the Jacobi kernel's rotation
threshold, 1e-13 sqrt(rows): at most twice that, plus 200 roundings of 2^-47.  Middle
bonds of q rows (blocks of odd and even size, one CTA to a whole cluster), and bonds
that double up to r and drop to b (every plan of Q's formation).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as g
    g.build()
    from paper_2205_11990_gb300 import vpmps
    c = vpmps.Context()
    yield c
    c.close()


def middle(q):
    half = max(2, int(np.ceil(np.log2(q))))
    bonds = [min(2 ** k, q) for k in range(half + 1)]
    return bonds + bonds[-2::-1]


def drop(r, b):
    bonds = [1]
    while bonds[-1] < r:
        bonds.append(min(2 * bonds[-1], r))
    bonds.append(b)
    while bonds[-1] > 1:
        bonds.append((bonds[-1] + 1) // 2)
    return bonds


CASES = [middle(q) for q in (2, 5, 13, 24, 31, 49, 96, 121, 193, 255, 448)] + \
        [drop(r, b) for r, b in ((15, 3), (33, 7), (65, 2), (129, 130), (257, 31), (513, 5), (1025, 2), (2049, 3))]


@pytest.mark.parametrize("bonds", CASES, ids=lambda b: str(max(b)))
@pytest.mark.parametrize("grade", [0.0, 9.0])
def test_rows_orthonormal(ctx, bonds, grade):
    rng = np.random.default_rng(max(bonds) + int(grade))
    cores = [rng.standard_normal((bonds[k], 2, bonds[k + 1])) / np.sqrt(2 * bonds[k]) for k in range(len(bonds) - 1)]
    k = int(np.argmax(bonds))
    cores[k - 1] = cores[k - 1] * np.logspace(0, -grade, bonds[k])
    m = ctx.mps_from_cores(cores)
    ctx.compress(m, 1 << 20, 1e-12)
    for c in m.cores()[1:]:
        a = c.reshape(c.shape[0], -1)
        assert np.max(np.abs(a @ a.T - np.eye(a.shape[0]))) <= 2e-13 * np.sqrt(max(a.shape)) + 200 * 2.0 ** -47
