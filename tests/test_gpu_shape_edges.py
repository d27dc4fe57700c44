"""Sizes at which a kernel changes its form: batch widths around the lane
groups and packs, Krylov vectors around what one block and one grid hold in
registers, slice widths around the row kernels' classes, sort windows around
the size that is ranked in shared memory, exact dots whose digits do not fit
one window.  Integer, set and rounded-once results must equal the CPU
oracle's; solutions agree with it to 1e-9 relative L2: both residuals are at
most 1e-10 |b| and the condition numbers stay below 5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_17517_gb300 as G  # noqa: E402
from oracle import airg as O  # noqa: E402
from synthetic import workload  # noqa: E402
from tests.test_gpu_parity import Case, _check_setup, _check_solve  # noqa: E402
from tests.test_gpu_sparse_products import random_matrix  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.build()
    G.lib()


class General:
    """GPU and oracle hierarchies of a general matrix."""

    def __init__(self, A, **opts):
        self.A = A
        self.h = G.airg_setup(torch.tensor(A.rowptr, device="cuda"),
                              torch.tensor(A.col.astype(np.int32), device="cuda"),
                              torch.tensor(A.val, device="cuda"), G.airg_options_default(**opts))
        self.Ho = O.setup(A, O.Options(**{k: v for k, v in opts.items() if k != "precision"}))

    def check_solve(self, b):
        x, info = G.airg_solve(self.h, torch.tensor(b, device="cuda"), rtol=1e-10)
        assert info.converged
        X = x.cpu().numpy().reshape(-1, self.A.n_rows)
        for q, bq in enumerate(b.reshape(-1, self.A.n_rows)):
            assert np.linalg.norm(bq - O.spmv(self.A, X[q])) <= 1e-10 * np.linalg.norm(bq) * (1 + 1e-6)
            xo, _ = O.solve(self.Ho, self.A, bq, rtol=1e-10)
            assert np.linalg.norm(X[q] - xo) <= 1e-9 * np.linalg.norm(xo)


@pytest.mark.parametrize("prec", [G.AIRG_FP64, G.AIRG_MIXED_FP32])
def test_batch_widths(prec):
    """One lane, odd widths without packs, whole and partly filled groups of
    16-byte packs, more than 32 and 64 lanes."""
    c = General(random_matrix(333, 5, 1), max_levels=3, trunc_rtol=0.0, coarse_poly_order=4, precision=prec)
    rng = np.random.default_rng(2)
    for k in (2, 3, 4, 6, 7, 8, 12, 16, 31, 32, 33, 36, 63, 64, 65, 66, 68, 127, 128):
        c.check_solve(rng.standard_normal((k, 333)))


# one block holds 2048 elements; 152 blocks of 512 threads hold one, two, four
# or eight elements a thread, beyond that each dot is a launch
@pytest.mark.parametrize("n", [1, 2, 511, 2048, 2049, 77824, 77825, 155649, 311297, 622592, 622593])
def test_gram_schmidt_columns(n):
    c = General(random_matrix(n, 2, n), max_levels=1, coarse_poly_order=4)
    _check_setup(c)
    c.check_solve(np.random.default_rng(n).standard_normal(n))


def banded(n, width):
    """`width` off-diagonal entries a row (fewer in the first rows)."""
    r = np.repeat(np.arange(n), width + 1)
    c = r - np.tile(np.arange(width, -1, -1), n)
    keep = c >= 0
    r, c = r[keep], c[keep]
    v = np.where(r == c, 1.5 * max(width, 1), -np.random.default_rng(width).uniform(0.1, 1.0, r.size))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    return O.CSR(n, n, rp.astype(np.int64), c.astype(np.int64), v)


# widest slices of one and two entries, slices of four on average and their
# neighbours; long rows with fewer and with more warps than fill the GPU
@pytest.mark.parametrize("prec", [G.AIRG_FP64, G.AIRG_MIXED_FP32])
@pytest.mark.parametrize("n,width", [(31, 0), (33, 1), (65, 1), (1000, 1), (999, 2), (129, 3), (1000, 4), (1000, 5),
                                     (777, 8), (1000, 9), (1000, 17), (1000, 70), (90000, 70)])
def test_slice_widths(n, width, prec):
    c = General(banded(n, width), max_levels=1, coarse_poly_order=4, precision=prec)
    c.check_solve(np.random.default_rng(n).standard_normal(n))


@pytest.mark.parametrize("window", ["0", "1", "2", "33", "4096", "4097", "100000"])
def test_sort_windows(window, monkeypatch):
    monkeypatch.setenv("AIRG_SORT_WINDOW", window)
    _check_solve(Case(workload("grid", (160, 120))))


@pytest.mark.parametrize("n", [2, 31, 33, 4097, 600_001])
def test_exact_dot_digit_spread(n):
    """Products from 2^-1050 to 2^1020 of both signs, sums that cancel down to
    one small product of either sign, and sums whose carries run through a
    long stretch of equal digits."""
    rng = np.random.default_rng(n)
    e = rng.integers(-525, 500, n).astype(float)
    x = rng.standard_normal(n) * np.exp2(e)
    y = rng.standard_normal(n) * np.exp2(e)
    cases = [(x, y)]
    for tiny in (2.0 ** -1000, -2.0 ** -1000):
        xc, yc = np.concatenate([x, x, [1.0]]), np.concatenate([y, -y, [tiny]])
        p = rng.permutation(xc.size)
        cases.append((xc[p], yc[p]))
    cases.append((np.array([2.0 ** 500, -2.0 ** -500] + [0.0] * n), np.array([2.0 ** 500, 2.0 ** -500] + [1.0] * n)))
    cases.append((np.array([-2.0 ** 500, 2.0 ** -500] + [0.0] * n), np.array([2.0 ** 500, 2.0 ** -500] + [1.0] * n)))
    for x, y in cases:
        got = G.airg_dot_exact(torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda"))
        assert got == O.xdot(x, y)
