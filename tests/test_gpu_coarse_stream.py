"""AIRG_COARSE_STREAM=1 at sizes where large FP64 operators take fewer than 8
warps per slice: the coarsest operator keeps the 8 that the streamed form
shares its arithmetic with, and with 8 everywhere the solution is that of the
row kernels, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_17517_gb300 as G  # noqa: E402
from tests.test_gpu_shape_edges import banded  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.build()
    G.lib()


# 938 slices of 71 entries a row (4 warps by size), 1563 of 51 (2 warps),
# 65,536 rows (the last with 16-bit column indices without slice bases), and
# one below the rule's line
@pytest.mark.parametrize("n,width,by_size", [(9000, 70, 8), (30000, 70, 4), (50001, 49, 2), (65536, 49, 2)])
@pytest.mark.parametrize("mode", ["1", "2"])
def test_streamed_coarse_operator(n, width, by_size, mode, monkeypatch):
    A = banded(n, width)
    arrays = [torch.tensor(a, device="cuda") for a in (A.rowptr, A.col.astype(np.int32), A.val)]
    b = torch.tensor(np.random.default_rng(n).standard_normal(n), device="cuda")

    def solve():
        h = G.airg_setup(*arrays, G.airg_options_default(max_levels=1, coarse_poly_order=6))
        d = G.airg_operator_layout_info(h, 0, "coarse")
        x, info = G.airg_solve(h, b, rtol=1e-10)
        assert info.converged
        G.airg_free(h)
        return d, x

    assert solve()[0]["warps_per_slice"] == by_size
    monkeypatch.setenv("AIRG_COARSE_STREAM", mode)
    d = solve()[0]
    # what the streamed form needs of the layout
    assert d["warps_per_slice"] == 8 and d["index_bytes"] == 2 and d["slice_bases"] == 0
    # the top-level operator, which is the same matrix here, with 8 warps too
    monkeypatch.setenv("AIRG_MAX_PARTS", "8")
    streamed = solve()[1]
    monkeypatch.delenv("AIRG_COARSE_STREAM")
    assert torch.equal(streamed, solve()[1])
