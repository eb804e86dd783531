"""Gradients of guide batches with zero-weight records: the weighted records
are shared out evenly over the thread blocks wherever they lie in the batch,
so a batch gives the gradient of its weighted records alone; a grid gradient
that is not 16-byte aligned gives the same as an aligned one."""
import ctypes as C

import numpy as np
import pytest

from paper_1912_04000_gb300 import scenes

pytestmark = pytest.mark.gpu
LOG2_T = 10


@pytest.fixture(scope="module")
def R():
    from paper_1912_04000_gb300.renderer import Renderer
    r = Renderer(0)
    wl = scenes.prism_room(width=8, height=8, n_bands=5, spp=1)
    r.load(wl)
    r.lo, r.hi = wl.scene.verts.min(0), wl.scene.verts.max(0)
    r.guide_init(seed=4, log2_table=LOG2_T)
    rng = np.random.default_rng(11)
    grid, W = r.guide_get_params()
    r.guide_set_params(0.3 * rng.standard_normal(grid.shape).astype(np.float32), W)
    return r


def _records(rng, n, lo, hi, weighted):
    rec = np.zeros((n, 12), np.float32)
    rec[:, 0:3] = lo + rng.random((n, 3)) * (hi - lo)
    nrm, om = rng.standard_normal((2, n, 3))
    rec[:, 4:7] = nrm / np.linalg.norm(nrm, axis=1, keepdims=True)
    rec[:, 7] = rng.integers(0, 9, n)
    rec[:, 8:11] = om / np.linalg.norm(om, axis=1, keepdims=True)
    rec[weighted, 3] = rng.exponential(size=len(weighted))
    return rec


CASES = {
    "one": (1, "all"), "short tile": (127, "all"), "over a tile": (129, "all"), "a tile per block and one": (152 * 128 + 1, "all"),
    "none": (3000, "none"), "last only": (70001, "last"), "one chunk of many": (40 * 1024 + 5, "chunk"),
    "a tenth": (30000, "tenth"), "chunks of two rounds": (1024 * 1024 + 77, "sparse"),
}


@pytest.mark.parametrize("name", CASES)
def test_weighted_records_alone(R, name):
    n, kind = CASES[name]
    rng = np.random.default_rng(n)
    weighted = {"all": lambda: np.arange(n), "none": lambda: np.arange(0), "last": lambda: np.array([n - 1]),
                "chunk": lambda: np.arange(17 * 1024 + 3, 18 * 1024 + 400),
                "tenth": lambda: np.flatnonzero(rng.random(n) < 0.1),
                "sparse": lambda: np.flatnonzero(rng.random(n) < 0.004)}[kind]()
    rec = _records(rng, n, R.lo, R.hi, weighted)
    loss, dg, dw = R.guide_grad(rec)
    dg, dw = dg.cpu().numpy().astype(np.float64), dw.cpu().numpy().astype(np.float64)
    if kind == "none":
        assert loss == 0.0 and not dg.any() and not dw.any()
        return
    # the weighted records alone, in another order: other tiles, the same sums.
    # FP32 sums of up to 19,457 terms: 2^-24 sqrt(19457) ~ 1e-5 of the norm,
    # ten times that for cancelling terms
    alone = rec[rng.permutation(weighted)]
    loss1, dg1, dw1 = R.guide_grad(alone)
    dg1, dw1 = dg1.cpu().numpy().astype(np.float64), dw1.cpu().numpy().astype(np.float64)
    assert loss == pytest.approx(loss1, rel=1e-4)
    assert np.linalg.norm(dw) > 0 and np.linalg.norm(dg) > 0
    assert np.linalg.norm(dw - dw1) <= 1e-4 * np.linalg.norm(dw1)
    assert np.linalg.norm(dg - dg1) <= 1e-4 * np.linalg.norm(dg1)


def test_unaligned_grid_gradient(R):
    torch = R.torch
    rng = np.random.default_rng(3)
    rec = torch.as_tensor(_records(rng, 5000, R.lo, R.hi, np.arange(0, 5000, 3)), device="cuda")
    loss, dg, dw = R.guide_grad(rec)
    buf = torch.zeros(dg.numel() + 8, device="cuda")
    out = buf[1:1 + dg.numel()]
    got = C.c_float()
    R._check("rt_guide_grad", R.lib.rt_guide_grad(R._h, rec.data_ptr(), 5000, C.byref(got), out.data_ptr(), None))
    assert got.value == pytest.approx(loss, rel=1e-5)
    assert torch.linalg.vector_norm(out - dg) <= 1e-4 * torch.linalg.vector_norm(dg)
    assert buf[0] == 0 and not buf[1 + dg.numel():].any()
