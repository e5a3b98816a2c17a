"""GPU parity: the scaling-vector update (Algorithm 2, inner repeat) against the oracle."""
import numpy as np
import pytest
import torch

from paper_2412_04180_b200 import inputs

pytestmark = pytest.mark.gpu
BITS = [1, 2, 3, 4]


def _labels(oracle, w, g, bits):
    res = oracle.cluster_rows(w, g, BITS, 15, row_bits=bits)
    rows = w.shape[0]
    return np.stack([res["codes"][int(b) - 1, i] for i, b in enumerate(bits)]).astype(np.uint8)


@pytest.mark.parametrize("rows,cols,steps", [(16, 64, 1), (40, 520, 7), (300, 257, 45), (700, 1024, 120)])
def test_scale_update_matches_oracle(ctx, oracle, rows, cols, steps):
    w, g = inputs.make_rows(rows, cols, 50 + rows, outlier_frac=0.01)
    bits = (np.arange(rows) % 4 + 1).astype(np.uint8)
    labels = _labels(oracle, w, g, bits)
    a0 = inputs.make_scale(cols, 3, spread=0.05)
    want, trace = oracle.scale_update(w, g, labels, a0.astype(np.float64), steps=steps)
    ctx.reserve(rows, cols)
    alpha = torch.from_numpy(a0.copy()).cuda()
    got_trace = ctx.scale_update(torch.from_numpy(w).cuda(), torch.from_numpy(g).cuda(),
                                 torch.from_numpy(labels).cuda(), alpha, steps=steps)
    torch.cuda.synchronize()
    assert ctx.get_status() == 0
    # both sides carry alpha in binary64 and differ only in summation order (Adam's normalised
    # step amplifies that where a gradient entry is near zero); the result is returned as binary32
    np.testing.assert_allclose(got_trace.cpu().numpy(), trace, rtol=1e-7)
    np.testing.assert_allclose(alpha.cpu().numpy().astype(np.float64), want, rtol=1e-6, atol=0)


@pytest.mark.parametrize("rows,cols,kind", [(1, 8, "mixed"), (3, 63, "mixed"), (25, 65, "mixed"), (149, 33, "mixed"), (3560, 68, "mixed"),
                                            (7, 1024, "one"), (5, 2050, "column"), (9, 700, "runs"), (4, 4100, "rare")])
def test_scale_update_label_layouts(ctx, oracle, rows, cols, kind):
    """The label-ordered copy at its edges: rows that are shared by several warps, taken whole, or both; clusters that
    are empty, a single one, one per column class, contiguous, or a few elements beside a large one."""
    rng = np.random.default_rng(rows + cols)
    w, g = inputs.make_rows(rows, cols, 60 + cols)
    j = np.arange(cols)
    labels = {"mixed": lambda: rng.integers(0, np.array([2, 4, 8, 16])[np.arange(rows) % 4][:, None], size=(rows, cols)),
              "one": lambda: np.full((rows, cols), 15), "column": lambda: np.broadcast_to(j % 16, (rows, cols)),
              "runs": lambda: np.broadcast_to(j * 16 // cols, (rows, cols)),
              "rare": lambda: np.where(rng.random((rows, cols)) < 0.002, rng.integers(0, 16, size=(rows, cols)), 7)}[kind]().astype(np.uint8)
    a0 = inputs.make_scale(cols, 5, spread=0.05)
    want, trace = oracle.scale_update(w, g, labels, a0.astype(np.float64), steps=2)
    ctx.reserve(rows, cols)
    alpha = torch.from_numpy(a0.copy()).cuda()
    got = ctx.scale_update(torch.from_numpy(w).cuda(), torch.from_numpy(g).cuda(), torch.from_numpy(np.ascontiguousarray(labels)).cuda(), alpha, steps=2)
    torch.cuda.synchronize()
    assert ctx.get_status() == 0
    np.testing.assert_allclose(got.cpu().numpy(), trace, rtol=1e-7, atol=1e-12)
    np.testing.assert_allclose(alpha.cpu().numpy().astype(np.float64), want, rtol=1e-6, atol=0)


@pytest.mark.parametrize("rows,cols,kind", [(40, 128, "mixed"), (17, 129, "mixed"), (300, 389, "rare"), (50, 512, "one"), (50, 513, "column"),
                                            (3553, 516, "mixed"), (3600, 1024, "mixed"), (3600, 1025, "rare")])
def test_scale_update_narrow_matrices(ctx, oracle, rows, cols, kind):
    """Row lengths and row counts around the rules for short rows, and blocks of the gradient kernel that hold several row shares."""
    test_scale_update_label_layouts(ctx, oracle, rows, cols, kind)


def test_scale_update_wide_rows(ctx, oracle):
    rows, cols = 6, 22016
    w, g = inputs.make_rows(8192, cols, 5001, 0, rows, importance_sigma=2.0)
    bits = np.array([1, 2, 3, 4, 4, 3], np.uint8)
    labels = _labels(oracle, w, g, bits)
    a0 = np.ones(cols, np.float32)
    want, trace = oracle.scale_update(w, g, labels, a0.astype(np.float64), steps=5)
    ctx.reserve(rows, cols)
    alpha = torch.from_numpy(a0.copy()).cuda()
    got = ctx.scale_update(torch.from_numpy(w).cuda(), torch.from_numpy(g).cuda(), torch.from_numpy(labels).cuda(),
                           alpha, steps=5)
    np.testing.assert_allclose(got.cpu().numpy(), trace, rtol=1e-7)
    np.testing.assert_allclose(alpha.cpu().numpy().astype(np.float64), want, rtol=1e-6)


@pytest.mark.parametrize("rows,cols,steps", [(16, 64, 3), (40, 520, 12), (130, 264, 40), (300, 1000, 25)])
def test_scale_update_lfull_matches_oracle(ctx, oracle, rows, cols, steps):
    """The Adam steps on the L-full loss (Section 4.3).  Both sides round the residual to the same binary16 operand;
    the GPU accumulates D H in binary32 on the tensor cores (relative error ~1e-6 of the magnitude sums) where the
    oracle sums in binary64, so the loss is compared at 2e-5 (observed: 2e-6) and alpha, whose Adam steps turn a relative
    gradient error delta into lr * delta per step, at 1e-4 relative + 1e-4 absolute (observed: 2e-5)."""
    w, g = inputs.make_rows(rows, cols, 150 + rows, outlier_frac=0.01)
    bits = (np.arange(rows) % 4 + 1).astype(np.uint8)
    labels = _labels(oracle, w, g, bits)
    H = inputs.make_gram(cols, 160 + cols)
    a0 = inputs.make_scale(cols, 5, spread=0.05)
    want, trace = oracle.scale_update_lfull(w, g, labels, a0.astype(np.float64), H, steps=steps)
    ctx.reserve(rows, cols)
    alpha = torch.from_numpy(a0.copy()).cuda()
    got_trace = ctx.scale_update_lfull(torch.from_numpy(w).cuda(), torch.from_numpy(g).cuda(), torch.from_numpy(labels).cuda(),
                                       alpha, torch.from_numpy(H).cuda(), steps=steps)
    torch.cuda.synchronize()
    assert ctx.get_status() == 0
    got_trace = got_trace.cpu().numpy()
    got = alpha.cpu().numpy().astype(np.float64)
    print("max rel trace diff", np.max(np.abs(got_trace - trace) / trace), "max alpha diff", np.max(np.abs(got - want)))
    np.testing.assert_allclose(got_trace, trace, rtol=2e-5)
    np.testing.assert_allclose(got, want, rtol=1e-4, atol=1e-4)
    assert trace[-1] < trace[0] or steps < 5


def test_scale_update_lfull_argument_errors(ctx, skimlib):
    rows, cols = 8, 64
    w, g = inputs.make_rows(rows, cols, 3)
    ctx.reserve(rows, cols)
    W, G = torch.from_numpy(w).cuda(), torch.from_numpy(g).cuda()
    L = torch.zeros((rows, cols), dtype=torch.uint8, device="cuda")
    H = torch.eye(cols, dtype=torch.float16, device="cuda")
    a = torch.ones(cols, device="cuda")
    with pytest.raises(skimlib.SkimError) as e:
        ctx.scale_update_lfull(W, G, L, a, H, steps=1, scratch=torch.empty(256, dtype=torch.uint8, device="cuda"))
    assert e.value.code == -5
    with pytest.raises(skimlib.SkimError) as e:
        ctx.scale_update_lfull(W[:, :60].contiguous(), G[:, :60].contiguous(), L[:, :60].contiguous(), a[:60].contiguous(),
                               H[:60, :60].contiguous(), steps=1)
    assert e.value.code == -2


@pytest.mark.parametrize("rows,cols,steps", [(257, 776, 4), (3560, 264, 2)])
def test_scale_update_lfull_tiles_and_shared_rows(ctx, oracle, rows, cols, steps):
    """More than one tile of the contraction either way, its last tiles halved; rows taken whole and rows shared by warps."""
    test_scale_update_lfull_matches_oracle(ctx, oracle, rows, cols, steps)
