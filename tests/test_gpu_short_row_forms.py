"""Short rows on and off the interleaved slices: the plans and batches that the rule turns
away (they run the older forms), slices made again after the values or the rows changed,
and runs that have to repeat bit for bit.  References and tolerances as in
test_gpu_operator_paths."""
import numpy as np
import pytest
import torch
from test_gpu_operator_paths import L, check_operators, uvw_cells


pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_3424_gb300 import wproj
    return wproj


def on_device(uvw):
    return torch.from_numpy(np.ascontiguousarray(uvw)).cuda()


def crowd(rng, uvw, k):
    """The first k rows within half a wavelength-cell of row 0: one crowded tile."""
    uvw[:k, :2] = uvw[0, :2] * 0.9 + rng.uniform(0, 0.5, (k, 2)) / L
    return uvw


def same_twice(op, x, y):
    a, b = op.phi(x), op.phi_adj(y)
    assert torch.equal(op.phi(x), a) and torch.equal(op.phi_adj(y), b)


# plans that slices do not serve: rows spread over a large grid (patches of more than four
# cells an entry) with a crowded tile of several chunks, and rows of one or two entries,
# which take eight places each; every storage and value type of the older forms
@pytest.mark.parametrize("N,M,k,wmax,e,fmt,value", [
    (512, 1300, 400, 2.0, 0.99, "auto", "f32"), (512, 1300, 400, 2.0, 0.99, "runs", "f16"),
    (512, 1300, 400, 2.0, 0.99, "runs", "bf16"), (512, 1300, 400, 2.0, 0.99, "columns", "f32"),
    (512, 1300, 400, 2.0, 0.99, "auto", "f16"), (64, 3000, 0, 0.0, 0.05, "auto", "f32"),
    (64, 3000, 0, 0.0, 0.05, "auto", "bf16")])
def test_plans_without_slices(wp, N, M, k, wmax, e, fmt, value):
    rng = np.random.default_rng(M + k)
    uvw = crowd(rng, uvw_cells(rng, M, N, wmax), k) if k else uvw_cells(rng, M, N, wmax)
    p = wp.Plan(N, L, box="rule", index_format=fmt, value_dtype=value)
    p.build_kernels(on_device(uvw), e)
    assert not p.slices()["used"]
    check_operators(p, N, 4, rng)
    same_twice(p, torch.randn(N, N, device="cuda"), torch.randn(M, dtype=torch.complex64, device="cuda"))
    p.close()


# the same bits from two passes of plans on slices: tiles of one and of several chunks
@pytest.mark.parametrize("N,M,k,value", [(64, 1500, 700, "f32"), (256, 20000, 9000, "bf16"), (32, 60, 0, "f16")])
def test_slices_repeat(wp, N, M, k, value):
    rng = np.random.default_rng(M)
    p = wp.Plan(N, L, box="rule", value_dtype=value)
    p.build_kernels(on_device(crowd(rng, uvw_cells(rng, M, N, 2.0), k) if k else uvw_cells(rng, M, N, 2.0)), 0.99)
    assert p.slices()["used"]
    same_twice(p, torch.randn(N, N, device="cuda"), torch.randn(M, dtype=torch.complex64, device="cuda"))
    p.close()


# batches sparser than the usual ones stay on slices (rows of one entry, few rows a tile);
# a tile's chunk of more than 12288 rows turns the whole batch to the older forms.  Both
# against single plans in the column form
@pytest.mark.parametrize("W,wmax,ms,k,used", [(4, 0.0, (40, 9, 30), 0, True), (1, 0.0, (500, 60, 9), 0, True),
                                              (1, 0.0, (20000, 60, 9), 19000, False)])
def test_sparse_batches(wp, W, wmax, ms, k, used):
    ns = (64, 32, 128)
    rng = np.random.default_rng(sum(ms))
    uvw = [uvw_cells(rng, m, n, wmax) for m, n in zip(ms, ns)]
    if k:
        crowd(rng, uvw[0], k)
    b = wp.Batch(ns, L, kb_support=W)
    b.build_kernels(on_device(np.concatenate(uvw)), ms, 0.9)
    assert b.slices()["used"] == used
    x = torch.from_numpy(rng.standard_normal(b.pixels).astype(np.float32)).cuda()
    y = torch.view_as_complex(torch.from_numpy(rng.standard_normal((b.m, 2)).astype(np.float32)).cuda())
    same_twice(b, x, y)
    py, px = b.split_vis(b.phi(x)), b.split_images(b.phi_adj(y))
    for i, (n, u) in enumerate(zip(ns, uvw)):
        p = wp.Plan(n, L, kb_support=W, box="rule", index_format="columns")
        p.build_kernels(on_device(u), 0.9)
        ry, rx = p.phi(b.split_images(x)[i].contiguous()), p.phi_adj(b.split_vis(y)[i].contiguous())
        assert float((py[i] - ry).norm() / ry.norm()) <= 1e-5
        assert float((px[i] - rx).norm() / rx.norm()) <= 1e-5
        p.close()
    b.close()


# a non-finite image or visibility of one problem stays in that problem
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_batch_keeps_nonfinite_values_apart(wp, bad):
    ns, ms = (32, 64, 32), (200, 500, 60)
    rng = np.random.default_rng(5)
    b = wp.Batch(ns, L)
    b.build_kernels(on_device(np.concatenate([uvw_cells(rng, m, n, 1.0) for m, n in zip(ms, ns)])), ms, 0.99)
    assert b.slices()["used"]
    x, y = torch.randn(b.pixels, device="cuda"), torch.randn(b.m, dtype=torch.complex64, device="cuda")
    vy, vx = b.split_vis(b.phi(x)), b.split_images(b.phi_adj(y))
    b.split_images(x)[1][5, 7] = bad
    b.split_vis(y)[1][11] = complex(bad, 0.0)
    wy, wx = b.split_vis(b.phi(x)), b.split_images(b.phi_adj(y))
    for i in (0, 2):
        assert torch.equal(vy[i], wy[i]) and torch.equal(vx[i], wx[i])
    assert not bool(torch.isfinite(torch.view_as_real(wy[1])).any()) and not bool(torch.isfinite(wx[1]).any())
    b.close()


# a plan built again with larger, smaller and nearly equal G (buffers kept where the next
# G fits) is the plan a new one would be, across storage forms
@pytest.mark.parametrize("fmt,value", [("auto", "f32"), ("columns", "f32"), ("auto", "bf16"), ("mask", "f32")])
def test_rebuilt_plan_is_a_new_plan(wp, fmt, value):
    N = 64
    rng = np.random.default_rng(9)
    p = wp.Plan(N, L, box="rule" if fmt != "mask" else "G", index_format=fmt, value_dtype=value)
    x = torch.randn(N, N, device="cuda")
    for M, wmax in ((700, 1.0), (2500, 4.0), (690, 1.0), (700, 1.0), (3, 0.5), (650, 1.1)):
        uvw = on_device(uvw_cells(rng, M, N, wmax))
        q = wp.Plan(N, L, box="rule" if fmt != "mask" else "G", index_format=fmt, value_dtype=value)
        y = torch.randn(M, dtype=torch.complex64, device="cuda")
        for o in (p, q):
            o.build_kernels(uvw, 0.99)
        assert p.slices() == q.slices()
        assert torch.equal(p.phi(x), q.phi(x)) and torch.equal(p.phi_adj(y), q.phi_adj(y))
        cp, cq = p.csr(), q.csr()
        assert torch.equal(cp.row_ptr, cq.row_ptr) and torch.equal(cp.col, cq.col) and torch.equal(cp.val, cq.val)
        q.close()
    p.close()


# the learned build replaces stored values after the slices (or the cell copy) were made:
# both operators against the rows that the plan exports.  A network of random weights with
# every mask logit high passes every row, so that all values change
@pytest.mark.parametrize("M,N,used", [(400, 32, True), (9, 512, False)])
def test_learned_values_reach_the_operators(wp, M, N, used):
    rng = np.random.default_rng(M)
    uvw = uvw_cells(rng, M, N, 1.0)
    ref = wp.Plan(N, L, box=32, index_format="columns")
    ref.build_kernels(on_device(uvw), 0.9)
    n = int(wp.lib().wproj_mlp_num_params())
    prm = 0.05 * torch.randn(n, generator=torch.Generator().manual_seed(1))
    prm[-1024:] = 50.0          # b4 of the mask logits
    net = wp.MLP(prm)
    p = wp.Plan(N, L, box=32, index_format="columns")
    info, _ = p.build_kernels_learned(net, on_device(uvw), 0.9, rel_l2_max=1e6)
    assert p.slices()["used"] == used
    assert info["learned"] == M
    assert not bool((p.csr().val == ref.csr().val).any())
    check_operators(p, N, 4, rng)
    for o in (ref, p, net):
        o.close()
