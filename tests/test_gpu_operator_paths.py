"""Phi and Phi^H through every storage and work split against the stored G itself:
the rows the plan exports (FP64 copies of its own values) applied by SciPy between
the oracle's FP64 transforms, so that only the operator kernels are under test.

Tolerance: FP32 sums and transforms.  A transform of up to 12 radix-4 / radix-2
stages and a sum of n terms in blocks each lose a few units of 2^-24 of the 2-norm;
1e-5 (170 units) covers both with the stored values taken as exact."""
import numpy as np
import pytest
import scipy.sparse
import torch

from oracle import wproj_oracle as O
from paper_1307_3424_gb300 import synth

pytestmark = pytest.mark.gpu

L = synth.fov_L()


@pytest.fixture(scope="module")
def wp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_3424_gb300 import wproj
    return wproj


def exported(plan):
    c = plan.csr()
    col, val = c.rows(0, c.m)
    val = val.cpu()
    if c.value_dtype == "f32":
        val = val.numpy().astype(np.complex128)
    else:
        v = val.float().numpy().astype(np.float64)
        rs = np.repeat(c.row_scale.cpu().numpy().astype(np.float64), np.diff(c.row_ptr.cpu().numpy()))
        val = (v[:, 0] + 1j * v[:, 1]) * rs
    return scipy.sparse.csr_matrix((val, col.cpu().numpy().astype(np.int64), c.row_ptr.cpu().numpy()),
                                   shape=(c.m, c.n_cols))


def uvw_cells(rng, M, N, wmax, edge=0.0):
    """Uniform disk, w_c ~ U[0, wmax] cells; a share `edge` of the rows at the band's
    corner, where kernels wrap around the grid."""
    uv = synth.uv_points(rng, M, synth.band_limit(N, L), N, "uniform")
    k = int(edge * M)
    uv[:k] = -synth.band_limit(N, L) * (1 - 3.0 * rng.uniform(0, 1, (k, 2)) / N)
    w = 2.0 * rng.uniform(0, wmax, M) / (L * L)
    return np.ascontiguousarray(np.concatenate([uv, w[:, None]], axis=1))


def check_operators(plan, N, W, rng, tol=1e-5):
    geo = O.Geometry(N, L, W=W)
    G = exported(plan)
    x = rng.standard_normal((N, N)).astype(np.float32)
    y = (rng.standard_normal(G.shape[0]) + 1j * rng.standard_normal(G.shape[0])).astype(np.complex64)
    xg, yg = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    yr, xr = O.phi(geo, G, x.astype(np.float64)), np.real(O.phi_adj(geo, G, y.astype(np.complex128)))
    for _ in range(2):      # a second pass on the same buffers gives the same bits
        py, px = plan.phi(xg).cpu().numpy(), plan.phi_adj(yg).cpu().numpy()
        assert np.linalg.norm(py - yr) <= tol * np.linalg.norm(yr)
        assert np.linalg.norm(px - xr) <= tol * np.linalg.norm(xr)
        assert np.abs(py - yr).max() <= 30 * tol * np.abs(yr).max()   # no row and no cell left out
        assert np.abs(px - xr).max() <= 30 * tol * np.abs(xr).max()


# dense rows: 16^2 grid (one 16-cell tile), one to ~100 chunks a tile, each format
@pytest.mark.parametrize("N,M,wmax,fmt,value", [(8, 5, 0.5, "auto", "f32"), (16, 700, 2.0, "columns", "f32"),
                                                (32, 40, 4.0, "mask", "f32"), (64, 300, 30.0, "mask", "f32"),
                                                (64, 300, 30.0, "mask", "bf16"), (128, 33, 60.0, "columns", "f16")])
def test_dense_rows(wp, N, M, wmax, fmt, value):
    rng = np.random.default_rng(N + M)
    plan = wp.Plan(N, L, value_dtype=value, index_format=fmt)
    plan.build_kernels(torch.from_numpy(uvw_cells(rng, M, N, wmax)).cuda(), 0.99)
    check_operators(plan, N, 4, rng)
    plan.close()


# short rows (boxes of at most 64 x 64 cells) on interleaved slices: grids whose
# patches wrap round the whole axis (32^2, 64^2) and larger ones; one row, a tile of
# rows split over several chunks, rows at the grid's edge; runs of 2 to 64 cells
# (w up to 4 cells; e = 1 keeps whole boxes), each value type and storage
@pytest.mark.parametrize("N,M,wmax,W,e,fmt,value", [
    (16, 40, 1.0, 4, 0.99, "auto", "f32"), (32, 1, 0.0, 4, 0.99, "auto", "f32"), (32, 900, 4.0, 4, 0.99, "auto", "f32"),
    (32, 300, 4.0, 8, 1.0, "columns", "f32"), (64, 1500, 4.0, 6, 0.999, "auto", "f32"),
    (64, 1500, 0.3, 4, 0.9, "auto", "bf16"), (128, 6001, 4.0, 4, 0.99, "auto", "f16"),
    (128, 3000, 2.0, 8, 0.99, "runs", "bf16"), (256, 20000, 1.0, 4, 0.99, "columns", "f32"),
    (256, 2000, 4.0, 4, 1.0, "auto", "f32"), (512, 9, 3.0, 4, 0.99, "auto", "f32"), (512, 9, 3.0, 4, 0.99, "auto", "bf16"),
])
def test_short_rows(wp, N, M, wmax, W, e, fmt, value):
    rng = np.random.default_rng(N + M + W)
    uvw = uvw_cells(rng, M, N, wmax, edge=0.2)
    if M > 1000:
        uvw[: M // 2, :2] = uvw[0, :2]      # half of the rows in one tile: several chunks
        uvw[: M // 2, :2] += rng.uniform(0, 0.5, (M // 2, 2)) / L
        uvw = uvw[np.abs(uvw[:, :2]).max(axis=1) < synth.band_limit(N, L) * (1 - 1e-9)]
    plan = wp.Plan(N, L, kb_support=W, box="rule", value_dtype=value, index_format=fmt)
    plan.build_kernels(torch.from_numpy(np.ascontiguousarray(uvw)).cuda(), e)
    check_operators(plan, N, W, rng)
    plan.close()


# a batch takes slices only when every problem can (a 16^2 grid, one tile of 16 x 16
# cells, cannot)
@pytest.mark.parametrize("ns", [(16, 32, 64), (64, 16, 128), (8, 64)])
def test_batch_matches_single_plans(wp, ns):
    rng = np.random.default_rng(sum(ns))
    ms = [7 * n + 3 for n in ns]
    uvw = [uvw_cells(rng, m, n, 1.0, edge=0.2) for m, n in zip(ms, ns)]
    b = wp.Batch(ns, L)
    b.build_kernels(torch.from_numpy(np.concatenate(uvw)).cuda(), ms, 0.99)
    b.tune()
    x = torch.from_numpy(rng.standard_normal(b.pixels).astype(np.float32)).cuda()
    y = torch.view_as_complex(torch.from_numpy(rng.standard_normal((b.m, 2)).astype(np.float32)).cuda())
    px, py = b.split_images(b.phi_adj(y)), b.split_vis(b.phi(x))
    for i, (n, u) in enumerate(zip(ns, uvw)):
        p = wp.Plan(n, L, box="rule")
        p.build_kernels(torch.from_numpy(u).cuda(), 0.99)
        ry, rx = p.phi(b.split_images(x)[i].contiguous()), p.phi_adj(b.split_vis(y)[i].contiguous())
        assert float((py[i] - ry).norm() / ry.norm()) <= 1e-5
        assert float((px[i] - rx).norm() / rx.norm()) <= 1e-5
        p.close()
    b.close()


# boxes built by one block each (32^2 and 64^2 cells): kept energy, cardinality and
# values against the oracle, with whole boxes (e = 1), single entries (small e), w = 0
# (mirror-symmetric kernels: ties at the cut) and each tap count
@pytest.mark.parametrize("N,e,W,wmax", [(16, 0.99, 4, 0.0), (32, 0.05, 4, 4.0), (32, 0.9, 8, 4.0), (64, 0.999, 6, 4.0),
                                        (64, 1.0, 4, 2.0), (128, 0.99, 4, 4.0)])
def test_small_boxes(wp, N, e, W, wmax):
    from test_gpu_parity import check_build
    rng = np.random.default_rng(N + W)
    uvw = uvw_cells(rng, 40, N, wmax, edge=0.2)
    plan = wp.Plan(N, L, kb_support=W, box="rule")
    plan.build_kernels(torch.from_numpy(uvw).cuda(), e)
    check_build(plan, O.Geometry(N, L, W=W), uvw, e, "rule")
    plan.close()

# passes launched one behind the other (blocks of a kernel start before the one ahead
# has ended) against the same passes each waited for, bit for bit: inputs overwritten
# right before and after a pass, eager and as a captured graph with copies between;
# dense rows with and without partial tiles, short rows, a batch
@pytest.mark.parametrize("N,M,box,value", [(64, 500, "G", "f32"), (32, 20, "G", "bf16"), (256, 3000, "rule", "f32"),
                                           (128, 900, "rule", "f16"), (0, 0, "batch", "f32")])
def test_back_to_back_passes(wp, N, M, box, value):
    rng = np.random.default_rng(N + M)
    if box == "batch":
        ns = (64, 128, 32)
        op = wp.Batch(ns, L)
        op.build_kernels(torch.from_numpy(np.concatenate([uvw_cells(rng, 9 * n, n, 1.0) for n in ns])).cuda(),
                         [9 * n for n in ns], 0.99)
        x = torch.empty(op.pixels, dtype=torch.float32, device="cuda")
    else:
        op = wp.Plan(N, L, box=box, value_dtype=value)
        op.build_kernels(torch.from_numpy(uvw_cells(rng, M, N, 20.0 if box == "G" else 2.0)).cuda(), 0.99)
        x = torch.empty((N, N), dtype=torch.float32, device="cuda")
    xs = torch.from_numpy(rng.standard_normal((4,) + tuple(x.shape)).astype(np.float32)).cuda()
    y = torch.empty(op.m, dtype=torch.complex64, device="cuda")
    z = torch.empty_like(x)
    out = torch.empty((8,) + tuple(x.shape), dtype=torch.float32, device="cuda")
    yo = torch.empty((8, op.m), dtype=torch.complex64, device="cuda")

    def passes(wait):
        for i in range(8):
            x.copy_(xs[i % 4])
            for step in range(3):      # Phi and Phi^H of each other's results
                op.phi(x, y)
                wait()
                op.phi_adj(y, z)
                wait()
                x.copy_(z) if step == 1 else x.add_(z, alpha=0.5)
                wait()
            yo[i].copy_(y)
            y.zero_()
            out[i].copy_(z)

    passes(torch.cuda.synchronize)
    torch.cuda.synchronize()
    want, wanty = out.clone(), yo.clone()
    out.zero_()
    yo.zero_()
    passes(lambda: None)
    torch.cuda.synchronize()
    assert torch.equal(out, want) and torch.equal(yo, wanty)
    out.zero_()
    yo.zero_()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        passes(lambda: None)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want) and torch.equal(yo, wanty)
    op.close()


# the GEMM's staged TMA stores (128 and 256 columns a tile, more tiles than SMs) and its
# element by element ones (an output or a bias off the 16-byte boundary): the same bits
@pytest.mark.parametrize("m,n,k,bf16", [(128, 128, 64, False), (512, 384, 256, True), (20480, 256, 64, True),
                                        (4096, 1280, 128, False)])
def test_gemm_unaligned_output(wp, m, n, k, bf16):
    g = torch.Generator().manual_seed(m + n)
    a, b = (torch.randn(r, k, generator=g).to(torch.bfloat16).cuda() for r in (m, n))
    bias = torch.randn(n, generator=g).cuda()
    ref = wp.gemm_bf16(a, b, bias, out_bf16=bf16)
    room = torch.full((m * n + 16,), 7.0, dtype=ref.dtype, device="cuda")
    bias1 = torch.cat([bias[:1], bias])
    for off, bs in ((1, bias), (0, bias1[1:])):
        room.fill_(7.0)
        c = room[off:off + m * n]
        st = wp.lib().wproj_gemm_bf16(m, n, k, a.data_ptr(), b.data_ptr(), bs.data_ptr(), c.data_ptr(), int(bf16),
                                      torch.cuda.current_stream().cuda_stream)
        assert st == 0
        assert torch.equal(c.view(m, n), ref)
        assert bool((room[:off] == 7).all()) and bool((room[off + m * n:] == 7).all())
    err = (ref.double().cpu() - (a.double().cpu() @ b.double().cpu().T + bias.double().cpu())).norm() / ref.double().norm().cpu()
    assert float(err) <= (4e-3 if bf16 else 1e-5)
