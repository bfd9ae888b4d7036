"""Plans built and used beside other work: another stream's capture, operators still
running on another stream, other plans on other host threads, little free memory."""
import threading

import numpy as np
import pytest
import torch

from paper_1307_3424_gb300 import synth

pytestmark = pytest.mark.gpu

L = synth.fov_L()


@pytest.fixture(scope="module")
def wp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1307_3424_gb300 import wproj
    return wproj


def uvw_cells(seed, M, N, wmax):
    """Uniform disk, w_c ~ U[0, wmax] cells, on the device."""
    rng = np.random.default_rng(seed)
    uv = synth.uv_points(rng, M, synth.band_limit(N, L), N, "uniform")
    w = 2.0 * rng.uniform(0, wmax, M) / (L * L)
    return torch.from_numpy(np.ascontiguousarray(np.concatenate([uv, w[:, None]], axis=1))).cuda()


# a build, of a new plan or of one that holds a G, while another stream is captured in
# relaxed mode: neither disturbs the other
@pytest.mark.parametrize("again", [False, True])
def test_build_beside_a_capture(wp, again):
    N, M = 64, 300
    uvw = uvw_cells(0, M, N, 1.0)
    p, q = wp.Plan(N, L, box="rule"), wp.Plan(N, L, box="rule")
    q.build_kernels(uvw, 0.99)
    if again:
        p.build_kernels(uvw, 0.99)
    x = torch.randn(N, N, generator=torch.Generator().manual_seed(1)).cuda()
    y = torch.empty(M, dtype=torch.complex64, device="cuda")
    want = q.phi(x).clone()
    side, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        q.phi(x, y)
        p.build_kernels(uvw, 0.99, stream=side)
    g.replay()
    assert torch.equal(y, want)
    assert torch.equal(p.phi(x), want)
    p.close()
    q.close()


# a plan built again while an operator of its last G still waits on another stream: the
# operator reads the G it was launched with
@pytest.mark.parametrize("box,value", [("rule", "f32"), ("rule", "bf16"), ("G", "f32")])
def test_build_waits_for_operators_in_flight(wp, box, value):
    N, M = 64, 600
    p = wp.Plan(N, L, box=box, value_dtype=value)
    p.build_kernels(uvw_cells(0, M, N, 1.0), 0.99)
    x = torch.randn(N, N, generator=torch.Generator().manual_seed(2)).cuda()
    want = p.phi(x).clone()
    y = torch.empty_like(want)
    other = uvw_cells(1, M, N, 1.0)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(400_000_000)      # about 0.2 s
        p.phi(x, y, stream=side)
    p.build_kernels(other, 0.99)
    torch.cuda.synchronize()
    assert torch.equal(y, want)
    p.close()


# two plans on two host threads, with small and with large (over 48 KB) needs of shared
# memory: no launch of either is refused, and both give what they give alone.  A power
# iteration is one call of some hundred operator passes, so the threads' launches mix.
@pytest.mark.parametrize("value", ["f32", "bf16"])
def test_plans_on_host_threads(wp, value):
    plans = []
    for N, M, wmax, W, e in ((128, 6000, 4.0, 8, 1.0), (32, 900, 1.0, 4, 0.99)):
        p = wp.Plan(N, L, kb_support=W, box="rule", value_dtype=value)
        p.build_kernels(uvw_cells(N, M, N, wmax), e)
        plans.append((p, p.power_norm2(500)))
    got, refused = [[], []], []

    def work(i):
        s = torch.cuda.Stream()
        for _ in range(8):
            try:
                got[i].append(plans[i][0].power_norm2(500, stream=s))
            except wp.WprojError as err:
                refused.append(str(err))

    threads = [threading.Thread(target=work, args=(i,)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not refused, (len(refused), refused[0])
    for (p, alone), g in zip(plans, got):
        assert g == [alone] * 8
        p.close()


def leave_free(gib):
    """A tensor that takes all of the device's memory but `gib` GiB."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(free - int(gib * 2 ** 30), dtype=torch.uint8, device="cuda")


# short rows built with room for G and the older copies but not for the slices (f32 run
# lengths, 4.35e7 entries: they fit 1.92 GiB, with slices 2.12; a batch of 2.7e7 entries:
# 3.7 and 4.2 GiB): the same G and operators, in a form that fits
def test_build_without_room_for_slices(wp):
    N, M = 512, 300000
    uvw = uvw_cells(0, M, N, 4.0)
    x = torch.randn(N, N, generator=torch.Generator().manual_seed(3)).cuda()
    yv = torch.randn(M, dtype=torch.complex64, generator=torch.Generator().manual_seed(4)).cuda()
    results = []
    for gib in (None, 2.0):
        p = wp.Plan(N, L, box="rule")
        fill = leave_free(gib) if gib else None
        p.build_kernels(uvw, 0.9)
        del fill
        torch.cuda.empty_cache()
        c = p.csr()
        results.append((p.phi(x), p.phi_adj(yv), c.col.clone(), c.val.clone()))
        p.close()
    (y0, z0, c0, v0), (y1, z1, c1, v1) = results
    assert torch.equal(c0, c1) and torch.equal(v0, v1)
    assert float((y1 - y0).norm() / y0.norm()) <= 1e-5
    assert float((z1 - z0).norm() / z0.norm()) <= 1e-5


def test_batch_without_room_for_slices(wp):
    N, ms = 256, [60000] * 8
    uvw = torch.cat([uvw_cells(i, m, N, 4.0) for i, m in enumerate(ms)])
    x = torch.randn(8 * N * N, generator=torch.Generator().manual_seed(5)).cuda()
    yv = torch.randn(sum(ms), dtype=torch.complex64, generator=torch.Generator().manual_seed(6)).cuda()
    results = []
    for gib in (None, 3.95):
        b = wp.Batch([N] * 8, L)
        fill = leave_free(gib) if gib else None
        b.build_kernels(uvw, ms, 0.9)
        del fill
        torch.cuda.empty_cache()
        results.append((b.phi(x), b.phi_adj(yv)))
        b.close()
    (y0, z0), (y1, z1) = results
    assert float((y1 - y0).norm() / y0.norm()) <= 1e-5
    assert float((z1 - z0).norm() / z0.norm()) <= 1e-5


# operators launched right after a build, on the build's own stream (which the legacy
# stream does not order): every table that the build wrote is complete.  Segment lists
# of the tile stream, tiles of several chunks on slices, a batch's size classes
@pytest.mark.parametrize("box,fmt,N,M", [("G", "mask", 64, 3000), ("rule", "auto", 64, 8000), ("batch", "", 64, 2000)])
def test_operators_right_after_a_build(wp, box, fmt, N, M):
    side = torch.cuda.Stream()
    uvws = [uvw_cells(i, M, N, 2.0) for i in range(6)]
    if box == "batch":
        op = wp.Batch([N, 32], L)
        build = lambda u: op.build_kernels(u, [M - 300, 300], 0.9, stream=side)
        x = torch.randn(op.pixels, generator=torch.Generator().manual_seed(7)).cuda()
    else:
        op = wp.Plan(N, L, box=box, index_format=fmt)
        build = lambda u: op.build_kernels(u, 0.9, stream=side)
        x = torch.randn(N, N, generator=torch.Generator().manual_seed(7)).cuda()
    if box == "batch":      # the second problem's band is half as wide
        for u in uvws:
            u[M - 300:, :2] *= 0.5
    yv = torch.randn(M, dtype=torch.complex64, generator=torch.Generator().manual_seed(8)).cuda()
    y, z = torch.empty_like(yv), torch.empty_like(x)
    torch.cuda.synchronize()
    for u in uvws:
        build(u)
        op.phi(x, y, stream=side)
        op.phi_adj(yv, z, stream=side)
        torch.cuda.synchronize()
        assert torch.equal(op.phi(x), y) and torch.equal(op.phi_adj(yv), z)
    op.close()


# the launch count of wproj_phi_noalloc is wproj_phi's: one degridding kernel on slices and
# run lengths, two on the column form and the tile stream
@pytest.mark.parametrize("M,wmax,box,fmt,value", [(900, 1.0, "rule", "auto", "f32"), (900, 1.0, "rule", "columns", "bf16"),
                                                  (9, 3.0, "rule", "auto", "f32"), (9, 3.0, "rule", "columns", "f32"),
                                                  (90, 1.0, "G", "mask", "f32")])
def test_launch_counts(wp, M, wmax, box, fmt, value):
    N = 64
    p = wp.Plan(N, L, box=box, index_format=fmt, value_dtype=value)
    p.build_kernels(uvw_cells(0, M, N, wmax), 0.99)
    x, y = torch.zeros(N, N, device="cuda"), torch.empty(M, dtype=torch.complex64, device="cuda")
    counts = []
    for call in (wp.lib().wproj_phi, wp.lib().wproj_phi_noalloc):
        before = p.stats()["launches"]
        assert call(p.handle, x.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream) == wp.OK
        counts.append(p.stats()["launches"] - before)
    assert counts[0] == counts[1]
    p.close()


# which form serves a plan or batch: slices for short rows, except where their patches would
# hold more than four cells an entry, and nowhere else; the bytes are at least those of the
# entries' values and 2-byte indices
@pytest.mark.parametrize("N,M,wmax,box,fmt,value,used", [
    (64, 900, 1.0, "rule", "auto", "f32", True), (64, 900, 1.0, "rule", "runs", "bf16", True),
    (64, 900, 1.0, "rule", "columns", "f16", True), (512, 9, 3.0, "rule", "auto", "f32", False),
    (512, 9, 3.0, "rule", "columns", "bf16", False), (64, 90, 1.0, "G", "mask", "f32", False),
    (64, 90, 1.0, "G", "columns", "f32", False), (8, 40, 1.0, "rule", "auto", "f32", False)])
def test_slices_reported(wp, N, M, wmax, box, fmt, value, used):
    p = wp.Plan(N, L, box=box, index_format=fmt, value_dtype=value)
    p.build_kernels(uvw_cells(0, M, N, wmax), 0.99)
    s = p.slices()
    least = p.csr().nnz * ((8 if value == "f32" else 4) + 2)
    assert s["used"] == used
    assert (min(s["degrid_bytes"], s["grid_bytes"]) >= least) if used else (s["degrid_bytes"] == s["grid_bytes"] == 0)
    p.close()


@pytest.mark.parametrize("ns,used", [((64, 32), True), ((64, 8), False)])
def test_batch_slices_reported(wp, ns, used):
    b = wp.Batch(ns, L)
    b.build_kernels(torch.cat([uvw_cells(n, 5 * n, n, 1.0) for n in ns]), [5 * n for n in ns], 0.99)
    s = b.slices()
    assert s["used"] == used
    assert (min(s["degrid_bytes"], s["grid_bytes"]) >= 10 * b.info()["nnz"]) if used else s["grid_bytes"] == 0
    b.close()
