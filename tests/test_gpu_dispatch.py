"""Edges of the kernels' size rules: row packings and pass chunks of anisotropic cells, the
slab pass on transforms as long as the data, the network's product kernels at widths and grids
that fill no tile, the batch's default launch against one CTA a cell."""
import zlib

import numpy as np
import pytest

import microstructures as ms
from oracle import fno, matfree

from layout import full_to_half, random_real_field

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

A2 = np.array([[2.0, 0.3], [0.3, 1.0]])
A3 = np.array([[2.0, 0.3, 0.1], [0.3, 1.0, -0.2], [0.1, -0.2, 1.5]])


@pytest.fixture(scope="module")
def hb():
    import paper_1404_3614_gb300 as hb
    return hb


@pytest.fixture(scope="module")
def solver(hb):
    s = hb.Bounds(0)
    yield s
    s.close()


# a plane of one point, planes and rows left over from quads, one row pair, long ragged rows
@pytest.mark.parametrize("N", [(1, 3), (5, 1), (37, 19), (203, 5), (3, 5, 1), (9, 5, 11), (17, 3, 13), (13, 29, 7),
                               (63, 7, 5)])
def test_ragged_anisotropic_operator_matches_oracle(hb, solver, N):
    """FP64 and float-float 1e-12, FP32 5e-6 of the largest entry: the bars of the operator's
    step tests (rounding of six transforms and the coefficient, with a factor to spare)."""
    d = len(N)
    A0, A1 = (A2, A2 @ A2) if d == 2 else (A3, A3 @ A3)
    p = ms.make_problem(d, N, (1.0, 0.7, 1.2)[:d], A0, [ms.box((0.1, 0.05, 0.0)[:d], (0.3, 0.2, 0.5)[:d], A1, d),
                                                        ms.ball((-0.25, -0.2, 0.1)[:d], 0.12, 0.2, d)])
    rng = np.random.default_rng([zlib.crc32(b"ragged"), *N])
    op = matfree.MatFreeOperator(p, "primal")
    info = hb.hom_problem_info(solver.ctx, p)
    nws = hb.hom_step_workspace_size(solver.ctx, p, d)
    ws = torch.empty(nws, dtype=torch.uint8, device="cuda")
    fields = [random_real_field(rng, d, N) for _ in range(d)]
    ref = np.stack([full_to_half(op.apply(u, project=True), d) for u in fields])
    x64 = torch.from_numpy(np.stack([full_to_half(u, d) for u in fields]).astype(np.complex128)).cuda()
    scale = max(np.abs(ref).max(), np.abs(x64.cpu().numpy()).max())
    for prec, cdt, rdt, tol in ((hb.HOM_FP64, torch.complex128, torch.float64, 1e-12),
                                (hb.HOM_FF, torch.complex128, torch.float32, 1e-12),
                                (hb.HOM_FP32, torch.complex64, torch.float32, 5e-6)):
        cshape = (info["ncomp"],) + tuple(info["M"][:d][::-1]) + ((2,) if prec == hb.HOM_FF else ())
        coef = torch.empty(cshape, dtype=rdt, device="cuda")
        hb.hom_coefficient(solver.ctx, p, 0, prec, coef.data_ptr(), ws.data_ptr(), nws)
        x = x64.to(cdt)
        y = torch.zeros_like(x)
        hb.hom_matvec(solver.ctx, p, 0, prec, 1, d, coef.data_ptr(), x.data_ptr(), y.data_ptr(), ws.data_ptr(), nws)
        torch.cuda.synchronize()
        assert np.abs(y.cpu().numpy() - ref).max() < tol * scale, (N, prec)


@pytest.mark.parametrize("N", [25, 81])
def test_slab_pass_on_transforms_as_long_as_the_data(hb, solver, N):
    """GaNi on N = 25 and 81: every frequency of the slab's transforms is kept. The FP64 inner
    CG (separate passes) solves the same cell: 1e-6, the bar of the mixed GaNi tests (an energy
    error of order tol^2 and the FP32 floor of the inner residual, refined in FP64)."""
    p = ms.random_spheres_3d(2, N=N, n_balls=6, phi=0.25, contrast=30.0)
    ref = solver(p, precision=hb.HOM_FP64, tol=1e-9, discretization=1)
    out = solver(p, precision=hb.HOM_MIXED, tol=1e-7, discretization=1)
    for key in ("gani_A", "gani_B", "upper", "lower"):
        assert np.abs(out[key] - ref[key]).max() <= 1e-6 * np.linalg.norm(ref[key]), key


@pytest.mark.parametrize("batch,cfg", [
    (1, dict(N=15, cin=1, width=7, modes=1, layers=1, proj=9, cout=5)),           # no vector stores, two row copies
    (5, dict(N=23, cin=2, width=40, modes=5, layers=2, proj=70, cout=8)),         # columns over several tiles
    (3, dict(N=81, cin=1, width=5, modes=3, layers=2, proj=16, cout=8)),          # inner length over a staged chunk
    (2, dict(N=135, cin=1, width=12, modes=33, layers=1, proj=20, cout=8)),       # rows over one tile, split sums
    (70, dict(N=9, cin=1, width=16, modes=2, layers=2, proj=32, cout=8)),         # mixing rows over a half tile
    (2, dict(N=11, cin=1, width=33, modes=3, layers=1, proj=33, cout=18, d=3)),   # odd columns in 3D
], ids=lambda v: str(v) if isinstance(v, int) else f"N{v['N']}w{v['width']}")
def test_network_products_match_cpu_reference(hb, batch, cfg):
    """Output 2e-2 and gradients 5e-2 of each tensor's largest entry against float64: BF16
    operands (2^-9 each) through up to eight products in a row, the bars of the network's tests."""
    ctx = hb.hom_create(0)
    try:
        c = hb.binding.net_config(**cfg)
        npar, wsb = hb.binding.hom_net_sizes(ctx, c, batch)
        grid = (batch,) + (cfg["N"],) * cfg.get("d", 2)
        params = torch.empty(npar, dtype=torch.float32, device="cuda")
        hb.binding.hom_net_init(ctx, c, 5, params.data_ptr())
        g = torch.Generator().manual_seed(cfg["N"])
        x = torch.randn(grid + (cfg["cin"],), generator=g, dtype=torch.float64)
        t = torch.randn(grid + (cfg["cout"],), generator=g, dtype=torch.float64) * 0.1
        ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
        out = torch.empty(grid + (cfg["cout"],), dtype=torch.float32, device="cuda")
        dx, dt = x.float().cuda(), t.float().cuda()
        hb.binding.hom_net_forward(ctx, c, params.data_ptr(), batch, dx.data_ptr(), out.data_ptr(), ws.data_ptr(), wsb)
        grad = torch.empty_like(params)
        loss = hb.binding.hom_net_gradient(ctx, c, params.data_ptr(), batch, dx.data_ptr(), dt.data_ptr(),
                                           grad.data_ptr(), ws.data_ptr(), wsb)
        rloss, rgrad, rout = fno.loss_and_grad(cfg, params.cpu().double(), x, t)
        assert (out.cpu().double() - rout).abs().max() <= 2e-2 * rout.abs().max()
        assert abs(loss - rloss) <= 2e-2 * rloss
        G = grad.cpu().double()
        for name, val in fno.offsets(**cfg).items():
            if name == "total":
                continue
            s, n = val
            scale = max(rgrad[s:s + n].abs().max().item(), 1e-12)
            assert (G[s:s + n] - rgrad[s:s + n]).abs().max().item() <= 5e-2 * scale, name
    finally:
        hb.hom_destroy(ctx)


@pytest.mark.parametrize("cells", [1, 3, 40, 160])
def test_default_batch_launch_matches_one_cta_a_cell(hb, solver, cells):
    """The threads and CTAs a cell gets by default follow the batch's size. FP64 at tol 1e-12:
    1e-10 of one CTA of 256 threads for each (bounds are quadratic in the residual; what is left
    is the rounding of differently grouped sums)."""
    probs = [ms.random_rectangles_2d(s, N=(9, 15, 23, 41)[s % 4]) for s in range(cells)]
    base = solver.batched(probs, precision=hb.HOM_FP64, tol=1e-12)
    try:
        hb.binding.hom_set_batch_threads(solver.ctx, 256)
        hb.binding.hom_set_batch_cluster(solver.ctx, 1, 225)
        one = solver.batched(probs, precision=hb.HOM_FP64, tol=1e-12)
    finally:
        hb.binding.hom_set_batch_threads(solver.ctx, 0)
        hb.binding.hom_set_batch_cluster(solver.ctx, 0, 0)
    assert (base["status"] == one["status"]).all()
    for i in range(cells):
        for key in ("upper", "lower"):
            assert np.abs(base[key][i] - one[key][i]).max() <= 1e-10 * np.linalg.norm(one[key][i]), (i, key)


@pytest.mark.parametrize("N", [(16, 16), (48, 32), (80, 13), (64, 96), (16, 12, 32)])
@pytest.mark.parametrize("arith", [0, 2])
def test_mixed_gani_on_grids_with_powers_of_two(hb, solver, N, arith):
    """GaNi transforms as long as an even grid, whose float-float residuals have factors 16 and
    more: the FP64 solve to 1e-6 (the bar of the mixed GaNi tests), by default and with every
    residual in float-float."""
    d = len(N)
    p = ms.make_problem(d, N, 1.0, 1.0, [ms.box((0.1, 0.05, 0.0)[:d], (0.3, 0.2, 0.5)[:d], 20.0, d),
                                         ms.ball((-0.25, -0.2, 0.1)[:d], 0.12, 0.2, d)])
    ref = solver(p, precision=hb.HOM_FP64, tol=1e-9, discretization=1)
    hb.binding.hom_set_refine_arith(solver.ctx, arith)
    try:
        out = solver(p, precision=hb.HOM_MIXED, tol=1e-7, discretization=1)
    finally:
        hb.binding.hom_set_refine_arith(solver.ctx, 0)
    assert out["status"] == 0
    for key in ("gani_A", "gani_B", "upper", "lower"):
        assert np.abs(out[key] - ref[key]).max() <= 1e-6 * np.linalg.norm(ref[key]), key


@pytest.mark.parametrize("N", [5, 13, 41, 113])
def test_slab_pass_warp_counts(hb, solver, N):
    """Every count of warps a CTA that can be asked for (at M = 225 the automatic one in place of 20)
    computes the operator of the separate passes: 2e-6 of the largest entry, the bar of the slab test."""
    p = ms.random_spheres_3d(7, N=N, n_balls=5, phi=0.2, contrast=100.0)
    info = hb.hom_problem_info(solver.ctx, p)
    nws = hb.hom_step_workspace_size(solver.ctx, p, 3)
    ws = torch.empty(nws, dtype=torch.uint8, device="cuda")
    coef = torch.empty((info["ncomp"],) + tuple(info["M"][::-1]), dtype=torch.float32, device="cuda")
    hb.hom_coefficient(solver.ctx, p, 0, hb.HOM_FP32, coef.data_ptr(), ws.data_ptr(), nws)
    x = torch.randn((3, 3, N, N, (N + 1) // 2), generator=torch.Generator().manual_seed(N), dtype=torch.complex64).cuda()
    out = {}
    try:
        for slab in (0, 1, 4, 8, 12, 16, 20):
            hb.hom_set_slab_pass(solver.ctx, slab)
            y = torch.zeros_like(x)
            hb.hom_matvec(solver.ctx, p, 0, hb.HOM_FP32, 1, 3, coef.data_ptr(), x.data_ptr(), y.data_ptr(), ws.data_ptr(), nws)
            torch.cuda.synchronize()
            out[slab] = y
    finally:
        hb.hom_set_slab_pass(solver.ctx, 1)
    for slab, y in out.items():
        assert (y - out[0]).abs().max() <= 2e-6 * out[0].abs().max(), slab


# the packed row pass past 48 KB: two planes a double pencil, three and four, a plane alone; the
# unpacked one: a single pair of rows, no double pencil in 110 KB, three pairs of three rows
@pytest.mark.parametrize("N,aniso", [((521, 81), True), ((521, 161), False), ((527, 305), True), ((521, 9), False),
                                     ((1175, 5), True), ((1001, 79), False), ((221, 5, 5), True), ((405, 3, 5), False),
                                     ((441, 5, 3), True), ((441, 9, 9), True), ((527, 9, 7), False)])
def test_long_rows_match_oracle(hb, solver, N, aniso):
    """FP32 operator: 5e-6 of the largest entry, the bar of the operator's step tests."""
    d = len(N)
    A0, A1 = (((A2, A2 @ A2) if d == 2 else (A3, A3 @ A3)) if aniso else (1.0, 20.0))
    p = ms.make_problem(d, N, (1.0, 0.7, 1.2)[:d], A0, [ms.box((0.1, 0.05, 0.0)[:d], (0.3, 0.2, 0.5)[:d], A1, d),
                                                        ms.ball((-0.25, -0.2, 0.1)[:d], 0.12, 0.2, d)])
    rng = np.random.default_rng([zlib.crc32(b"long"), *N])
    op = matfree.MatFreeOperator(p, "primal")
    info = hb.hom_problem_info(solver.ctx, p)
    nws = hb.hom_step_workspace_size(solver.ctx, p, d)
    ws = torch.empty(nws, dtype=torch.uint8, device="cuda")
    fields = [random_real_field(rng, d, N) for _ in range(d)]
    ref = np.stack([full_to_half(op.apply(u, project=True), d) for u in fields])
    x = torch.from_numpy(np.stack([full_to_half(u, d) for u in fields]).astype(np.complex64)).cuda()
    coef = torch.empty((info["ncomp"],) + tuple(info["M"][:d][::-1]), dtype=torch.float32, device="cuda")
    hb.hom_coefficient(solver.ctx, p, 0, hb.HOM_FP32, coef.data_ptr(), ws.data_ptr(), nws)
    y = torch.zeros_like(x)
    hb.hom_matvec(solver.ctx, p, 0, hb.HOM_FP32, 1, d, coef.data_ptr(), x.data_ptr(), y.data_ptr(), ws.data_ptr(), nws)
    torch.cuda.synchronize()
    scale = max(np.abs(ref).max(), x.abs().max().item())
    assert np.abs(y.cpu().numpy() - ref).max() < 5e-6 * scale


# full and partial tiles, K over one chunk, a ragged last chunk, strides that allow no vector loads
@pytest.mark.parametrize("M,N,K,pad", [(128, 64, 64, 0), (128, 64, 128, 0), (256, 128, 192, 1), (200, 70, 100, 0), (129, 65, 65, 3),
                                       (40, 24, 333, 0), (384, 192, 250, 4), (3, 2, 700, 0), (700, 64, 63, 2)])
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_gemm_tiles(hb, solver, M, N, K, pad, ta, tb):
    """The BF16 product against the same rounded operands in FP64: FP32 sums of K terms, at most
    K 2^-23 of the sum of the terms' magnitudes."""
    g = torch.Generator().manual_seed(M + N + K)
    A = torch.randn((K, M) if ta else (M, K), generator=g)
    B = torch.randn((N, K) if tb else (K, N), generator=g)
    dA, dB = (torch.nn.functional.pad(t, (0, pad)).cuda() for t in (A, B))
    C = torch.full((M, N + pad), 7.0, device="cuda")
    hb.binding.hom_gemm_bf16(solver.ctx, M, N, K, dA.data_ptr(), dA.shape[1], ta, dB.data_ptr(), dB.shape[1], tb, C.data_ptr(),
                             N + pad)
    torch.cuda.synchronize()
    a, b = (t.bfloat16().double() for t in (A.T if ta else A, B.T if tb else B))
    err = (C[:, :N].cpu().double() - a @ b).abs()
    assert (err <= K * 2.0 ** -23 * (a.abs() @ b.abs())).all()
    assert (C[:, N:] == 7.0).all()
