"""GPU parity: mwu_gemm / mwu_conv_implicit through the C ABI against the CPU checker.

Tolerances: bf16 output -- relative Frobenius error <= 2e-3 and max element error
<= 1e-2 * max|y| (output rounding alone is about 1.5e-3); fp32 output -- 1e-5 relative
Frobenius, so that an indexing or decode mistake cannot hide under output rounding.
"""
import numpy as np
import pytest
import torch

import packed_format as F
from oracle import mwu_oracle as O
from paper_2106_08301_b200 import binding as B
from paper_2106_08301_b200 import inputs

pytestmark = pytest.mark.gpu


def project_and_pack(W, b, ku, kp):
    rows, cols = W.shape
    desc = B.make_desc(rows, cols, b, ku, kp)
    bufs = B.ProjectionBuffers(desc, want_q=False)
    Wd = W.cuda().contiguous()
    bufs.project(Wd)
    packed = bufs.pack(Wd)
    torch.cuda.synchronize()
    assert int(bufs.dev_status.item()) == 0
    p = O.project(W.numpy(), b, ku, kp)
    return desc, bufs, packed, p


def errors(Y, ref):
    Y = Y.astype(np.float64)
    fro = np.linalg.norm(Y - ref) / max(np.linalg.norm(ref), 1e-300)
    mx = np.abs(Y - ref).max() / max(np.abs(ref).max(), 1e-300)
    return fro, mx


def run_gemm(desc, bufs, packed, X, y_dtype, ldy=None):
    M = X.shape[0]
    N = desc.rows
    ldy = ldy or N
    Y = torch.full((M, ldy), float("nan"), dtype=torch.float32 if y_dtype else torch.bfloat16, device="cuda")
    Xd = X.cuda().contiguous()
    B.mwu_gemm(desc, packed, Xd, M, X.shape[1], Y, ldy, y_dtype, bufs.dev_status)
    torch.cuda.synchronize()
    assert int(bufs.dev_status.item()) == 0
    return Y.float().cpu().numpy()[:, :N]


def check_gemm(W, b, ku, kp, M, seed=0):
    desc, bufs, packed, p = project_and_pack(W, b, ku, kp)
    X = inputs.normal_activations_bf16((M, W.shape[1]), 4242 + seed)
    What = O.decoded_weights(p, b)
    ref = O.gemm(X.to(torch.float64).numpy(), What)
    Y32 = run_gemm(desc, bufs, packed, X, 1)
    fro, mx = errors(Y32, ref)
    assert fro <= 1e-5, (fro, mx)
    Y16 = run_gemm(desc, bufs, packed, X, 0)
    fro, mx = errors(Y16, ref)
    assert fro <= 2e-3 and mx <= 1e-2, (fro, mx)
    return desc, bufs, packed, p


def test_gemm_config1_linear():
    wl = inputs.WORKLOADS["c1_linear"]
    Mb = wl.n_blocks
    check_gemm(wl.weights(), wl.block, B.mwu_count_from_permille(Mb, wl.unified_permille),
               B.mwu_count_from_permille(Mb, wl.pruned_permille), wl.m)


@pytest.mark.parametrize("b", [2, 4, 8, 16])
def test_gemm_block_widths_and_ragged_shapes(b):
    # N = 384 -> three 128-row weight tiles (an odd count: last CTA tile has one record);
    # M = 300 -> ragged last row tile; K = 192 -> three stages
    W = inputs.normal_weights(384, 192, 0.02, 50 + b)
    Mb = W.numel() // b
    check_gemm(W, b, Mb * 6 // 10, Mb * 3 // 10, 300, seed=b)


def test_gemm_ragged_weight_rows():
    W = inputs.normal_weights(200, 128, 0.02, 61)       # N not a multiple of 128, single CTA tile
    Mb = W.numel() // 8
    check_gemm(W, 8, Mb // 2, Mb // 4, 130)
    W = inputs.normal_weights(72, 64, 0.02, 62)         # one record, N = 72
    check_gemm(W, 4, 100, 50, 5)


def test_gemm_all_classes_degenerate():
    W = inputs.normal_weights(256, 256, 0.02, 63)
    Mb = W.numel() // 16
    check_gemm(W, 16, 0, 0, 64)            # all dense: an ordinary GEMM
    check_gemm(W, 16, Mb, 0, 64)           # all unified
    check_gemm(W, 16, Mb, Mb, 64)          # all pruned: exactly zero, every stage skipped
    desc, bufs, packed, p = project_and_pack(W, 16, Mb, Mb)
    X = inputs.normal_activations_bf16((64, 256), 1)
    assert np.all(run_gemm(desc, bufs, packed, X, 0) == 0)


def test_gemm_skips_dead_stages_and_slices():
    """Structured pruning: whole 64-column stages and single 16-column slices are zero in every
    row, so the kernel's skip paths run; results must not change."""
    W = inputs.normal_weights(256, 512, 0.02, 64)
    W[:, 64:192] = 0.0                  # stages 1 and 2 dead in every tile
    W[:, 272:288] = 0.0                 # slice 1 of stage 4 dead
    W[:128, 448:512] = 0.0              # stage 7 dead in the first row tile only (not skippable with 2-tile CTAs)
    b = 16
    Mb = W.numel() // b
    n_zero = int((W.reshape(-1, b).abs().sum(dim=1) == 0).sum())
    desc, bufs, packed, p = check_gemm(W, b, n_zero + 500, n_zero, 200)
    rec = F.records(packed.cpu().numpy())
    assert rec[1, 3] == 0 and rec[2, 3] == 0 and rec[8 + 1, 3] == 0 and rec[4, 3] == 0b1101


def test_gemm_output_leading_dimension():
    W = inputs.normal_weights(256, 128, 0.02, 65)
    desc, bufs, packed, p = project_and_pack(W, 8, 2000, 1000)
    X = inputs.normal_activations_bf16((100, 128), 3)
    ref = O.gemm(X.to(torch.float64).numpy(), O.decoded_weights(p))
    Y = run_gemm(desc, bufs, packed, X, 1, ldy=264)
    assert errors(Y, ref)[0] <= 1e-5


def test_gemm_argument_errors():
    W = inputs.normal_weights(128, 64, 0.02, 66)
    desc, bufs, packed, p = project_and_pack(W, 4, 100, 50)
    X = inputs.normal_activations_bf16((16, 64), 3).cuda()
    Y = torch.empty((16, 128), dtype=torch.bfloat16, device="cuda")
    assert B.mwu_gemm(desc, packed, X, 16, 60, Y, 128, 0, bufs.dev_status, check=False) == 2   # ldx < cols
    assert B.mwu_gemm(desc, packed, X, 16, 64, Y, 100, 0, bufs.dev_status, check=False) == 2   # ldy < rows
    assert B.mwu_gemm(desc, packed, X, 16, 64, Y, 132, 0, bufs.dev_status, check=False) == 3   # ldy % 8
    assert B.mwu_gemm(desc, packed, X, 16, 64, Y, 128, 7, bufs.dev_status, check=False) == 1
    assert B.mwu_gemm(desc, packed, X, 0, 64, Y, 128, 0, bufs.dev_status, check=False) == 0    # no-op


def test_gemm_config3_shape_reduced_rows():
    """1x1 conv as GEMM (K = 256, N = 1024) on a reduced M, every output compared (the full
    M = 200704 runs in test_gpu_decode_once.py on sampled rows)."""
    wl = inputs.WORKLOADS["c3_conv1x1"]
    Mb = wl.n_blocks
    check_gemm(wl.weights(), wl.block, B.mwu_count_from_permille(Mb, wl.unified_permille),
               B.mwu_count_from_permille(Mb, wl.pruned_permille), 1000)


def conv_case(W, b, ku, kp, x, kh, kw, stride, pad, expect_ws=None):
    """Both entry points: mwu_conv_implicit (decode fused into the kernel) and mwu_conv_implicit_ws
    (weights expanded once into a workspace; falls back to the first for shapes it does not serve)."""
    desc, bufs, packed, p = project_and_pack(W, b, ku, kp)
    n, c, h, w = x.shape
    oh = (h + 2 * pad - kh) // stride + 1
    ow = (w + 2 * pad - kw) // stride + 1
    ref = O.conv2d_direct(x.to(torch.float64).numpy(), O.decoded_weights(p), kh, kw, stride, pad)
    xd = x.cuda().contiguous()
    ws_bytes = B.mwu_conv_workspace_bytes(desc, n, c, h, w, kh, kw, stride, pad)
    if expect_ws is not None:
        assert (ws_bytes > 0) == expect_ws
    ws = torch.empty(ws_bytes, dtype=torch.uint8, device="cuda") if ws_bytes else None
    for use_ws in (False, True):
        for y_dtype, tol in [(1, 1e-5), (0, 2e-3)]:
            Y = torch.full((n, W.shape[0], oh, ow), float("nan"),
                           dtype=torch.float32 if y_dtype else torch.bfloat16, device="cuda")
            if use_ws:
                B.mwu_conv_implicit_ws(desc, packed, xd, n, c, h, w, kh, kw, stride, pad, Y, y_dtype, ws,
                                       bufs.dev_status)
            else:
                B.mwu_conv_implicit(desc, packed, xd, n, c, h, w, kh, kw, stride, pad, Y, y_dtype, bufs.dev_status)
            torch.cuda.synchronize()
            assert int(bufs.dev_status.item()) == 0
            fro, mx = errors(Y.float().cpu().numpy(), ref)
            assert fro <= tol and mx <= 1e-2, (use_ws, y_dtype, fro, mx)
    return desc, bufs, packed, p, xd, ref


def test_conv_small_cases():
    # 3x3 s1 p1, K = 64*9 = 576; M = 2*9*7 = 126 (ragged)
    W = inputs.normal_weights(128, 576, 0.05, 70)
    x = inputs.normal_activations_bf16((2, 64, 9, 7), 71)
    Mb = W.numel() // 4
    conv_case(W, 4, Mb * 6 // 10, Mb * 3 // 10, x, 3, 3, 1, 1)
    # stride 2, no padding, 256 filters (two records per CTA tile), b = 16
    W = inputs.normal_weights(256, 576, 0.05, 72)
    Mb = W.numel() // 16
    conv_case(W, 16, Mb // 2, Mb // 4, x, 3, 3, 2, 0)
    # 1x1 convolution equals a GEMM over channels
    W = inputs.normal_weights(128, 64, 0.05, 73)
    conv_case(W, 8, 300, 100, x, 1, 1, 1, 0)


@pytest.mark.parametrize("filters,cin,h,w,k,pad,b", [(128, 64, 13, 12, 3, 1, 4),     # second tile of an image has 3 of 10 rows
                                                     (256, 128, 28, 28, 3, 1, 16),   # two filter tiles, two channel chunks, 4-row tiles
                                                     (200, 64, 9, 11, 5, 2, 8),      # 5x5 taps, filters ragged inside a tile
                                                     (128, 64, 10, 10, 3, 0, 2),     # no padding: 8x8 output
                                                     (128, 192, 6, 40, 1, 0, 8)])    # 1x1, three channel chunks, 3-row tiles
def test_conv_workspace_path_shapes(filters, cin, h, w, k, pad, b):
    W = inputs.normal_weights(filters, cin * k * k, 0.05, 740 + filters + cin + k)
    x = inputs.normal_activations_bf16((3, cin, h, w), 741 + h)
    Mb = W.numel() // b
    conv_case(W, b, Mb * 6 // 10, Mb * 3 // 10, x, k, k, 1, pad, expect_ws=True)


def test_conv_workspace_path_declines_other_shapes():
    x = inputs.normal_activations_bf16((2, 64, 9, 7), 71)
    W = inputs.normal_weights(128, 576, 0.05, 72)
    d = B.make_desc(128, 576, 16, 1000, 500)
    assert B.mwu_conv_workspace_bytes(d, 2, 64, 9, 7, 3, 3, 2, 0) == 0          # stride 2
    assert B.mwu_conv_workspace_bytes(d, 2, 64, 9, 200, 3, 3, 1, 1) == 0        # 200 output pixels per row
    assert B.mwu_conv_workspace_bytes(d, 2, 64, 9, 7, 3, 3, 1, 1) > 0
    d2 = B.make_desc(128, 288, 16, 500, 200)                                     # 32 channels
    assert B.mwu_conv_workspace_bytes(d2, 2, 32, 9, 7, 3, 3, 1, 1) == 0


def test_bounded_wait_runs_out_and_the_context_stays_usable():
    """Every wait of a kernel on its own barriers has a limit.  Here the producer of the convolution
    kernel leaves one stage's loads out (a barrier that nothing completes) and the limit is cut to
    about a millisecond: the kernel must come back by itself with MWU_DEV_TIMEOUT set, and the next
    call on the same stream must give the right result."""
    W = inputs.normal_weights(128, 576, 0.05, 760)
    x = inputs.normal_activations_bf16((4, 64, 8, 8), 761)
    Mb = W.numel() // 4
    desc, bufs, packed, p = project_and_pack(W, 4, Mb // 2, Mb // 4)
    ref = O.conv2d_direct(x.to(torch.float64).numpy(), O.decoded_weights(p), 3, 3, 1, 1)
    xd = x.cuda()
    ws = torch.empty(B.mwu_conv_workspace_bytes(desc, 4, 64, 8, 8, 3, 3, 1, 1), dtype=torch.uint8, device="cuda")
    assert ws.numel() > 0
    Y = torch.zeros((4, 128, 8, 8), dtype=torch.float32, device="cuda")
    B.mwu_debug_conv_wait(2_000_000, 3)                  # ~1 ms; the fourth stage of every CTA never arrives
    try:
        B.mwu_conv_implicit_ws(desc, packed, xd, 4, 64, 8, 8, 3, 3, 1, 1, Y, 1, ws, bufs.dev_status)
        torch.cuda.synchronize()
    finally:
        B.mwu_debug_conv_wait(0, -1)
    assert int(bufs.dev_status.item()) & B.MWU_DEV_TIMEOUT
    bufs.dev_status.zero_()
    B.mwu_conv_implicit_ws(desc, packed, xd, 4, 64, 8, 8, 3, 3, 1, 1, Y, 1, ws, bufs.dev_status)
    torch.cuda.synchronize()
    assert int(bufs.dev_status.item()) == 0
    assert errors(Y.cpu().numpy(), ref)[0] <= 1e-5


def test_conv_config2():
    wl = inputs.WORKLOADS["c2_conv3x3"]
    Mb = wl.n_blocks
    x = wl.activations()
    n, c, h, w, kh, kw, stride, pad = wl.conv
    conv_case(wl.weights(), wl.block, B.mwu_count_from_permille(Mb, wl.unified_permille),
              B.mwu_count_from_permille(Mb, wl.pruned_permille), x, kh, kw, stride, pad)


@pytest.mark.parametrize("b", [2, 4, 8, 16])
def test_gemm_few_stages(b):
    """The streaming kernel: M = 900 leaves a ragged last tile of eight, K = 320 gives five stages."""
    W = inputs.normal_weights(512, 320, 0.02, 80 + b)
    Mb = W.numel() // b
    check_gemm(W, b, Mb * 7 // 10, Mb * 4 // 10, 900, seed=20 + b)


def test_gemm_dead_stages_and_all_pruned():
    """The streaming kernel over several tiles of activation rows."""
    W = inputs.normal_weights(512, 512, 0.02, 90)
    W[:, 128:256] = 0.0                 # stages 2 and 3 dead in every record
    W[:256, 448:464] = 0.0              # one dead slice in the first two weight tiles only
    b = 16
    Mb = W.numel() // b
    n_zero = int((W.reshape(-1, b).abs().sum(dim=1) == 0).sum())
    check_gemm(W, b, n_zero + 700, n_zero, 1030)
    check_gemm(W, b, Mb, Mb, 600)       # everything pruned: zeros, no MMA issued at all
    check_gemm(W, b, 0, 0, 513)         # everything dense


def assert_fused(rows, cols, M):
    """Too many record decodes for the streaming kernel (nine an SM), too long a reduction for the one that keeps the weights:
    without a workspace the fused kernels multiply."""
    assert cols > 256 and M > 640
    assert -(-rows // 128) * -(-M // 128) * (cols // 64) > 9 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("b", [2, 4, 8, 16])
@pytest.mark.parametrize("rows,cols,M", [(512, 320, 9000),       # pairs of CTAs: five stages (more than the four slots), a ragged last tile
                                         (512, 1024, 2900),      # ... sixteen stages
                                         (640, 1024, 2300),      # a CTA to a tile: an odd number of record tiles
                                         (1000, 1024, 2100),     # ... weight rows that end inside a tile
                                         (128, 1024, 11000)])    # ... one record tile
def test_gemm_fused_tiles(rows, cols, M, b):
    assert_fused(rows, cols, M)
    W = inputs.normal_weights(rows, cols, 0.02, 80 + b)
    Mb = W.numel() // b
    check_gemm(W, b, Mb * 7 // 10, Mb * 4 // 10, M, seed=20 + b)


@pytest.mark.parametrize("rows,M", [(512, 5500), (640, 4500)])         # pairs of CTAs, a CTA to a tile
def test_gemm_fused_tiles_dead_stages_and_all_pruned(rows, M):
    assert_fused(rows, 512, M)
    W = inputs.normal_weights(rows, 512, 0.02, 90)
    W[:, 128:256] = 0.0                 # stages 2 and 3 dead in every record
    W[:256, 448:464] = 0.0              # one dead slice in the first tile only
    b = 16
    Mb = W.numel() // b
    n_zero = int((W.reshape(-1, b).abs().sum(dim=1) == 0).sum())
    check_gemm(W, b, n_zero + 700, n_zero, M)
    check_gemm(W, b, Mb, Mb, M)         # everything pruned: zeros, no MMA issued at all
    check_gemm(W, b, 0, 0, M)           # everything dense


@pytest.mark.parametrize("K,b", [(256, 8), (192, 16)])
def test_gemm_short_reduction_two_weight_tiles(K, b):
    """Small reduction, many activation rows: half of the CTAs keep one weight tile, half the other, and walk the activation
    tiles (K = 256: one store box a warp, K = 192: two)."""
    W = inputs.normal_weights(512, K, 0.02, 95 + b)
    Mb = W.numel() // b
    check_gemm(W, b, Mb * 3 // 4, Mb // 2, 77000 + 37, seed=31 + b)


@pytest.mark.parametrize("b,rows,cols,M,ku,kp", [(2, 136, 64, 1, 7, 3),           # one stage, one row, a padded weight tile
                                                 (2, 128, 320, 16, 10, 0),        # every block unified: the longest u lists
                                                 (4, 200, 448, 17, 0, 0),         # every block dense: the longest payloads
                                                 (8, 384, 1088, 48, 6, 3),        # 17 stages over a cluster, the last CTA with fewer
                                                 (16, 256, 2304, 128, 8, 6),      # the most rows of one CTA
                                                 (16, 1000, 4096, 65, 9, 8),
                                                 (4, 128, 192, 100, 10, 10)])     # everything pruned: no MMA at all
def test_gemm_few_rows(b, rows, cols, M, ku, kp):
    """Few activation rows: the streaming kernel, with and without dead stages (ku, kp in tenths)."""
    W = inputs.normal_weights(rows, cols, 0.02, 300 + b)
    if cols > 256 and kp < ku:
        W[:, 64:144] = 0.0                       # a dead stage and a dead slice wherever blocks of zeros are pruned
    Mb = W.numel() // b
    check_gemm(W, b, Mb * ku // 10, Mb * kp // 10, M, seed=40 + b)


def uneven_weights(rows, cols, seed, balanced=False):
    """Each run of 64 columns on a scale of its own, from 1e-4 to 30; balanced: a quarter of them on each."""
    gen = torch.Generator().manual_seed(seed)
    W = torch.randn(rows, cols, generator=gen) * 0.02
    which = torch.randperm(cols // 64, generator=gen) % 4 if balanced else torch.randint(0, 4, (cols // 64,), generator=gen)
    return W * torch.tensor([0.0001, 1.0, 30.0, 0.01])[which].repeat_interleave(64)[None, :]


@pytest.mark.parametrize("b,M,pr,un", [(16, 20, 4, 7), (16, 3, 1, 2), (16, 100, 6, 9), (8, 20, 4, 7), (4, 5, 3, 6), (2, 17, 3, 6)])
def test_gemm_few_rows_uneven_records(b, M, pr, un):
    """Records that differ, in runs of nine stages or less: dead ones, nearly empty ones, all-dense and all-unified ones that
    need several batches (pr, un in tenths)."""
    rows, cols = 296, 64 * 70
    W = uneven_weights(rows, cols, b * 100 + M)
    Mb = W.numel() // b
    check_gemm(W, b, Mb * un // 10, Mb * pr // 10, M)


@pytest.mark.parametrize("b,M,pr,un", [(16, 20, 4, 7), (16, 100, 5, 8), (8, 20, 4, 7), (4, 5, 3, 6), (2, 128, 3, 6)])
def test_gemm_few_rows_long_runs(b, M, pr, un):
    """Runs of 65 stages: fp32 results of more than 6912 columns are summed in two pieces at most.  Dead stages among the
    first 32 and behind them, so that the list of the live ones is closed up over several rounds, and at least six records to a
    decode group, so that every way of clearing a tile follows every other."""
    rows, cols = 296, 64 * 130
    W = uneven_weights(rows, cols, b * 100 + M, balanced=True)
    Mb = W.numel() // b
    _, _, packed, _ = check_gemm(W, b, Mb * un // 10, Mb * pr // 10, M)
    live = F.records(packed.cpu().numpy())[:3 * 130, 3].reshape(3, 2, 65) != 0
    assert (live.sum(axis=2) >= 6 * 5).all()
    assert not live[:, :, :32].all(axis=2).any() and not live[:, :, 32:].all(axis=2).any()


@pytest.mark.parametrize("rows,cols,b,M", [(96, 128, 8, 37900),          # one record tile: half a tile of outputs
                                           (640, 192, 4, 12801),         # five record tiles, a ragged last row, two boxes a warp
                                           (1000, 256, 2, 9604),         # ragged weight rows; one box a warp
                                           (16384, 64, 16, 620),         # 64 weight tiles: CTAs change weights on the way
                                           (128, 64, 4, 37888),          # exactly two tiles an SM, the fewest
                                           (264, 256, 16, 20000)])
def test_gemm_short_reduction(rows, cols, b, M):
    """Weights kept in shared memory: at least two tiles of 128 x 256 outputs an SM, with dead stages and slices where there is room."""
    W = inputs.normal_weights(rows, cols, 0.02, 500 + b)
    if cols > 128:
        W[:, 64:144] = 0.0                       # a dead stage and a dead slice
    Mb = W.numel() // b
    assert -(-rows // 256) * -(-M // 128) >= 2 * torch.cuda.get_device_properties(0).multi_processor_count
    desc, bufs, packed, p = check_gemm(W, b, Mb * 7 // 10, Mb // 2, M, seed=60 + b)
    # gaps behind the rows of X and Y; what lies in them is neither read nor written
    X = inputs.normal_activations_bf16((M, cols + 8), 4243)
    X[:, cols:] = float("nan")
    ref = O.gemm(X[:, :cols].to(torch.float64).numpy(), O.decoded_weights(p, b))
    for dtype, tol in ((torch.bfloat16, 2e-3), (torch.float32, 1e-5)):
        Y = torch.full((M, rows + 8), float("nan"), dtype=dtype, device="cuda")
        B.mwu_gemm(desc, packed, X.cuda(), M, cols + 8, Y, rows + 8, int(dtype == torch.float32), bufs.dev_status)
        assert int(bufs.dev_status.item()) == 0
        assert bool(torch.isnan(Y[:, rows:]).all())
        assert errors(Y[:, :rows].float().cpu().numpy(), ref)[0] <= tol


@pytest.mark.parametrize("rows,cols,M,fp32", [(64, 64, 100352, 0),        # one store a tile
                                              (192, 192, 40000, 0),       # one in the second half of a tile
                                              (2248, 128, 17000, 0),      # weight rows end 8 columns into a box of 64
                                              (200, 192, 38000, 1),       # three stores of 32 columns, the last of 8
                                              (1064, 128, 12000, 1),      # two, the second of 8
                                              (1056, 128, 12000, 1)])     # one
def test_gemm_short_reduction_odd_stores(rows, cols, M, fp32):
    """Output that leaves through two boxes of shared memory, an odd number of stores to a tile: every value, several times."""
    b = 8
    W = inputs.normal_weights(rows, cols, 0.02, 900 + rows)
    Mb = W.numel() // b
    desc, bufs, packed, p = project_and_pack(W, b, Mb // 2, Mb // 4)
    X = inputs.normal_activations_bf16((M, cols), 901 + rows)
    What = O.decoded_weights(p, b)
    Xf = X.to(torch.float64).numpy()
    ref = O.gemm(Xf, What)
    # rounding to bf16, 2^-8 of the value, and what each of `cols` fp32 additions may drop, 2^-23 of the sum's magnitude
    bound = (0.0 if fp32 else 2.0 ** -8) * np.abs(ref) + cols * 2.0 ** -22 * O.gemm(np.abs(Xf), np.abs(What))
    Xd, first = X.cuda(), None
    for _ in range(5):
        Y = torch.full((M, rows), float("nan"), dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
        B.mwu_gemm(desc, packed, Xd, M, cols, Y, rows, fp32, bufs.dev_status)
        assert int(bufs.dev_status.item()) == 0
        if first is None:
            first = Y
            assert (np.abs(Y.double().cpu().numpy() - ref) <= bound).all()
        assert torch.equal(Y, first)


@pytest.mark.parametrize("rows,cols,M,first_live", [(1024, 256, 12000, 1024),     # two stages dead everywhere
                                                    (1024, 256, 12000, 256),      # ... dead in the first weight tile only
                                                    (5000, 256, 2000, 4864),      # ... alive in the 153rd record and later
                                                    (33000, 256, 390, 33000),     # dead everywhere, more than 1024 records
                                                    (520, 192, 13000, 0)])        # everything pruned
def test_gemm_short_reduction_dead_stages(rows, cols, M, first_live):
    """Stages that no weight tile multiplies, or only some do."""
    b = 16
    W = inputs.normal_weights(rows, cols, 0.02, 950)
    W[:first_live, 64:192] = 0.0
    Mb = W.numel() // b
    zero = first_live * 128 // b
    desc, bufs, packed, p = project_and_pack(W, b, zero + (Mb - zero) // 2 if first_live else Mb, zero if first_live else Mb)
    X = inputs.normal_activations_bf16((M, cols), 951)
    ref = O.gemm(X.to(torch.float64).numpy(), O.decoded_weights(p, b))
    assert errors(run_gemm(desc, bufs, packed, X, 0), ref)[0] <= 2e-3
    assert errors(run_gemm(desc, bufs, packed, X, 1), ref)[0] <= 1e-5


@pytest.mark.parametrize("b", [2, 4, 8, 16])
@pytest.mark.parametrize("pr,un", [(0, 0), (0, 10), (3, 6)])
def test_gemm_short_reduction_uneven_records(b, pr, un):
    """Records of every filling, several rounds of either list or of both: all dense, all unified, and a mixture of empty, nearly
    empty and full ones (pr, un in tenths)."""
    rows, cols, M = 904, 192, 9600
    gen = torch.Generator().manual_seed(b + pr)
    W = torch.randn(rows, cols, generator=gen) * 0.02
    if pr:
        W *= torch.tensor([0.0001, 1.0, 30.0, 0.01])[torch.randint(0, 4, (8, 3), generator=gen)].repeat_interleave(128, 0)[:rows].repeat_interleave(64, 1)
    Mb = W.numel() // b
    check_gemm(W, b, Mb * un // 10, Mb * pr // 10, M, seed=70 + b)


@pytest.mark.parametrize("M", [40, 38000])       # the streaming kernel, the one that keeps the weights
@pytest.mark.parametrize("b", [2, 4, 8, 16])
def test_gemm_record_with_more_blocks_than_it_has(b, M):
    """A damaged record table whose ranges stay inside the lists: a record that claims its neighbour's blocks too is reported."""
    W = inputs.normal_weights(256, 192, 0.02, 980 + b)
    Mb = W.numel() // b
    desc, bufs, packed, _ = project_and_pack(W, b, Mb, 0)              # all unified: every record is full
    rec = F.records(packed.cpu().numpy())
    at = F.parse_header(packed.cpu().numpy())["off_rec"]
    words = packed[at:at + rec.size * 4].view(torch.int32).view(-1, 4)
    assert words[1, 0] == rec[1, 0] == 128 * 64 // b
    words[1, 0] = int(rec[2, 0])
    Y = torch.zeros((M, 256), dtype=torch.bfloat16, device="cuda")
    X = inputs.normal_activations_bf16((M, 192), 981).cuda()
    B.mwu_gemm(desc, packed, X, M, 192, Y, 256, 0, bufs.dev_status)
    torch.cuda.synchronize()
    assert int(bufs.dev_status.item()) == B.MWU_DEV_BOUNDS


@pytest.mark.parametrize("filters,cin,h,w,k,stride,pad,n,b", [(128, 64, 13, 11, 3, 2, 1, 2, 4),    # four planes, odd sizes
                                                              (136, 128, 9, 9, 3, 1, 1, 1, 8),     # two chunks over a cluster, ragged filters
                                                              (256, 64, 30, 29, 3, 1, 1, 24, 16),  # several tiles to a CTA, two filter tiles
                                                              (128, 80, 12, 10, 2, 2, 0, 3, 2),    # a chunk of 16 channels, four taps
                                                              (128, 64, 7, 8, 1, 2, 0, 2, 4),      # 1x1 with a stride: one plane of four
                                                              (128, 64, 9, 7, 3, 1, 4, 2, 4),      # more padding than kernel
                                                              (128, 64, 6, 700, 3, 1, 1, 1, 8),    # long rows: one gather per kernel row
                                                              (128, 64, 10, 9, 3, 3, 1, 2, 16)])
def test_conv_fused_shapes(filters, cin, h, w, k, stride, pad, n, b):
    """The kernel without scratch memory: strides, planes, halos and chunks at their edges."""
    W = inputs.normal_weights(filters, cin * k * k, 0.05, 780 + filters + cin + k + h)
    x = inputs.normal_activations_bf16((n, cin, h, w), 781 + h)
    Mb = W.numel() // b
    conv_case(W, b, Mb * 6 // 10, Mb * 3 // 10, x, k, k, stride, pad)


@pytest.mark.parametrize("filters,cin,h,w,k,pad,n,b", [(128, 64, 17, 120, 11, 5, 1, 8),     # a halo too large for one fetch: a fetch per kernel row
                                                       (128, 64, 5, 6, 3, 3, 2, 4),         # padding as wide as the kernel
                                                       (256, 128, 56, 55, 3, 1, 8, 16),     # tiles of 256 pixels
                                                       (130, 64, 31, 33, 5, 2, 2, 2)])
def test_conv_line_shapes(filters, cin, h, w, k, pad, n, b):
    W = inputs.normal_weights(filters, cin * k * k, 0.05, 790 + filters + cin + k + h)
    x = inputs.normal_activations_bf16((n, cin, h, w), 791 + h)
    Mb = W.numel() // b
    if k * k <= 9:
        conv_case(W, b, Mb * 6 // 10, Mb * 3 // 10, x, k, k, 1, pad, expect_ws=True)
        return
    # plain weights: the projection is beside the point here
    desc, bufs, packed, p = project_and_pack(W, b, Mb * 6 // 10, Mb * 3 // 10)
    What = O.decoded_weights(p)
    ref = O.conv2d_direct(x.to(torch.float64).numpy(), What, k, k, 1, pad)
    ws = torch.empty(B.mwu_conv_dense_workspace_bytes(filters, n, cin, h, w, k, k, 1, pad), dtype=torch.uint8, device="cuda")
    Wd = torch.from_numpy(What).to(torch.bfloat16).cuda()
    for call in ("dense", "packed"):
        Y = torch.full(ref.shape, float("nan"), dtype=torch.float32, device="cuda")
        if call == "dense":
            B.mwu_conv_dense(filters, Wd, cin * k * k, x.cuda(), n, cin, h, w, k, k, 1, pad, Y, 1, ws, bufs.dev_status)
        else:
            B.mwu_conv_implicit_ws(desc, packed, x.cuda(), n, cin, h, w, k, k, 1, pad, Y, 1, ws, bufs.dev_status)
        torch.cuda.synchronize()
        assert int(bufs.dev_status.item()) == 0
        assert errors(Y.cpu().numpy(), ref)[0] <= 1e-5, call


@pytest.mark.parametrize("cols", [6144, 6208, 6912, 6976, 8192, 16384])
@pytest.mark.parametrize("workspace", [True, False])
def test_gemm_long_fp32_sums_of_few_rows_are_as_exact_as_whole_ones(cols, workspace):
    """40 rows, whose sums may be taken in pieces, and the same rows by the kernel that never splits, both against fp64."""
    W = inputs.normal_weights(128, cols, 0.02, 910).cuda()
    Mb = W.numel() // 4
    desc = B.make_desc(128, cols, 4, Mb // 2, Mb // 4)
    bufs = B.ProjectionBuffers(desc)
    bufs.project(W)
    packed = bufs.pack(W)
    Wd = torch.empty(128, cols, dtype=torch.bfloat16, device="cuda")
    B.mwu_decode(desc, packed, Wd, cols, bufs.dev_status)
    X = inputs.normal_activations_bf16((40, cols), 911).cuda()
    Y, Z = torch.zeros(40, 128, device="cuda"), torch.zeros(40, 128, device="cuda")
    ws = torch.empty(B.mwu_gemm_workspace_bytes(desc, 40), dtype=torch.uint8, device="cuda") if workspace else None
    B.mwu_gemm_ws(desc, packed, X, 40, cols, Y, 128, 1, ws, bufs.dev_status)
    B.mwu_gemm_dense(128, cols, Wd, cols, X, 40, cols, Z, 128, 1, bufs.dev_status)
    torch.cuda.synchronize()
    assert int(bufs.dev_status.item()) == 0
    ref = X.double() @ Wd.double().t()
    few, whole = (float((y.double() - ref).norm() / ref.norm()) for y in (Y, Z))
    # a sum in pieces meets a smaller accumulator at every step; the margin is for sums that were not split at all
    assert few <= 1.02 * whole and whole <= 2.0 ** -23 * cols / 16



def test_conv_padding_of_two_to_the_32_pixels():
    """Paddings may be 32767 wide: 2 x 2 pixels become 65536 x 65536, whose number does not fit 32 bits."""
    W = inputs.normal_weights(8, 64, 0.05, 797)
    desc, bufs, packed, p = project_and_pack(W[:1].contiguous(), 4, 8, 4)
    x = inputs.normal_activations_bf16((1, 64, 2, 2), 798)
    Y = torch.full((1, 1, 65536, 65536), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.mwu_conv_implicit(desc, packed, x.cuda(), 1, 64, 2, 2, 1, 1, 1, 32767, Y, 0, bufs.dev_status)
    torch.cuda.synchronize()
    assert int(bufs.dev_status.item()) == 0
    ref = np.einsum("ok,nkhw->nohw", O.decoded_weights(p), x.to(torch.float64).numpy())
    inner = Y[:, :, 32767:32769, 32767:32769]
    assert errors(inner.float().cpu().numpy(), ref)[1] <= 1e-2
    inner.zero_()
    assert all(int(torch.count_nonzero(Y[0, 0, r:r + 8192])) == 0 for r in range(0, 65536, 8192))


@pytest.mark.parametrize("kh,kw,h,w,n", [(1, 1400, 3, 1450, 1),      # the widest kernel row that one fetch holds
                                         (1, 1450, 3, 1500, 1),      # a fetch per tap
                                         (2, 1450, 4, 1500, 1),
                                         (1, 1450, 64, 1500, 2)])    # the same with tiles of 256 pixels
def test_conv_wide_kernels_with_workspace(kh, kw, h, w, n):
    torch.manual_seed(800 + kh + kw + h)
    rows, cin, cols = 16, 64, 64 * kh * kw
    W = torch.randn(rows, cols, device="cuda") * 0.02
    x = torch.randn(n, cin, h, w, device="cuda").bfloat16()
    desc = B.make_desc(rows, cols, 16, rows * cols // 32, rows * cols // 64)
    bufs = B.ProjectionBuffers(desc)
    bufs.project(W)
    packed = bufs.pack(W)
    Wd = torch.empty(128, cols, dtype=torch.bfloat16, device="cuda")
    B.mwu_decode(desc, packed, Wd, cols, bufs.dev_status)
    # im2col is all it takes: the kernel spans almost the whole row
    A = x.double().unfold(2, kh, 1).unfold(3, kw, 1).permute(0, 2, 3, 1, 4, 5)
    ref = torch.stack([A[i].reshape(A.shape[1], A.shape[2], cols) @ Wd[:rows].double().t() for i in range(n)]).permute(0, 3, 1, 2)
    args = (x, n, cin, h, w, kh, kw, 1, 0)
    ws = torch.empty(max(B.mwu_conv_workspace_bytes(desc, *args[1:]), B.mwu_conv_dense_workspace_bytes(rows, *args[1:])),
                     dtype=torch.uint8, device="cuda")
    for call in ("dense", "packed"):
        Y = torch.full(ref.shape, float("nan"), device="cuda")
        if call == "dense":
            B.mwu_conv_dense(rows, Wd, cols, *args, Y, 1, ws, bufs.dev_status)
        else:
            B.mwu_conv_implicit_ws(desc, packed, *args, Y, 1, ws, bufs.dev_status)
        torch.cuda.synchronize()
        assert int(bufs.dev_status.item()) == 0
        # an MMA adds 16 products and may cut its accumulator off at 2^-23 of itself; the partial sums of independent
        # products are no larger, in the mean, than the whole
        assert float((Y.double() - ref).norm() / ref.norm()) <= 2.0 ** -23 * cols / 16, call


@pytest.mark.parametrize("rows,cols,m,launches", [(1024, 64, 4096, 2), (1024, 64, 1024, 1),       # two tiles an SM; one
                                                  (256, 256, 8192, 1), (256, 256, 16384, 2),
                                                  (512, 512, 2048, 2), (512, 512, 512, 1)])       # split to two CTAs an SM
def test_gemm_many_rows_of_a_small_weight(rows, cols, m, launches):
    """Where the streaming kernel (one launch) gives way to expanding the weights (two): results on both sides of the line."""
    torch.manual_seed(920)
    W = torch.randn(rows, cols, device="cuda") * 0.02
    Mb = rows * cols // 4
    desc = B.make_desc(rows, cols, 4, Mb * 6 // 10, Mb * 4 // 10)
    bufs = B.ProjectionBuffers(desc)
    bufs.project(W)
    packed = bufs.pack(W)
    Wd = torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda")
    B.mwu_decode(desc, packed, Wd, cols, bufs.dev_status)
    X = torch.randn(m, cols, device="cuda").bfloat16()
    Y = torch.full((m, rows), float("nan"), dtype=torch.bfloat16, device="cuda")
    ws = torch.empty(B.mwu_gemm_workspace_bytes(desc, m), dtype=torch.uint8, device="cuda")
    before = B.mwu_kernel_launches()
    B.mwu_gemm_ws(desc, packed, X, m, cols, Y, rows, 0, ws, bufs.dev_status)
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert B.mwu_kernel_launches() - before == launches
    torch.cuda.synchronize()
    assert int(bufs.dev_status.item()) == 0
    ref = X.double() @ Wd.double().t()
    assert float((Y.double() - ref).norm() / ref.norm()) <= 2e-3
