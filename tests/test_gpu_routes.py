"""GPU parity at the edges of the size rules that choose a kernel: the dynamic
quantizers' routes (clusters that each read x, x in registers or shared memory,
two phases over x) and the GEMM's tile configurations and K stages (256 NVFP4
elements as 96 + 96 + 64, partial stages, the scale rings' wrap-around).

Codes and scales are compared bit for bit with the oracle's; GEMM outputs are
within the tolerance of the exact product (2e-3 of the operands' row norms) on
a few rows per 128-row tile."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2609_21849_gb300 import qlin, synthetic

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_util import (GEMM_TOL, assert_nvfp4_equal, bf16_bits, f32, gemm_errors, to_dev, u8)

# x of n chunks (8 values): 1 MB is 65536 chunks, the cluster route's last
# size; x in registers reaches 12288 chunks per SM, in shared memory 14336.
SMS = (torch.cuda.get_device_properties(0).multi_processor_count
       if torch.cuda.is_available() else 152)
ROUTES = [(1, 64), (3, 64), (17, 448), (256, 2048), (257, 2048), (1023, 512),
          (12288 * SMS // 512, 4096), (12288 * SMS // 512 + 1, 4096),
          (14336 * SMS // 512, 4096), (14336 * SMS // 512 + 1, 4096)]


@pytest.mark.parametrize("M,K", ROUTES)
def test_dynamic_routes_match_oracle(M, K):
    # twice with one workspace, the smaller amax second: the scratch is left
    # zero, and a stale maximum would show
    ws = qlin.alloc_workspace()
    q4, q8 = qlin.alloc_nvfp4(M, K), qlin.alloc_fp8(M, K, False)
    for seed, scale in ((5, 1), (6, 64)):
        bits = synthetic.act_entry_outliers(seed, M, K)
        x = (to_dev(bits).float() / scale).bfloat16()
        bits = bf16_bits(x)
        qlin.qlin_quantize_act_nvfp4(x, None, q4, ws)
        qlin.qlin_quantize_act_fp8(x, None, q8, ws)
        assert qlin.qlin_sync_status() == 0
        assert_nvfp4_equal(q4, oracle.quant_nvfp4(bits), f"{M}x{K}")
        c8, s8 = oracle.quant_fp8(bits)[:2]
        assert f32(q8.scale)[0] == np.float32(s8)
        assert np.array_equal(u8(q8.codes), c8)
    assert int(ws.count_nonzero()) == 0


def test_one_workspace_for_every_route():
    # every dynamic route and the dynamic chain in turn on one workspace, with
    # maxima that fall: each leaves it zero for the next
    ws = qlin.alloc_workspace()
    shapes = [(256, 512), (1025, 512), (4608, 3072), (13000 * SMS // 512, 4096), (9217, 4096)]
    xs = [synthetic.act_entry_outliers(50 + i, *s) for i, s in enumerate(shapes)]
    (w,) = synthetic.weights(60, [(576, 512)], 0.02)
    W = qlin.qlin_quantize_weight(to_dev(w), qlin.QLIN_FMT_NVFP4)
    want4 = [oracle.quant_nvfp4(x) for x in xs]
    want8 = [oracle.quant_fp8(x)[:2] for x in xs]
    for order in ((4, 3, 2, 1, 0), (0, 2, 4, 1, 3)):
        for i in order:
            x = to_dev(xs[i])
            q4 = qlin.qlin_quantize_act_nvfp4(x, None, None, ws)
            q8 = qlin.qlin_quantize_act_fp8(x, None, None, ws)
            A = qlin.qlin_quantize_act_nvfp4(to_dev(xs[1]), None, None, ws)
            y, yq = qlin.qlin_linear_dynamic(A, W, workspace=ws)
            assert qlin.qlin_sync_status() == 0
            assert_nvfp4_equal(q4, want4[i], str(shapes[i]))
            assert f32(q8.scale)[0] == np.float32(want8[i][1])
            assert np.array_equal(u8(q8.codes), want8[i][0])
            assert_nvfp4_equal(yq, oracle.quant_nvfp4(bf16_bits(y)), "chain")
            assert int(ws.count_nonzero()) == 0


@pytest.mark.parametrize("bits", [0x0001, 0x8001, 0x007F, 0x8080, 0x7F7F, 0xFF7F, 0x7F80, 0xFF80,
                                  0x7FC0, 0xFF81, 0x7FFF])
@pytest.mark.parametrize("M,K", [(3, 64), (1000, 3072), (9217, 4096)])
def test_maximum_of_extreme_values(M, K, bits):
    # one subnormal, largest finite value, infinity or NaN among zeros, at an
    # odd element: scale = max |x| / 448 in fp32, NaN if x holds one
    x = torch.zeros((M, K), dtype=torch.int16, device="cuda")
    x[M - 1, K - 13] = bits - 65536 if bits > 32767 else bits
    ws = qlin.alloc_workspace()
    q = qlin.qlin_quantize_act_fp8(x.view(torch.bfloat16), None, None, ws)
    assert qlin.qlin_sync_status() == 0
    amax = np.array([(bits & 0x7FFF) << 16], np.uint32).view(np.float32)
    assert np.array_equal(f32(q.scale), amax / np.float32(448), equal_nan=True)
    q4 = qlin.qlin_quantize_act_nvfp4(x.view(torch.bfloat16), None, None, ws)
    assert qlin.qlin_sync_status() == 0
    assert np.array_equal(f32(q4.tensor_scale), amax / np.float32(2688), equal_nan=True)
    assert int(ws.count_nonzero()) == 0


@pytest.mark.parametrize("M,K", [(1025, 512), (4608, 3072), (12288 * SMS // 512 + 64, 4096),
                                 (9217, 4096)])
def test_grid_wait_that_expires_gives_the_same_codes(M, K):
    # with the shortest wait limit, CTAs that miss the others' arrival read x in
    # their place (test_gpu_grid_wait.py forces each such path and counts it):
    # same codes, no error, scratch left zero
    bits = synthetic.act_entry_outliers(7, M, K)
    x, ws = to_dev(bits), qlin.alloc_workspace()
    want4 = qlin.qlin_quantize_act_nvfp4(x, None, None, ws)
    want8 = qlin.qlin_quantize_act_fp8(x, None, None, ws)
    assert qlin.qlin_sync_status() == 0
    qlin.qlin_set_wait_timeout_ns(1000)
    try:
        q4 = qlin.qlin_quantize_act_nvfp4(x, None, None, ws)
        q8 = qlin.qlin_quantize_act_fp8(x, None, None, ws)
        assert qlin.qlin_sync_status() == 0
    finally:
        qlin.qlin_set_wait_timeout_ns(2000000000)
    assert_nvfp4_equal(q4, oracle.quant_nvfp4(bits), f"{M}x{K}")
    for a, b in ((q4.codes, want4.codes), (q4.tensor_scale, want4.tensor_scale),
                 (q8.codes, want8.codes), (q8.scale, want8.scale)):
        assert torch.equal(a, b)
    assert int(ws.count_nonzero()) == 0


@pytest.mark.parametrize("M", [1, 2055, 2048 * SMS // 4, 2048 * SMS // 4 + 5])
@pytest.mark.parametrize("shift", [0, 8])
def test_static_nvfp4_alignment_and_partial_tile(shift, M):
    # one block per thread up to 2048 threads per SM, tiles beyond; x 32-byte
    # aligned (there one 32-byte load per block) and only 16-byte aligned (two
    # 16-byte loads); the last CTA's share and the last tile are partial
    K = 64
    bits = synthetic.act_entry_outliers(9, M, K)
    buf = torch.zeros(M * K + 16, dtype=torch.bfloat16, device="cuda")
    x = buf[shift:shift + M * K].view(M, K)
    x.copy_(to_dev(bits))
    s = np.float32(0.03)
    q = qlin.qlin_quantize_act_nvfp4(x, torch.tensor([s], device="cuda"))
    assert qlin.qlin_sync_status() == 0
    assert_nvfp4_equal(q, oracle.quant_nvfp4(bits, s), f"shift {shift}")


@pytest.mark.parametrize("N,K", [(1, 64), (40003, 64), (200, 512), (200, 576), (3001, 1024),
                                 (200, 1088), (200, 3072), (33, 3136), (9, 12288)])
def test_fp8_weight_rows(N, K):
    # rows held in registers (two, four or twelve chunks a lane) up to K = 512,
    # 1024 and 3072, read twice beyond; more rows than warps
    (w,) = synthetic.weights(11, [(N, K)], 0.02)
    q = qlin.qlin_quantize_weight(to_dev(w), qlin.QLIN_FMT_FP8)
    codes, scales = oracle.quant_fp8_rows(w)[:2]
    assert np.array_equal(u8(q.codes), codes) and np.array_equal(f32(q.scale), scales)


def _rows(M):
    r = {0, M - 1} | {t * 128 + (37 * t) % 128 for t in range((M + 127) // 128)}
    return np.array(sorted(i for i in r if i < M))


# (M, N): 64-wide, 128-wide and pair tiles (with a partial pair), and a single
# N tile whose W every CTA shares; K: one
# partial stage, full ones, every remainder of a stage, and K long enough that
# every ring wraps
@pytest.mark.parametrize("M,N", [(40, 192), (300, 2560), (3000, 1024), (4700, 2112),
                                 (18400, 64)])
@pytest.mark.parametrize("K", [64, 192, 256, 832, 2688])
@pytest.mark.parametrize("fmt", ["nvfp4", "fp8"])
def test_gemm_tiles_and_stages(fmt, M, N, K):
    x = synthetic.act_entry_outliers(21, M, K)
    (w,) = synthetic.weights(22, [(N, K)], 0.02)
    rows = _rows(M)
    if fmt == "nvfp4":
        A = qlin.qlin_quantize_act_nvfp4(to_dev(x))
        W = qlin.qlin_quantize_weight(to_dev(w), qlin.QLIN_FMT_NVFP4)
        y = qlin.qlin_gemm_nvfp4(A, W)
        c, s, ts = oracle.quant_nvfp4(x)
        ref = oracle.gemm_nvfp4((c[rows], s[rows], ts), oracle.quant_nvfp4(w))
    else:
        A = qlin.qlin_quantize_act_fp8(to_dev(x))
        W = qlin.qlin_quantize_weight(to_dev(w), qlin.QLIN_FMT_FP8)
        y = qlin.qlin_gemm_fp8(A, W)
        c, s = oracle.quant_fp8(x)[:2]
        ref = oracle.gemm_fp8((c[rows], s), oracle.quant_fp8_rows(w))
    assert qlin.qlin_sync_status() == 0
    err, exact = gemm_errors(bf16_bits(y)[rows], *ref)
    assert err.max() <= GEMM_TOL and exact >= 0.99, (err.max(), exact)


def test_back_to_back_launches_see_new_operands():
    # the scales of single-CTA tiles are read through L1: two activations
    # quantized in turn into one operand, no wait between the launches
    M, N, K = 256, 384, 1024
    xs = [to_dev(synthetic.act_entry_outliers(s, M, K)) for s in (31, 32)]
    (w,) = synthetic.weights(33, [(N, K)], 0.02)
    W = qlin.qlin_quantize_weight(to_dev(w), qlin.QLIN_FMT_NVFP4)
    A, ws = qlin.alloc_nvfp4(M, K), qlin.alloc_workspace()
    want = []
    for x in xs:
        want.append(qlin.qlin_gemm_nvfp4(qlin.qlin_quantize_act_nvfp4(x, None, None, ws), W))
        torch.cuda.synchronize()
    got = [torch.empty_like(want[0]) for _ in range(40)]
    for i, y in enumerate(got):
        qlin.qlin_quantize_act_nvfp4(xs[i & 1], None, A, ws)
        qlin.qlin_gemm_nvfp4(A, W, y)
    assert qlin.qlin_sync_status() == 0
    assert all(torch.equal(y, want[i & 1]) for i, y in enumerate(got))
