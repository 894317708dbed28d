"""The dynamic quantizers when their grid is not resident together: CTAs that
wait too long read x in the missing ones' place, so no call waits for another
kernel to leave the machine, and codes, scales and scratch are as ever.

The paths are forced by wait limits of zero (and counted), by a kernel that
holds most of the SMs, and by quantizers and a GEMM on streams of their own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2609_21849_gb300 import probe, qlin, synthetic

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from gpu_util import assert_nvfp4_equal, f32, to_dev, u8

SMS = (torch.cuda.get_device_properties(0).multi_processor_count
       if torch.cuda.is_available() else 152)
# x in registers (NVFP4) or shared memory (FP8), x in shared memory, two phases;
# ragged sizes, the first with fewer pieces than CTAs
SHAPES = [(1025, 512), (4601, 3072), (13000 * SMS // 512, 4096), (9217, 4096)]


def _out(fmt, M, K):
    return qlin.alloc_nvfp4(M, K) if fmt == "nvfp4" else qlin.alloc_fp8(M, K, False)


def _check(fmt, q, bits, label):
    if fmt == "nvfp4":
        assert_nvfp4_equal(q, oracle.quant_nvfp4(bits), label)
    else:
        c, s = oracle.quant_fp8(bits)[:2]
        assert f32(q.scale)[0] == np.float32(s), label
        assert np.array_equal(u8(q.codes), c), label


@pytest.mark.parametrize("M,K", SHAPES)
@pytest.mark.parametrize("fmt", ["nvfp4", "fp8"])
def test_waits_that_expire(fmt, M, K):
    pieces = -(-M * K // 8 // 4096)
    sync = torch.zeros(8, dtype=torch.int32, device="cuda")
    bits = synthetic.act_entry_outliers(11, M, K)
    x = to_dev(bits)
    # the largest value alone in the first, then in the last piece
    for row in (0, M - 1):
        b = bits.copy()
        b[row, 5] = 0x4500
        x.view(torch.int16).copy_(torch.from_numpy(b.view(np.int16)))
        # no wait for the grid: every CTA helps, each piece is read at most once
        q = _out(fmt, M, K)
        helped, read, alone = probe.grid_max(x, q, sync, 0, 1_000_000)
        assert helped > 1 and 1 <= read <= pieces and alone == 0, (helped, read, alone)
        _check(fmt, q, b, f"help {M}x{K} row {row}")
        assert int(sync.count_nonzero()) == 0
        # no piece left and no wait: every CTA reads all of x (the smallest shape)
        if M * K <= 1 << 20:
            q = _out(fmt, M, K)
            sync[3] = pieces
            helped, read, alone = probe.grid_max(x, q, sync, 0, 0)
            assert helped == alone > 1 and read == 0, (helped, read, alone)
            _check(fmt, q, b, f"alone {M}x{K} row {row}")
            assert int(sync.count_nonzero()) == 0
    # undisturbed, no CTA gives up
    q = _out(fmt, M, K)
    assert probe.grid_max(x, q, sync, 1_000_000, 1_000_000) == (0, 0, 0)
    _check(fmt, q, b, f"plain {M}x{K}")


@pytest.mark.parametrize("M,K", SHAPES)
@pytest.mark.parametrize("fmt", ["nvfp4", "fp8"])
def test_does_not_wait_for_held_sms(fmt, M, K):
    # all but 32 SMs held for 4 ms: the quantizer ends long before they are free
    bits = synthetic.act_entry_outliers(12, M, K)
    x, q, ws = to_dev(bits), _out(fmt, M, K), qlin.alloc_workspace()
    quantize = qlin.qlin_quantize_act_nvfp4 if fmt == "nvfp4" else qlin.qlin_quantize_act_fp8
    quantize(x, None, q, ws)   # one-time set-up
    torch.cuda.synchronize()
    held, own = torch.cuda.Stream(), torch.cuda.Stream()
    t0, t1, free = (torch.cuda.Event(enable_timing=True) for _ in range(3))
    probe.hold_sms(SMS - 32, 4_000_000, held)
    free.record(held)
    t0.record(own)
    quantize(x, None, q, ws, own)
    t1.record(own)
    t1.synchronize()
    assert not free.query()
    # (a wait of 1 ms for the grid, then all of x in every CTA, took longer)
    assert t0.elapsed_time(t1) < 0.9, t0.elapsed_time(t1)
    torch.cuda.synchronize()
    assert qlin.qlin_sync_status() == 0
    _check(fmt, q, bits, f"{M}x{K}")
    assert int(ws.count_nonzero()) == 0


@pytest.mark.parametrize("fmt", ["nvfp4", "fp8"])
def test_two_quantizers_and_a_gemm_on_their_own_streams(fmt):
    quantize = qlin.qlin_quantize_act_nvfp4 if fmt == "nvfp4" else qlin.qlin_quantize_act_fp8
    shapes = [(4608, 3072), (18432, 3072), (1025, 512)]
    bits = [synthetic.act_entry_outliers(40 + i, *s) for i, s in enumerate(shapes)]
    xs = [to_dev(b) for b in bits]
    ws = [qlin.alloc_workspace() for _ in xs]
    (w,) = synthetic.weights(43, [(3072, 3072)], 0.02)
    W = qlin.qlin_quantize_weight(to_dev(w), qlin.QLIN_FMT_NVFP4)
    A = qlin.qlin_quantize_act_nvfp4(xs[0])
    want = qlin.qlin_gemm_nvfp4(A, W)
    y = torch.empty_like(want)
    streams = [torch.cuda.Stream(priority=p) for p in (0, -1, 0, 0)]
    qs = [[_out(fmt, *s) for _ in range(20)] for s in shapes]
    torch.cuda.synchronize()
    for i in range(20):
        for x, q, wsp, s in zip(xs, qs, ws, streams):
            quantize(x, None, q[i], wsp, s)
        qlin.qlin_gemm_nvfp4(A, W, y, streams[3])
    torch.cuda.synchronize()
    assert qlin.qlin_sync_status() == 0
    for b, q, s in zip(bits, qs, shapes):
        _check(fmt, q[0], b, str(s))
        for r in q[1:]:
            assert torch.equal(r.codes, q[0].codes)
    assert torch.equal(y, want)
    assert all(int(w.count_nonzero()) == 0 for w in ws)


def test_a_waiting_quantizer_comes_before_the_next_gemm():
    # two GEMMs on one stream, then a quantizer on another while the first runs:
    # it starts when that one ends, not when both have
    (w,) = synthetic.weights(47, [(12288, 3072)], 0.02)
    W = qlin.qlin_quantize_weight(to_dev(w), qlin.QLIN_FMT_NVFP4)
    bits = synthetic.act_normal(46, 18432, 3072)
    A = qlin.qlin_quantize_act_nvfp4(to_dev(bits))
    y = torch.empty((18432, 12288), dtype=torch.bfloat16, device="cuda")
    x, q, ws = to_dev(bits[:4608]), qlin.alloc_nvfp4(4608, 3072), qlin.alloc_workspace()
    gemms, own = torch.cuda.Stream(), torch.cuda.Stream()
    first = []
    for _ in range(9):
        torch.cuda.synchronize()
        t0, t1, t2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        t0.record(gemms)
        qlin.qlin_gemm_nvfp4(A, W, y, gemms)
        qlin.qlin_gemm_nvfp4(A, W, y, gemms)
        t2.record(gemms)
        qlin.qlin_quantize_act_nvfp4(x, None, q, ws, own)
        t1.record(own)
        torch.cuda.synchronize()
        first.append(t0.elapsed_time(t1) < t0.elapsed_time(t2))
    assert sum(first) >= 7, first
    assert qlin.qlin_sync_status() == 0
    _check("nvfp4", q, bits[:4608], "beside GEMMs")
