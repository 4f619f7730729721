"""Rows that teams of 1, 2, 4, 8 or 16 warps share (past 2 KiB, up to one
stage) against the oracle, bit-identical across policies: the
lengths at which the team, the vectors a lane holds, or the part left in the
stage changes; batches that mix team sizes (and long rows); rows with NaN,
+inf, all -inf, and finite masks; and the bounded wait."""
import numpy as np
import pytest

from gpu_util import (FINITE_MASKS, bits, check_all_against_oracle, check_finite_masks, run, to_device,
                      to_host)
from paper_2002_07062_gb300 import bsm, workload

pytestmark = pytest.mark.gpu

POLICIES = [bsm.POLICY_RR, bsm.POLICY_DYNAMIC, bsm.POLICY_CBMF_LB, bsm.POLICY_WHOLE_GPU]
# 16-byte vectors per row around every switch; 7232 fill a stage (113 KiB)
EDGES = [129, 192, 193, 256, 257, 384, 385, 512, 513, 768, 769, 1024, 1025, 1536, 1537, 2048, 2049, 3072, 3073,
         4096, 4097, 4608, 7231, 7232]


@pytest.fixture(scope="module", autouse=True)
def setup():
    import torch
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)
    bsm.bsm_device_status_clear()
    yield
    bsm.bsm_cache_clear()


def _same_bits(w, x):
    import torch
    ys = [run(w, x, p) for p in POLICIES]
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0, bsm.bsm_device_debug()
    for y in ys[1:]:
        assert torch.equal(bits(y), bits(ys[0]))
    return ys[0]


@pytest.mark.parametrize("nvec", EDGES)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
@pytest.mark.parametrize("flags", [0, workload.CAUSAL])
def test_row_lengths_at_the_edges(nvec, dtype, flags):
    C = nvec * (4 if dtype == workload.F32 else 8)
    # 37 rows: stages of several rows end ragged; the mask crosses a row
    w = workload.uniform("team", dtype, 3, 37, C, 3.0, 0x7EA0 + nvec + flags, flags).materialize()
    check_all_against_oracle(w, to_host(_same_bits(w, to_device(w.x))))


@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
def test_causal_square(dtype):
    """Slices as high as wide: every position of the diagonal in a row of the
    team routine, wholly masked vectors included."""
    C = 2400
    w = workload.uniform("team causal", dtype, 1, C, C, 3.0, 0x7EB0 + dtype, workload.CAUSAL).materialize()
    check_all_against_oracle(w, to_host(_same_bits(w, to_device(w.x))))


@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
@pytest.mark.parametrize("long_rows", [False, True])
def test_team_sizes_mixed_in_one_batch(dtype, long_rows):
    per = 4 if dtype == workload.F32 else 8
    rng = np.random.default_rng(0x7EC0 + dtype)
    nvec = rng.choice(EDGES[:-4] + [8, 40, 100], 300)
    if long_rows:
        nvec[rng.choice(300, 6, replace=False)] = 9000
    rows = rng.integers(1, 6, 300).astype(np.int32)
    cols = (nvec * per).astype(np.int32)
    sizes = rows.astype(np.int64) * cols
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.int64)
    w = workload.Workload("team mix", dtype, rows, cols, off, 0, 0x7EC1, 3.0)
    w.materialize()
    check_all_against_oracle(w, to_host(_same_bits(w, to_device(w.x))))


@pytest.mark.parametrize("nvec", [300, 1000, 2000, 5000])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_non_finite_and_lowest_value_rows(nvec, dtype):
    import torch
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    C = nvec * (4 if dtype == "f32" else 8)
    low = torch.finfo(t).min
    x = torch.randn(9, C, device="cuda").to(t)
    x[1, C - 1] = float("nan")
    x[2, 5] = float("inf")
    x[3, :] = -float("inf")
    x[3, C // 2] = 1.0
    x[4, :] = -float("inf")
    x[5, :] = low
    x[5, C - 3] = 2.0                         # one element left by such a mask
    x[6, : C // 2] = low
    x[7, 8:] = low                            # whole warps see the mask only
    y = torch.full_like(x, -1.0)
    bsm.bsm_softmax_ex(x, y, 1, 9, C, bsm.F32 if dtype == "f32" else bsm.BF16, bsm.POLICY_DYNAMIC)
    torch.cuda.synchronize()
    assert torch.isnan(y[[1, 2, 4]]).all()
    assert float(y[3, C // 2]) == 1.0 and int(y[3].count_nonzero()) == 1
    assert float(y[5, C - 3]) == 1.0 and int(y[5].count_nonzero()) == 1
    ref = torch.softmax(x[[0, 6, 7, 8]].double(), -1)
    err = (y[[0, 6, 7, 8]].double() - ref).abs()
    assert float(err.max()) <= 2e-6 if dtype == "f32" else bool((err <= ref * 2.0 ** -8 + 1e-30).all())


@pytest.mark.parametrize("mask", FINITE_MASKS)
@pytest.mark.parametrize("nvec", [100, 300, 1000, 2000, 5000, 7000])
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
def test_finite_masks(mask, nvec, dtype):
    check_finite_masks(mask, dtype, 9, nvec * (4 if dtype == workload.F32 else 8))


def test_withheld_stage_times_out_on_team_rows():
    import time
    import torch
    w = workload.uniform("team fail", workload.F32, 4, 200, 12000, 2.0, 0x7ED0).materialize()
    x = to_device(w.x)
    y = torch.zeros_like(x)
    p = bsm.bsm_plan_create(x, y, w.rows, w.cols, w.dtype, bsm.POLICY_DYNAMIC)
    bsm.bsm_plan_debug(p, bsm.DEBUG_WITHHOLD_STAGE, 100_000_000)      # 0.1 s waits
    t0 = time.time()
    p.execute()
    torch.cuda.synchronize()
    assert time.time() - t0 < 5.0
    assert bsm.bsm_device_status() & bsm.DEV_TIMEOUT
    bsm.bsm_plan_debug(p, bsm.DEBUG_NONE)
    bsm.bsm_device_status_clear()
    p.execute()
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0
    check_all_against_oracle(w, to_host(y))
    p.close()


# backward: 16-byte vectors of y (and of dy) around every switch; 3616 fill half a stage
BWD_EDGES = [65, 96, 97, 128, 129, 192, 193, 256, 257, 400, 512, 513, 800, 1024, 1025, 1600, 2048, 2049, 3615, 3616]


@pytest.mark.parametrize("nvec", BWD_EDGES)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
def test_backward_row_lengths_at_the_edges(nvec, dtype):
    import torch
    from test_backward_gpu import _check, _inputs
    C = nvec * (4 if dtype == workload.F32 else 8)
    w = workload.uniform("team bwd", dtype, 3, 37, C, 3.0, 0x7EE0 + nvec).materialize()
    y, dy = _inputs(w)
    yd, dyd = to_device(y), to_device(dy)
    outs = []
    for p in POLICIES:
        dx = torch.full_like(yd, float("nan"))
        bsm.bsm_softmax_backward(yd, dyd, dx, w.nslices, 37, C, dtype, p)
        outs.append(dx)
    bsm.bsm_softmax_backward(yd, dyd, dyd, w.nslices, 37, C, dtype, bsm.POLICY_DYNAMIC)   # in place
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0
    for o in outs[1:] + [dyd]:
        assert torch.equal(bits(o), bits(outs[0]))
    _check(w, y, dy, to_host(outs[0]))


@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
def test_backward_team_sizes_mixed_in_one_batch(dtype):
    import torch
    from test_backward_gpu import _check, _inputs
    per = 4 if dtype == workload.F32 else 8
    rng = np.random.default_rng(0x7EF0 + dtype)
    nvec = rng.choice(BWD_EDGES + [8, 40], 200)
    nvec[rng.choice(200, 4, replace=False)] = 5000           # and rows longer than half a stage
    rows = rng.integers(1, 6, 200).astype(np.int32)
    cols = (nvec * per).astype(np.int32)
    sizes = rows.astype(np.int64) * cols
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.int64)
    w = workload.Workload("team bwd mix", dtype, rows, cols, off, 0, 0x7EF1, 3.0)
    w.materialize()
    y, dy = _inputs(w)
    yd, dyd = to_device(y), to_device(dy)
    outs = []
    for p in POLICIES:
        dx = torch.full_like(yd, float("nan"))
        bsm.bsm_softmax_backward_ragged(yd, dyd, dx, w.offsets, w.rows, w.cols, dtype, p)
        outs.append(dx)
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0
    for o in outs[1:]:
        assert torch.equal(bits(o), bits(outs[0]))
    _check(w, y, dy, to_host(outs[0]))
