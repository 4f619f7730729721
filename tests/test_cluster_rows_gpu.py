"""Batches of rows longer than a stage that clusters of 2 to 16 CTAs share,
against the oracle (sampled rows) and bit-identical across policies: the
lengths at which the cluster grows and parts of unequal length, the causal
mask across parts, NaN, +inf, all -inf and finite masks, unequal rows,
the self-checking kernel, a withheld stage and a corrupted record."""
import numpy as np
import pytest

from gpu_util import (FINITE_MASKS, bits, check_finite_masks, check_rows_against_oracle, run, sample_rows,
                      to_device, to_host)
from paper_2002_07062_gb300 import bsm, workload

pytestmark = pytest.mark.gpu

POLICIES = [bsm.POLICY_DYNAMIC, bsm.POLICY_RR, bsm.POLICY_CBMF, bsm.POLICY_CBMF_LB, bsm.POLICY_WHOLE_GPU]
# 16-byte vectors per row: just past a stage, odd parts, either side of the
# largest row of two CTAs, then rows of 4, 8 and 16 (forward rows of more than
# 16384 vectors are those that groups take otherwise: some of these do)
FWD = [7233, 8195, 14463, 14465, 16383, 28845, 40001, 70003]
BWD = [3617, 4099, 7231, 7233, 14401, 20003, 29001]


@pytest.fixture(scope="module", autouse=True)
def setup():
    import torch
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)
    bsm.bsm_device_status_clear()
    yield
    bsm.bsm_cache_clear()


def _rows(nvec=0):
    import torch
    # (rows for groups: a few waves of them, whichever kernel runs)
    return 150 if nvec > 16384 else 2 * torch.cuda.get_device_properties(0).multi_processor_count + 5


@pytest.mark.parametrize("nvec", FWD)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
@pytest.mark.parametrize("flags", [0, workload.CAUSAL])
def test_forward_row_lengths(nvec, dtype, flags):
    import torch
    C = nvec * (4 if dtype == workload.F32 else 8)
    w = workload.uniform("cluster", dtype, 5, (_rows(nvec) + 4) // 5, C, 3.0, 0xC10 + nvec + flags, flags).materialize()
    x = to_device(w.x)
    ys = [run(w, x, p) for p in POLICIES]
    bsm.bsm_set_device_checks(True)
    ys.append(run(w, x, bsm.POLICY_DYNAMIC))
    torch.cuda.synchronize()
    bsm.bsm_set_device_checks(False)
    assert bsm.bsm_device_status() == 0, bsm.bsm_device_debug()
    for y in ys[1:]:
        assert torch.equal(bits(y), bits(ys[0]))
    check_rows_against_oracle(w, to_host(ys[0]), sample_rows(w, 24, nvec))
    s = ys[0].view(-1, C).double().sum(1)
    assert float((s - 1).abs().max()) < (1e-5 if dtype == workload.F32 else 0.02)     # every row written


# (vectors a row, rows, CTAs a cluster): rows that fill the clusters' waves
# better than the groups'
LARGER = [(28845, 144, 4), (28863, 36, 4), (40002, 30, 8), (57001, 15, 8), (70003, 7, 16), (113001, 7, 16)]


@pytest.mark.parametrize("nvec,R,K", LARGER)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
@pytest.mark.parametrize("flags", [0, workload.CAUSAL])
def test_forward_rows_on_larger_clusters(nvec, R, K, dtype, flags):
    import torch
    C = nvec * (4 if dtype == workload.F32 else 8)
    w = workload.uniform("larger", dtype, 1, R, C, 3.0, 0xC20 + nvec + flags, flags).materialize()
    x = to_device(w.x)
    p = bsm.bsm_plan_create(x, x, w.rows, w.cols, dtype, bsm.POLICY_DYNAMIC, flags=flags)
    kernel = bsm.bsm_plan_kernel(p, 2)
    p.close()
    if torch.cuda.get_device_properties(0).multi_processor_count == 152 and not (dtype == workload.BF16 and nvec == 40002):
        assert kernel == (bsm.KERNEL_CLUSTER, K)
    ys = [run(w, x, p) for p in POLICIES]
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0, bsm.bsm_device_debug()
    for y in ys[1:]:
        assert torch.equal(bits(y), bits(ys[0]))
    check_rows_against_oracle(w, to_host(ys[0]), sample_rows(w, 7, nvec))
    s = ys[0].view(-1, C).double().sum(1)
    assert float((s - 1).abs().max()) < (1e-5 if dtype == workload.F32 else 0.02)     # every row written


@pytest.mark.parametrize("nvec", BWD)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
def test_backward_row_lengths(nvec, dtype):
    import torch
    from test_backward_gpu import _check
    C = nvec * (4 if dtype == workload.F32 else 8)
    R = _rows()
    t = torch.float32 if dtype == workload.F32 else torch.bfloat16
    g = torch.Generator(device="cuda").manual_seed(nvec)
    y = torch.softmax(torch.randn(R, C, generator=g, device="cuda") * 3, -1).to(t)
    dy = torch.randn(R, C, generator=g, device="cuda").to(t)
    p = bsm.bsm_plan_create(y, dy, [R], [C], dtype, bsm.POLICY_DYNAMIC, op=bsm.OP_BACKWARD, x2=dy)
    assert bsm.bsm_plan_kernel(p)[0] == bsm.KERNEL_CLUSTER
    p.close()
    outs = []
    for p in POLICIES:
        dx = torch.full_like(y, float("nan"))
        bsm.bsm_softmax_backward(y, dy, dx, 1, R, C, dtype, p)
        outs.append(dx)
    bsm.bsm_softmax_backward(y, dy, dy2 := dy.clone(), 1, R, C, dtype, bsm.POLICY_DYNAMIC)
    bsm.bsm_set_device_checks(True)
    dx = torch.full_like(y, float("nan"))
    bsm.bsm_softmax_backward(y, dy, dx, 1, R, C, dtype, bsm.POLICY_DYNAMIC)
    torch.cuda.synchronize()
    bsm.bsm_set_device_checks(False)
    assert bsm.bsm_device_status() == 0, bsm.bsm_device_debug()
    for o in outs[1:] + [dx]:
        assert torch.equal(bits(o), bits(outs[0]))
    assert not torch.isnan(outs[0]).any() and not torch.isnan(dy2).any()
    pick = [0, 1, R // 2, R - 1]
    w = workload.Workload("cluster bwd", dtype, np.full(4, 1, np.int32), np.full(4, C, np.int32),
                          np.arange(4, dtype=np.int64) * C, 0, 0, 1.0)
    _check(w, *(to_host(v[pick].reshape(-1)) for v in (y, dy)), to_host(outs[0][pick].reshape(-1)))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("nvec", [9000, 15000])
def test_non_finite_and_lowest_value_rows(dtype, nvec):
    import torch
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    C, R = nvec * (4 if dtype == "f32" else 8), _rows()
    low = torch.finfo(t).min
    x = torch.randn(R, C, device="cuda").to(t)
    x[1, C - 1] = float("nan")
    x[2, 5] = float("inf")
    x[3, :] = -float("inf")
    x[3, C // 2] = 1.0
    x[4, :] = -float("inf")
    x[5, :] = low
    x[5, C - 3] = 2.0
    x[6, 8:] = low
    y = torch.full_like(x, -1.0)
    bsm.bsm_softmax(x, y, 1, R, C, bsm.F32 if dtype == "f32" else bsm.BF16, bsm.POLICY_DYNAMIC)
    torch.cuda.synchronize()
    assert torch.isnan(y[[1, 2, 4]]).all()
    assert float(y[3, C // 2]) == 1.0 and int(y[3].count_nonzero()) == 1
    assert float(y[5, C - 3]) == 1.0 and int(y[5].count_nonzero()) == 1
    rest = [0] + list(range(6, R))
    ref = torch.softmax(x[rest].double(), -1)
    err = (y[rest].double() - ref).abs()
    assert float(err.max()) <= 2e-6 if dtype == "f32" else bool((err <= ref * 2.0 ** -8 + 1e-30).all())


@pytest.mark.parametrize("mask", FINITE_MASKS)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
@pytest.mark.parametrize("nvec", [9000, 15000, 28845, 70003])       # clusters of 2 and 4, of 4 to 16 or groups
def test_finite_masks(mask, dtype, nvec):
    check_finite_masks(mask, dtype, _rows(nvec), nvec * (4 if dtype == workload.F32 else 8))


def test_backward_withheld_stage_and_corrupted_record():
    import time
    import torch
    R, C = _rows(), 20000
    y = torch.softmax(torch.randn(R, C, device="cuda"), -1)
    dy = torch.randn(R, C, device="cuda")
    dx = torch.full_like(y, -7.0)
    p = bsm.bsm_plan_create(y, dx, [R], [C], bsm.F32, bsm.POLICY_DYNAMIC, op=bsm.OP_BACKWARD, x2=dy)
    bsm.bsm_plan_debug(p, bsm.DEBUG_WITHHOLD_STAGE, 100_000_000)
    t0 = time.time()
    p.execute()
    torch.cuda.synchronize()
    assert time.time() - t0 < 5.0
    assert bsm.bsm_device_status() & bsm.DEV_TIMEOUT
    bsm.bsm_plan_debug(p, bsm.DEBUG_NONE)
    bsm.bsm_device_status_clear()
    dx.fill_(-7.0)
    bsm.bsm_plan_debug(p, bsm.DEBUG_CORRUPT_PATCH, 11)
    p.execute()
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == bsm.DEV_BOUNDS
    bsm.bsm_device_status_clear()
    skipped = (dx == -7.0).all(1).nonzero().flatten().tolist()
    assert skipped == [11]
    keep = [r for r in range(R) if r != 11]
    yd, gd = y[keep].double(), dy[keep].double()
    ref = yd * (gd - (yd * gd).sum(-1, keepdim=True))
    assert float((dx[keep].double() - ref).abs().max()) < 1e-7
    p.close()


@pytest.mark.parametrize("rows,C,K", [(0, 40000, 2), (64, 262144, 16)])
def test_forward_withheld_stage(rows, C, K):
    """Every wait of every CTA ends, with copies and other CTAs' partials in
    flight; the next execute is right."""
    import time
    import torch
    R = rows or _rows()
    w = workload.uniform("cluster fail", workload.F32, 1, R, C, 2.0, 0xC1F).materialize()
    x = to_device(w.x)
    y = torch.zeros_like(x)
    p = bsm.bsm_plan_create(x, y, w.rows, w.cols, w.dtype, bsm.POLICY_DYNAMIC)
    assert bsm.bsm_plan_kernel(p, 2 if rows else 0) == (bsm.KERNEL_CLUSTER, K)
    for _ in range(3):
        bsm.bsm_plan_debug(p, bsm.DEBUG_WITHHOLD_STAGE, 20_000_000)      # 0.02 s waits
        t0 = time.time()
        p.execute()
        torch.cuda.synchronize()
        assert time.time() - t0 < 5.0
        assert bsm.bsm_device_status() & bsm.DEV_TIMEOUT
        bsm.bsm_plan_debug(p, bsm.DEBUG_NONE)
        bsm.bsm_device_status_clear()
        y.fill_(float("nan"))
        p.execute()
        torch.cuda.synchronize()
        assert bsm.bsm_device_status() == 0
        check_rows_against_oracle(w, to_host(y), sample_rows(w, 16, 1))
        assert float((y.view(R, C).double().sum(1) - 1).abs().max()) < 1e-5
    p.close()


@pytest.mark.parametrize("others,kernel", [(58, bsm.KERNEL_STREAM), (500, bsm.KERNEL_CLUSTER)])
def test_backward_rows_beside_one_much_longer(others, kernel):
    """One row of 800 KiB sets the size of the clusters: rows that leave them
    nearly empty stay with one CTA each."""
    import torch
    n = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 6
    cols = np.full(n, others * 256, np.int32)
    cols[n // 3] = 800 * 256
    rows = np.ones(n, np.int32)
    off = np.concatenate([[0], np.cumsum(cols.astype(np.int64))[:-1]])
    total = int(cols.astype(np.int64).sum())
    dy = torch.randn(total, device="cuda")
    y = torch.rand(total, device="cuda") / 1000
    dx = torch.full_like(y, float("nan"))
    p = bsm.bsm_plan_create(y, dx, rows, cols, bsm.F32, bsm.POLICY_DYNAMIC, op=bsm.OP_BACKWARD, x2=dy)
    assert bsm.bsm_plan_kernel(p)[0] == kernel
    p.execute()
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0
    for o, c in zip(off.tolist(), cols.tolist()):
        yd, gd = y[o:o + c].double(), dy[o:o + c].double()
        ref = yd * (gd - (yd * gd).sum())
        # (two roundings of 2^-24 and the dot product's error, a few 2^-24 of it)
        assert float((dx[o:o + c].double() - ref).norm()) <= 4e-7 * float(ref.norm())
    p.close()
