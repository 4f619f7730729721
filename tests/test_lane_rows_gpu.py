"""Rows that one lane group's registers hold (every class and its edges, 16
bytes to 2 KiB), against the oracle and bit-identical across policies, whose
patches end such rows at different places; causal, non-finite and lowest-value
rows, and the backward pass."""
import pytest

from gpu_util import bits, check_all_against_oracle, run, to_device, to_host
from paper_2002_07062_gb300 import bsm, workload

pytestmark = pytest.mark.gpu

POLICIES = [bsm.POLICY_RR, bsm.POLICY_DYNAMIC, bsm.POLICY_CBMF_LB, bsm.POLICY_WHOLE_GPU]
NVEC = [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 24, 25, 31, 32, 33, 48, 49, 63, 64, 65, 96, 97, 127, 128]


@pytest.fixture(scope="module", autouse=True)
def setup():
    import torch
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)
    bsm.bsm_device_status_clear()
    yield
    bsm.bsm_cache_clear()


@pytest.mark.parametrize("nvec", NVEC)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
@pytest.mark.parametrize("flags", [0, workload.CAUSAL])
def test_row_lengths_of_every_class(nvec, dtype, flags):
    import torch
    C = nvec * (4 if dtype == workload.F32 else 8)
    w = workload.uniform("lanes", dtype, 7, 333, C, 3.0, 0x1A0 + nvec + flags, flags).materialize()
    x = to_device(w.x)
    ys = [run(w, x, p) for p in POLICIES]
    bsm.bsm_set_device_checks(True)
    ys.append(run(w, x, bsm.POLICY_DYNAMIC))
    torch.cuda.synchronize()
    bsm.bsm_set_device_checks(False)
    assert bsm.bsm_device_status() == 0, bsm.bsm_device_debug()
    for y in ys[1:]:
        assert torch.equal(bits(y), bits(ys[0]))
    check_all_against_oracle(w, to_host(ys[0]))


@pytest.mark.parametrize("nvec", [2, 6, 12, 20, 40, 100])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_non_finite_and_lowest_value_rows(nvec, dtype):
    import torch
    t = torch.float32 if dtype == "f32" else torch.bfloat16
    C = nvec * (4 if dtype == "f32" else 8)
    low = torch.finfo(t).min
    x = torch.randn(7, C, device="cuda").to(t)
    x[1, C - 1] = float("nan")
    x[2, 0] = float("inf")
    x[3, :] = -float("inf")
    x[3, C // 2] = 1.0
    x[4, :] = -float("inf")
    x[5, :] = low
    x[5, C - 3] = 2.0
    y = torch.full_like(x, -1.0)
    bsm.bsm_softmax_ex(x, y, 1, 7, C, bsm.F32 if dtype == "f32" else bsm.BF16, bsm.POLICY_DYNAMIC)
    torch.cuda.synchronize()
    assert torch.isnan(y[[1, 2, 4]]).all()
    for r, c in ((3, C // 2), (5, C - 3)):
        assert float(y[r, c]) == 1.0 and int(y[r].count_nonzero()) == 1
    ref = torch.softmax(x[[0, 6]].double(), -1)
    err = (y[[0, 6]].double() - ref).abs()
    assert float(err.max()) <= 2e-6 if dtype == "f32" else bool((err <= ref * 2.0 ** -8 + 1e-30).all())


@pytest.mark.parametrize("nvec", NVEC)
@pytest.mark.parametrize("dtype", [workload.F32, workload.BF16])
def test_backward_row_lengths_of_every_class(nvec, dtype):
    import torch
    from test_backward_gpu import _check, _inputs
    C = nvec * (4 if dtype == workload.F32 else 8)
    w = workload.uniform("lanes bwd", dtype, 7, 333, C, 2.0, 0x1B0 + nvec).materialize()
    y, dy = _inputs(w)
    yd, dyd = to_device(y), to_device(dy)
    outs = []
    for p in POLICIES:
        dx = torch.full_like(yd, float("nan"))
        bsm.bsm_softmax_backward(yd, dyd, dx, w.nslices, 333, C, dtype, p)
        outs.append(dx)
    bsm.bsm_softmax_backward(yd, dyd, dyd, w.nslices, 333, C, dtype, bsm.POLICY_DYNAMIC)   # in place
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0
    for dx in outs[1:] + [dyd]:
        assert torch.equal(bits(dx), bits(outs[0]))
    _check(w, y, dy, to_host(outs[0]))
