"""The batched product on pairs of CTAs (tiles of 256 rows: products bound by
the tensor cores): integer operands make every result exact, equal to the
oracle and, bit for bit, to single-CTA tiles (a caller's own split) and
between policies.  Tile counts under, over and ragged against the pairs, both
tile widths, K of a few blocks, of a ring's remainder and long."""
import numpy as np
import pytest

from oracle import bmm_oracle as O
from paper_2002_07062_gb300 import bsm, workload as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [  # B, M, N, K
    (1, 512, 512, 4096), (1, 256, 512, 4160), (8, 1024, 1024, 832), (19, 1280, 512, 640), (26, 512, 1280, 384),
    (32, 768, 384, 1088), (3, 2304, 1152, 704), (77, 512, 512, 576),
]


def _run(w, da, db, policy, split=None):
    dt = torch.float32 if w.out_dtype == W.F32 else torch.int16
    c = torch.full((w.B * w.M * w.N,), -1, dtype=dt, device="cuda")
    if split:
        bsm.bsm_bmm_ex(da, db, c, w.B, w.M, w.N, w.K, w.out_dtype, policy, *split)
    else:
        bsm.bsm_bmm(da, db, c, w.B, w.M, w.N, w.K, w.out_dtype, policy)
    return c


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("out", [W.F32, W.BF16])
def test_pair_tiles_are_exact(shape, out):
    import __graft_entry__ as g
    g.build()
    B, M, N, K = shape
    w = W.BmmWorkload("pair", B, M, N, K, out, seed=0x9A1 + B + K, kind="int")
    a, bt = w.operands()
    da, db = (torch.from_numpy(t.view(np.int16)).cuda() for t in (a, bt))
    c = _run(w, da, db, bsm.POLICY_DYNAMIC)
    one = _run(w, da, db, bsm.POLICY_DYNAMIC, (2, 2, 1))
    others = [_run(w, da, db, p) for p in (bsm.POLICY_WHOLE_GPU, bsm.POLICY_RR, bsm.POLICY_CBMF, bsm.POLICY_CBMF_LB,
                                           bsm.POLICY_MINIMAX)]
    again = _run(w, da, db, bsm.POLICY_DYNAMIC)
    torch.cuda.synchronize()
    assert bsm.bsm_device_status() == 0
    for o in [one, again] + others:
        assert torch.equal(c, o)
    pick = sorted({0, B // 2, B - 1})
    a3, b3 = a.reshape(B, M * K)[pick].reshape(-1), bt.reshape(B, N * K)[pick].reshape(-1)
    ref = O.bmm_f64(a3, b3, len(pick), M, N, K)
    h = c.cpu().numpy().reshape(B, M, N)[pick]
    if out == W.F32:
        assert np.array_equal(h, ref.astype(np.float32))
    else:
        assert np.array_equal(h.view(np.uint16), O.round_bf16(ref))
