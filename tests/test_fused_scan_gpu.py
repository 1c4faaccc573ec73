"""The forward's two launch forms against each other. A forward with at least
two CTAs of the fused block scan per SM runs clean and noisy tokens in one
kernel (three launches); below that the noisy blocks have a launch of their own
(four). A batch row alone is such a small problem, so every row of a large
batch has to have the bits that it has alone, and the cached active block the
bits of the row's last noisy block. Blocks of every kind (tiles of 4 and 7
tokens, one segment, several segments with and without a remainder), both state
sizes, every type, ragged channel groups and last chunks; all of it against the
fp64 oracle too."""

import numpy as np
import pytest

import parity as P
from paper_2607_02805_gb300.inputs import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import Layer, to_numpy  # noqa: E402

F32 = binding.BDSCAN_F32


def _row(wl, b):
    w = object.__new__(Workload)
    w.__dict__.update(wl.__dict__)
    w.t32 = {k: (np.ascontiguousarray(v[b:b + 1]) if v.ndim >= 3 else v) for k, v in wl.t32.items()}
    w.batch = 1
    return w


@pytest.mark.parametrize("L,Bs,D,N,dt,od", [
    (256, 4, 136, 16, "bf16", None),
    (256, 4, 132, 8, "f32", None),
    (252, 7, 132, 16, "f32", None),
    (259, 7, 136, 8, "bf16", F32),
    (272, 16, 136, 16, "bf16", None),
    (272, 16, 136, 8, "bf16", None),
    (256, 16, 132, 16, "f32", None),
    (256, 16, 136, 16, "bf16", F32),
    (260, 20, 136, 16, "bf16", None),
    (240, 20, 132, 8, "f32", None),
    (240, 48, 136, 16, "bf16", F32),
    (192, 48, 132, 16, "f32", None),
    (256, 128, 136, 8, "bf16", None),
])
def test_fused_and_apart_forwards_agree(L, Bs, D, N, dt, od):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tc = binding.bdscan_chunk_tokens(Bs)
    per_row = -(-L // tc) * -(-D // 128)
    Bt = -(-2 * sms // per_row)
    P.oracle_threads()
    wl = Workload(Bt, L, Bs, D, N, dtype=dt, seed=L + Bs + D, with_grads=False)
    lay = Layer(wl, out_dtype=od)
    lay.forward()
    assert binding.bdscan_last_launch_count() == 3
    torch.cuda.synchronize()
    for b in (0, Bt - 1):
        one = Layer(_row(wl, b), out_dtype=od)
        one.forward()
        assert binding.bdscan_last_launch_count() == 4
        y = torch.zeros((1, Bs, D), dtype=one.out_torch, device="cuda")
        last = {k: (v[:, L - Bs:].contiguous() if v.ndim == 3 else v) for k, v in one.t.items()}
        code = F32 if dt == "f32" else binding.BDSCAN_BF16
        binding.active_block(binding.make_dims(1, Bs, Bs, D, N, code, od), lay.states[b:b + 1, -2].contiguous(), last, y)
        torch.cuda.synchronize()
        assert torch.equal(one.y_c, lay.y_c[b:b + 1])
        assert torch.equal(one.states, lay.states[b:b + 1])
        assert torch.equal(one.y_n, lay.y_n[b:b + 1])
        assert torch.equal(y, lay.y_n[b:b + 1, L - Bs:])
    u = P.BF16_U if lay.out_torch == torch.bfloat16 else 0.0
    y_c, y_n, st = P.oracle_forward(wl)
    P.assert_close("y_c", to_numpy(lay.y_c), y_c, P.FWD_TOL, u)
    P.assert_close("y_n", to_numpy(lay.y_n), y_n, P.FWD_TOL, u)
    P.assert_close("states", to_numpy(lay.states), st, P.FWD_TOL)
