"""Small problems take their own launches: every block a backward chunk of its
own with its three parts in three CTAs (dx_n joined afterwards), and the noisy
blocks of the forward apart from the clean rescan. Sizes on both sides of
those lines, blocks of one token, of a part of a segment, of several segments
and of the longest that takes part, ragged channel groups, state gradients,
every type, against the fp64 oracle; the noisy outputs apart are the bits of
the cached active block."""

import pytest

import parity as P
from paper_2607_02805_gb300.inputs import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import Layer, to_numpy  # noqa: E402


@pytest.mark.parametrize("Bt,L,Bs,D,N,dt,od", [
    (1, 17, 1, 8, 16, "bf16", None),                  # blocks of one token
    (2, 36, 12, 132, 8, "f32", None),                 # part of a segment, a second channel group of 4
    (1, 152 * 16, 16, 40, 16, "bf16", None),          # 456 CTAs: the last problem that is split
    (1, 153 * 16, 16, 40, 16, "bf16", None),          # 459: the first that is not
    (3, 96, 48, 200, 16, "f32", None),                # three segments
    (1, 384, 128, 64, 16, "bf16", binding.BDSCAN_F32),  # the longest block that is split
    (1, 512, 256, 64, 8, "f32", None),                # above it
    (2, 40 * 16, 16, 1024, 16, "f32", None),          # fp32 with one staging buffer, several blocks per chunk
    (2, 90 * 7, 7, 520, 16, "f32", None),             # the same in tiles of short blocks
])
def test_small_problems_match_oracle(Bt, L, Bs, D, N, dt, od):
    P.oracle_threads()
    wl = Workload(Bt, L, Bs, D, N, dtype=dt, seed=L + D, with_dstates=True)
    lay = Layer(wl, out_dtype=od)
    lay.forward()
    lay.alloc_backward()
    for g in lay.g.values():
        g.fill_(float("nan"))
    lay.backward()
    torch.cuda.synchronize()
    u = P.BF16_U if lay.out_torch == torch.bfloat16 else 0.0
    y_c, y_n, st = P.oracle_forward(wl)
    P.assert_close("y_c", to_numpy(lay.y_c), y_c, P.FWD_TOL, u)
    P.assert_close("y_n", to_numpy(lay.y_n), y_n, P.FWD_TOL, u)
    P.assert_close("states", to_numpy(lay.states), st, P.FWD_TOL)
    ref = P.oracle_backward(wl, st, use_dstates=True)
    for k, v in lay.g.items():
        P.assert_close("d" + k, to_numpy(v), ref[k], P.GRAD_TOL, 0.0 if k in P.PARAMS else u)


def test_back_to_back_small_steps_keep_their_order():
    """Small launches may be placed before their predecessor has ended; two
    steps that share every buffer but the inputs, enqueued without a wait,
    give the bits of the same steps run one at a time."""
    wls = [Workload(1, 256, 16, 32, 8, dtype="f32", seed=s) for s in (5, 6)]
    lay = Layer(wls[0])
    lay.alloc_backward()
    ins = [lay.t, Layer(wls[1]).t]

    def outputs():
        return [lay.y_c, lay.y_n, lay.states] + list(lay.g.values())

    def step(t):
        lay.t = t
        lay.forward()
        lay.backward(use_dstates=False)

    step(ins[1])
    torch.cuda.synchronize()
    alone = [v.clone() for v in outputs()]
    torch.cuda.synchronize()
    for _ in range(20):
        step(ins[0])
        step(ins[1])
    torch.cuda.synchronize()
    assert all(torch.equal(a, v) for a, v in zip(alone, outputs()))
