"""The chunk scan's split of a channel's states over CTAs: whole, halves and
quarters of 16 states, whole and halves of 8, chosen by the number of CTAs.
Sizes on both sides of each line (152 and 304 CTAs of 128 channels, 128
tokens per chunk), ragged channel counts, against the fp64 oracle; a
sequence's first chunks give the same bits alone and inside a longer one,
which takes another split."""

import pytest

import parity as P
from paper_2607_02805_gb300.inputs import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import to_device, to_numpy  # noqa: E402


def states(wl, dims, t, L):
    ws = torch.empty(binding.bdscan_boundary_states_workspace_size(dims, 1), dtype=torch.uint8, device="cuda")
    out = torch.full((1, L // wl.block, wl.d_inner, wl.d_state), float("nan"), device="cuda")
    binding.boundary_states(dims, t, t["init_state"], None, out, 1, ws)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("chunks,D,N,dt", [
    (1, 20, 16, "f32"),       # one CTA of a few channels
    (76, 160, 16, "bf16"),    # 152 CTAs: the last count of quarters
    (77, 160, 16, "bf16"),    # 154: halves
    (152, 136, 16, "bf16"),   # 304: the last count of halves
    (153, 136, 16, "f32"),    # 306: whole
    (76, 160, 8, "f32"),      # eight states: halves
    (77, 160, 8, "bf16"),     # whole
])
def test_split_matches_oracle_and_longer_stream(chunks, D, N, dt):
    import oracle
    P.oracle_threads()
    Bs, code = 16, binding.BDSCAN_BF16 if dt == "bf16" else binding.BDSCAN_F32
    tc = binding.bdscan_chunk_tokens(Bs)
    L, few = chunks * tc, min(chunks, 2) * tc
    wl = Workload(1, L, Bs, D, N, dtype=dt, seed=chunks, with_grads=False, with_init=True, parts=("clean",))
    t = {k: to_device(wl.dev_bits(k), code, "cuda") for k in wl.t32}
    every = states(wl, binding.make_dims(1, L, Bs, D, N, code), t, L)
    d = P.slice_channels(wl, None)
    ref, _ = oracle.boundary_states(Bs, d["x_c"], d["dt_c"], d["B_c"], d["C_c"], d["A_f"], d["D_f"],
                                    d["init_state"], emit_all=True)
    P.assert_close("states", to_numpy(every), ref, P.FWD_TOL)
    short = {k: v[:, :few].contiguous() if k in ("x_c", "dt_c", "B_c", "C_c") else v for k, v in t.items()}
    head = states(wl, binding.make_dims(1, few, Bs, D, N, code), short, few)
    assert torch.equal(head, every[:, : head.shape[1]])
