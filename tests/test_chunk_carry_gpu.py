"""The chunk carry's ring of staged chunk rows: chunk counts around the ring's
stages (16 rows, four stages), channel counts that leave the last CTA's 64
(channel, state) elements partly empty, a partial last chunk, an initial
state, against the fp64 oracle; the build that keeps only the final state
(which writes no chunk start states) gives the bits of the one that keeps
all of them."""

import pytest

import parity as P
from paper_2607_02805_gb300.inputs import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import to_device, to_numpy  # noqa: E402


@pytest.mark.parametrize("Bt,chunks,tail,Bs,D,N,dt", [
    (1, 1, 0, 16, 8, 16, "bf16"),     # one chunk, two whole CTAs
    (2, 15, 1, 16, 12, 8, "f32"),     # 96 elements: the second CTA half empty; one block past the chunks
    (2, 16, 0, 32, 20, 16, "f32"),    # exactly one stage
    (1, 49, 3, 16, 24, 16, "bf16"),   # one row more than the stages in flight
    (1, 80, 0, 64, 36, 8, "f32"),     # the ring wraps
    (1, 32, 1, 16, 24, 16, "bf16"),   # the last count without the ring
    (2, 33, 0, 32, 20, 16, "f32"),    # the first with it, one row past two stages
    (2, 47, 1, 16, 12, 8, "f32"),     # the ring with the second CTA half empty
    (3, 0, 2, 16, 8, 16, "bf16"),     # no full chunk
])
def test_chunk_carry_matches_oracle(Bt, chunks, tail, Bs, D, N, dt):
    import oracle
    P.oracle_threads()
    code = binding.BDSCAN_BF16 if dt == "bf16" else binding.BDSCAN_F32
    L = chunks * binding.bdscan_chunk_tokens(Bs) + tail * Bs
    wl = Workload(Bt, L, Bs, D, N, dtype=dt, seed=chunks + 1, with_grads=False, with_init=True, parts=("clean",))
    t = {k: to_device(wl.dev_bits(k), code, "cuda") for k in wl.t32}
    dims = binding.make_dims(Bt, L, Bs, D, N, code)
    ws = torch.empty(binding.bdscan_boundary_states_workspace_size(dims, 1), dtype=torch.uint8, device="cuda")
    every = torch.full((Bt, L // Bs, D, N), float("nan"), device="cuda")
    last = torch.full((Bt, 1, D, N), float("nan"), device="cuda")
    binding.boundary_states(dims, t, t["init_state"], None, every, 1, ws)
    binding.boundary_states(dims, t, t["init_state"], None, last, 0, ws)
    torch.cuda.synchronize()
    assert torch.equal(last[:, 0], every[:, -1])
    d = P.slice_channels(wl, None)
    ref, _ = oracle.boundary_states(Bs, d["x_c"], d["dt_c"], d["B_c"], d["C_c"], d["A_f"], d["D_f"],
                                    d["init_state"], emit_all=True)
    P.assert_close("states", to_numpy(every), ref, P.FWD_TOL)
