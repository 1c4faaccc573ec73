"""The cache build without a workspace over more chunks than the plain chunk
carry takes: the final state alone, with and without a partial last chunk, and
every state, has the launches and the bits of the build with a workspace."""

import pytest

from paper_2607_02805_gb300.inputs import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import to_device  # noqa: E402


@pytest.mark.parametrize("chunks,tail,emit_all", [(40, 0, 0), (40, 3, 0), (40, 3, 1), (8, 0, 0)])
def test_noalloc_over_many_chunks(chunks, tail, emit_all):
    Bt, Bs, D, N = 2, 16, 136, 16
    L = chunks * binding.bdscan_chunk_tokens(Bs) + tail * Bs
    wl = Workload(Bt, L, Bs, D, N, dtype="bf16", seed=chunks + tail, with_grads=False, with_init=True,
                  parts=("clean",))
    dims = binding.make_dims(Bt, L, Bs, D, N, binding.BDSCAN_BF16)
    t = {k: to_device(wl.dev_bits(k), binding.BDSCAN_BF16, "cuda") for k in wl.t32}
    want, got = [torch.full((Bt, L // Bs if emit_all else 1, D, N), float("nan"), device="cuda") for _ in range(2)]
    ws = torch.empty(binding.bdscan_boundary_states_workspace_size(dims, emit_all), dtype=torch.uint8, device="cuda")
    binding.boundary_states(dims, t, t["init_state"], None, want, emit_all, ws)
    launches = binding.bdscan_last_launch_count()
    rc = binding.bdscan_boundary_states_noalloc(
        dims, binding.make_clean(t), t["A_f"].data_ptr(), t["D_f"].data_ptr(), t["init_state"].data_ptr(), None,
        got.data_ptr(), emit_all, torch.cuda.current_stream().cuda_stream)
    assert rc == 0, binding.bdscan_last_error()
    assert binding.bdscan_last_launch_count() == launches
    torch.cuda.synchronize()
    assert torch.equal(got, want)
