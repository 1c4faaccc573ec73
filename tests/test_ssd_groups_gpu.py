"""Head groups of the SSD backward: one head, one group, several groups with a
ragged last one, more heads than a block-state CTA holds (13), blocks of one
and two tiles, both state sizes, state gradients, against the fp64 oracle."""

import pytest

import parity as P
from paper_2607_02805_gb300.inputs import SsdWorkload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import to_device, to_numpy  # noqa: E402

NAMES = P.FWD_NAMES


@pytest.mark.parametrize("Bt,nb,Bs,H,N", [
    (1, 1, 128, 1, 64),      # one CTA
    (1, 3, 256, 14, 128),    # two tiles per block; 14 heads are above the block-state CTA's 13
    (5, 16, 128, 5, 128),    # 80 blocks: every head of a block in one CTA
    (13, 12, 128, 3, 64),    # 156 blocks: a second wave
    (2, 4, 256, 17, 64),     # ragged groups
])
def test_ssd_head_groups_match_oracle(Bt, nb, Bs, H, N):
    from oracle import ssd as oracle_ssd
    P.oracle_threads()
    L = nb * Bs
    wl = SsdWorkload(Bt, L, Bs, H, N, seed=H + nb, with_grads=True, with_dstates=True)
    f32 = ("A_f", "A_r", "D_f", "D_r", "dstates")
    t = {k: to_device(wl.dev_bits(k) if k != "dstates" else wl.t32[k],
                      binding.BDSCAN_F32 if k in f32 else binding.BDSCAN_BF16, "cuda") for k in wl.t32}
    dims = binding.make_ssd_dims(Bt, L, Bs, H, N)
    y = torch.empty_like(t["x_c"])
    st = torch.empty((Bt, nb, H, 64, N), device="cuda")
    ws = torch.empty(binding.bdscan_ssd_forward_workspace_size(dims), dtype=torch.uint8, device="cuda")
    binding.ssd_forward(dims, t, y, torch.empty_like(y), st, ws)
    g = {k: torch.full(t[k].shape, float("nan"), dtype=torch.float32 if k in f32 else torch.bfloat16, device="cuda")
         for k in NAMES}
    wsb = torch.empty(binding.bdscan_ssd_backward_workspace_size(dims), dtype=torch.uint8, device="cuda")
    binding.ssd_backward(dims, t, st, t["dy_c"], t["dy_n"], t["dstates"], g, wsb)
    torch.cuda.synchronize()
    assert binding.bdscan_ssd_wait_flag(1) == 0
    ref = oracle_ssd.backward(Bs, *[wl.f64(k) for k in NAMES], to_numpy(st), wl.f64("dy_c"), wl.f64("dy_n"),
                              wl.t32["dstates"].astype("float64"))
    for k in NAMES:
        P.assert_close("d" + k, to_numpy(g[k]), ref[k], P.GRAD_TOL, 0.0 if k in f32 else P.BF16_U)


@pytest.mark.parametrize("nb,Bt,H,N", [(64, 1, 1, 64), (65, 2, 2, 64), (70, 1, 3, 128), (97, 1, 1, 64)])
def test_ssd_long_state_pass_matches_oracle(nb, Bt, H, N):
    """The state recurrence on both sides of the length where it streams its
    blocks through a ring (64), with part of a ring stage left over; states and
    outputs against the oracle, the final-state build bit for bit."""
    from oracle import ssd as oracle_ssd
    P.oracle_threads()
    L = nb * 128
    wl = SsdWorkload(Bt, L, 128, H, N, seed=nb, with_init=True)
    t = {k: to_device(wl.dev_bits(k) if k != "init_state" else wl.t32[k],
                      binding.BDSCAN_F32 if k in ("A_f", "A_r", "D_f", "D_r", "init_state") else binding.BDSCAN_BF16,
                      "cuda") for k in wl.t32}
    dims = binding.make_ssd_dims(Bt, L, 128, H, N)
    every = torch.full((Bt, nb, H, 64, N), float("nan"), device="cuda")
    last = torch.full((Bt, 1, H, 64, N), float("nan"), device="cuda")
    y = torch.empty_like(t["x_c"])
    for emit, st, out in ((1, every, y), (0, last, None)):
        ws = torch.empty(binding.bdscan_ssd_boundary_states_workspace_size(dims, emit), dtype=torch.uint8, device="cuda")
        binding.ssd_boundary_states(dims, t, t["init_state"], out, st, emit, ws)
    torch.cuda.synchronize()
    assert binding.bdscan_ssd_wait_flag(1) == 0
    assert torch.equal(last[:, 0], every[:, -1])
    ref = oracle_ssd.boundary_states(128, *[wl.f64(k) for k in ("x_c", "dt_c", "B_c", "C_c", "A_f", "D_f")],
                                     init_state=wl.t32["init_state"].astype("float64"), emit_all=True, want_y=True)
    P.assert_close("states", to_numpy(every), ref[0], P.FWD_TOL)
    P.assert_close("y_c", to_numpy(y), ref[1], P.FWD_TOL, P.BF16_U)
