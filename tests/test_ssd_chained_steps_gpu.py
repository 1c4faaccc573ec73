"""The SSD active block is the one launch that lets the next grid be placed
beside it, so a chain of steps depends on every step's wait: here step k + 1
reads the output of step k as its noisy input and writes over the input of step
k. Eager and captured in a graph, the chain has to give the bits of the same
steps with a synchronisation between them. (Every other kernel releases its
successor only by ending.)"""

import pytest

from paper_2607_02805_gb300.inputs import SsdWorkload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import to_device  # noqa: E402

STEPS, ROUNDS = 12, 10
PARAMS = ("A_f", "D_f", "A_r", "D_r")


@pytest.mark.parametrize("Bt,Bs,H,N", [(1, 256, 2, 128), (1, 256, 26, 128), (3, 128, 14, 64), (2, 256, 80, 64)])
def test_each_step_waits_for_the_one_before(Bt, Bs, H, N):
    wl = SsdWorkload(Bt, Bs, Bs, H, N, seed=Bs + H)
    t = {k: to_device(wl.dev_bits(k), binding.BDSCAN_F32 if k in PARAMS else binding.BDSCAN_BF16, "cuda")
         for k in wl.t32}
    for k in ("D_f", "D_r"):  # the chain neither grows nor dies out
        t[k].fill_(0.45)
    for k in ("B_f", "B_r"):
        t[k].mul_(0.05)
    dims = binding.make_ssd_dims(Bt, Bs, Bs, H, N)
    state = torch.linspace(-1, 1, Bt * H * 64 * N, device="cuda").reshape(Bt, H, 64, N).contiguous()
    x0, bufs = t["x_n"].clone(), [torch.empty_like(t["x_n"]) for _ in range(2)]
    ins = [dict(t, x_n=b) for b in bufs]

    def start():
        bufs[0].copy_(x0)
        bufs[1].fill_(float("nan"))

    def chain(stream, wait=False):
        for k in range(STEPS):
            binding.ssd_active_block(dims, state, ins[k & 1], bufs[1 - (k & 1)], stream)
            if wait:
                torch.cuda.synchronize()

    start()
    chain(None, wait=True)
    ref = [b.clone() for b in bufs]
    torch.cuda.synchronize()
    assert all(torch.isfinite(b.float()).all() for b in ref)
    assert not torch.equal(ref[0], x0) and float(ref[0].float().abs().max()) > 1e-3
    for _ in range(ROUNDS):
        start()
        chain(None)
        torch.cuda.synchronize()
        assert all(torch.equal(b, r) for b, r in zip(bufs, ref))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        chain(side)
    for _ in range(ROUNDS):
        start()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(b, r) for b, r in zip(bufs, ref))
    assert binding.bdscan_ssd_wait_flag(1) == 0
