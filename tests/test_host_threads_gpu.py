"""Host threads on one device. A kernel's largest dynamic shared memory is an
attribute of the kernel, shared by every thread: a call must neither lower it
under a launch of another thread nor leave it below what it launches with
itself. Each thread has its own stream, tensors and workspaces; every call has
to succeed and to give the bits of the same call made alone."""

import ctypes
import threading

import pytest

from paper_2607_02805_gb300.inputs import Workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - collected on CPU machines
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2607_02805_gb300 import binding  # noqa: E402
from paper_2607_02805_gb300.layer import Layer  # noqa: E402


def _train(Bt, L, Bs, D, N, dt, seed):
    """A training step and its outputs."""
    lay = Layer(Workload(Bt, L, Bs, D, N, dtype=dt, seed=seed))
    lay.alloc_backward()

    def step(stream):
        lay.forward(stream)
        lay.backward(stream, use_dstates=False)

    return step, [lay.y_c, lay.y_n, lay.states] + list(lay.g.values())


def _backward(Bt, L, Bs, D, N, dt, seed):
    """The backward alone, with its arguments made once: the threads then spend
    their time inside the library, where the interpreter's lock is released."""
    lay = Layer(Workload(Bt, L, Bs, D, N, dtype=dt, seed=seed))
    lay.alloc_backward()
    lay.forward()
    g, lib, p = lay.g, binding.load(), binding._ptr
    gc = binding.bdscan_clean_grads(*[p(g[k]) for k in ("x_c", "dt_c", "B_c", "C_c")])
    gn = binding.bdscan_noisy_grads(*[p(g[k]) for k in ("x_n", "dt_f", "B_f", "C_f", "dt_r", "B_r", "C_r")])
    gp = binding.bdscan_param_grads(*[p(g[k]) for k in ("A_f", "D_f", "A_r", "D_r")])
    structs = [lay.dims, binding.make_clean(lay.t), binding.make_noisy(lay.t), binding.make_params(lay.t), gc, gn, gp]
    dims, cl, nz, pr, gc, gn, gp = [ctypes.byref(v) for v in structs]

    def step(stream):
        rc = lib.bdscan_backward(dims, cl, nz, pr, p(lay.states), p(lay.t["dy_c"]), p(lay.t["dy_n"]), None, gc, gn, gp,
                                 p(lay.ws_b), lay.ws_b.numel() * 4, binding._stream(stream))
        assert rc == 0, (rc, binding.bdscan_last_error())

    step.keep = structs
    return step, list(g.values())


def _forward(Bt, L, Bs, D, N, dt, seed):
    lay = Layer(Workload(Bt, L, Bs, D, N, dtype=dt, seed=seed, with_grads=False))
    return lay.forward, [lay.y_c, lay.y_n, lay.states]


def _active(Bt, Bs, D, N, dt, seed):
    wl = Workload(Bt, Bs, Bs, D, N, dtype=dt, seed=seed, with_grads=False, parts=("noisy",))
    lay = Layer(wl)
    state = torch.linspace(-1, 1, Bt * D * N, device="cuda").reshape(Bt, D, N).contiguous()
    return (lambda stream: binding.active_block(lay.dims, state, lay.t, lay.y_n, stream)), [lay.y_n]


def _in_threads(jobs, calls):
    alone = []
    for step, outs in jobs:
        step(None)
        torch.cuda.synchronize()
        alone.append([o.clone() for o in outs])
    errors, barrier = [], threading.Barrier(len(jobs))

    def work(step):
        try:
            stream = torch.cuda.Stream()
            barrier.wait()
            for _ in range(calls):
                step(stream)
            stream.synchronize()
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(step,)) for step, _ in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    for (_, outs), ref in zip(jobs, alone):
        assert all(torch.equal(o, r) for o, r in zip(outs, ref))


@pytest.mark.parametrize("L,Bs,D,N,dt", [
    (16, 16, 8, 8, "f32"),     # one segment
    (24, 12, 8, 8, "f32"),     # a part of a segment
    (32, 32, 8, 16, "f32"),    # two segments
    (16, 16, 8, 16, "bf16"),
])
def test_backwards_of_equal_sizes(L, Bs, D, N, dt):
    """fp32 calls choose between two staging plans with different amounts of
    shared memory; looking at the other plan may not show."""
    _in_threads([_backward(1, L, Bs, D, N, dt, seed) for seed in (1, 2, 3, 4)], 10000)


def test_training_steps_of_block_sizes_that_share_an_instance():
    _in_threads([_train(1, L, Bs, 64, 16, "f32", 4) for L, Bs in ((256, 32), (256, 64), (384, 128))], 1000)


def test_forwards_of_block_sizes_that_share_an_instance():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = 2 * sms  # the fused scan of both streams
    _in_threads([_forward(rows, Bs, Bs, 64, 16, "bf16", 5) for Bs in (32, 64, 128)], 1500)


def test_active_blocks_of_sizes_that_share_an_instance():
    _in_threads([_active(1, Bs, 64, 16, "f32", 6) for Bs in (96, 160, 256)], 4000)
