"""The mixer's token sweeps where they can go wrong: both sweep lengths (8
tokens for small problems, 32 once there is work for every SM), streams whose
length is no multiple of the sweep, blocks that start inside a sweep and
windows that span several blocks, channel counts that leave warps partly
empty, every input and output type, against the fp64 oracle (every gradient)."""

import pytest

import parity as P
import test_mixer_gpu as M
from paper_2607_02805_gb300.inputs import MixerWorkload

pytestmark = pytest.mark.gpu

from paper_2607_02805_gb300 import binding  # noqa: E402


@pytest.mark.parametrize("Bt,L,Bs,D,N,dt,od", [
    (10, 2052, 12, 256, 8, "bf16", None),              # 32-token sweeps, the last one of 4 tokens
    (12, 2048 + 16, 16, 260, 8, "f32", None),          # 32-token sweeps, fp32, a ragged channel tile
    (3, 39, 3, 72, 16, "bf16", binding.BDSCAN_F32),    # 8-token sweeps, the last one of 7
    (1, 5, 1, 8, 8, "bf16", None),                     # shorter than one sweep, blocks of one token
    (2, 9, 9, 36, 8, "f32", None),                     # one block, one token past a sweep
])
def test_mixer_sweeps_match_oracle(Bt, L, Bs, D, N, dt, od):
    P.oracle_threads()
    wl = MixerWorkload(Bt, L, Bs, D, N, dtype=dt, seed=L)
    _, _, out_c, out_n, st, g, u = M._run(wl, od)
    M._check(wl, out_c, out_n, st, g, u)
