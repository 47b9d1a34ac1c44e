"""Edges of the search kernels' loops: chunk, group and buffer boundaries.

Each case is compared with the same search through another route of the library that
shares no loop with the one under test (byte-identical records are the contract).
"""
import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module")
def ctx(kb):
    c = kb.Context(0)
    yield c
    c.close()


def _stack(kb, ctx, st, storage):
    N, H, W = st.sci.shape
    s = kb.Stack(ctx, N, H, W, storage)
    s.make_psi_phi(torch.from_numpy(st.sci).to(DEV), torch.from_numpy(st.var).to(DEV), None, st.psf)
    return s


def _records(kb, ctx, s, st, V, k, nu_min=-math.inf, flags=0):
    N, H, W = st.sci.shape
    job = kb.Job(ctx, H, W, N, V, k, flags & kb.KB_RESCORE_FP64)
    job.search(s, st.times, st.vx[:V], st.vy[:V], k, nu_min, flags)
    out = job.results()
    torch.cuda.synchronize()
    job.free()
    return out


@pytest.mark.parametrize("V", [1, 31, 32, 33, 97])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_pruning_at_the_edges_of_its_velocity_groups(kb, ctx, storage, V):
    """Bounds are taken for 32 velocities at once, within chunks of the offset table."""
    st = synth.small_stack(40 + V, 12, 41, 200, K=5, nan_frac=0.02, n_angles=10, n_speeds=10, s_hi=60.0, n_sources=6,
                           flux=60.0)
    s = _stack(kb, ctx, st, storage)
    for nu_min in (3.0, 6.0):
        ref = _records(kb, ctx, s, st, V, 4, nu_min)
        assert _records(kb, ctx, s, st, V, 4, nu_min, kb.KB_PRUNE).tobytes() == ref.tobytes()
    s.free()
