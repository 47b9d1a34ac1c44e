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


# epochs (groups of 4, 8, 16 and 32 lanes build the offset table), start pixels off the 64-pixel
# and 8-row tiles, velocities around the buffers' 4 and 5 entries and the table's chunks, list
# lengths of both merge networks, speeds that leave the image at some or all epochs
SHAPES = [(1, 9, 65, 3, 1, 8.0), (2, 8, 64, 4, 8, 8.0), (4, 17, 33, 5, 4, 200.0), (5, 40, 129, 100, 8, 60.0),
          (9, 7, 300, 64, 9, 30.0), (12, 33, 70, 129, 16, 500.0), (17, 24, 191, 43, 12, 90.0), (34, 16, 130, 90, 7, 40.0),
          (100, 9, 66, 30, 8, 25.0)]


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("N,H,W,V,k,s_hi", SHAPES)
def test_gather_kernel_equals_the_pipelined_kernel(kb, ctx, storage, N, H, W, V, k, s_hi):
    """The register-gather kernel against the TMA kernel, which has its own gathers and lists."""
    st = synth.small_stack(7 * N + k, N, H, W, K=5, nan_frac=0.05, n_angles=10, n_speeds=13, s_hi=s_hi, n_sources=3,
                           flux=40.0)
    s = _stack(kb, ctx, st, storage)
    for nu_min in (-math.inf, 2.0):
        ctx.set_search_variant(5)
        ref = _records(kb, ctx, s, st, V, k, nu_min)
        ctx.set_search_variant(0)
        assert _records(kb, ctx, s, st, V, k, nu_min).tobytes() == ref.tobytes()
    s.free()


@pytest.mark.parametrize("n0", [2, 6])
def test_epochs_at_the_reference_time(kb, ctx, n0):
    """n0 of 6 epochs at the earliest time: the table holds the others only, or nothing at all."""
    times = np.concatenate([np.zeros(n0), np.linspace(0.3, 1.5, 6 - n0)])
    st = synth.small_stack(90 + n0, 6, 21, 80, K=5, times=times, n_angles=6, n_speeds=6, s_hi=40.0, n_sources=2, flux=40.0)
    s = _stack(kb, ctx, st, "f32")
    ctx.set_search_variant(5)
    ref = _records(kb, ctx, s, st, 36, 8)
    ctx.set_search_variant(0)
    assert _records(kb, ctx, s, st, 36, 8).tobytes() == ref.tobytes()
    s.free()


@pytest.mark.parametrize("storage", ["bf16", "f16"])
@pytest.mark.parametrize("k", [1, 6, 8, 10])
def test_key_lists_at_their_lengths(kb, ctx, storage, k):
    """Candidate lists of 3 to 15 keys: the rescored records are those of the FP32 planes in FP64."""
    st = synth.small_stack(60 + k, 9, 37, 150, K=5, nan_frac=0.02, n_angles=10, n_speeds=13, s_hi=70.0, n_sources=5,
                           flux=40.0)
    s, f = _stack(kb, ctx, st, storage), _stack(kb, ctx, st, "f32")
    got = _records(kb, ctx, s, st, 130, k, flags=kb.KB_RESCORE_FP64)
    ref = _records(kb, ctx, f, st, 130, k, flags=kb.KB_RESCORE_FP64)
    assert got.tobytes() == ref.tobytes()
    for o in (s, f):
        o.free()
