"""Where the width of the search's offsets changes: planes between 2 and 4 GiB, where byte offsets pass
2^31, and just above 4 GiB, where short lists take 64-bit offsets and the others keep 32-bit ones.

Only 4 of the 128 epochs carry data; the others are masked everywhere and add exact zeros, so every
record must equal, bit for bit, that of the 4-epoch stack (nobs apart, which counts masked epochs too).
"""
import math

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
N, W, REAL = 128, 4096, [0, 41, 87, 127]
FIELDS = ("x0", "y0", "vidx", "vx", "vy", "psi", "phi", "nu", "alpha")


def _host(kb, job, H, k):
    out = torch.empty(H * W * k * kb.RESULT_DTYPE.itemsize, dtype=torch.uint8, device=DEV)
    job.results(out)
    return out.cpu().numpy().view(kb.RESULT_DTYPE).reshape(H, W, k)


@pytest.mark.parametrize("H", [700, 1000])
@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_widths_around_4_gib(kb, storage, H):
    below = N * (H + 16) * (W + 260) * 8 < 2 ** 32
    small = synth.small_stack(H, len(REAL), H, W, K=5, var_lo=80, var_hi=120, nan_frac=0.005, times=[0.0, 0.4, 1.1, 2.0],
                              n_angles=4, n_speeds=4, s_lo=20.0, s_hi=200.0, n_sources=20, flux=60.0)
    times = np.sort(np.random.default_rng(H).uniform(0.0, 2.0, N))
    times[REAL] = small.times
    psf = np.stack([small.psf[0]] * N)
    psf[REAL] = small.psf
    sci = torch.zeros((N, H, W), dtype=torch.float32, device=DEV)
    var = torch.full((N, H, W), math.inf, dtype=torch.float32, device=DEV)
    sci[REAL], var[REAL] = torch.from_numpy(small.sci).to(DEV), torch.from_numpy(small.var).to(DEV)
    ctx = kb.Context(0)
    big, ref = kb.Stack(ctx, N, H, W, storage), kb.Stack(ctx, len(REAL), H, W, storage)
    big.make_psi_phi(sci, var, None, psf)
    ref.make_psi_phi(sci[REAL].contiguous(), var[REAL].contiguous(), None, small.psf)
    del sci, var
    for k, flags in ((4, 0), (12, 0)) + (((8, kb.KB_RESCORE_FP64),) if storage != "f32" else ()):
        got, want = (kb.Job(ctx, H, W, s.N, small.vx.size, k, flags) for s in (big, ref))
        want.search(ref, small.times, small.vx, small.vy, k, -math.inf, flags)
        w = _host(kb, want, H, k)
        got.search(big, times, small.vx, small.vy, k, -math.inf, flags)
        g = _host(kb, got, H, k)
        for f in FIELDS:
            assert np.array_equal(g[f], w[f]), (k, flags, f)
        batch = kb.Batch(ctx, [dict(job=got, stack=big, times=times, vx=small.vx, vy=small.vy, topk=k, flags=flags)],
                         autotune=False)
        assert batch.groups()[0].index_bits == (32 if below or k > 4 else 64)
        batch.run()
        g = _host(kb, got, H, k)
        for f in FIELDS:
            assert np.array_equal(g[f], w[f]), (k, flags, f)
        batch.free()
        got.free()
        want.free()
    big.free()
    ref.free()
    ctx.close()
