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


@pytest.mark.parametrize("N,H,W,k", [(5, 9, 255, 3), (16, 6, 257, 8), (17, 5, 300, 16), (32, 4, 70, 1), (33, 6, 40, 5),
                                     (70, 3, 33, 2)])
def test_filter_against_direct_sums(kb, ctx, N, H, W, k):
    """Epochs held in registers (up to 16, up to 32) or gathered again, strips of 256 pixels: sums,
    rejections and scores of the direct FP64 form, which rounds alike step by step."""
    st = synth.small_stack(200 + N, N, H, W, K=5, nan_frac=0.1, n_angles=6, n_speeds=6, s_hi=12.0, n_sources=3, flux=60.0)
    s = _stack(kb, ctx, st, "f32")
    job = kb.Job(ctx, H, W, N, st.vx.size, k)
    job.search(s, st.times, st.vx, st.vy)
    rec, got = job.results(), job.filter_lightcurves(s, 2.5)
    planes = np.empty((N, H, W, 2), np.float32)
    s.copy_planes(0, planes)
    dx, dy = kb.offsets(st.times, st.vx, st.vy)
    y, x, _ = np.meshgrid(np.arange(H), np.arange(W), np.arange(k), indexing="ij")
    v, order, q = np.maximum(rec["vidx"], 0), np.argsort(st.times, kind="stable"), {}
    P, F = np.zeros((H, W, k)), np.zeros((H, W, k))
    for e in order:
        yy, xx = y + dy[v, e], x + dx[v, e]
        ok = (rec["vidx"] >= 0) & (yy >= 0) & (yy < H) & (xx >= 0) & (xx < W)
        q[e] = np.where(ok[..., None], planes[e][np.clip(yy, 0, H - 1), np.clip(xx, 0, W - 1)].astype(np.float64), 0.0), ok
        P, F = P + q[e][0][..., 0], F + q[e][0][..., 1]
    Pk, Fk, n, bits = np.zeros_like(P), np.zeros_like(P), np.zeros(P.shape, int), np.zeros(P.shape + (4,), np.uint32)
    for e in order:
        (pe, fe), ok = (q[e][0][..., 0], q[e][0][..., 1]), q[e][1]
        rest = F - fe
        out = ok & (fe > 0) & (rest > 0) & ((pe * F - P * fe) ** 2 > 6.25 * F * fe * rest)
        keep = ok & ~out
        Pk, Fk, n = Pk + np.where(keep, pe, 0.0), Fk + np.where(keep, fe, 0.0), n + keep
        bits[..., e // 32] |= np.where(out, np.uint32(1 << (e % 32)), np.uint32(0)).astype(np.uint32)
    assert np.array_equal(got["rejected"], bits) and np.array_equal(got["nobs"], n)
    assert np.array_equal(got["nrejected"], sum(((bits >> b) & 1).sum(-1) for b in range(32)))
    assert np.array_equal(got["psi"], Pk) and np.array_equal(got["phi"], Fk)
    ok = Fk > 0
    assert np.array_equal(got["nu"][ok], Pk[ok] / np.sqrt(Fk[ok])) and np.all(got["nu"][~ok] == -np.inf)
    assert np.array_equal(got["alpha"][ok], Pk[ok] / Fk[ok]) and (bits.any() or H * W < 200)
    assert np.array_equal(got["x0"], x) and np.array_equal(got["y0"], y) and np.array_equal(got["vidx"], rec["vidx"])
    job.free()
    s.free()


@pytest.mark.parametrize("n", [1, 31, 33, 700])
@pytest.mark.parametrize("eps", [2.0, 5.0])
def test_cluster_on_a_lattice(kb, ctx, n, eps):
    """Whole-pixel spacings: many pairs lie at eps exactly, cells hold up to hundreds of points."""
    rng = np.random.default_rng(n)
    rec = np.zeros(n, kb.RESULT_DTYPE)
    rec["x0"], rec["y0"] = rng.integers(0, 24, n), rng.integers(0, 24, n)
    rec["vx"], rec["vy"] = rng.integers(0, 3, n), rng.integers(0, 3, n)
    rec["vidx"], rec["nu"] = rng.integers(-1, 40, n), rng.normal(5.0, 2.0, n)
    dev = torch.from_numpy(rec.view(np.uint8).copy()).to(DEV)
    for ms in (1, 4, 40):
        label, keep, core, groups = ctx.cluster(dev, 1.0, 1.0, eps, ms, core=True)
        p = np.stack([rec["x0"], rec["y0"], rec["vx"], rec["vy"]], 1).astype(np.float64)
        d2, ok = ((p[:, None] - p[None]) ** 2).sum(-1), rec["vidx"] >= 0   # exact: small whole numbers
        near = (d2 <= eps * eps) & ok[:, None] & ok[None]
        want_core = ok & (near.sum(1) >= ms)
        want = np.where(ok, np.arange(n), -1)
        link = near & want_core[:, None] & want_core[None]
        for _ in range(n):
            low = np.where(link, want[None], n).min(1, initial=n)
            new = np.where(want_core, np.minimum(want, low), want)
            if np.array_equal(new, want):
                break
            want = new
        for i in np.flatnonzero(ok & ~want_core):
            c = np.flatnonzero(near[i] & want_core)
            if c.size:
                want[i] = want[c[np.lexsort((c, d2[i, c]))[0]]]
        assert np.array_equal(label.cpu().numpy(), want)
        assert np.array_equal(core.cpu().numpy(), want_core)
        assert groups == np.unique(want[ok]).size == int(keep.sum())


@pytest.mark.parametrize("N,H,W,K", [(1, 1, 1, 3), (3, 33, 63, 7), (2, 70, 66, 13), (9, 130, 129, 21), (1, 1200, 64, 5),
                                     (4, 97, 1027, 17)])
def test_streaming_images_equal_the_tile_kernel(kb, ctx, N, H, W, K):
    """Aligned and ragged widths, short and split columns, against the tile kernel: the same PSF within
    23 x 23 taps, whose added zeros change no sum.  Planes, and the 16-bit codes, copied to both kinds of memory."""
    st = synth.small_stack(N + K, N, H, W, K=K, nan_frac=0.05, mask_frac=0.05, n_sources=1, flux=50.0)
    wide = np.zeros((N, 23, 23), np.float32)
    o = (23 - K) // 2
    wide[:, o:o + K, o:o + K] = st.psf
    mask = torch.from_numpy((np.arange(N * H * W).reshape(N, H, W) % 37 == 0).astype(np.uint8)).to(DEV)
    got = []
    for psf in (st.psf, wide):
        s = kb.Stack(ctx, N, H, W, "f16")
        s.make_psi_phi(torch.from_numpy(st.sci).to(DEV), torch.from_numpy(st.var).to(DEV), mask, psf)
        for which, dt, kind in ((0, torch.float32, np.float32), (1, torch.int16, np.int16)):
            d = torch.empty((N, H, W, 2), dtype=dt, device=DEV)
            h = np.empty((N, H, W, 2), kind)
            s.copy_planes(which, d)
            s.copy_planes(which, h)
            assert np.array_equal(d.cpu().numpy(), h)
            got.append(h)
        s.free()
    assert np.array_equal(got[0], got[2]) and np.array_equal(got[1], got[3])


# epochs on both sides of the steps of the buffers' rule (13, 17 and 33 past the reference time, and 65), list
# lengths whose lists leave buffers of 5, 4, 3 and 2 entries there
@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("N", [12, 15, 24, 34, 66])
def test_buffers_by_the_number_of_epochs(kb, ctx, storage, N):
    """Long lists (15 and 20 of them rescoring candidates) and key lists, whose buffers shorten with the epochs."""
    st = synth.small_stack(300 + N, N, 17, 130, K=5, nan_frac=0.02, n_angles=10, n_speeds=13, s_hi=60.0, n_sources=3,
                           flux=40.0)
    s, f = _stack(kb, ctx, st, storage), _stack(kb, ctx, st, "f32")
    for k in (9, 12, 14, 15, 16):
        ctx.set_search_variant(5)
        ref = _records(kb, ctx, s, st, 130, k).tobytes()
        for variant in (0, 4):
            ctx.set_search_variant(variant)
            assert _records(kb, ctx, s, st, 130, k).tobytes() == ref, (k, variant)
        ctx.set_search_variant(0)
        job = kb.Job(ctx, 17, 130, N, 130, k)
        batch = kb.Batch(ctx, [dict(job=job, stack=s, times=st.times, vx=st.vx, vy=st.vy, topk=k)], autotune=False)
        batch.run()
        assert job.results().tobytes() == ref, k
        torch.cuda.synchronize()
        batch.free()
        job.free()
    for k in (8, 12, 16):
        got = _records(kb, ctx, s, st, 130, k, flags=kb.KB_RESCORE_FP64)
        assert got.tobytes() == _records(kb, ctx, f, st, 130, k, flags=kb.KB_RESCORE_FP64).tobytes(), k
    for o in (s, f):
        o.free()


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("N,V", [(29, 70), (30, 70), (33, 70), (64, 40), (66, 33), (100, 21), (128, 40), (128, 3), (35, 1)])
def test_pruning_with_many_epochs(kb, ctx, storage, N, V):
    """Fewer than 32 velocities in a chunk of the table: several lanes share a velocity's bound."""
    st = synth.small_stack(500 + N, N, 19, 200, K=5, nan_frac=0.02, n_angles=10, n_speeds=10, s_hi=60.0, n_sources=6,
                           flux=60.0)
    s = _stack(kb, ctx, st, storage)
    for k, nu_min in ((1, 4.0), (4, 5.0), (8, 9.0), (10, 9.0)):
        ref = _records(kb, ctx, s, st, V, k, nu_min)
        assert _records(kb, ctx, s, st, V, k, nu_min, kb.KB_PRUNE).tobytes() == ref.tobytes()
    s.free()


@pytest.mark.parametrize("N,H,W,k", [(3, 40, 1, 1), (5, 11, 2, 16), (4, 3, 256, 7), (4, 5, 257, 5), (20, 4, 511, 3), (6, 2, 513, 9)])
def test_filter_on_strips_of_any_width(kb, ctx, N, H, W, k):
    """Images narrower than a strip, and wider ones that leave a ragged strip: with nothing rejected
    the filter returns the search's own trajectories, summed in 64 bits."""
    st = synth.small_stack(230 + W, N, H, W, K=3, nan_frac=0.1, n_angles=5, n_speeds=5, s_hi=6.0, n_sources=1, flux=30.0)
    s = _stack(kb, ctx, st, "f32")
    job = kb.Job(ctx, H, W, N, st.vx.size, k)
    job.search(s, st.times, st.vx, st.vy)
    rec, got = job.results(), job.filter_lightcurves(s, 1e6)
    y, x, _ = np.meshgrid(np.arange(H), np.arange(W), np.arange(k), indexing="ij")
    assert np.array_equal(got["x0"], x) and np.array_equal(got["y0"], y) and np.array_equal(got["vidx"], rec["vidx"])
    assert np.array_equal(got["nobs"], np.where(rec["vidx"] >= 0, rec["nobs"], 0)) and not got["nrejected"].any()
    # N FP32 additions against FP64 ones: N roundings of the partial sums, each at most the sum of the sizes
    planes = np.empty((N, H, W, 2), np.float32)
    s.copy_planes(0, planes)
    bound = N * 2.0 ** -24 * np.abs(planes).sum(0).max((0, 1)) * N
    assert np.abs(got["psi"] - rec["psi"]).max() <= bound[0] and np.abs(got["phi"] - rec["phi"]).max() <= bound[1]
    job.free()
    s.free()


def test_filter_where_products_are_subnormal(kb, ctx):
    """Two epochs whose phi lie 40 decades apart: the test's FP32 form has subnormal products on the way, and
    must leave them to FP64.  Values within 2e-4 of the rejection limit, decided as the direct sums decide."""
    rng = np.random.default_rng(5)
    H, W, nsigma = 64, 64, 1e-10
    phi = np.stack([10.0 ** rng.uniform(-36, -31, (H, W)), 10.0 ** rng.uniform(10, 14, (H, W))])
    var = (1.0 / phi).astype(np.float32)
    # |psi_0| F = nsigma sqrt(F phi_0 (F - phi_0)) up to 2e-4, psi_1 = 0
    psi0 = nsigma * np.sqrt(phi[0]) * (1.0 + rng.uniform(-2e-4, 2e-4, (H, W)))
    sci = np.stack([psi0 * var[0], np.zeros((H, W))]).astype(np.float32)
    s = kb.Stack(ctx, 2, H, W, "f32")
    s.make_psi_phi(torch.from_numpy(sci).to(DEV), torch.from_numpy(var).to(DEV), None, np.ones((2, 1, 1), np.float32))
    job = kb.Job(ctx, H, W, 2, 1, 1)
    job.search(s, np.array([0.0, 1.0]), np.zeros(1), np.zeros(1))
    got = job.filter_lightcurves(s, nsigma)[..., 0]
    p = np.empty((2, H, W, 2), np.float32)
    s.copy_planes(0, p)
    pe, fe = p[..., 0].astype(np.float64), p[..., 1].astype(np.float64)
    P, F = pe[0] + pe[1], fe[0] + fe[1]
    rest = F - fe
    out = (fe > 0) & (rest > 0) & ((pe * F - P * fe) ** 2 > nsigma * nsigma * F * fe * rest)
    assert np.array_equal(got["rejected"][..., 0], (out[0] + 2 * out[1]).astype(np.uint32)) and out.any() and not out.all()
    job.free()
    s.free()


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("N,H,W,V,k,s_hi", SHAPES)
def test_every_shape_equals_the_pipelined_kernel(kb, ctx, storage, N, H, W, V, k, s_hi):
    """The explicit shapes, which never share a tile's velocities between CTAs: several chunks of the table and
    full buffers in the plain kernel (FP32's fourth shape is the automatic one, 16-bit's second and fourth are)."""
    st = synth.small_stack(7 * N + k, N, H, W, K=5, nan_frac=0.05, n_angles=10, n_speeds=13, s_hi=s_hi, n_sources=3,
                           flux=40.0)
    s = _stack(kb, ctx, st, storage)
    ctx.set_search_variant(5)
    ref = _records(kb, ctx, s, st, V, k).tobytes()
    for variant in (1, 2, 3, 4):
        ctx.set_search_variant(variant)
        assert _records(kb, ctx, s, st, V, k).tobytes() == ref, variant
    ctx.set_search_variant(0)
    s.free()


@pytest.mark.parametrize("storage,k,flags", [("f32", 4, 0), ("f32", 12, 0), ("bf16", 8, 0), ("f16", 11, 0), ("bf16", 8, 1),
                                             ("f16", 4, 1), ("f32", 8, 1)])
def test_automatic_search_beyond_one_wave(kb, ctx, storage, k, flags):
    """More tiles than the GPU holds at once, so that the automatic search keeps a tile to one CTA: value and
    key lists over several chunks of the table."""
    st = synth.small_stack(850 + k, 13, 330, 1300, K=5, nan_frac=0.01, n_angles=10, n_speeds=13, s_hi=80.0, n_sources=20,
                           flux=60.0)
    s = _stack(kb, ctx, st, storage)
    if flags:   # rescored: the records of the FP32 planes' own candidates, in FP64
        f = _stack(kb, ctx, st, "f32")
        ctx.set_search_variant(4)
        ref = _records(kb, ctx, f, st, 130, k, flags=kb.KB_RESCORE_FP64)
        f.free()
    else:
        ctx.set_search_variant(5)
        ref = _records(kb, ctx, s, st, 130, k)
    ctx.set_search_variant(0)
    assert _records(kb, ctx, s, st, 130, k, flags=kb.KB_RESCORE_FP64 if flags else 0).tobytes() == ref.tobytes()
    s.free()
