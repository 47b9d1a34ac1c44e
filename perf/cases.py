"""The work that users of this framework have it do, as measurable cases.

Kinds of a case (every call goes through paper_1901_02492_gb300.binding):

  images     likelihood images of a stack.  storage "f32": make_psi_phi_static into the caller's
             planes; "bf16" / "f16": Stack.make_psi_phi, then the 16-bit codes read with copy_planes.
  job        one whole request: Stack.make_psi_phi, Job.search, the kept records on the device.
  search     Job.search of a stack whose likelihood images are there already, and its records.
  batch      Batch.run of several uneven searches, and the records of each.
  filter     Job.filter_lightcurves over every kept trajectory of a search.
  vet        candidates of a search grouped (Context.cluster), then stamped (Job.stamps).

Sizes, velocity grids, noise and sources follow the repository's own workloads (the 5 x 64 x 64
stack, the DECam-shaped 12 x 4096 x 4096 stack, the uneven batch and the serving stream).
"""
import math

import numpy as np
import torch

from paper_1901_02492_gb300 import binding as kb

DEV = "cuda:0"
FWHM_PER_SIGMA = 2.0 * math.sqrt(2.0 * math.log(2.0))


def listed():
    return [
        # the smallest request: the whole pipeline on a cut-out, where launches and latency count
        dict(name="job_tiny", kind="job", N=5, H=64, W=64, K=7, sigma=1.0, V=256, k=4, storage="f32", slow=True,
             out="full"),
        # the small request of the serving stream: a 512 x 512 patch, 16-bit planes, FP64 ranking
        dict(name="job_512_rescored", kind="job", N=9, H=512, W=512, K=13, sigma=1.5, V=640, k=8, storage="bf16",
             rescore=True, out="compact"),
        # likelihood images of one DECam-shaped stack
        dict(name="images_decam", kind="images", N=12, H=4096, W=4096, K=17, sigma=1.7, storage="f32"),
        # a ragged, masked patch into 16-bit planes
        dict(name="images_ragged_bf16", kind="images", N=8, H=1531, W=2047, K=13, sigma=1.5, storage="bf16",
             mask=True),
        # trailed or astigmatic PSFs, which do not separate
        dict(name="images_elongated", kind="images", N=12, H=2048, W=2048, K=17, sigma=1.7, storage="f32",
             elongated=True),
        # the headline search: every start pixel of the DECam-shaped stack, 1024 velocities
        dict(name="search_decam", kind="search", N=12, H=4096, W=4096, K=17, sigma=1.7, V=1024, k=8, storage="f32",
             out="compact"),
        # one search of the uneven batch's range: longer lists, a ragged patch
        dict(name="search_long_lists", kind="search", N=14, H=2111, W=2045, K=13, sigma=1.5, V=512, k=12,
             storage="f32", out="full"),
        # the middle request of the serving stream: 16-bit planes, FP64 ranking
        dict(name="search_rescored", kind="search", N=10, H=4096, W=2048, K=13, sigma=1.6, V=640, k=8,
             storage="bf16", rescore=True, out="compact"),
        # the thresholded search of a new stack: only trajectories of nu >= 10 are kept
        dict(name="job_threshold", kind="job", N=12, H=2048, W=2048, K=17, sigma=1.7, V=1024, k=8, storage="f32",
             nu_min=10.0, out="compact"),
        # several uneven stacks in one captured launch
        dict(name="batch_uneven", kind="batch", count=5, H=1024, W=2048, n_lo=5, n_hi=20, v_lo=256, v_hi=1024,
             k_lo=4, k_hi=16, storage="f32"),
        # outlier rejection on the light curves of every kept trajectory
        dict(name="filter_2048", kind="filter", N=12, H=2048, W=2048, K=17, sigma=1.7, V=256, k=8, storage="f32"),
        # candidates grouped, then stamped with their moments
        dict(name="vet_candidates", kind="vet", N=12, H=2048, W=2048, K=17, sigma=1.7, V=256, k=8, storage="f32",
             n=262144, stamps=16384, radius=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _psf_draw(rng):
    sigma = round(rng.uniform(1.2, 2.0), 3)
    return 2 * math.ceil(rng.choice((3, 4)) * sigma) + 1, sigma


def draw(rng):
    kind = rng.choice(("images", "images", "job", "job", "search", "search", "batch", "filter", "vet"))
    K, sigma = _psf_draw(rng)
    if kind == "images":
        H, W, N = _log(rng, 64, 4096), _log(rng, 64, 4096), rng.randint(2, 12)
        return dict(kind=kind, N=N, H=H, W=W, K=K, sigma=sigma, storage=rng.choice(("f32", "f32", "bf16", "f16")),
                    elongated=rng.random() < 0.3, mask=rng.random() < 0.5)
    if kind in ("job", "search"):
        storage = rng.choice(("f32", "f32", "bf16", "f16"))
        H, W = _log(rng, 48, 2000), _log(rng, 48, 2000)
        c = dict(kind=kind, N=rng.randint(4, 20), H=H, W=W, K=K, sigma=sigma, V=_log(rng, 64, 1024),
                 k=rng.randint(1, 16), storage=storage, rescore=storage != "f32" and rng.random() < 0.7,
                 out=rng.choice(("compact", "full")), slow=H * W < 20000)
        if storage == "f32" and kind == "job" and rng.random() < 0.3:
            c["nu_min"] = round(rng.uniform(7.0, 11.0), 2)
        return c
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 5), H=_log(rng, 200, 1500), W=_log(rng, 200, 2048), n_lo=5,
                    n_hi=20, v_lo=128, v_hi=1024, k_lo=4, k_hi=16, storage=rng.choice(("f32", "bf16")))
    H, W = _log(rng, 256, 2048), _log(rng, 256, 2048)
    c = dict(kind=kind, N=rng.randint(5, 16), H=H, W=W, K=K, sigma=sigma, V=_log(rng, 64, 512), k=rng.randint(2, 8),
             storage="f32")
    if kind == "vet":
        c.update(n=min(_log(rng, 2000, 300000), H * W * c["k"]), radius=rng.randint(4, 15), median=rng.random() < 0.5)
        c["stamps"] = min(_log(rng, 500, 16384), c["n"])
    return c


# ---- inputs ------------------------------------------------------------------------------------


def _times(N, seed):
    """Four visits 1.5 h apart on the first night, the rest on two more nights."""
    r = np.random.default_rng(seed + 17)
    t = [j * 1.5 / 24.0 for j in range(min(4, N))]
    for i in range(N - len(t)):
        t.append(1 + i % 2 + (i // 2) * 0.0625 + r.uniform(0.0, 0.02))
    return np.sort(np.array(t))


def _grid(V, slow):
    """A grid of about sqrt(V) angles: V velocities, index = angle * speeds + speed."""
    na = max(1, int(math.sqrt(V)))
    ns = -(-V // na)
    if slow:
        th, sp = np.linspace(-math.pi, math.pi, na, endpoint=False), np.linspace(1.0, 10.0, ns)
    else:
        th, sp = np.linspace(-math.pi / 4, math.pi / 4, na), np.linspace(90.0, 550.0, ns)
    T, S = np.meshgrid(th, sp, indexing="ij")
    return (S * np.cos(T)).ravel()[:V].copy(), (S * np.sin(T)).ravel()[:V].copy()


def _psfs(N, K, sigma, elongated, seed):
    r = np.random.default_rng(seed + 29)
    d = np.arange(-(K // 2), K // 2 + 1, dtype=np.float64)
    yy, xx = np.meshgrid(d, d, indexing="ij")
    out = []
    for _ in range(N):
        s = sigma * r.uniform(0.9, 1.1)
        if elongated:
            q, th = r.uniform(0.6, 0.9), r.uniform(0.2, math.pi / 2 - 0.2)
            u, w = math.cos(th) * xx + math.sin(th) * yy, -math.sin(th) * xx + math.cos(th) * yy
            g = np.exp(-0.5 * ((u / s) ** 2 + (w / (q * s)) ** 2))
        else:
            g = np.outer(np.exp(-0.5 * (d / s) ** 2), np.exp(-0.5 * (d / s) ** 2))
        out.append((g / g.sum()).astype(np.float32))
    return np.stack(out)


def _images(c, seed, times):
    """Science and variance planes (sky noise, 1 % bad pixels as NaN disks, moving sources), mask."""
    N, H, W = c["N"], c["H"], c["W"]
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    var_t = torch.empty(N, device=DEV).uniform_(80.0, 120.0, generator=g)
    var = torch.rand((N, H, W), device=DEV, generator=g)
    var.mul_(0.2).add_(0.9).mul_(var_t.view(N, 1, 1))
    sci = torch.randn((N, H, W), device=DEV, generator=g)
    sci.mul_(var_t.sqrt().view(N, 1, 1))
    r = np.random.default_rng(seed + 41)
    ns = max(1, min(200, H * W // 20000))
    speed, ang = r.uniform(90.0, 550.0, ns), r.uniform(-math.pi / 4, math.pi / 4, ns)
    if c.get("slow"):
        speed, ang = r.uniform(1.0, 10.0, ns), r.uniform(-math.pi, math.pi, ns)
    x0, y0, snr = r.uniform(0, W, ns), r.uniform(0, H, ns), r.uniform(1.5, 8.0, ns)
    s = float(c["sigma"])
    flux = torch.tensor(snr * math.sqrt(4.0 * math.pi * s * s * 100.0), device=DEV)
    o = torch.arange(-7, 8, device=DEV)
    for e in range(N):
        cx = torch.tensor(x0 + speed * np.cos(ang) * times[e], device=DEV)
        cy = torch.tensor(y0 + speed * np.sin(ang) * times[e], device=DEV)
        px, py = cx.round().long()[:, None] + o, cy.round().long()[:, None] + o
        gx, gy = torch.exp(-0.5 * ((px - cx[:, None]) / s) ** 2), torch.exp(-0.5 * ((py - cy[:, None]) / s) ** 2)
        v = (flux / (2.0 * math.pi * s * s))[:, None, None] * gy[:, :, None] * gx[:, None, :]
        yy, xx = py[:, :, None].expand_as(v), px[:, None, :].expand_as(v)
        ok = (yy >= 0) & (yy < H) & (xx >= 0) & (xx < W)
        # added as integers of 2^-20: the same sums in any order
        flat = torch.zeros(H * W, dtype=torch.int64, device=DEV)
        flat.index_add_(0, (yy * W + xx)[ok], (v[ok] * 1048576.0).round().long())
        sci[e].view(-1).add_((flat.double() / 1048576.0).float())
        rad = torch.randint(1, 4, (max(1, int(0.01 * H * W / 15.67)),), device=DEV, generator=g)
        by = torch.randint(0, H, rad.shape, device=DEV, generator=g)
        bx = torch.randint(0, W, rad.shape, device=DEV, generator=g)
        d = torch.arange(-3, 4, device=DEV)
        yy = (by[:, None, None] + d[None, :, None]).expand(-1, 7, 7)
        xx = (bx[:, None, None] + d[None, None, :]).expand(-1, 7, 7)
        inside = (d[:, None] ** 2 + d[None, :] ** 2)[None] <= (rad * rad)[:, None, None]
        ok = inside & (yy >= 0) & (yy < H) & (xx >= 0) & (xx < W)
        sci[e].view(-1)[(yy * W + xx)[ok]] = float("nan")
    mask = None
    if c.get("mask"):
        mask = (torch.rand((N, H, W), device=DEV, generator=g) < 0.01).to(torch.uint8)
    return sci, var, mask


def _stack_inputs(c, seed):
    times = _times(c["N"], seed)
    psf = _psfs(c["N"], c["K"], c["sigma"], c.get("elongated", False), seed)
    return (times, psf) + _images(c, seed, times)


def _batch_cases(c, seed):
    """The uneven members of a batch (drawn from the case alone, so that its cost is the case's)."""
    r = np.random.default_rng(c["H"] * 8191 + c["W"])
    out = []
    for _ in range(c["count"]):
        sigma = float(r.uniform(1.2, 2.0))
        out.append(dict(N=int(r.integers(c["n_lo"], c["n_hi"] + 1)), H=c["H"], W=c["W"],
                        K=2 * math.ceil(4 * sigma) + 1, sigma=sigma, V=int(r.integers(c["v_lo"], c["v_hi"] + 1)),
                        k=int(r.integers(c["k_lo"], c["k_hi"] + 1)), storage=c["storage"]))
    return out


# ---- the program's state -----------------------------------------------------------------------

_CTX = []


def _ctx():
    """The one context that a program keeps."""
    if not _CTX:
        _CTX.append(kb.Context(0))
    return _CTX[0]


def _flags(c):
    return (kb.KB_RESCORE_FP64 if c.get("rescore") else 0) | (kb.KB_PRUNE if c.get("nu_min") else 0)


class _Search:
    """A stack, the job that searches it and the buffer its records go to."""

    def __init__(self, c, seed):
        self.c = c
        self.times, self.psf, self.sci, self.var, self.mask = _stack_inputs(c, seed)
        self.vx, self.vy = _grid(c["V"], c.get("slow"))
        self.nu_min, self.flags = c.get("nu_min") or -math.inf, _flags(c)
        self.stack = kb.Stack(_ctx(), c["N"], c["H"], c["W"], c["storage"])
        self.job = kb.Job(_ctx(), c["H"], c["W"], c["N"], c["V"], c["k"], self.flags & kb.KB_RESCORE_FP64)
        self.full = c.get("out") == "full"
        size = kb.RESULT_DTYPE.itemsize if self.full else kb.COMPACT_DTYPE.itemsize
        self.n = c["H"] * c["W"] * c["k"]
        self.out = torch.empty(self.n * size, dtype=torch.uint8, device=DEV)

    def images(self):
        self.stack.make_psi_phi(self.sci, self.var, self.mask, self.psf)

    def search(self):
        self.job.search(self.stack, self.times, self.vx, self.vy, self.c["k"], self.nu_min, self.flags)

    def records(self):
        if self.full:
            self.job.results(self.out)
            w, d = self.out.view(torch.int32).view(self.n, 12), self.out.view(torch.float64).view(self.n, 6)
            f = self.out.view(torch.float32).view(self.n, 12)
            return dict(x0=w[:, 0], y0=w[:, 1], vidx=w[:, 2], nobs=w[:, 3], vx=f[:, 4], vy=f[:, 5], psi=f[:, 6],
                        phi=f[:, 7], nu=d[:, 4], alpha=d[:, 5])
        self.job.results_compact_async(self.out)
        f = self.out.view(torch.float32).view(self.n, 4)
        return dict(psi=f[:, 0], phi=f[:, 1], nu=f[:, 2], vidx=self.out.view(torch.int16).view(self.n, 8)[:, 6],
                    nobs=self.out.view(self.n, 16)[:, 14])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "images":
        times, psf, sci, var, mask = _stack_inputs(case, seed)
        N, H, W = sci.shape
        st = dict(kind=kind, sci=sci, var=var, mask=mask, psf=psf, stack=None)
        if case["storage"] == "f32":
            st["out"] = torch.empty((N, H, W, 2), dtype=torch.float32, device=DEV)
        else:
            st["stack"] = kb.Stack(_ctx(), N, H, W, case["storage"])
            st["out"] = torch.empty((N, H, W, 2), dtype=torch.int16, device=DEV)
        return st
    if kind == "batch":
        members = [_Search(dict(c, out="compact"), seed + 101 * i) for i, c in enumerate(_batch_cases(case, seed))]
        for m in members:
            m.images()
        torch.cuda.synchronize()
        batch = kb.Batch(_ctx(), [dict(job=m.job, stack=m.stack, times=m.times, vx=m.vx, vy=m.vy, topk=m.c["k"])
                                  for m in members])
        return dict(kind=kind, members=members, batch=batch)
    s = _Search(case, seed)
    if kind != "job":
        s.images()
    st = dict(kind=kind, s=s)
    if kind in ("filter", "vet"):
        s.search()
    if kind == "filter":
        st["out"] = torch.empty(s.n * kb.FILTERED_DTYPE.itemsize, dtype=torch.uint8, device=DEV)
    if kind == "vet":
        # the n most likely trajectories, best first, as kb_result records in hand
        full = torch.empty(s.n * kb.RESULT_DTYPE.itemsize, dtype=torch.uint8, device=DEV)
        s.job.results(full)
        best = torch.sort(full.view(torch.float64).view(s.n, 6)[:, 4], descending=True, stable=True)[1][:case["n"]]
        rec = full.view(s.n, kb.RESULT_DTYPE.itemsize)[best].contiguous()
        st["cand"] = rec.view(-1)
        head = rec[:case["stamps"]].contiguous().view(torch.int32).view(-1, 12).cpu().numpy()
        st["pick"] = [np.ascontiguousarray(head[:, i]) for i in range(3)]
        sig = float(case["sigma"])
        st["cuts"] = dict(max_offset=1.5, min_var=0.2 * sig * sig, max_var=3.0 * sig * sig, max_mu11=1.5 * sig * sig)
    return st


def run(state):
    kind = state["kind"]
    if kind == "images":
        if state["stack"] is None:
            kb.make_psi_phi_static(state["sci"], state["var"], state["mask"], state["psf"], state["out"])
        else:
            state["stack"].make_psi_phi(state["sci"], state["var"], state["mask"], state["psf"])
            state["stack"].copy_planes(1, state["out"])
        return state["out"]
    if kind == "batch":
        state["batch"].run()
        return [m.records() for m in state["members"]]
    s = state["s"]
    if kind == "job":
        s.images()
    if kind in ("job", "search"):
        s.search()
        return s.records()
    if kind == "filter":
        o = s.job.filter_lightcurves(s.stack, 5.0, state["out"])
        w, d = o.view(torch.int32).view(s.n, 18), o.view(torch.float64).view(s.n, 9)
        return dict(vidx=w[:, 2], nobs=w[:, 3], nrejected=w[:, 4], rejected=w[:, 6:10], psi=d[:, 5], phi=d[:, 6],
                    nu=d[:, 7], alpha=d[:, 8])
    # weights and radius of the repository's own clustering workload
    label, keep, _, groups = _ctx().cluster(state["cand"], 0.5, 1.0 / 15.0, 1.5, 4)
    c, (x0, y0, v) = s.c, state["pick"]
    stamps, mo = s.job.stamps(s.sci, s.mask, x0, y0, v, c["radius"], median=bool(c.get("median")), cuts=state["cuts"],
                              aperture=3.0)
    return dict(label=label, keep=keep, groups=groups, stamps=stamps, passed=mo["passed"],
                **{f: mo[f] for f in ("m00", "mx", "my", "mu20", "mu02", "mu11")})


# ---- what a pass cannot do without -------------------------------------------------------------


def _images_work(c):
    px = c["N"] * c["H"] * c["W"]
    taps = c["K"] ** 2 if c.get("elongated") else 2 * c["K"]
    read = 8 + (1 if c.get("mask") else 0)
    return px * (read + 8), px * (4.0 * taps + 4)


def _search_work(c):
    px, plane = c["H"] * c["W"], 8 if c["storage"] == "f32" else 4
    size = 48 if c.get("out") == "full" else 16
    # psi and phi added once per trajectory and epoch inside the image, the score and a comparison
    inside = 0.0
    vx, vy = _grid(c["V"], c.get("slow"))
    for t in _times(c["N"], 0):
        inside += float(np.sum(np.maximum(0.0, c["W"] - np.abs(vx * t)) * np.maximum(0.0, c["H"] - np.abs(vy * t))))
    extra = px * c["k"] * c["N"] * 2.0 if c.get("rescore") else 0.0
    byte = c["N"] * px * (plane + (8 if c.get("rescore") else 0)) + px * c["k"] * size
    return byte, 2.0 * inside + 3.0 * c["V"] * px + extra


def work(case):
    kind = case["kind"]
    if kind == "images":
        b, f = _images_work(case)
        return {"bytes": b if case["storage"] == "f32" else b - 4 * case["N"] * case["H"] * case["W"], "flops": f}
    if kind == "batch":
        got = [_search_work(dict(c, out="compact")) for c in _batch_cases(case, 0)]
        return {"bytes": sum(g[0] for g in got), "flops": sum(g[1] for g in got)}
    if kind == "search":
        b, f = _search_work(case)
        return {"bytes": b, "flops": f}
    if kind == "job":
        (b0, f0), (b1, f1) = _images_work(case), _search_work(case)
        return {"bytes": b0 + b1, "flops": f0 + f1}
    px = case["H"] * case["W"]
    if kind == "filter":
        return {"bytes": px * (case["N"] * 8 + case["k"] * (16 + 72)), "flops": px * case["k"] * case["N"] * 12.0}
    S2 = (2 * case["radius"] + 1) ** 2
    return {"bytes": case["n"] * (48 + 5) + case["stamps"] * (S2 * 4.0 * (case["N"] + 1) + 68),
            "flops": case["n"] * 81 * 11.0 + case["stamps"] * S2 * (case["N"] + 12.0)}


# ---- the same in 64 bits -----------------------------------------------------------------------


def _planes64(c, psf, sci, var, mask):
    """psi and phi in 64 bits, each [N][H][W]."""
    N, H, W, r = c["N"], c["H"], c["W"], c["K"] // 2
    psi, phi = torch.empty((N, H, W), dtype=torch.float64, device=DEV), torch.empty((N, H, W), dtype=torch.float64,
                                                                                    device=DEV)
    for e in range(N):
        n, v = sci[e].double(), var[e].double()
        bad = ~torch.isfinite(n) | ~torch.isfinite(v) | ~(v > 0)
        if mask is not None:
            bad |= mask[e] != 0
        w = torch.where(bad, 0.0, 1.0 / v)
        for dst, plane, p in ((psi, torch.where(bad, 0.0, n * w), 1), (phi, w, 2)):
            pad = torch.nn.functional.pad(plane, (r, r, r, r))
            T = psf[e].astype(np.float64) ** p
            acc = torch.zeros((H, W), dtype=torch.float64, device=DEV)
            for i in range(c["K"]):
                for j in range(c["K"]):
                    acc.add_(pad[i:i + H, j:j + W], alpha=float(T[i, j]))
            dst[e] = acc
    return psi, phi


def _offsets(times, vx, vy):
    """Pixel offsets of every velocity and epoch in the fixed point of include/kb.h."""
    tq = [int(math.floor((t - min(times)) * 2 ** 20 + 0.5)) for t in times]

    def q(v):
        return int(math.copysign(math.floor(abs(v) * 65536.0 + 0.5), v))

    return [[((q(a) * t + (1 << 35)) >> 36, (q(b) * t + (1 << 35)) >> 36) for t in tq] for a, b in zip(vx, vy)]


def _topk64(c, psi, phi, times, nu_min):
    """The k best nu of every start pixel, best first: [H][W][k] in 64 bits."""
    H, W = c["H"], c["W"]
    best = torch.full((c["k"], H, W), -math.inf, dtype=torch.float64, device=DEV)
    for offs in _offsets(times, *_grid(c["V"], c.get("slow"))):
        P, F = torch.zeros((H, W), dtype=torch.float64, device=DEV), torch.zeros((H, W), dtype=torch.float64,
                                                                                 device=DEV)
        for e, (dx, dy) in enumerate(offs):
            x0, x1, y0, y1 = max(0, -dx), min(W, W - dx), max(0, -dy), min(H, H - dy)
            if x0 < x1 and y0 < y1:
                P[y0:y1, x0:x1] += psi[e, y0 + dy:y1 + dy, x0 + dx:x1 + dx]
                F[y0:y1, x0:x1] += phi[e, y0 + dy:y1 + dy, x0 + dx:x1 + dx]
        nu = torch.where(F > 0, P / F.sqrt(), -math.inf)
        nu = torch.where(nu >= nu_min, nu, -math.inf)
        for i in range(c["k"]):
            lo = torch.minimum(best[i], nu)
            torch.maximum(best[i], nu, out=best[i])
            nu = lo
    return best.permute(1, 2, 0).reshape(-1)


def _records64(c, seed):
    times, psf, sci, var, mask = _stack_inputs(c, seed)
    psi, phi = _planes64(c, psf, sci, var, mask)
    nu = _topk64(c, psi, phi, times, c.get("nu_min") or -math.inf)
    keys = ("x0", "y0", "vidx", "nobs", "vx", "vy", "psi", "phi", "alpha") if c.get("out") == "full" else \
        ("psi", "phi", "vidx", "nobs")
    # velocities, sums and fluxes hang on which of two nearly equal trajectories is named: the score does not
    return dict({k: None for k in keys}, nu=nu)


def _filtered64(c, s):
    """The filter on the trajectories that the search named, from the planes that it searched."""
    N, H, W, k = c["N"], c["H"], c["W"], c["k"]
    planes = torch.empty((N, H, W, 2), dtype=torch.float32, device=DEV)
    s.stack.copy_planes(0, planes)
    vidx = s.records()["vidx"].long().view(H, W, k)
    offs = torch.tensor(_offsets(s.times, s.vx, s.vy), device=DEV)
    y, x = torch.arange(H, device=DEV)[:, None, None], torch.arange(W, device=DEV)[None, :, None]
    out = []
    for i in range(k):
        v = vidx[..., i:i + 1]
        got = []
        for e in range(N):
            yy, xx = y + offs[v.clamp(min=0), e, 1], x + offs[v.clamp(min=0), e, 0]
            ok = (v >= 0) & (yy >= 0) & (yy < H) & (xx >= 0) & (xx < W)
            q = planes[e][yy.clamp(0, H - 1), xx.clamp(0, W - 1)].double()[:, :, 0]
            got.append(torch.where(ok, q, 0.0))
        tot = sum(got)
        P, F = tot[..., 0], tot[..., 1]
        kept = torch.zeros_like(tot)
        for q in got:
            p, f, rest = q[..., 0], q[..., 1], F - q[..., 1]
            reject = (f > 0) & (rest > 0) & ((p * F - P * f) ** 2 > 25.0 * F * f * rest)
            kept += torch.where(reject[..., None], 0.0, q)
        out.append(kept)
    kept = torch.stack(out, 2).view(-1, 2)
    P, F = kept[:, 0], kept[:, 1]
    return dict(vidx=None, nobs=None, nrejected=None, rejected=None, psi=P, phi=F,
                nu=torch.where(F > 0, P / F.sqrt(), -math.inf), alpha=torch.where(F > 0, P / F, 0.0))


def exact(case, seed):
    kind = case["kind"]
    if kind == "images":
        if case["storage"] != "f32":
            return None   # integer codes
        times, psf, sci, var, mask = _stack_inputs(case, seed)
        return torch.stack(_planes64(case, psf, sci, var, mask), dim=-1)
    if kind in ("job", "search"):
        return _records64(case, seed)
    if kind == "batch":
        return [_records64(dict(c, out="compact"), seed + 101 * i) for i, c in enumerate(_batch_cases(case, seed))]
    if kind == "filter":
        return _filtered64(case, prepare(case, seed)["s"])
    # stamps of the candidates that the search names, from the science images
    st = prepare(case, seed)
    x0, y0, v = (torch.from_numpy(a).to(DEV).long() for a in st["pick"])
    sci, c, r = st["s"].sci, case, case["radius"]
    offs = torch.tensor(_offsets(st["s"].times, st["s"].vx, st["s"].vy), device=DEV)
    d = torch.arange(-r, r + 1, device=DEV)
    out = []
    for lo in range(0, x0.numel(), 2048):
        sl = slice(lo, lo + 2048)
        vals = []
        for e in range(c["N"]):
            yy = (y0[sl] + offs[v[sl], e, 1])[:, None, None] + d[None, :, None]
            xx = (x0[sl] + offs[v[sl], e, 0])[:, None, None] + d[None, None, :]
            ok = (yy >= 0) & (yy < c["H"]) & (xx >= 0) & (xx < c["W"])
            val = sci[e][yy.clamp(0, c["H"] - 1), xx.clamp(0, c["W"] - 1)].double()
            vals.append(torch.where(ok & torch.isfinite(val), val, math.inf))
        a = torch.sort(torch.stack(vals, -1), -1)[0]
        m = torch.isfinite(a).sum(-1)
        if c.get("median"):
            pick = torch.stack([torch.gather(a, -1, i.clamp(0, c["N"] - 1)[..., None])[..., 0]
                                for i in ((m - 1) // 2, m // 2)]).mean(0)
        else:
            pick = torch.where(torch.isfinite(a), a, 0.0).sum(-1) / m.clamp(min=1)
        out.append(torch.where(m > 0, pick, 0.0))
    stamps = torch.cat(out)
    x, y = d.double()[None, None, :], d.double()[None, :, None]
    w = stamps.float().double() * ((x * x + y * y) <= 9.0)
    tot = w.sum((1, 2))
    mx, my = (x * w).sum((1, 2)) / tot, (y * w).sum((1, 2)) / tot
    cx, cy = x - mx[:, None, None], y - my[:, None, None]
    mom = dict(m00=tot, mx=mx, my=my, mu20=(cx * cx * w).sum((1, 2)) / tot, mu02=(cy * cy * w).sum((1, 2)) / tot,
               mu11=(cx * cy * w).sum((1, 2)) / tot)
    return dict(label=None, keep=None, groups=None, stamps=stamps, passed=None, **mom)
