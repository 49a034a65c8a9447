"""The work that a texturing pipeline has this library do, as measurable cases.

A pipeline renders (or rasterises here) the position maps of its meshes, builds
the correspondences of a batch of assets once, and then runs a sampler loop:
full steps, where every view went through the denoiser, and cached steps, where
only the anchors did and the library transports their change to the others.
Each case is one of these calls, or a whole loop, through the Python binding on
torch tensors.  Sizes are those of the workloads the repository is benchmarked
and tested on, with ragged ones beside them.

Geometry is made here from the seed: blobs, unions of boxes and spheres, and
tori, seen by the camera layouts of multi-view texture diffusion.  Latents and
x0 are N(0, 1) and an anchor's update N(0, 0.1^2).

`exact` recomputes a case in torch: the choices the interface defines in
binary32 (projection, tap choice, the tolerance test, the nearest face) in
binary32 in the interface's order, every value that follows in binary64.
"""
import math

import numpy as np
import torch

from paper_2608_13255_gb300 import geocache as gc

DEV = "cuda"
LAYOUTS = {  # camera layouts (azimuth, elevation) by number of views; other numbers: a ring at elevation +-15
    6: [(0.0, 0.0), (90.0, 0.0), (180.0, 0.0), (270.0, 0.0), (0.0, 90.0), (0.0, -90.0)],
    12: [(45.0 * i, 20.0 if i % 2 == 0 else -20.0) for i in range(8)]
        + [(0.0, 70.0), (180.0, 70.0), (90.0, -70.0), (270.0, -70.0)],
}
FOV, DIST = math.radians(40.0), 1.05 / math.sin(math.radians(20.0))
TOL = 0.01  # the correspondence tolerance, a fraction of the asset's diagonal


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # one asset of a 6-view, 64 x 64 latent pipeline, one cached DDIM step: the smallest call of the sampler
        # loop, where latency and launches count
        _step("step_one_asset_64", B=1, N=6, H=64, W=64, C=4, a=2),
        # 12 views with 16-channel latents, 8 assets, flow matching: wide latents, four anchors
        _step("step_12_views_16_channels", B=8, N=12, H=128, W=128, C=16, a=4, sampler="fm"),
        # the throughput batch: 128 assets x 6 views
        _step("step_128_assets", B=128, N=6, H=128, W=128, C=4, a=2),
        # ragged maps, f32 latents, the x0 cache and the latents updated in place, the velocity kept for a
        # multistep solver
        _step("step_ragged_f32", B=5, N=5, H=75, W=53, C=6, a=2, dtype="f32", sampler="fm", pred=True, in_place=True),
        # a caller that keeps only the one-byte masks (no records, no workspace), 3 anchors
        _step("step_masks_8_assets", B=8, N=6, H=96, W=96, C=4, a=3, sampler="fm", mode="mask"),
        # a full refresh step of 64 assets: the denoiser ran on every view, x0 is stored and x_t reconstructed
        dict(name="full_step_64_assets", op="full", B=64, N=6, H=128, W=128, C=4, dtype="bf16", sampler="ddim",
             pred=False, store=True),
        # the correspondences of one asset, as a per-asset pipeline builds them before its loop
        dict(name="build_one_asset_64", op="build", B=1, N=6, H=64, W=64, K=4, tables=False),
        # the correspondences of a batch
        dict(name="build_64_assets", op="build", B=64, N=6, H=128, W=128, K=4, tables=False),
        # position maps of 16 noisy blob meshes of 81,920 faces at the token grid
        dict(name="raster_16_meshes", op="raster", B=16, N=6, H=128, W=128, s=1, subdiv=6, rough=True),
        # smooth ones rendered at 512 x 512 (image resolution) and pooled to the token grid
        dict(name="raster_512_pooled", op="raster", B=4, N=6, H=128, W=128, s=4, subdiv=6, rough=False),
        # maps a pipeline rendered itself, 96 views of 512 x 512, brought to 64 x 64 tokens
        dict(name="pool_512_to_64", op="pool", n=96, H=64, W=64, s=8),
        # a whole 30-step DDIM loop of one asset, every fifth step full: rotation, the anchors' rows packed for
        # the denoiser, cached and full steps
        dict(name="loop_one_asset_64", op="loop", B=1, N=6, H=64, W=64, C=4, a=2, steps=30, every=5),
    ]


def _step(name, B, N, H, W, C, a, dtype="bf16", sampler="ddim", mode="sparse", update="delta", pred=False,
          in_place=False, K=4):
    return dict(name=name, op="step", B=B, N=N, H=H, W=W, C=C, a=a, K=K, dtype=dtype, sampler=sampler, mode=mode,
                update=update, pred=pred, in_place=in_place)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit(cap, per):  # the largest batch a drawn case may have
    return max(1, int(cap // max(1, per)))


def draw(rng):
    op = rng.choice(["step", "step", "step", "step", "full", "build", "build", "raster", "raster", "pool", "loop"])
    H, W = _log(rng, 48, 136), _log(rng, 48, 136)
    if rng.random() < 0.5:  # square maps of a multiple of 8, as most pipelines have
        H = W = 8 * max(6, round(H / 8))
    N = rng.choice([4, 5, 6, 6, 6, 8, 10, 12])
    sampler = rng.choice(["ddim", "fm"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    if op == "step":
        C, a = rng.choice([3, 4, 4, 4, 6, 8, 16]), rng.randint(1, min(4, N - 1))
        mode = rng.choice(["sparse", "sparse", "sparse", "sparse", "mask", "table", "geometry"])
        K = rng.choice([4, 4, 4, 1])
        cap = 25e6 if mode == "sparse" else 2e6
        B = _log(rng, 1, _fit(cap, N * C * H * W * (1 if dtype == "bf16" else 2)))
        c = _step("", min(B, 96), N, H, W, C, a, dtype, sampler, mode, rng.choice(["delta"] * 4 + ["copy"]),
                  rng.random() < 0.25, rng.random() < 0.25, K)
        del c["name"]
        return c
    if op == "full":
        C = rng.choice([3, 4, 8, 16])
        return dict(op="full", B=_log(rng, 1, _fit(20e6, N * C * H * W)), N=N, H=H, W=W, C=C, dtype=dtype,
                    sampler=sampler, pred=rng.random() < 0.25, store=rng.random() < 0.5)
    if op == "build":
        tables = rng.random() < 0.25
        return dict(op="build", B=_log(rng, 1, min(64, _fit(3e6 if tables else 25e6, N * N * H * W))), N=N, H=H, W=W,
                    K=rng.choice([4, 4, 4, 1]), tables=tables)
    if op == "raster":
        s, subdiv = rng.choice([1, 1, 2, 3, 4]), rng.choice([3, 4, 5, 6])
        per = N * max(H * W * s * s, 20 * 4 ** subdiv)
        return dict(op="raster", B=_log(rng, 1, min(16, _fit(5e6, per))), N=N, H=H, W=W, s=s, subdiv=subdiv,
                    rough=rng.random() < 0.5)
    if op == "pool":
        s = rng.choice([2, 3, 4, 8])
        return dict(op="pool", n=_log(rng, 1, _fit(20e6, H * W * s * s)), H=H, W=W, s=s)
    return dict(op="loop", B=1, N=N, H=H, W=W, C=4, a=rng.randint(1, 3), steps=rng.choice([15, 20, 30]),
                every=rng.choice([3, 4, 5]))


# --------------------------------------------------------------- geometry --
def _cameras(B, N, H, W, rng):
    """Look-at cameras [B, N, 16] f32: the layout of N views, its azimuth turned by a random angle per asset."""
    views = LAYOUTS.get(N) or [(360.0 * i / N, 15.0 if i % 2 == 0 else -15.0) for i in range(N)]
    out = np.zeros((B, N, 16), np.float32)
    for b in range(B):
        turn = rng.uniform(0.0, 360.0)
        for v, (az, el) in enumerate(views):
            az, el = math.radians(az + turn), math.radians(el)
            c = DIST * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
            f = -c / np.linalg.norm(c)
            up = np.array([0.0, 0.0, 1.0]) if abs(f[2]) < 0.9999 else np.array([math.cos(az), math.sin(az), 0.0])
            right = np.cross(f, up)
            right /= np.linalg.norm(right)
            R = np.stack([right, np.cross(f, right), f])
            focal = min(H, W) / 2.0 / math.tan(FOV / 2)
            out[b, v] = np.concatenate([R.reshape(-1), -R @ c, [focal, focal, W / 2.0, H / 2.0]])
    return torch.from_numpy(out).to(DEV)


def _bumps(B, rng):
    """Parameters [B, 6, 5] of a blob's radius 0.8 + sum_k amp sin(wave . d + phase): amp, wave[3], phase."""
    p = np.concatenate([rng.uniform(0.02, 0.07, (B, 6, 1)), rng.normal(0.0, 3.0, (B, 6, 3)),
                        rng.uniform(0.0, 6.28, (B, 6, 1))], -1)
    return torch.from_numpy(p.astype(np.float32)).to(DEV)


def _radius(bumps, d):
    """Blob radius in directions d [B, M, 3]."""
    r = torch.full(d.shape[:2], 0.8, device=DEV)
    for k in range(bumps.shape[1]):
        r = r + bumps[:, k, 0:1] * torch.sin((d * bumps[:, k, None, 1:4]).sum(-1) + bumps[:, k, 4:5])
    return r / 1.1


def _position_maps(B, N, H, W, cams, rng):
    """Position maps [B, N, H, W, 3] f32 and validity u8 of B solids (blob, boxes and spheres, torus in turn): the
    first crossing of an implicit surface along each token's ray, by marching and bisection."""
    kind = [b % 3 for b in range(B)]
    bumps = _bumps(B, rng)
    centre = torch.from_numpy(rng.uniform(-0.45, 0.45, (B, 4, 3)).astype(np.float32)).to(DEV)
    half = torch.from_numpy(rng.uniform(0.15, 0.35, (B, 4, 3)).astype(np.float32)).to(DEV)
    jj, ii = torch.meshgrid(torch.arange(H, device=DEV) + 0.5, torch.arange(W, device=DEV) + 0.5, indexing="ij")
    pos = torch.zeros((B, N, H, W, 3), device=DEV)
    valid = torch.zeros((B, N, H, W), dtype=torch.uint8, device=DEV)
    for k in range(3):
        sel = [b for b in range(B) if kind[b] == k]
        if not sel:
            continue
        cam = cams[sel]
        R, t, intr = cam[..., :9].reshape(-1, N, 3, 3), cam[..., 9:12], cam[..., 12:]
        d = torch.stack([(ii - intr[..., 2, None, None]) / intr[..., 0, None, None],
                         (jj - intr[..., 3, None, None]) / intr[..., 1, None, None],
                         torch.ones((len(sel), N, H, W), device=DEV)], -1).reshape(len(sel), N, H * W, 3)
        d = torch.nn.functional.normalize(torch.matmul(d, R), dim=-1).reshape(len(sel), -1, 3)
        o = -torch.matmul(t[:, :, None, :], R).expand(-1, -1, H * W, -1).reshape(len(sel), -1, 3)

        def inside(s):
            p = o + s[..., None] * d
            if k == 0:
                q = p.norm(dim=-1)
                return q < _radius(bumps[sel], p / q.clamp_min(1e-6)[..., None])
            if k == 1:
                hit = torch.zeros(p.shape[:2], dtype=torch.bool, device=DEV)
                for j in range(4):
                    x = (p - centre[sel, j, None]).abs()
                    hit |= (x < half[sel, j, None]).all(-1) if j % 2 else x.norm(dim=-1) < half[sel, j, None, 0]
                return hit
            return (p[..., :2].norm(dim=-1) - 0.66) ** 2 + p[..., 2] ** 2 < 0.3 ** 2

        lo, hi = (torch.full(d.shape[:2], DIST + x, device=DEV) for x in (-1.05, 1.05))
        hit = torch.zeros(d.shape[:2], dtype=torch.bool, device=DEV)
        for j in range(48):
            s = torch.full(d.shape[:2], DIST - 1.05 + 2.1 * (j + 1) / 48, device=DEV)
            now = inside(s) & ~hit
            lo, hi = torch.where(now, s - 2.1 / 48, lo), torch.where(now, s, hi)
            hit |= now
        for _ in range(16):
            mid = 0.5 * (lo + hi)
            now = inside(mid)
            lo, hi = torch.where(now, lo, mid), torch.where(now, mid, hi)
        p = torch.where(hit[..., None], o + hi[..., None] * d, torch.zeros_like(d))
        pos[sel] = p.reshape(len(sel), N, H, W, 3)
        valid[sel] = hit.to(torch.uint8).reshape(len(sel), N, H, W)
    return pos, valid


_SPHERES = {}


def _icosphere(subdiv):
    """Vertices [V, 3], faces [F, 3] and neighbours [V, 6] of a subdivided icosahedron."""
    if subdiv not in _SPHERES:
        p = (1.0 + 5.0 ** 0.5) / 2.0
        V = np.array([[-1, p, 0], [1, p, 0], [-1, -p, 0], [1, -p, 0], [0, -1, p], [0, 1, p], [0, -1, -p], [0, 1, -p],
                      [p, 0, -1], [p, 0, 1], [-p, 0, -1], [-p, 0, 1]], np.float64)
        F = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                      [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5],
                      [2, 4, 11], [6, 2, 10], [8, 6, 7], [9, 8, 1]], np.int64)
        V /= np.linalg.norm(V, axis=1, keepdims=True)
        for _ in range(subdiv):
            e = np.sort(np.concatenate([F[:, [0, 1]], F[:, [1, 2]], F[:, [2, 0]]]), axis=1)
            _, first, inv = np.unique(e[:, 0] * len(V) + e[:, 1], return_index=True, return_inverse=True)
            mid = V[e[first, 0]] + V[e[first, 1]]
            ab, bc, ca = (len(V) + inv.reshape(-1)[k * len(F):(k + 1) * len(F)] for k in range(3))
            V = np.concatenate([V, mid / np.linalg.norm(mid, axis=1, keepdims=True)])
            a, b, c = F.T
            F = np.concatenate([np.stack(x, 1) for x in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
        e = np.concatenate([F[:, [i, j]] for i in range(3) for j in range(3) if i != j])
        e = e[np.unique(e[:, 0] * len(V) + e[:, 1], return_index=True)[1]]  # directed edges, by their first vertex
        first = np.searchsorted(e[:, 0], np.arange(len(V)))
        degree = np.diff(np.append(first, len(e)))
        near = e[np.minimum(first[:, None] + np.arange(6), first[:, None] + degree[:, None] - 1), 1]
        _SPHERES[subdiv] = (torch.from_numpy(V.astype(np.float32)).to(DEV), torch.from_numpy(F.astype(np.int32)).to(DEV),
                            torch.from_numpy(near).to(DEV))
    return _SPHERES[subdiv]


def _noise(B, near, gen):
    """Radii [B, V] of a rough blob: N(0, 1) per vertex, four rounds of averaging with the neighbours, scaled to a
    standard deviation of 0.15."""
    r = _randn(gen, B, len(near))
    for _ in range(4):
        r = 0.5 * r + 0.5 * sum(r[:, near[:, k]] for k in range(6)) / 6.0
    r = 1.0 + 0.15 * (r - r.mean(1, keepdim=True)) / r.std(1, keepdim=True)
    return r / r.amax(1, keepdim=True)


# ----------------------------------------------------------------- inputs --
def _anchors(c):
    s = -(-c["N"] // c["a"])
    return sorted(((j * s) % c["N"]) for j in range(c["a"]))


def _sampler(c, k=0.4):
    """Parameters of one sampler step, about 40% into the schedule."""
    if c["sampler"] == "ddim":
        return dict(sampler="ddim", a_t=0.31 + 0.1 * k, a_prev=0.38 + 0.1 * k)
    return dict(sampler="fm_euler", sigma=1.0 - k, sigma_next=0.98 - k)


def _pred_kind(c):
    return ("eps" if c["sampler"] == "ddim" else "velocity") if c["pred"] else None


def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _randn(gen, *shape, dtype=torch.float32):
    return torch.randn(shape, generator=gen, device=DEV).to(dtype)


def _inputs(c, seed):
    """What the call reads, from the seed alone."""
    rng, gen = np.random.default_rng(seed), torch.Generator(DEV).manual_seed(seed)
    op, s = c["op"], {}
    if op in ("step", "build", "loop"):
        s["cams"] = _cameras(c["B"], c["N"], c["H"], c["W"], rng)
        s["pos"], s["valid"] = _position_maps(c["B"], c["N"], c["H"], c["W"], s["cams"], rng)
    if op in ("step", "full", "loop"):
        shape = (c["B"], c["N"], c["C"], c["H"], c["W"])
        s["x_t"] = _randn(gen, *shape, dtype=_dtype(c) if op != "loop" else torch.bfloat16)
        s["x0"] = _randn(gen, *shape)
    if op == "step":
        s["x0_new"] = (s["x0"][:, _anchors(c)] + 0.1 * _randn(gen, c["B"], c["a"], *shape[2:])).contiguous()
    if op == "loop":
        s["drift"] = 0.1 * _randn(gen, c["steps"], *shape)
    if op == "raster":
        V, F, near = _icosphere(c["subdiv"])
        r = (_noise(c["B"], near, gen) if c["rough"]
             else _radius(_bumps(c["B"], rng), V[None].expand(c["B"], -1, -1)))
        s["verts"] = (V * r[..., None]).reshape(-1, 3)
        shift = torch.arange(c["B"], device=DEV, dtype=torch.int32)[:, None, None] * len(V)
        s["faces"] = (F[None] + shift).reshape(-1, 3).contiguous()
        s["face_off"] = torch.arange(c["B"] + 1, device=DEV, dtype=torch.int64) * len(F)
        s["cams"] = _cameras(c["B"], c["N"], c["H"], c["W"], rng)
    if op == "pool":
        hi, wi = c["s"] * c["H"], c["s"] * c["W"]
        y, x = torch.meshgrid(torch.linspace(-1, 1, hi, device=DEV), torch.linspace(-1, 1, wi, device=DEV), indexing="ij")
        at = torch.from_numpy(rng.uniform(-0.2, 0.2, (c["n"], 2)).astype(np.float32)).to(DEV)
        depth = 0.6 - (x - at[:, 0, None, None]) ** 2 - (y - at[:, 1, None, None]) ** 2
        s["valid"] = (depth > 0).to(torch.uint8)
        s["pos"] = torch.stack([x.expand_as(depth), y.expand_as(depth), depth], -1) * s["valid"][..., None]
    return s


def prepare(case, seed):
    c = case
    s = _inputs(c, seed)
    s["case"] = c
    if c["op"] == "step":
        B, N, H, W = s["valid"].shape
        if c["mode"] in ("sparse", "table"):
            s["corr"] = gc.build_sparse_corr(s["pos"], s["valid"], s["cams"], K=c["K"], tables=c["mode"] == "table")
            if c["mode"] == "table":
                t = s["corr"]
                s["corr"] = gc.make_corr(s["pos"], s["valid"], s["cams"], t.tau, idx=t.idx, w=t.w, K=c["K"],
                                         mode=gc.CORR_TABLE)
        else:
            keep = torch.empty((B, N, N, H, W), dtype=torch.uint8, device=DEV) if c["mode"] == "mask" else None
            s["corr"] = gc.build_corr(gc.make_corr(s["pos"], s["valid"], s["cams"], torch.zeros(B, device=DEV), K=c["K"],
                                                   keep=keep))
        s["ws"] = None
        if c["mode"] == "sparse":
            s["ws"] = torch.empty(max(4, s["corr"].workspace_floats(c["C"])), device=DEV)
    if c["op"] == "build":
        s["records"] = torch.zeros((_capacity(c), 4), dtype=torch.int32, device=DEV)
    if c["op"] in ("step", "full"):
        s["pred"] = torch.empty_like(s["x0"]) if c["pred"] else None
        s["recon"] = gc.make_recon(**_sampler(c), pred_kind=_pred_kind(c), pred_out=s["pred"])
        in_place = c.get("in_place", False)
        s["x_next"] = s["x_t"] if in_place else torch.empty_like(s["x_t"])
        s["x0_out"] = s["x0"] if in_place else torch.empty_like(s["x0"]) if c["op"] == "step" or c["store"] else None
    if c["op"] == "loop":
        s["corr"] = gc.build_sparse_corr(s["pos"], s["valid"], s["cams"])
        s["ws"] = torch.empty(max(4, s["corr"].workspace_floats(c["C"])), device=DEV)
        s["lat"], s["cache"] = torch.empty_like(s["x_t"]), [torch.empty_like(s["x0"]) for _ in range(2)]
        s["rows"] = torch.empty_like(s["x_t"][:, :c["a"]])
        s["x0_new"] = torch.empty_like(s["x0"][:, :c["a"]])
        s["recons"] = [gc.make_recon("ddim", **p) for p in _alpha_bars(c["steps"])]
    return s


def _capacity(c):
    """Records that a program which keeps the records of many builds sets aside for one."""
    return c["B"] * c["N"] * (c["N"] - 1) * c["H"] * c["W"] // 4


def _alpha_bars(S):
    ab = np.cumprod(1.0 - np.linspace(0.00085 ** 0.5, 0.012 ** 0.5, 1000) ** 2)
    ts = np.round(np.linspace(999, 0, S)).astype(int)
    return [dict(a_t=float(ab[t]), a_prev=float(ab[ts[k + 1]]) if k + 1 < S else 1.0) for k, t in enumerate(ts)]


# -------------------------------------------------------------------- run --
def run(state):
    s, c = state, state["case"]
    op = c["op"]
    if op == "step":
        gc.transport_step(s["corr"], _anchors(c), c["C"], s["x0_new"], s["x0"], s["x0_out"], s["x_t"], s["x_next"],
                          s["recon"], workspace=s["ws"], update=c["update"])
        return {"x0": s["x0_out"], "x_next": s["x_next"], "pred": s["pred"]}
    if op == "full":
        gc.reconstruct(s["x_t"], s["x0"], s["x_next"], s["recon"], x0_store=s["x0_out"])
        return {"x_next": s["x_next"], "pred": s["pred"], "x0": s["x0_out"]}
    if op == "build":
        corr = gc.build_sparse_corr(s["pos"], s["valid"], s["cams"], K=c["K"], tables=c["tables"])
        t = corr._keep  # the tensors that the handle was built over
        rec = s["records"]
        rec[:len(t["records"])].copy_(t["records"])
        return {"tau": t["tau"], "keep": t["keep"], "tile_ptr": t["tile_ptr"], "idx": t["idx"], "w": t["w"],
                "taps": rec[:, :2], "frac": rec[:, 2:].view(torch.float32)}
    if op == "raster":
        pos, valid = gc.raster_posmaps(s["verts"], s["faces"], s["face_off"], s["cams"], c["H"], c["W"], s=c["s"])
        return {"pos": pos, "valid": valid}
    if op == "pool":
        pos, valid = gc.pool_posmaps(s["pos"], s["valid"], c["s"])
        return {"pos": pos, "valid": valid}
    # the sampler loop: the stand-in for the denoiser is x0 = the last x0 plus a drift given for the step
    sched = {"kind": "every_k", "k": c["every"]}
    lat, cur, nxt = s["lat"], s["cache"][0], s["cache"][1]
    lat.copy_(s["x_t"])
    cur.copy_(s["x0"])
    for k in range(c["steps"]):
        anchors, full = gc.rotate_anchors(c["N"], c["a"], k, c["steps"], sched)
        if full:
            torch.add(cur, s["drift"][k], out=nxt)
            gc.reconstruct(lat, nxt, lat, s["recons"][k])
        else:
            gc.pack_anchors(lat, s["rows"], anchors)
            gc.pack_anchors(cur, s["x0_new"], anchors)
            s["x0_new"].add_(s["drift"][k][:, :c["a"]])
            gc.transport_step(s["corr"], anchors, c["C"], s["x0_new"], cur, nxt, lat, lat, s["recons"][k],
                              workspace=s["ws"])
        cur, nxt = nxt, cur
    return {"x": lat, "x0": cur, "rows": s["rows"]}


# ------------------------------------------------------------------- work --
def work(case):
    c = case
    op = c["op"]
    px = c.get("B", 1) * c.get("N", 1) * c["H"] * c["W"]  # texels of all views
    if op in ("step", "full"):
        lat = 2 if c["dtype"] == "bf16" else 4
        per = px * c["C"]
        if op == "full":
            return {"bytes": per * (4 + 2 * lat + 4 * c["pred"] + 4 * c["store"]), "flops": 8 * per}
        f = c["a"] / c["N"]
        # other views: x0(t-1) in, x0(t) out, the latents in and out; anchors: the fresh x0 as well
        bytes_ = per * (8 + 2 * lat + 4 * c["pred"]) + per * f * (4 if c["update"] == "delta" else 0)
        pairs = px * (1 - f) * c["a"]  # (target token, anchor)
        bytes_ += {"sparse": 0, "mask": pairs, "table": pairs * c["K"] * 8, "geometry": px * 13}[c["mode"]]
        return {"bytes": bytes_, "flops": 10 * per}
    if op == "build":
        # positions and validity in, a mask byte per (token, source view) out, the tables where asked for
        return {"bytes": px * (13 + c["N"] + (8 * c["K"] * c["N"] if c["tables"] else 0)),
                "flops": 0.4 * px * (c["N"] - 1) * 80}
    if op == "raster":
        faces = 20 * 4 ** c["subdiv"]
        return {"bytes": c["B"] * (faces * 12 + faces / 2 * 12) + px * 13,
                "flops": c["B"] * c["N"] * faces * 60 + px * c["s"] ** 2 * 60}
    if op == "pool":
        return {"bytes": c["n"] * c["H"] * c["W"] * 13 * (c["s"] ** 2 + 1), "flops": c["n"] * c["H"] * c["W"] * 3 * c["s"] ** 2}
    per = px * c["C"]
    full = -(-c["steps"] // c["every"])
    f = c["a"] / c["N"]
    return {"bytes": full * per * (8 + 12) + (c["steps"] - full) * per * (12 + f * (4 + 4 + 20)),
            "flops": c["steps"] * per * 10}


# -------------------------------------------------------------- tolerance --
def tolerance(case):
    c = case
    if c["op"] in ("build", "raster", "pool"):
        return "exact"  # the interface fixes every choice and rounding of these
    if c["op"] == "loop":
        # bf16 latents carried through 30 steps: a rounding that falls the other way travels on
        return {"rel": 2e-3, "max": 5e-2}
    if c["dtype"] == "bf16":
        # f32 x0 differs by sums in another order (1e-7); a bf16 result by one last place at a tie
        return {"rel": 1e-4, "max": 1.6e-2}
    # a transported increment carries the rounding of its footprint's fractions: up to 1e-6 off the binary64 value
    return {"rel": 4e-6, "max": 2e-4}


# ------------------------------------------------------------------ exact --
def _f32_project(cam, X):
    """Projection of points X [B, M, 3] by cameras cam [B, 16], one binary32 rounding per operation."""
    xc = []
    for r in range(3):
        t = cam[:, 3 * r, None] * X[..., 0]
        t = t + cam[:, 3 * r + 1, None] * X[..., 1]
        t = t + cam[:, 3 * r + 2, None] * X[..., 2]
        xc.append(t + cam[:, 9 + r, None])
    uv = [cam[:, 12 + k, None] * (xc[k] / xc[2]) + cam[:, 14 + k, None] for k in range(2)]
    return xc, uv[0], uv[1]


def _tau(s):
    inf = torch.tensor(float("inf"), device=DEV)
    fg = s["valid"].bool().flatten(1)[..., None]
    p = s["pos"].flatten(1, 3)
    d = torch.where(fg, p, -inf).amax(1) - torch.where(fg, p, inf).amin(1)
    diag2 = d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2]
    tau = torch.tensor(TOL, device=DEV) * torch.sqrt(diag2)
    d = d.double()
    return torch.where(fg.any(1)[:, 0], tau, 0), np.float64(np.float32(TOL)) * d.pow(2).sum(1).sqrt()


def _taps(s, K, v, u, tau):
    """Taps of target view v in source view u: kept [B, HW, K] bool, index q, weights w (binary64), top-left index
    and fractions (binary64)."""
    B, N, H, W = s["valid"].shape
    X = s["pos"][:, v].reshape(B, -1, 3)
    src, ok = s["pos"][:, u].reshape(B, -1, 3), s["valid"][:, u].reshape(B, -1).bool()
    cam = s["cams"][:, u]
    xc, uu, vv = _f32_project(cam, X)
    _, u64, v64 = _f32_project(cam.double(), X.double())
    shift = 0.5 if K == 4 else 0.0
    x, y = uu - shift, vv - shift
    lo = -1.0 if K == 4 else 0.0
    there = s["valid"][:, v].reshape(B, -1).bool() & (xc[2] > 0) & (x >= lo) & (x < W) & (y >= lo) & (y < H)
    i0, j0 = (torch.where(there, torch.floor(t), 0).long() for t in (x, y))
    fx, fy = (u64 - shift - i0, v64 - shift - j0)
    f32x, f32y = x - torch.floor(x), y - torch.floor(y)
    kept, q, w = [], [], []
    for k in range(K):
        col, row = i0 + (k & 1), j0 + (k >> 1)
        inside = there & (col >= 0) & (col < W) & (row >= 0) & (row < H)
        if K == 4:
            inside &= ((f32x if k & 1 else 1.0 - f32x) != 0) & ((f32y if k >> 1 else 1.0 - f32y) != 0)
        at = torch.where(inside, row * W + col, 0)
        d = torch.gather(src, 1, at[..., None].expand(-1, -1, 3)) - X
        near = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2] <= (tau * tau)[:, None]
        kept.append(inside & near & torch.gather(ok, 1, at))
        q.append(at)
        w.append((fx if k & 1 else 1.0 - fx) * (fy if k >> 1 else 1.0 - fy) if K == 4 else torch.ones_like(fx))
    kept, q, w = torch.stack(kept, -1), torch.stack(q, -1), torch.stack(w, -1)
    w = torch.where(kept, w, 0.0)
    w = w / torch.where(kept.any(-1), w.sum(-1), 1.0)[..., None]
    return kept, q, w, j0 * W + i0, fx, fy


def _exact_step(s, c, taps, anchors, x0, x0_new, x_t, recon):
    """x0(t), x_{t-1} and the prediction of one cached step in binary64."""
    B, N, C, H, W = x0.shape
    out = x0.clone()
    out[:, anchors] = x0_new
    change = x0_new if c.get("update") == "copy" else x0_new - x0[:, anchors]
    for v in range(N):
        if v in anchors:
            continue
        total = torch.zeros((B, C, H * W), dtype=torch.float64, device=DEV)
        n = torch.zeros((B, H * W), dtype=torch.float64, device=DEV)
        for j, u in enumerate(anchors):
            kept, q, w = taps(v, u)[:3]
            n += kept.any(-1)
            for k in range(q.shape[-1]):
                at = q[:, None, :, k].expand(-1, C, -1)
                total += w[:, None, :, k] * torch.gather(change[:, j].flatten(2), 2, at)
        mean = total / n.clamp_min(1.0)[:, None]
        base = torch.where((n > 0)[:, None], 0.0, x0[:, v].flatten(2)) if c.get("update") == "copy" else x0[:, v].flatten(2)
        out[:, v] = (base + mean).reshape(B, C, H, W)
    return (out,) + _exact_recon(recon, x_t, out)


def _exact_recon(r, x_t, x0):
    if r["sampler"] == "ddim":
        eps = (x_t - math.sqrt(r["a_t"]) * x0) / math.sqrt(1.0 - r["a_t"])
        return math.sqrt(r["a_prev"]) * x0 + math.sqrt(1.0 - r["a_prev"]) * eps, eps
    vel = (x_t - x0) / r["sigma"]
    return x_t + (r["sigma_next"] - r["sigma"]) * vel, vel


def exact(case, seed):
    c = case
    s = _inputs(c, seed)
    op = c["op"]
    if op == "full":
        x, p = _exact_recon(_sampler(c), s["x_t"].double(), s["x0"].double())
        return {"x_next": x, "pred": p if c["pred"] else None, "x0": s["x0"].double() if c["store"] else None}
    if op == "pool":
        n, H, W, q = c["n"], c["H"], c["W"], c["s"]
        v = s["valid"].reshape(n, H, q, W, q)
        cnt = v.sum((2, 4), dtype=torch.float64)
        mean = torch.stack([(s["pos"][..., k].reshape(n, H, q, W, q) * v).sum((2, 4), dtype=torch.float64)
                            for k in range(3)], -1) / cnt.clamp_min(1.0)[..., None]
        fg = (cnt > 0) & (2 * cnt >= q * q)
        return {"pos": torch.where(fg[..., None], mean, 0.0), "valid": fg.to(torch.uint8)}
    if op == "raster":
        return _exact_raster(s, c)
    tau, tau64 = _tau(s)
    if op == "build":
        return _exact_build(s, c, tau, tau64)
    if op == "step":
        x0, x_next, pred = _exact_step(s, c, lambda v, u: _taps(s, c["K"], v, u, tau), _anchors(c), s["x0"].double(),
                                       s["x0_new"].double(), s["x_t"].double(), _sampler(c))
        return {"x0": x0, "x_next": x_next, "pred": pred if c["pred"] else None}
    lat, cur, kept = s["x_t"].double(), s["x0"].double(), {}

    def taps(v, u):
        if (v, u) not in kept:
            kept[v, u] = _taps(s, 4, v, u, tau)
        return kept[v, u]

    rows, r, N, a = None, 0, c["N"], c["a"]
    for k, p in enumerate(_alpha_bars(c["steps"])):
        p = dict(p, sampler="ddim")
        if k % c["every"] == 0:
            cur = cur + s["drift"][k].double()
            lat = _exact_recon(p, lat, cur)[0]
            continue
        step = -(-N // a)
        anchors = []
        for j in range(a):  # strided rotation; a repeated view gives way to the smallest free one
            x = (r % step + j * step) % N
            anchors.append(x if x not in anchors else min(y for y in range(N) if y not in anchors))
        anchors = sorted(anchors)
        r += 1
        rows = lat[:, anchors]
        x0_new = cur[:, anchors] + s["drift"][k][:, :a].double()
        cur, lat, _ = _exact_step(s, c, taps, anchors, cur, x0_new, lat, p)
    return {"x": lat, "x0": cur, "rows": rows}


def _exact_build(s, c, tau, tau64):
    B, N, H, W = s["valid"].shape
    HW, K = H * W, c["K"]
    keep = torch.zeros((B, N, N, HW), dtype=torch.uint8, device=DEV)
    tl = torch.zeros((B, N, N, HW), dtype=torch.int64, device=DEV)
    frac = torch.zeros((B, N, N, HW, 2), dtype=torch.float64, device=DEV)
    idx = w = None
    if c["tables"]:
        idx = torch.full((B, N, N, HW, K), -1, dtype=torch.int32, device=DEV)
        w = torch.zeros((B, N, N, HW, K), dtype=torch.float64, device=DEV)
    for v in range(N):
        for u in range(N):
            if u == v:
                continue
            kept, q, wt, q0, fx, fy = _taps(s, K, v, u, tau)
            keep[:, v, u] = sum(kept[..., k].to(torch.uint8) << k for k in range(K))
            tl[:, v, u] = q0
            if K == 4:
                frac[:, v, u] = torch.stack([fx, fy], -1)
            if c["tables"]:
                idx[:, v, u], w[:, v, u] = torch.where(kept, q, -1).int(), wt
    rows = keep.flatten() != 0
    at = rows.nonzero()[:, 0]
    token = at % HW
    mask = keep.flatten()[at].long() << 28
    word = token | mask
    word = torch.where(word >= 2 ** 31, word - 2 ** 32, word)
    T = -(-HW // gc.TILE_TOKENS)
    n = torch.zeros((B, N, N, T * gc.TILE_TOKENS), dtype=torch.int64, device=DEV)
    n[..., :HW] = keep != 0
    ends = n.reshape(-1, gc.TILE_TOKENS).sum(1).cumsum(0)
    taps, fr = torch.zeros((_capacity(c), 2), dtype=torch.int32), torch.zeros((_capacity(c), 2), dtype=torch.float64)
    taps[:len(at)] = torch.stack([word, tl.flatten()[at]], 1).int().cpu()
    fr[:len(at)] = frac.reshape(-1, 2)[at].cpu()
    return {"tau": tau64, "keep": keep.reshape(B, N, N, H, W),
            "tile_ptr": torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), ends]).int(),
            "idx": None if idx is None else idx.reshape(B, N, N, H, W, K),
            "w": None if w is None else w.reshape(B, N, N, H, W, K),
            "taps": taps, "frac": fr}


def _exact_raster(s, c):
    B, N, ss = c["B"], c["N"], c["s"]
    H, W = c["H"] * ss, c["W"] * ss
    F = len(s["faces"]) // B
    pos = torch.zeros((B, N, H, W, 3), dtype=torch.float64, device=DEV)
    valid = torch.zeros((B, N, H, W), dtype=torch.uint8, device=DEV)
    for b in range(B):
        tri = s["verts"][s["faces"][b * F:(b + 1) * F].long()]  # [F, 3, 3]
        for v in range(N):
            cam = s["cams"][b, v].clone()
            cam[12:] *= ss
            pos[b, v], valid[b, v] = _exact_view(tri, cam, H, W)
    if ss == 1:
        return {"pos": pos, "valid": valid}
    fine = valid.reshape(B, N, c["H"], ss, c["W"], ss)
    cnt = fine.sum((3, 5), dtype=torch.float64)
    fg = (cnt > 0) & (2 * cnt >= ss * ss)
    total = pos.reshape(B, N, c["H"], ss, c["W"], ss, 3).sum((3, 5))
    return {"pos": torch.where(fg[..., None], total / cnt.clamp_min(1.0)[..., None], 0.0), "valid": fg.to(torch.uint8)}


def _plane(P):
    """Normal n and offset n . P0 of camera-space triangles P [F, 3, 3], term by term in P's own precision."""
    e1, e2 = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
    n = [e1[:, (k + 1) % 3] * e2[:, (k + 2) % 3] - e1[:, (k + 2) % 3] * e2[:, (k + 1) % 3] for k in range(3)]
    return n, n[0] * P[:, 0, 0] + n[1] * P[:, 0, 1] + n[2] * P[:, 0, 2]


def _camera_points(tri, cam):
    out = []
    for r in range(3):
        t = cam[3 * r] * tri[..., 0]
        t = t + cam[3 * r + 1] * tri[..., 1]
        t = t + cam[3 * r + 2] * tri[..., 2]
        out.append(t + cam[9 + r])
    return torch.stack(out, -1)


def _exact_view(tri, cam, H, W):
    """The nearest face of every pixel centre (binary32), and where its plane meets the pixel's ray (binary64)."""
    P = _camera_points(tri, cam)
    U, V = (cam[12 + k] * (P[..., k] / P[..., 2]) + cam[14 + k] for k in range(2))
    area = (U[:, 1] - U[:, 0]) * (V[:, 2] - V[:, 0]) - (V[:, 1] - V[:, 0]) * (U[:, 2] - U[:, 0])
    ilo, ihi = torch.ceil(U.amin(1) - 0.5).clamp_min(0), torch.floor(U.amax(1) - 0.5).clamp_max(W - 1)
    jlo, jhi = torch.ceil(V.amin(1) - 0.5).clamp_min(0), torch.floor(V.amax(1) - 0.5).clamp_max(H - 1)
    ok = (P[..., 2] > 1e-6).all(1) & (area != 0) & (ilo <= ihi) & (jlo <= jhi)
    n, nd = _plane(P)
    f = ok.nonzero()[:, 0]
    bw = (ihi - ilo + 1).long()[f]
    size = bw * (jhi - jlo + 1).long()[f]
    face = torch.repeat_interleave(f, size)  # every (face, pixel of its box)
    start = torch.repeat_interleave(size.cumsum(0) - size, size)
    k = torch.arange(len(face), device=DEV) - start
    wide = torch.repeat_interleave(bw, size)
    i, j = ilo.long()[face] + k % wide, jlo.long()[face] + k // wide
    pu, pv = i.float() + 0.5, j.float() + 0.5

    def edge(a, b):
        return (U[face, b] - U[face, a]) * (pv - V[face, a]) - (V[face, b] - V[face, a]) * (pu - U[face, a])

    w = torch.stack([edge(1, 2), edge(2, 0), edge(0, 1)])
    inside = torch.where(area[face] > 0, (w >= 0).all(0), (w <= 0).all(0))
    d0, d1 = (pu - cam[14]) / cam[12], (pv - cam[15]) / cam[13]
    den = n[0][face] * d0 + n[1][face] * d1 + n[2][face]
    depth = nd[face] / den
    inside &= (den != 0) & (depth > 0) & (depth <= 3e38)
    face, i, j, depth = face[inside], i[inside], j[inside], depth[inside]
    key = (depth.view(torch.int32).long() << 32) | face
    z = torch.full((H * W,), 2 ** 63 - 1, dtype=torch.int64, device=DEV)
    z.scatter_reduce_(0, j * W + i, key, "amin")
    hit = (z != 2 ** 63 - 1).nonzero()[:, 0]
    cam, face = cam.double(), z[hit] & 0xffffffff
    P = _camera_points(tri[face].double(), cam)
    n, nd = _plane(P)
    d0 = ((hit % W) + 0.5 - cam[14]) / cam[12]
    d1 = ((hit // W) + 0.5 - cam[15]) / cam[13]
    depth = nd / (n[0] * d0 + n[1] * d1 + n[2])
    x = torch.stack([depth * d0, depth * d1, depth], -1) - cam[9:12]
    pos = torch.zeros((H * W, 3), dtype=torch.float64, device=DEV)
    pos[hit] = x @ cam[:9].reshape(3, 3)
    valid = torch.zeros(H * W, dtype=torch.uint8, device=DEV)
    valid[hit] = 1
    return pos.reshape(H, W, 3), valid.reshape(H, W)
