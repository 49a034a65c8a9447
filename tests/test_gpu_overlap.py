"""Dependent calls back to back: some kernels become resident while the one
before them still runs, so a chain of steps that each read what the step
before wrote, without a host synchronisation between them, must equal the same
chain synchronised after every call, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2608_13255_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_13255_gb300 import build as gbuild
    gbuild.build()
    from paper_2608_13255_gb300 import geocache
    geocache.load()
    return geocache


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("mode,B,H,W,C,a,K,dtype", [
    ("sparse", 70, 36, 32, 4, 2, 4, "bf16"),    # 840 units: the record-parallel apply, two launches
    ("sparse", 12, 37, 29, 18, 3, 4, "f32"),    # 720 units: the increment plane, unaligned rows
    ("sparse_min", 20, 36, 32, 16, 2, 4, "bf16"),  # 960 units: the source-tile apply
    ("sparse", 2, 64, 64, 4, 2, 4, "f32"),      # 48 units: one launch, one token per thread
    ("mask", 2, 64, 64, 4, 3, 4, "f32"),        # the same from the masks
    ("mask", 46, 64, 64, 4, 2, 4, "bf16"),      # 1,104 units: the staged kernel
    ("mask", 40, 37, 29, 4, 2, 1, "f32"),       # 480 units, unaligned rows: one CTA per tile
    ("table", 3, 37, 29, 4, 2, 4, "bf16"),
    ("geometry", 3, 37, 29, 5, 5, 4, "f32"),    # two rounds of anchors
])
def test_dependent_steps_equal_synchronised_ones(gc, mode, B, H, W, C, a, K, dtype, in_place):
    w = synth.replicate_assets(synth.make_workload("batch128", B=2, H=H, W=W), B)
    N = w.N
    pos, valid, cams = (torch.from_numpy(x).cuda() for x in (w.pos, w.valid, w.cams))
    corr = gc.build_sparse_corr(pos, valid, cams, K=K, source_index=True, tables=mode == "table")
    corr.c.mode = {"mask": gc.CORR_MASK, "table": gc.CORR_TABLE, "geometry": gc.CORR_GEOMETRY}.get(mode, gc.CORR_SPARSE)
    minimal = mode == "sparse_min"
    ws = torch.empty(max(4, corr.min_workspace_floats(C) if minimal else corr.workspace_floats(C)), device="cuda")
    gen = torch.Generator("cuda").manual_seed(7)
    rnd = lambda *s: torch.randn(s, generator=gen, device="cuda")
    lat = torch.bfloat16 if dtype == "bf16" else torch.float32
    x0_init, x_init = rnd(B, N, C, H, W), rnd(B, N, C, H, W).to(lat)
    fresh = [rnd(B, a, C, H, W) for _ in range(3)]
    full = rnd(B, N, C, H, W)
    S = 24

    def chain(sync):
        cache, x = [x0_init.clone(), x0_init.clone()], [x_init.clone(), x_init.clone()]
        torch.cuda.synchronize()
        i = 0
        for t in range(S):
            o = i if in_place else 1 - i
            r = gc.make_recon("fm_euler", sigma=1.0 - t / S, sigma_next=1.0 - (t + 1) / S)
            if t % 6 == 5:  # a full step
                gc.reconstruct(x[i], full, x[o], r, x0_store=cache[o])
            else:
                anchors = sorted((t + k * (N // a)) % N for k in range(a))
                gc.transport_step(corr, anchors, C, fresh[t % 3], cache[i], cache[o], x[i], x[o], r, workspace=ws)
            if sync:
                torch.cuda.synchronize()
            i = o
        gc.device_status()
        return cache[i], x[i]

    ref = chain(True)
    assert torch.isfinite(ref[1]).all() and not torch.equal(ref[1], x_init)
    for _ in range(3):
        for got, want in zip(chain(False), ref):
            assert torch.equal(got.view(torch.uint8), want.view(torch.uint8))


@pytest.mark.parametrize("s", [2, 3, 8])
def test_pooling_behind_its_render_equals_a_synchronised_one(gc, s):
    # the fine maps are rendered into the same buffers again and again, each pooled by the next call
    H, W, N = 24, 40, 6
    V, F = synth.blob_mesh(3, 0.15, np.random.default_rng(5))
    dev = lambda x, t: torch.from_numpy(np.ascontiguousarray(x)).to(t).cuda()
    verts, faces = dev(V, torch.float32), dev(F, torch.int32)
    f_off = torch.tensor([0, len(F)], dtype=torch.int64, device="cuda")
    cams = [dev(np.stack([synth.look_at_camera(az + 15.0 * k, el, s * H, s * W) for az, el in synth.hunyuan_layout()])[None],
                torch.float32) for k in range(8)]

    def chain(sync):
        zb = torch.empty((1, N, s * H, s * W), dtype=torch.int64, device="cuda")
        hi, hv = torch.empty((1, N, s * H, s * W, 3), device="cuda"), torch.empty((1, N, s * H, s * W), dtype=torch.uint8,
                                                                                device="cuda")
        out = [(torch.empty((1, N, H, W, 3), device="cuda"), torch.empty((1, N, H, W), dtype=torch.uint8, device="cuda"))
               for _ in cams]
        torch.cuda.synchronize()
        for c, (p, v) in zip(cams, out):
            gc.raster_posmaps(verts, faces, f_off, c, s * H, s * W, zb, hi, hv)
            if sync:
                torch.cuda.synchronize()
            gc.pool_posmaps(hi, hv, s, p, v)
            if sync:
                torch.cuda.synchronize()
        gc.device_status()
        return out

    ref = chain(True)
    assert all(v.float().mean() > 0.05 for _, v in ref)
    for (p, v), (rp, rv) in zip(chain(False), ref):
        assert torch.equal(v, rv) and torch.equal(p.view(torch.int32), rp.view(torch.int32))
