"""The backward differentiates a pixel's hits in windows of 16 samples: gradients of calls
with several windows per work item, the last one ragged or not, against the oracle (the
usual bar), with a texture so small that many samples of a window share a texel cell and
some lie beyond its border."""
import numpy as np
import pytest

import oracle
from paper_2107_05509_gb300 import inputs as I
from tests.gpu_common import grad_ok, require_gpu, torch
from tests.test_gpu_shading_bits import _hand

pytestmark = pytest.mark.gpu


# 40 x 36: lists in the shaders' tile; 9 x 9 of 24.6 k triangles: more candidates than a
# list holds, rays through the tree, a lane's one after another (k_overflow)
@pytest.mark.parametrize("levels,W,H", [(0, 40, 36), (2, 9, 9)])
@pytest.mark.parametrize("spp", [1, 35, 64])
def test_gradients_of_several_windows(levels, W, H, spp):
    require_gpu()
    from paper_2107_05509_gb300 import binding as B
    h, seed = _hand(levels), 31
    cfg = I.SceneConfig("windows", views=1, width=W, height=H, spp=spp, edge_samples=0, elevation_deg=20.0, azimuths_deg=(10.0,))
    cams = I.pack_cameras(I.make_cameras(cfg, h.v_template.mean(0)))
    cams[:, 0:2] *= 2.0
    verts = oracle.skin(h, I.gt_params(5).astype(np.float32)).astype(np.float32)
    normals = oracle.vertex_normals(verts, h.faces, h.vf_offsets, h.vf_faces)
    bg, tex = I.background(5, 1, H, W), np.random.default_rng(5).random((3, 5, 3), dtype=np.float32)
    A = (np.random.default_rng(6).choice([-1.0, 0.0, 1.0], size=(1, H, W, 3)) * 1e-4).astype(np.float32)
    common = dict(spp=spp, edge_samples=0, ka=I.K_AMBIENT, kd=I.K_DIFFUSE, light_dir=I.LIGHT_DIR, light_rgb=I.LIGHT_RGB)
    o = oracle.make_opts(seed=seed, edge_eps=I.EDGE_EPS_PX, texture=tex, uv=h.uv, **common)
    dT_ref = np.zeros(tex.shape, np.float64)
    dv_ref, _ = oracle.render_bwd(h, verts, cams, H, W, bg, o, A, normals=normals, d_texture=dT_ref)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    model, ctx = B.Model(h), B.Context(h.V, h.F, h.E, 1, W, H)
    vt, ct, bt, tt, At, img, dv = t(verts), t(cams), t(bg), t(tex), t(A), torch.empty((1, H, W, 3), device="cuda"), torch.empty((h.V, 3), device="cuda")
    B.hr_build_bvh(ctx, model, vt)
    fixed = []
    for chunks, rays, flags in ((1, 4, 0), (1, 1, 0), (1, 4, B.HR_DETERMINISTIC), (1, 2, B.HR_DETERMINISTIC), (16, 4, 0)):
        ctx.set_tuning(max_chunks=chunks, bwd_rays_per_lane=rays)
        dt = torch.zeros_like(tt)
        go = B.render_opts(seed=seed, texture=tt, d_texture=dt, edge_eps_px=I.EDGE_EPS_PX, flags=flags | B.HR_BWD_REUSE_FWD, **common)
        B.hr_render_fwd(ctx, model, vt, ct, H, W, bt, go, img)
        B.hr_render_bwd(ctx, model, vt, ct, H, W, bt, go, At, dv)
        assert grad_ok(dv.cpu().numpy(), dv_ref).all(), (chunks, rays, flags)
        assert np.abs(dT_ref).max() > 0 and grad_ok(dt.cpu().numpy(), dT_ref).all(), (chunks, rays, flags)
        if flags:
            fixed.append(dv.clone())
    assert torch.equal(*fixed)
    assert B.hr_get_status(ctx) == B.HR_OK


@pytest.mark.parametrize("zoom,spp", [(2.0, 1), (30.0, 1), (30.0, 2), (30.0, 17), (300.0, 1)])
@pytest.mark.parametrize("size", [1e-6, 1.0, 1e4])
def test_fixed_point_sums_of_lanes_that_share_a_triangle(zoom, spp, size):
    """From many triangles per sub-tile to one under the whole image: fixed-point sums
    (a contribution is rounded to 2^-40) against the oracle at gradients of either sign
    and a range of sizes, the same bits again when other warps do the same work."""
    require_gpu()
    from paper_2107_05509_gb300 import binding as B
    h, (W, H), seed = _hand(0), (72, 52), 13
    cfg = I.SceneConfig("shared", views=1, width=W, height=H, spp=spp, edge_samples=0, elevation_deg=20.0, azimuths_deg=(10.0,))
    verts = oracle.skin(h, I.gt_params(5).astype(np.float32)).astype(np.float32)
    cams = I.pack_cameras(I.make_cameras(cfg, verts[h.faces[700]].mean(0)))
    cams[:, 0:2] *= zoom
    normals = oracle.vertex_normals(verts, h.faces, h.vf_offsets, h.vf_faces)
    bg = I.background(5, 1, H, W)
    A = (np.random.default_rng(6).normal(size=(1, H, W, 3)) * size).astype(np.float32)
    common = dict(spp=spp, edge_samples=0, ka=I.K_AMBIENT, kd=I.K_DIFFUSE, light_dir=I.LIGHT_DIR, light_rgb=I.LIGHT_RGB)
    ref, _ = oracle.render_bwd(h, verts, cams, H, W, bg, oracle.make_opts(seed=seed, edge_eps=I.EDGE_EPS_PX, **common), A, normals=normals)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    model, ctx = B.Model(h), B.Context(h.V, h.F, h.E, 1, W, H)
    vt, ct, bt, At, img, dv = t(verts), t(cams), t(bg), t(A), torch.empty((1, H, W, 3), device="cuda"), torch.empty((h.V, 3), device="cuda")
    go = B.render_opts(seed=seed, edge_eps_px=I.EDGE_EPS_PX, flags=B.HR_DETERMINISTIC | B.HR_BWD_REUSE_FWD, **common)
    B.hr_build_bvh(ctx, model, vt)
    B.hr_render_fwd(ctx, model, vt, ct, H, W, bt, go, img)
    fixed = []
    for blocks in (4, 1):
        ctx.set_tuning(bwd_blocks_per_sm=blocks)
        B.hr_render_bwd(ctx, model, vt, ct, H, W, bt, go, At, dv)
        fixed.append(dv.clone())
    assert np.abs(ref).max() > 0 and torch.equal(*fixed)
    if np.abs(ref).max() < 2.0 ** 22:   # (sums wrap at 2^23: 64 bits of 2^-40)
        assert grad_ok(dv.cpu().numpy(), ref).all()
    assert B.hr_get_status(ctx) == B.HR_OK
