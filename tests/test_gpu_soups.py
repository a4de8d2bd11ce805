"""Separate triangles of awkward shapes and places, against the oracle's brute force: the
pixels a triangle can cover are taken from its edges on the screen (moved outward by a
margin, or its box where that is not certain), and a mask that is too small loses hits
silently; the backward takes a triangle's own vectors down to |cos| = 1/32 to the view
and each sample's ray below."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2107_05509_gb300 import inputs as I
from tests.gpu_common import pixel_ok, require_gpu, torch

pytestmark = pytest.mark.gpu


def _soup(corners, seed):
    """A model of separate triangles ([n][3][3])."""
    h, r, V = I.make_hand(0), np.random.default_rng(seed), 3 * len(corners)
    v, faces = np.ascontiguousarray(corners, np.float32).reshape(V, 3), np.arange(V, dtype=np.int32).reshape(-1, 3)
    edges, edge_faces, off, vf = I.mesh_topology(faces, V)
    w = np.zeros((V, h.weights.shape[1]), np.float32)
    w[:, 0] = 1
    return dataclasses.replace(h, v_template=v, shapedirs=np.zeros((V, 3, h.shapedirs.shape[2]), np.float32), weights=w,
                               faces=faces, edges=edges, edge_faces=edge_faces, vf_offsets=off, vf_faces=vf,
                               albedo=r.random((V, 3), dtype=np.float32), uv=r.random((V, 2), dtype=np.float32))


def _view(W, H, azimuth=33.0):
    """(camera record, R, t, centre) of a view from 0.6 m of the origin."""
    cfg = I.SceneConfig("soup", views=1, width=W, height=H, spp=1, edge_samples=0, elevation_deg=17.0, azimuths_deg=(azimuth,))
    cams = I.pack_cameras(I.make_cameras(cfg, np.zeros(3)))
    return cams, cams[0, 4:13].reshape(3, 3).astype(np.float64), cams[0, 13:16].astype(np.float64), cams[0, 16:19].astype(np.float64)


def _corners(kind, r, R, t, c):
    n = 600
    size = lambda lo, hi: 10 ** r.uniform(lo, hi, (n, 1, 1))
    base, a = r.uniform(-0.15, 0.15, (n, 1, 3)), r.normal(size=(n, 1, 3)) * size(-3, -1)
    if kind in ("sizes", "wide"):       # from a hundredth of a pixel to the whole image
        return base + r.normal(size=(n, 3, 3)) * size(-5, -1)
    if kind == "slivers":               # three corners nearly on a line
        return base + np.concatenate([0 * a, a, r.uniform(-0.5, 1.5, (n, 1, 1)) * a + r.normal(size=a.shape) * size(-8, -4)], 1)
    if kind == "needles":               # two corners nearly the same
        return base + np.concatenate([0 * a, r.normal(size=a.shape) * size(-7, -4), a], 1)
    if kind == "edge-on":               # planes nearly through the centre
        d = (base - c) / np.linalg.norm(base - c, axis=-1, keepdims=True)
        return np.concatenate([base, base + a, base + 0.02 * d + 0.3 * a + r.normal(size=a.shape) * size(-9, -4)], 1)
    # corners just before and behind the camera's plane
    z = size(-4, 0) * r.choice([-1.0, 1.0, 1.0, 1.0], (n, 3, 1))
    return (np.concatenate([r.uniform(-1, 1, (n, 3, 2)) * np.abs(z), z], -1) - t) @ R


@pytest.mark.parametrize("kind", ["sizes", "slivers", "needles", "edge-on", "camera-plane", "wide"])
def test_no_hit_is_lost(kind):
    require_gpu()
    from paper_2107_05509_gb300 import binding as B
    W, H = (16384, 3) if kind == "wide" else (96, 80)
    cams, R, t, c = _view(W, H)
    h, seed = _soup(_corners(kind, np.random.default_rng(7), R, t, c), 7), 11
    opts = dict(seed=seed, spp=8, edge_samples=0, ka=1.0, kd=0.0, light_dir=I.LIGHT_DIR, light_rgb=(1.0, 1.0, 1.0))
    normals = oracle.vertex_normals(h.v_template, h.faces, h.vf_offsets, h.vf_faces)
    bg = np.zeros((1, H, W, 3), np.float32)
    ref = oracle.render_fwd(h.v_template, h.faces, normals, h.albedo, cams, H, W, bg, oracle.make_opts(edge_eps=I.EDGE_EPS_PX, **opts))
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    model, ctx = B.Model(h), B.Context(h.V, h.F, h.E, 1, W, H)
    v, img = dev(h.v_template), torch.empty((1, H, W, 3), device="cuda")
    B.hr_build_bvh(ctx, model, v)
    B.hr_render_fwd(ctx, model, v, dev(cams), H, W, dev(bg), B.render_opts(edge_eps_px=I.EDGE_EPS_PX, **opts), img)
    ok = pixel_ok(img.cpu().numpy(), ref)
    assert (ref > 0).any() and ok.all(), np.argwhere(~ok)[:5]
    assert B.hr_get_status(ctx) == B.HR_OK


@pytest.mark.parametrize("cos", [1 / 8, 1 / 31, 1 / 33, 1 / 64])
def test_gradients_at_grazing_angles(cos):
    """64 triangles of 20 mm at one angle to their views, on both sides of the limit: a
    triangle's interior gradient within 1e-4 of its norm (ten roundings of its vectors,
    2^-24 each, against a height that is `cos` of them: 4e-5 at 1/64)."""
    require_gpu()
    from paper_2107_05509_gb300 import binding as B
    W, n, r = 128, 8, np.random.default_rng(3)
    cams, R, t, c = _view(W, W)
    corners = []
    for i in range(n * n):
        x, y = (i % n + 0.5) * W / n, (i // n + 0.5) * W / n
        d = R.T @ np.array([(x - cams[0, 2]) / cams[0, 0], (y - cams[0, 3]) / cams[0, 1], 1.0])
        p, d = c + 0.6 * d, d / np.linalg.norm(d)
        a = np.cross(d, r.normal(size=3))
        a /= np.linalg.norm(a)
        b = cos * np.cross(d, a) + np.sqrt(1 - cos * cos) * d
        phi = r.random() * 2 * np.pi + 2 * np.pi / 3 * np.arange(3)[:, None]
        corners.append(p + 0.02 * (np.cos(phi) * a + np.sin(phi) * b))
    h = _soup(corners, 3)
    opts = dict(seed=9, spp=32, edge_samples=0, ka=I.K_AMBIENT, kd=I.K_DIFFUSE, light_dir=I.LIGHT_DIR, light_rgb=I.LIGHT_RGB)
    normals = oracle.vertex_normals(h.v_template, h.faces, h.vf_offsets, h.vf_faces)
    bg, A = np.zeros((1, W, W, 3), np.float32), (r.normal(size=(1, W, W, 3)) * 1e-3).astype(np.float32)
    ref, _ = oracle.render_bwd_interior(h.v_template, h.faces, normals, h.albedo, cams, W, W, bg,
                                        oracle.make_opts(edge_eps=I.EDGE_EPS_PX, **opts), A)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    model, ctx = B.Model(h), B.Context(h.V, h.F, h.E, 1, W, W)
    v, ct, bt, img, dv = dev(h.v_template), dev(cams), dev(bg), torch.empty((1, W, W, 3), device="cuda"), torch.empty((h.V, 3), device="cuda")
    go = B.render_opts(edge_eps_px=I.EDGE_EPS_PX, flags=B.HR_BWD_REUSE_FWD | B.HR_BWD_NO_EDGES | B.HR_BWD_NO_NORMALS, **opts)
    B.hr_build_bvh(ctx, model, v)
    B.hr_render_fwd(ctx, model, v, ct, W, W, bt, go, img)
    B.hr_render_bwd(ctx, model, v, ct, W, W, bt, go, dev(A), dv)
    ref, got = np.asarray(ref).reshape(-1, 9), dv.cpu().numpy().reshape(-1, 9)
    size = np.linalg.norm(ref, axis=1)
    assert (size > 0).sum() > 40 and (np.linalg.norm(got - ref, axis=1) <= 1e-4 * size).all()
    assert B.hr_get_status(ctx) == B.HR_OK
