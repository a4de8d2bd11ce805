"""The forward's pixels bit for bit against a float32 restatement of its shading in
numpy, every rounding stated: a last bit that moves turns the sign that the loss's
adjoint takes of a pixel, so images must not depend on how the kernels around the
shading are compiled, nor on which of them shades a pixel."""
import functools

import numpy as np
import pytest

import oracle
from oracle import _fma32
from paper_2107_05509_gb300 import inputs as I
from tests.gpu_common import require_gpu, torch

pytestmark = pytest.mark.gpu

F32 = np.float32
SPP, KA, LIGHT = 3, F32(0.8), np.array([0.9, 1.0, 1.1], F32)


@functools.lru_cache(maxsize=None)
def _hand(levels):
    h = I.make_hand(0)
    return I.subdivide_hand(h, levels) if levels else h


def _mul_add2(a, b, c, d):
    """a b + c d, the first product exact."""
    return _fma32(a, b, c * d)


def _texture_albedo(tex, uv, u, v):
    """Bilinear lookup at the interpolated texture coordinates (uv [n][3][2])."""
    th, tw, _ = tex.shape
    w = F32(1) - u - v
    x, y = (_fma32(_fma32(v, uv[:, 2, k], _fma32(u, uv[:, 1, k], w * uv[:, 0, k])), F32(n), F32(-0.5))
            for k, n in ((0, tw), (1, th)))
    xf, yf = np.floor(x), np.floor(y)
    fx, fy = x - xf, y - yf
    gx, gy = F32(1) - fx, F32(1) - fy
    i0, i1 = (np.clip(xf + k, 0, tw - 1).astype(int) for k in (0, 1))
    j0, j1 = (np.clip(yf + k, 0, th - 1).astype(int) for k in (0, 1))
    out = np.empty((len(u), 3), F32)
    for c in range(3):
        t00, t10, t01, t11 = tex[j0, i0, c], tex[j0, i1, c], tex[j1, i0, c], tex[j1, i1, c]
        p = _mul_add2(fx, t10, gx, t00) if c < 2 else _mul_add2(gx, t00, fx, t10)
        out[:, c] = _mul_add2(gy, p, fy, _mul_add2(gx, t01, fx, t11))
    return out


def _vertex_albedo(alb, u, v):
    w = F32(1) - u - v
    return np.stack([_fma32(v, alb[:, 2, c], _mul_add2(w, alb[:, 0, c], u, alb[:, 1, c])) for c in range(3)], 1)


# 40 x 36: lists in the shaders' tile; 9 x 9 of 24.6 k triangles: more candidates than a list holds,
# rays through the tree (k_overflow)
@pytest.mark.parametrize("levels,W,H", [(0, 40, 36), (2, 9, 9)])
@pytest.mark.parametrize("textured", [True, False])
def test_pixels_have_the_stated_roundings(levels, W, H, textured):
    require_gpu()
    from paper_2107_05509_gb300 import binding as B
    h, seed = _hand(levels), 77
    cfg = I.SceneConfig("bits", views=1, width=W, height=H, spp=SPP, edge_samples=0, elevation_deg=20.0, azimuths_deg=(10.0,))
    cam = I.pack_cameras(I.make_cameras(cfg, h.v_template.mean(0)))[0].astype(F32)
    cam[0:2] *= F32(2.0)
    verts = oracle.skin(h, I.gt_params(5)).astype(F32)
    rng = np.random.default_rng(5)
    bg, tex = rng.random((1, H, W, 3), dtype=F32), rng.random((13, 31, 3), dtype=F32)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    model, ctx = B.Model(h), B.Context(h.V, h.F, h.E, 1, W, H)
    vt, ct, bt, tt, img = t(verts), t(cam[None]), t(bg), t(tex), torch.empty((1, H, W, 3), device="cuda")
    B.hr_build_bvh(ctx, model, vt)
    # kd = 0: the shading factor is ka (the normal's reciprocal length is the hardware's)
    opts = B.render_opts(seed=seed, spp=SPP, edge_samples=0, ka=float(KA), kd=0.0, light_rgb=tuple(map(float, LIGHT)),
                         texture=tt if textured else None)
    # the samples' rays and hits, pixel by pixel, sample by sample
    n = H * W * SPP
    r = np.array([oracle.philox([p, 0, s, 0], [seed, 0])[:2] for p in range(H * W) for s in range(SPP)], np.uint32)
    j = (r >> 8).astype(F32) * F32(2.0 ** -24)
    pix = np.repeat(np.arange(H * W), SPP)
    dx = ((pix % W).astype(F32) + j[:, 0] - cam[2]) / cam[0]
    dy = ((pix // W).astype(F32) + j[:, 1] - cam[3]) / cam[1]
    R = cam[4:13]
    d = np.stack([_fma32(R[k], dx, _fma32(R[3 + k], dy, R[6 + k])) for k in range(3)], 1)
    tri, tuv = torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty((n, 3), device="cuda")
    B.hr_trace(ctx, t(np.broadcast_to(cam[16:19], (n, 3))), t(d), tri, tuv)
    tri, tuv = tri.cpu().numpy(), tuv.cpu().numpy()
    f, u, v, hit = h.faces[np.maximum(tri, 0)], tuv[:, 1], tuv[:, 2], (tri >= 0).reshape(-1, SPP)
    alb = _texture_albedo(tex, h.uv.astype(F32)[f], u, v) if textured else _vertex_albedo(h.albedo.astype(F32)[f], u, v)
    rad = (alb * LIGHT).reshape(-1, SPP, 3)
    acc = np.zeros((H * W, 3), F32)
    for s in range(SPP):
        acc = np.where(hit[:, s, None], _fma32(rad[:, s], KA, acc), acc)
    miss = (~hit).sum(1).astype(F32)[:, None] / F32(SPP)
    ref = _mul_add2(acc, F32(1) / F32(SPP), bg.reshape(-1, 3) * (miss > 0), miss)
    assert hit.any(1).sum() > 10
    for rays in (1, 2, 4):
        ctx.set_tuning(rays_per_lane=rays, max_chunks=1)   # a pixel's samples in one sum
        B.hr_render_fwd(ctx, model, vt, ct, H, W, bt, opts, img)
        assert (img.cpu().numpy().reshape(-1, 3) == ref).all(), (rays, (img.cpu().numpy().reshape(-1, 3) != ref).sum())
    assert B.hr_get_status(ctx) == B.HR_OK
