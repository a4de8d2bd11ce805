"""Kernels at the sizes where their division of the work changes: fewer tiles than
SMs, one more than a multiple, odd counts."""
import dataclasses

import numpy as np
import pytest

from oracle import net as N
from paper_2107_05509_gb300 import inputs as I
from tests import test_gpu_gemm as TG
from tests import test_gpu_net as TN
from tests.gpu_common import hand, require_gpu, scene, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B_():
    require_gpu()
    from paper_2107_05509_gb300 import binding
    return binding


def _net_run(B_, copies):
    p, X, cams = TN._case(2, 2)
    net = B_.Net(2 * copies, 2)
    net.set_params(torch.as_tensor(p, device="cuda"))
    Xt = torch.as_tensor(X.astype(np.float32), device="cuda").to(torch.bfloat16)
    net.set_inputs_bf16(Xt.repeat(copies, 1, 1, 1))
    out = torch.empty((2 * copies, 61), device="cuda")
    net.forward(torch.as_tensor(np.concatenate([cams] * copies), device="cuda"), out)
    d_out = np.random.default_rng(7).normal(size=(2, 61)).astype(np.float32)
    net.backward(torch.as_tensor(np.concatenate([d_out] * copies), device="cuda"))
    g = torch.empty(net.P, device="cuda")
    net.get_params(grads=g)
    assert net.status() == B_.HR_OK
    return out.cpu().numpy(), g.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("copies", [3, 9, 40])
def test_convolutions_are_sums_over_their_images(B_, copies):
    """The gathered convolutions on copies of the four images that the network's tests
    check against the oracle: 12 images (most SMs idle), 36 (tiles and splits do not
    divide evenly), 160 (rings and accumulators wrap, more images than SMs).  Outputs
    equal the single case's bit for bit in every copy.  Gradients are sums of equal
    addends: they are `copies` times the single ones up to float32 accumulation of at
    most 655360 products in pieces of at most 4096 (256 steps of the tensor cores, each
    2^-24 of the running sum, 1.5e-5 per piece, with some cancellation): 1e-4 of the
    layer's largest."""
    out1, g1 = _net_run(B_, 1)
    out, g = _net_run(B_, copies)
    assert (out.reshape(copies, 2, 61) == out1).all()
    for name, (w, b, n_out, K) in N.offsets()[0].items():
        for lo, hi in ((w, w + n_out * K), (b, b + n_out)):
            err = np.abs(g[lo:hi] - copies * g1[lo:hi]).max()
            assert err <= 1e-4 * copies * np.abs(g1[lo:hi]).max(), (name, err)


@pytest.mark.parametrize("M,N,K,relu,bf16", [
    (2048, 2048, 1024, False, True),    # the smallest that takes pairs, whole tiles
    (2049, 2303, 1088, True, True),     # ragged on both sides, rows of C at odd addresses
    (16389, 200, 1024, False, False),   # one column of tiles, the last with 5 rows
    (2000, 5003, 512, True, False),     # two rounds of tiles, a short reduction
])
def test_gemm_on_pairs(B_, M, N, K, relu, bf16):
    """Tolerance: that of the small tiles' test (float32 accumulation of K products)."""
    TG.test_gemm_matches_float64((B_, B_.Context(8, 8, 8, 1, 8, 8)), M, N, K, 1, relu, bf16)


@pytest.mark.parametrize("F", [1, 2, 3, 33, 255, 257, 1024, 1025, 2048, 2049, 4097, 8193])
def test_trees_reach_every_triangle(B_, F):
    """Full builds and refits around the powers of two of the sort, one and two leaves
    per thread, the largest merged build (2048), search builds beyond and the multi-block
    one (8193): separate triangles on two layers of a grid, in random order, each hit by a
    ray of its own at t = 9.  A refit keeps the tree for other positions."""
    rng = np.random.default_rng(F)
    n = (F + 1) // 2
    side = int(np.ceil(np.sqrt(n)))
    order = rng.permutation(F)

    def soup(order):
        cell, layer = order // 2, order % 2
        c = np.stack([cell % side, cell // side, layer.astype(np.float64)], 1)
        tri = np.array([[-0.2, -0.2, 0], [0.3, -0.1, 0], [-0.1, 0.3, 0]])
        orig = c + np.where(layer == 1, 9.0, -9.0)[:, None] * [0, 0, 1]
        dirs = np.where(layer == 1, -1.0, 1.0)[:, None] * [0, 0, 1]
        return (c[:, None] + tri).reshape(-1, 3), orig, dirs

    h = hand()
    faces = np.arange(3 * F, dtype=np.int32).reshape(F, 3)
    one = lambda a: np.repeat(a[:1], 3 * F, 0)
    v, _, _ = soup(order)
    model = B_.Model(dataclasses.replace(
        h, v_template=v.astype(np.float32), shapedirs=one(h.shapedirs), weights=one(h.weights), faces=faces,
        edges=faces[:, :2].copy(), edge_faces=np.stack([np.arange(F), np.full(F, -1)], 1).astype(np.int32),
        vf_offsets=np.arange(3 * F + 1, dtype=np.int32), vf_faces=np.repeat(np.arange(F, dtype=np.int32), 3),
        albedo=one(h.albedo), uv=None))
    ctx = B_.Context(3 * F, F, F, 1, 8, 8)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")
    counter = torch.full((1,), 3, dtype=torch.int32, device="cuda")
    for refit in (False, True):
        v, orig, dirs = soup(rng.permutation(F) if refit else order)
        if refit:
            B_.hr_update_bvh(ctx, model, t(v), counter, 8)
        else:
            B_.hr_build_bvh(ctx, model, t(v))
        tri = torch.empty(F, dtype=torch.int32, device="cuda")
        tuv = torch.empty((F, 3), device="cuda")
        B_.hr_trace(ctx, t(orig), t(dirs), tri, tuv)
        assert (tri.cpu().numpy() == np.arange(F)).all()
        assert np.abs(tuv.cpu().numpy()[:, 0] - 9.0).max() <= 1e-5
    assert B_.hr_get_status(ctx) == B_.HR_OK


@pytest.mark.parametrize("W,Wo", [(2, 1), (510, 85), (514, 257), (65536, 32768)])
def test_resampling_by_whole_factors(B_, W, Wo):
    """Segments of a row (one channel column to more than a block), more taps than a
    chunk (factor 6) and the longest rows.  Means of f x f uniform values
    to float32 accumulation (36 products with weights exact to 2^-24): 2e-6."""
    f = W // Wo
    rng = np.random.default_rng(W)
    img = rng.random((2, 2 * f, W, 3), dtype=np.float32)
    m = rng.integers(0, 255, (2, 2 * f, W)).astype(np.uint8)
    out, mout = torch.empty((2, 2, Wo, 3), device="cuda"), torch.empty((2, 2, Wo), dtype=torch.uint8, device="cuda")
    B_.hr_area_resample(torch.as_tensor(img, device="cuda"), out)
    B_.hr_mask_resample(torch.as_tensor(m, device="cuda"), mout)
    ref = img.astype(np.float64).reshape(2, 2, f, Wo, f, 3).mean((2, 4))
    assert np.abs(out.cpu().numpy() - ref).max() <= 2e-6
    assert (mout.cpu().numpy() == m.reshape(2, 2, f, Wo, f).max((2, 4))).all()


@pytest.mark.parametrize("name,samples", [("tiny", 60), ("ragged", 700), ("ragged", 150000)])
def test_edge_samples_do_not_depend_on_their_lanes(B_, name, samples):
    """Fixed-point sums: the same bits for 2 to 32 lanes per sample, and (150000 samples)
    for the one to four lanes that large calls come down to."""
    sc, h = scene(name), hand()
    model, ctx = B_.Model(h), B_.Context(h.V, h.F, h.E, sc.N, sc.W, sc.H)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    vt, cams, bg = t(sc.verts), t(sc.cams), t(sc.bg)
    adj = t(np.random.default_rng(3).normal(size=(sc.N, sc.H, sc.W, 3)).astype(np.float32))
    img, outs = torch.empty((sc.N, sc.H, sc.W, 3), device="cuda"), []
    B_.hr_build_bvh(ctx, model, vt)
    opts = lambda flags: B_.render_opts(seed=7, spp=2, edge_samples=samples, flags=flags)
    B_.hr_render_fwd(ctx, model, vt, cams, sc.H, sc.W, bg, opts(0), img)
    for lanes in (2, 4, 8, 16, 32):
        ctx.set_tuning(edge_lanes=lanes)
        outs.append(torch.empty((h.V, 3), device="cuda"))
        B_.hr_render_bwd(ctx, model, vt, cams, sc.H, sc.W, bg, opts(B_.HR_DETERMINISTIC | B_.HR_BWD_REUSE_FWD), adj, outs[-1])
    assert outs[0].abs().max() > 0 and all(torch.equal(outs[0], o) for o in outs[1:])
    assert B_.hr_get_status(ctx) == B_.HR_OK


@pytest.mark.parametrize("width", [100, 16])
def test_edge_samples_of_a_hand_alone_and_among_others(B_, width):
    """One hand's samples, alone (four lanes each) and in batches whose numbers of samples
    take the rule to two lanes and to one: the hand's fixed-point gradient has the same
    bits, with the silhouettes' lists (100 columns) and with sub-tiles of more candidates
    than a list holds, whose rays go through the tree (16)."""
    sc, h = scene("ragged"), hand()
    f, samples = width / sc.W, 777
    H = int(sc.H * f)
    cams = np.array(sc.cams, np.float32, copy=True)
    cams[:, :4] *= f    # fx, fy, cx, cy
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")
    rng = np.random.default_rng(width)
    bg, adj = rng.random((sc.N * H * width, 3)), rng.normal(size=(sc.N * H * width, 3))
    model, outs = B_.Model(h), []
    for n in (1, 24, 48):   # 2331, 55944 and 111888 samples
        bt = B_.Batch(h.V, h.F, h.E, [(sc.N, width, H, 2, samples, i) for i in range(n)])
        many = lambda a: t(np.concatenate([a] * n))
        verts, img, out = many(sc.verts[None]), torch.empty((bt.total_pixels, 3), device="cuda"), torch.empty((n, h.V, 3), device="cuda")
        o = B_.render_opts(seed=7, flags=B_.HR_DETERMINISTIC | B_.HR_BWD_REUSE_FWD | B_.HR_BWD_NO_INTERIOR)
        cam_t, bg_t, adj_t = many(cams), many(bg), many(adj)
        B_.hr_build_bvh_batch(bt, model, verts)
        B_.hr_render_fwd_batch(bt, model, verts, cam_t, bg_t, o, img)
        B_.hr_render_bwd_batch(bt, model, verts, cam_t, bg_t, o, adj_t, out)
        assert B_.hr_get_status(bt) == B_.HR_OK
        outs.append(out[0].clone())
    assert outs[0].abs().max() > 0 and all(torch.equal(outs[0], o) for o in outs[1:])


@pytest.mark.parametrize("width", [208, 104, 56, 24])
def test_lists_of_every_length(B_, width):
    """Sub-tiles of a hand seen ever smaller: lists of up to 32, 64, 128 and more records
    (sorted in one, two or four registers per lane, or in shared memory) and beyond what a
    list holds.  Pixels against the oracle's, with its tolerance."""
    import oracle
    from tests.gpu_common import pixel_ok
    sc, h = scene("tiny"), hand()
    model = B_.Model(h)
    f = width / sc.W
    cams = np.array(sc.cams, np.float32, copy=True)
    cams[:, :4] *= f    # fx, fy, cx, cy
    H = int(sc.H * f)
    ctx = B_.Context(h.V, h.F, h.E, sc.N, width, H)
    bg = np.random.default_rng(width).random((sc.N, H, width, 3), dtype=np.float32)
    o = sc.opts()
    ref = oracle.render_fwd(sc.verts, h.faces, sc.normals, h.albedo, cams, H, width, bg, o)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    img = torch.empty((sc.N, H, width, 3), device="cuda")
    B_.hr_build_bvh(ctx, model, t(sc.verts))
    B_.hr_render_fwd(ctx, model, t(sc.verts), t(cams), H, width, t(bg), sc.gpu_opts(o), img)
    assert pixel_ok(img.cpu().numpy(), ref).all()
    assert B_.hr_get_status(ctx) == B_.HR_OK


@pytest.mark.parametrize("n", [1, 3, 40])
@pytest.mark.parametrize("V", [31, 128, 129, 778])
def test_skinning_blocks(B_, V, n):
    """Skinning and its adjoint for a model of V vertices at the edges of a block's (128 of
    the forward): against the oracle per hand.  Forward: float32 sums of 26
    terms of size ~0.1, 1e-6.  Adjoint: sums of V terms, 1e-5 of the largest."""
    import oracle
    h = hand()
    faces = h.faces[(h.faces < V).all(1)] if V < h.V else h.faces
    if len(faces) == 0:
        faces = np.array([[0, 1, 2]], np.int32)
    edges, ef, vfo, vff = I.mesh_topology(faces, V)
    h = dataclasses.replace(h, v_template=h.v_template[:V], shapedirs=h.shapedirs[:V], weights=h.weights[:V],
                            faces=np.ascontiguousarray(faces), edges=edges, edge_faces=ef, vf_offsets=vfo, vf_faces=vff,
                            albedo=h.albedo[:V], uv=None)
    model = B_.Model(h)
    rng = np.random.default_rng(V + n)
    x = np.concatenate([rng.normal(0, 1, (n, 10)), rng.normal(0, 0.4, (n, 48)), rng.normal(0, 0.1, (n, 3))], 1)
    x = x.astype(np.float32)
    g = rng.normal(size=(n, V, 3)).astype(np.float32)
    bt = B_.Batch(h.V, h.F, h.E, [(1, 8, 8, 1, 0, i) for i in range(n)])
    verts, dx = torch.empty((n, V, 3), device="cuda"), torch.empty((n, 61), device="cuda")
    B_.hr_skin_batch(bt, model, torch.as_tensor(x, device="cuda"), verts)
    B_.hr_skin_bwd_batch(bt, model, torch.as_tensor(x, device="cuda"), torch.as_tensor(g, device="cuda"), dx)
    for i in range(n):
        ref = oracle.skin(h, x[i].astype(np.float64))
        assert np.abs(verts[i].cpu().numpy() - ref).max() <= 1e-6
        d = oracle.skin_bwd(h, x[i].astype(np.float64), g[i].astype(np.float64))
        assert np.abs(dx[i].cpu().numpy() - d).max() <= 1e-5 * max(np.abs(d).max(), 1.0)
