"""The tracing kernels where their routes change: BVHs of one, several and part
blocks of leaves, scenes far from the origin, tiny and flat ones (the node
boxes' grid), and frames whose long walks are put aside, in part or all of
them, or find no room."""
import numpy as np
import pytest

import oracle
import paper_2405_10565_gb300 as hr
import scenegen
from gpu_util import HIT_AGREE_MIN, KBUF_AGREE_MIN, RMSE_FP32, compare, gpu_samples, oracle_prepare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_10565_gb300.build import build
    build()
    c = hr.hr_create(0)
    yield c
    hr.hr_destroy(c)


def _scene(n, S, seed=1, radius=4e-3, **kw):
    v = scenegen.make_strands(n, S, seed=seed, jitter=0.01, radius=radius, **kw)
    return scenegen.Scene(v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                          np.stack([np.full(n, 0.7), np.linspace(0, 6, n)], -1).astype(np.float32))


def _against_oracle(ctx, sc, res=40, k=3, fill=0.8):
    cam = scenegen.frame_camera(*sc.aabb(), res, res, perspective=True, fill=fill)
    lights = scenegen.point_lights(2, 0.5 * sum(sc.aabb()), seed=2)
    w = scenegen.Workload("paths", sc, cam, lights, 2, k, 0)
    a = hr.hr_asset_create(ctx, sc.verts, sc.mat, sc.shape)
    try:
        hr.hr_build_bvh(ctx, a, None)
        d = hr.render_desc(cam.pack(), lights, 2, k, w.sample_seed)
        sids = np.arange(res * res * 2)
        rg, hg = gpu_samples(ctx, a, d, sids)
        prep = oracle_prepare(w)
        ro, ho = oracle.render_samples(prep, cam.pack(), lights, sids, 2, k, w.sample_seed)
        near, full, rel, _ = compare(rg, hg, ro, ho)
        assert (ho[:, 0] >= 0).any()
        assert near >= HIT_AGREE_MIN and full >= KBUF_AGREE_MIN and rel <= RMSE_FP32
        img = np.zeros((res, res, 3), np.float32)
        hr.hr_render(ctx, a, d, img)
        mean = rg.reshape(-1, 2, 3).astype(np.float64).mean(1).reshape(img.shape)
        assert np.allclose(img, mean, rtol=1e-4, atol=1e-6 * max(1.0, float(mean.max())))
    finally:
        hr.hr_asset_destroy(ctx, a)


@pytest.mark.parametrize("n,S", [(2, 1), (51, 5), (64, 4), (257, 1), (73, 7), (171, 3), (683, 3)])
def test_bvh_of_part_and_several_blocks(ctx, n, S):
    """2, 255, 256, 257, 511, 513 and 2,049 leaves: one block of 256, its edge, more."""
    _against_oracle(ctx, _scene(n, S))


@pytest.mark.parametrize("shift,scale", [((100.0, -30.0, 7.0), 1.0), ((0.0, 0.0, 0.0), 1e-3),
                                         ((0.0, 0.0, 0.0), 1e3)])
def test_node_grid_far_from_the_origin_and_at_other_scales(ctx, shift, scale):
    sc = _scene(300, 6)
    sc.verts[..., :3] = sc.verts[..., :3] * scale + np.asarray(shift, np.float32)
    sc.verts[..., 3] *= scale
    _against_oracle(ctx, sc)


def test_flat_scene(ctx):
    """Every vertex in one plane and every strand along one axis."""
    sc = _scene(64, 8)
    sc.verts[..., 2] = 0.25
    sc.verts[..., 0] = np.linspace(-0.5, 0.5, 64, dtype=np.float32)[:, None]
    sc.verts[..., 1] = np.linspace(0.0, 1.0, 9, dtype=np.float32)[None]
    _against_oracle(ctx, sc)


@pytest.mark.parametrize("res,spp,k,setting", [
    (9, 1, 1, "strands"),    # less than a warp of pixels
    (64, 1, 4, "eth"),
    (48, 3, 2, "half"),
    (40, 32, 3, "eth"),      # a tile is one pixel
    (24, 33, 4, "eth"),      # two samples a lane: nothing is put aside
    (96, 4, 8, "eth"),       # the records of K = 8 outgrow the room of so small a frame
    (200, 8, 8, "half"),
])
def test_long_walks_finish_as_short_ones(ctx, res, spp, k, setting):
    """Small frames give every ray the least budget, so that most walks of a
    dense view are put aside; counting frames put none aside."""
    w = scenegen.clustered(n=4000, S=16, res=res, spp=spp, lod_setting=setting, n_clusters=60)
    a = hr.hr_asset_create(ctx, w.scene.verts, w.scene.mat, w.scene.shape)
    try:
        hr.hr_build_clusters(ctx, a, w.n_clusters)
        C, L, _ = hr.hr_hierarchy_info(ctx, a)
        hr.hr_build_bvh(ctx, a, scenegen.lod_preset(setting, C, L))
        img = [np.zeros((res, res, 3), np.float32) for _ in range(3)]
        for i, flags in enumerate((0, hr.HR_FLAG_COUNT, hr.HR_FLAG_FIXED_TILE_ORDER)):
            d = hr.render_desc(w.camera.pack(), w.lights, spp, k, 5, 0, flags)
            st = hr.hr_render(ctx, a, d, img[i], stats=True)
            assert st.stack_overflows == 0
            if i == 1:
                steps = (st.node_visits + st.prim_tests) / max(1, st.traced_samples)
                assert res < 20 or steps > 40  # the least budget
        assert img[1].max() > 0
        # the same hits; an FP32 depth that one order of tests made precise and
        # the other did not is within 2^-16 of it
        assert np.allclose(img[0], img[1], rtol=1e-4, atol=1e-6), np.abs(img[0] - img[1]).max()
        assert np.allclose(img[2], img[0], rtol=1e-4, atol=1e-6)
    finally:
        hr.hr_asset_destroy(ctx, a)


@pytest.mark.parametrize("res,spp,k", [(3, 1, 4), (16, 1, 1), (24, 2, 2), (33, 5, 8), (64, 8, 4), (20, 32, 3)])
def test_parts_of_tiles_equal_whole_tiles(res, spp, k):
    """Small frames hand out parts of a tile, with rays put aside from them;
    counting renders trace whole tiles."""
    from paper_2405_10565_gb300.build import build
    build()
    w = scenegen.clustered(n=1500, S=8, res=res, spp=spp, n_clusters=40)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, w.scene.verts, w.scene.mat, w.scene.shape)
        hr.hr_build_clusters(ctx, a, w.n_clusters)
        C, n_levels, _ = hr.hr_hierarchy_info(ctx, a)
        hr.hr_build_bvh(ctx, a, scenegen.lod_preset("half", C, n_levels))
        img = [np.zeros((res, res, 3), np.float32) for _ in range(4)]
        for i, flags in enumerate((hr.HR_FLAG_COUNT, hr.HR_FLAG_FIXED_TILE_ORDER, 0, 0)):
            d = hr.render_desc(w.camera.pack(), w.lights, spp, k, 7, 0, flags)
            hr.hr_render(ctx, a, d, img[i], stats=True)
        assert img[0].max() > 0
        # the same operations in the same order; the compiler may contract them differently
        assert np.allclose(img[1], img[0], rtol=1e-5, atol=1e-7), np.abs(img[1] - img[0]).max()
        assert np.array_equal(img[1], img[2]) and np.array_equal(img[1], img[3])
    finally:
        hr.hr_destroy(ctx)
