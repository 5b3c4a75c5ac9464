"""The tile searches and the medoid bound of the guide-driven hierarchy where
they can go wrong, bit for bit against the oracle: part tiles, row counts that
are no multiple of a group, strands too long for a tile, large clusters, and
strands that coincide (every decision a tie)."""
import numpy as np
import pytest

import oracle
import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_10565_gb300.build import build
    build()
    c = hr.hr_create(0)
    yield c
    hr.hr_destroy(c)


@pytest.mark.parametrize("n,S,G,iters,copies", [
    (33, 300, 3, 2, 1),     # longer than a tile holds, one strand in the last tile
    (97, 255, 13, 1, 1),    # the longest strands a tile holds
    (641, 7, 17, 0, 1),     # one row in the last group, no update round
    (2500, 5, 4, 4, 1),     # about 600 members a cluster: several rounds of the FP32 sums
    (300, 6, 9, 3, 2),      # every strand twice
    (64, 4, 8, 2, 64),      # one strand 64 times: all distances zero
])
def test_guides_and_clusters_bit_exact(ctx, n, S, G, iters, copies):
    v = scenegen.make_strands(max(n // copies, 1), S, seed=n, curl_amp=0.02, hang=0.08)
    v = np.ascontiguousarray(np.tile(v, (copies, 1, 1)))
    n = v.shape[0]
    a = hr.hr_asset_create(ctx, v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                           np.zeros((n, 2), np.float32))
    try:
        cl, order, guides = np.zeros(n, np.uint32), np.zeros(n, np.uint32), np.zeros(G, np.int32)
        try:
            want, want_guides, _ = oracle.build_guided_hierarchy(v, G, iters)
        except IndexError:  # fewer than three non-empty clusters
            with pytest.raises(hr.HairRTError):
                hr.hr_build_guided_clusters(ctx, a, G, iters)
            return
        for _ in range(2):  # again into the arrays of the first build
            hr.hr_build_guided_clusters(ctx, a, G, iters, 0, cl, order)
            hr.hr_guides_export(ctx, a, guides)
            assert np.array_equal(guides.astype(np.int64), want_guides)
            assert np.array_equal(order.astype(np.int64), want.order)
            assert np.array_equal(cl, want.cluster_of)
    finally:
        hr.hr_asset_destroy(ctx, a)


@pytest.mark.parametrize("n,S", [(300, 9), (24, 2100)])  # in one pass; strands too long for it
def test_skinning_to_the_rest_pose_keeps_the_image(ctx, n, S):
    v = scenegen.make_strands(n, S, seed=3, jitter=0.002, hang=0.08, radius=4e-3)
    sc = scenegen.Scene(v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                        np.zeros((n, 2), np.float32))
    cam = scenegen.frame_camera(*sc.aabb(), 48, 48, perspective=True, fill=0.7).pack()
    lights = scenegen.point_lights(2, np.zeros(3), seed=1)
    a = hr.hr_asset_create(ctx, v, sc.mat, sc.shape)
    try:
        hr.hr_build_guided_clusters(ctx, a, 5, 2)
        guides = np.zeros(5, np.int32)
        hr.hr_guides_export(ctx, a, guides)
        d = hr.render_desc(cam, lights, 4, 3, 1, 0, hr.HR_FLAG_KEEP_HIERARCHY)
        img = [np.zeros((48, 48, 3), np.float32) for _ in range(2)]
        hr.hr_render_frame(ctx, a, 0, 0.5, 0, d, img[0])
        hr.hr_asset_skin(ctx, a, np.ascontiguousarray(v[np.maximum(guides, 0)]))
        back = np.zeros_like(v)
        hr.hr_vertex_export(ctx, a, back)
        assert np.allclose(back, v, atol=2e-6)
        hr.hr_render_frame(ctx, a, 0, 0.5, 0, d, img[1])
        # vertices moved by a few 1e-7 change few pixels at the fibres' edges
        assert img[0].max() > 0
        assert np.linalg.norm(img[1] - img[0]) <= 0.1 * np.linalg.norm(img[0])
    finally:
        hr.hr_asset_destroy(ctx, a)
