"""The one-block builds at the edges of their ranges: clusters of up to 8,192
strands (1, 4 and 8 strands a thread) and BVHs of up to 1,024 leaves, against
the oracle, and a refit of a BVH built in one block."""
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


def _materials(n):
    return (scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
            np.stack([np.full(n, 0.7), np.linspace(0, 6, n)], -1).astype(np.float32))


@pytest.mark.parametrize("n,C,same", [(1, 1, 0), (31, 31, 0), (1024, 33, 0), (1025, 1, 0), (4096, 100, 7),
                                      (4097, 1000, 0), (8192, 255, 0), (8193, 255, 0), (7001, 17, 7001)])
def test_clusters_bit_exact(ctx, n, C, same):
    """Order, cluster ids and starts; `same` strands share one root (equal codes
    keep the order of their ids)."""
    v = scenegen.make_strands(n, 2, seed=n)
    v[:same, 0, :3] = v[0, 0, :3]
    a = hr.hr_asset_create(ctx, v, *_materials(n))
    try:
        h = oracle.build_hierarchy(v[:, 0, :3], C)
        for _ in range(2):  # the order kept and found unchanged
            cl, order = np.zeros(n, np.uint32), np.zeros(n, np.uint32)
            hr.hr_build_clusters(ctx, a, C, 0, cl, order)
            assert np.array_equal(order.astype(np.int64), h.order)
            assert np.array_equal(cl, h.cluster_of)
    finally:
        hr.hr_asset_destroy(ctx, a)


@pytest.mark.parametrize("n,S,same", [(1, 2, 0), (11, 3, 0), (64, 16, 0), (1023, 1, 0), (205, 5, 0),
                                      (300, 2, 300)])
def test_bvh_against_the_oracle(ctx, n, S, same):
    """2, 33, 1,024, 1,023, 1,025 and 600 leaves; `same` strands coincide."""
    v = scenegen.make_strands(n, S, seed=n + S, jitter=0.01, radius=4e-3)
    v[:same] = v[0]
    sc = scenegen.Scene(v, *_materials(n))
    res = 40
    cam = scenegen.frame_camera(*sc.aabb(), res, res, perspective=True, fill=0.8)
    lights = scenegen.point_lights(2, 0.5 * sum(sc.aabb()), seed=2)
    a = hr.hr_asset_create(ctx, v, sc.mat, sc.shape)
    try:
        sids = np.arange(res * res)
        for step in range(2):  # built, then refit to moved strands
            d = hr.render_desc(cam.pack(), lights, 1, 3, 1, 0, hr.HR_FLAG_REFIT if step else 0)
            img = np.zeros((res, res, 3), np.float32)
            st = hr.hr_render_frame(ctx, a, 0, 2.0, 0, d, img, stats=True)
            assert st.bvh_refit == step
            rg, hg = gpu_samples(ctx, a, d, sids)
            w = scenegen.Workload("small", sc, cam, lights, 1, 3, 0)
            ro, ho = oracle.render_samples(oracle_prepare(w), cam.pack(), lights, sids, 1, 3, 1)
            if same:  # any of the coinciding strands may be named first
                hg, ho = np.where(hg >= 0, hg % S, -1), np.where(ho >= 0, ho % S, -1)
            near, full, rel, _ = compare(rg, hg, ro, ho)
            assert near >= HIT_AGREE_MIN and full >= KBUF_AGREE_MIN and rel <= RMSE_FP32
            assert np.allclose(img.reshape(-1, 3), rg, rtol=1e-4, atol=1e-6)
            v = np.array(v)
            v[:, 1:, 0] += 0.02
            sc = scenegen.Scene(v, sc.mat, sc.shape)
            hr.hr_asset_update(ctx, a, v)
    finally:
        hr.hr_asset_destroy(ctx, a)
