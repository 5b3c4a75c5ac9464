"""Scenes with vertices that are not numbers: the segments that touch one are
never hit, and every other segment is, as the oracle has it without them."""
import numpy as np
import pytest

import oracle
import paper_2405_10565_gb300 as hr
import scenegen
from gpu_util import HIT_AGREE_MIN, KBUF_AGREE_MIN, RMSE_FP32, compare, gpu_samples

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2405_10565_gb300.build import build
    build()
    c = hr.hr_create(0)
    yield c
    hr.hr_destroy(c)


def _scene(n, S, seed=1):
    v = scenegen.make_strands(n, S, seed=seed, jitter=0.01, radius=4e-3)
    return scenegen.Scene(v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                          np.stack([np.full(n, 0.7), np.linspace(0, 6, n)], -1).astype(np.float32))


def _check(ctx, sc, odd, bad, update, fill=0.8, res=40, k=3, spp=2):
    """Render `sc` with its vertices replaced by `odd`; `bad` marks the
    vertices whose segments the oracle leaves out."""
    n, S = sc.n_strands, sc.n_segments
    cam = scenegen.frame_camera(*sc.aabb(), res, res, perspective=True, fill=fill)
    lights = scenegen.point_lights(2, 0.5 * sum(sc.aabb()), seed=2)
    clean = np.where(bad[..., None], sc.verts, odd)
    rows, ids = oracle.strand_prim_rows(clean, sc.shape, np.arange(n))
    keep = ~(bad[:, :-1] | bad[:, 1:]).reshape(-1)
    prep = oracle.Prepared(np.ascontiguousarray(rows[keep]), np.ascontiguousarray(ids[keep].astype(np.int64)),
                           sc.mat.astype(np.float64), None, None, None)
    a = hr.hr_asset_create(ctx, sc.verts if update else odd, sc.mat, sc.shape)
    try:
        if update:
            hr.hr_asset_update(ctx, a, odd)
        hr.hr_build_bvh(ctx, a, None)
        d = hr.render_desc(cam.pack(), lights, spp, k, 5)
        sids = np.arange(res * res * spp)
        rg, hg = gpu_samples(ctx, a, d, sids)
        ro, ho = oracle.render_samples(prep, cam.pack(), lights, sids, spp, k, 5)
        near, full, rel, _ = compare(rg, hg, ro, ho)
        assert (ho[:, 0] >= 0).any()
        assert near >= HIT_AGREE_MIN and full >= KBUF_AGREE_MIN and rel <= RMSE_FP32, (near, full, rel)
        img = np.zeros((res, res, 3), np.float32)
        hr.hr_render(ctx, a, d, img)
        mean = rg.reshape(-1, spp, 3).astype(np.float64).mean(1).reshape(img.shape)
        assert np.allclose(img, mean, rtol=1e-4, atol=1e-6 * max(1.0, float(mean.max())))
    finally:
        hr.hr_asset_destroy(ctx, a)


@pytest.mark.parametrize("update", [False, True])
@pytest.mark.parametrize("n,S", [(40, 8), (300, 8)])  # a BVH of one block; of several
@pytest.mark.parametrize("vertex,axes", [(0, (0, 1, 2)), (0, (1,)), (4, (0, 1, 2)), (8, (2,))])
def test_a_vertex_that_is_not_a_number(ctx, n, S, vertex, axes, update):
    sc = _scene(n, S)
    odd, bad = np.array(sc.verts), np.zeros((n, S + 1), bool)
    for s in (n // 3, n - 1):
        odd[s, vertex, list(axes)] = np.nan
        bad[s, vertex] = True
    _check(ctx, sc, odd, bad, update)
