"""Medoids of clusters whose sums of distances overflow in FP32 (each distance is
finite): where every sum is infinite it is a tie that the lowest strand id wins,
bit for bit as the oracle has it.  All clusters of three, one of five, and none."""
import numpy as np
import pytest

import oracle.guides as og
import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,G,scale", [(900, 3, 1.5e18), (900, 5, 1.5e18), (900, 3, 1e16)])
def test_medoids_of_infinite_sums(n, G, scale):
    from paper_2405_10565_gb300.build import build
    build()
    v = scenegen.make_strands(n, 4, seed=3, jitter=0.05)
    v[..., :3] *= np.float32(scale)
    with np.errstate(over="ignore"):
        of, _, want = og.guide_kmeans(v, G, 2)
        lowest = [int(np.nonzero(of == g)[0][0]) for g in range(G)]
    assert any(w == low for w, low in zip(want.tolist(), lowest)) == (scale > 1e17)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                               np.zeros((n, 2), np.float32))
        hr.hr_build_guided_clusters(ctx, a, G, 2)
        guides = np.zeros(G, np.int32)
        hr.hr_guides_export(ctx, a, guides)
        assert np.array_equal(guides.astype(np.int64), want)
    finally:
        hr.hr_destroy(ctx)
