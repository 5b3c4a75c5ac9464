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
