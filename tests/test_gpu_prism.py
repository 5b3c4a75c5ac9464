"""The skinning weights of the strands' vertices against the same formula in
80-bit floats, for few large clusters (shared out to many blocks) and many small
ones.  A pose with a cluster's guides at (0, 0, 0), (1, 0, 0) and (0, 1, 0) moves
a vertex to its weights themselves: every product and sum of the skinning is
exact there."""
import numpy as np
import pytest

import paper_2405_10565_gb300 as hr
import scenegen

pytestmark = pytest.mark.gpu


def exact_weights(p, g0, g1, g2):
    """(w1, w2, h) in 80-bit floats, the sine of the triangle's angle, and where it
    is degenerate (the weights are the offset p - g0)."""
    p, g0, g1, g2 = (np.asarray(x, np.longdouble) for x in (p, g0, g1, g2))
    e1, e2, q = g1 - g0, g2 - g0, p - g0
    n = np.cross(e1, e2)
    nn = np.sqrt((n * n).sum(-1))
    scale = np.sqrt((e1 * e1).sum(-1) * (e2 * e2).sum(-1))
    flat = ~(nn > 1e-6 * scale)
    with np.errstate(invalid="ignore", divide="ignore"):
        nh = n / nn[..., None]
        w = np.stack([(q * np.cross(e2, nh)).sum(-1) / nn, (q * np.cross(nh, e1)).sum(-1) / nn,
                      (q * nh).sum(-1)], -1)
        sine = nn / scale
    return np.where(flat[..., None], q, w), sine, flat


def read_weights(ctx, a, n, S, order, cluster_of, tri, guides, clusters):
    """{cluster: (strand ids, weights [m, S + 1, 3])} by one pose a cluster."""
    out = {}
    for c in clusters:
        ids = order[cluster_of[order] == c]
        pose = np.zeros((len(guides), S + 1, 4), np.float32)
        pose[tri[c, 1], :, 0] = 1.0
        pose[tri[c, 2], :, 1] = 1.0
        hr.hr_asset_skin(ctx, a, pose)
        v = np.zeros((n, S + 1, 4), np.float32)
        hr.hr_vertex_export(ctx, a, v)
        out[c] = ids, v[ids, :, :3]
    return out


@pytest.mark.parametrize("n,S,G", [(3000, 8, 3), (700, 300, 3), (2000, 40, 5), (3000, 8, 24), (40, 600, 4)])
def test_strand_weights(n, S, G):
    from paper_2405_10565_gb300.build import build
    build()
    v = scenegen.make_strands(n, S, seed=n, jitter=0.002, hang=0.08)
    ctx = hr.hr_create(0)
    try:
        a = hr.hr_asset_create(ctx, v, scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2)),
                               np.zeros((n, 2), np.float32))
        cluster_of, order = np.zeros(n, np.uint32), np.zeros(n, np.uint32)
        hr.hr_build_guided_clusters(ctx, a, G, 2, 0, cluster_of, order)
        C = hr.hr_hierarchy_info(ctx, a)[0]
        guides, tri = np.zeros(G, np.int32), np.zeros((C, 3), np.uint32)
        hr.hr_guides_export(ctx, a, guides, tri)
        seen = 0
        for c, (ids, w) in read_weights(ctx, a, n, S, order, cluster_of, tri, guides, range(C)).items():
            P = v[..., :3]
            g = [P[guides[t]][None] for t in tri[c]]
            want, sine, flat = exact_weights(P[ids], *g)
            ok = np.broadcast_to(~flat & (sine > 1e-3), w.shape[:2])  # FP64 loses 2^-53 / sine^2 itself
            err = np.abs(w[ok] - want[ok]).astype(np.float64)
            # rounded once to FP32; beside it the FP64 prism's loss where terms cancel
            big = np.abs(want[ok]).astype(np.float64)
            slack = 2.0 ** -53 * 32 / np.broadcast_to(sine, w.shape[:2])[ok][:, None] ** 2
            size = 1.0 + big.max(-1, keepdims=True)
            assert (err <= 0.5001 * np.spacing(big.astype(np.float32)) + slack * size).all()
            seen += int(ok.sum())
        assert seen > n * S // 4
    finally:
        hr.hr_destroy(ctx)
