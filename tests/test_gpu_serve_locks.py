"""Requests that make the server reclaim memory while another thread updates an
asset: the API's and the server's lock are taken in one order.  In a process of its
own, so that two threads that wait for one another end with it."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r'''
import threading
import numpy as np
import paper_2405_10565_gb300 as hr
import scenegen

n, S, W, H = 1500, 16, 64, 48
verts = [scenegen.make_strands(n, S, seed=s, radius=4e-3) for s in (1, 2, 3)]
mat = scenegen.material_from_melanin(np.full(n, 0.5), np.full(n, 0.2))
lights = scenegen.point_lights(1, np.zeros(3), seed=1)

def set_up(budget):
    ctx = hr.hr_create(0, budget)
    a = [hr.hr_asset_create(ctx, v, mat, np.zeros((n, 2), np.float32)) for v in verts]
    hr.hr_build_bvh(ctx, a[2], None)
    return ctx, a

probe, _ = set_up(0)
used = hr.hr_bytes_in_use(probe)
hr.hr_destroy(probe)
# room for one resident BVH: every request for the other asset reclaims it first
ctx, a = set_up(used + n * S * 132 + (1 << 20))
cams = [scenegen.frame_camera(v[..., :3].min((0, 1)), v[..., :3].max((0, 1)), W, H, perspective=True, fill=0.8).pack()
        for v in verts]
hr.hr_serve_start(ctx, 1, 1 << 20)
stop, updates = threading.Event(), [0]

def updater():
    while not stop.is_set():
        hr.hr_asset_update(ctx, a[2], verts[2])
        updates[0] += 1

t = threading.Thread(target=updater, daemon=True)
t.start()
first = {}
for i in range(120):
    k = i % 2
    out = np.zeros((H, W, 3), np.float32)
    st, res = hr.hr_poll(ctx, hr.hr_submit(ctx, a[k], hr.render_desc(cams[k], lights, 2, 2, 1), out, 2.0, 0), 20000)
    assert st == hr.HR_OK and res.status == hr.HR_OK, (i, st, res.status)
    assert np.array_equal(out, first.setdefault(k, out)) and out.max() > 0
stop.set()
t.join()
hr.hr_serve_stop(ctx)
hr.hr_destroy(ctx)
print("served", updates[0] > 0)
'''


def test_reclaim_beside_updates():
    from paper_2405_10565_gb300.build import build
    build()
    r = subprocess.run([sys.executable, "-c", PROGRAM], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "served True" in r.stdout, (r.stdout[-500:], r.stderr[-1500:])
