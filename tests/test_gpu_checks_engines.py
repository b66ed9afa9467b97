"""The bounds-checked build over both engines and the distance transform: every
case says which engine must have run (the wavefront engine scans rows, the merging
engine does not), gives the oracle's bytes and records no failed check. One
wavefront setting (RECON_P_REVISIT_SCANS) keeps a context on the wavefront engine
while its block height takes every value, the default among them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import sys
sys.path[:0] = [%(root)r, %(root)r + "/tests"]
import numpy as np, torch
import paper_1311_0378_gb300 as rc
rc.LIB_PATH = %(lib)r
import oracle, synth
from test_gpu_forest import KINDS, image, markers

def dev(a):
    t = torch.from_numpy(np.ascontiguousarray(a)).cuda(); torch.cuda.synchronize(); return t

def clean(what):
    assert rc.recon_checks()[:2] == (1, 0), (what, rc.recon_checks())

rc.recon_checks(reset=True)
c = rc.recon_init(0, 0, rc.RECON_FLAG_SYNC)
def both(I, J, conn, op, wavefront):
    want = (oracle.recon if op == rc.RECON_OP_DILATE else oracle.recon_erode)(I, J, conn) if op != rc.RECON_OP_FILL_HOLES \
        else oracle.fill_holes(I, conn)
    dI, dJ = dev(I), dev(J)
    rc.check(rc.recon_run_op(c, dI.data_ptr(), dJ.data_ptr(), I.shape[0], I.shape[1], conn, op), "run")
    assert (dJ.cpu().numpy() == want).all()
    assert (rc.recon_get_work(c, 1)[0]["scan_rows"] > 0) == wavefront

def operations(I, J, conn, wavefront):
    both(I, J, conn, rc.RECON_OP_DILATE, wavefront)
    both(255 - I, 255 - J, conn, rc.RECON_OP_ERODE, wavefront)
    both(I, np.zeros_like(I), conn, rc.RECON_OP_FILL_HOLES, wavefront)

base = synth.workload("single512").tiles[0]
rc.check(rc.recon_set_param(c, rc.RECON_P_REVISIT_SCANS, 1))
for marker in (synth.HDOME, synth.FILLHOLES):
    I, J = synth.tile_pair(synth.with_marker(base, marker), 1)
    for bh in (32, 64, 256, 128):
        rc.check(rc.recon_set_param(c, rc.RECON_P_BLOCK_H, bh))
        for conn in (4, 8):
            operations(I, J, conn, True)
    clean("wavefront")
rc.check(rc.recon_set_param(c, rc.RECON_P_REVISIT_SCANS, 0))
for marker in (synth.HDOME, synth.FILLHOLES):
    I, J = synth.tile_pair(synth.with_marker(base, marker), 1)
    for conn in (4, 8):
        operations(I, J, conn, False)
clean("merging 512")
rng = np.random.default_rng(1)
for kind in KINDS:                       # "board" overflows the pass lists
    for H, W in ((1, 1), (63, 65), (64, 64), (130, 257)):
        I = image(kind, H, W, rng)
        for J in markers(I, rng):
            for conn in (4, 8):
                operations(I, J, conn, False)
    clean("merging " + kind)
w = synth.workload("uneven1000")
specs = [s for s in w.tiles[:40] if s.H * s.W <= 1 << 20][:12]
pairs = [synth.tile_pair(s, w.seed) for s in specs]
keep = [(dev(I), dev(J)) for I, J in pairs]
rc.check(rc.recon_batch(c, [(a.data_ptr(), b.data_ptr(), s.H, s.W, s.W, s.conn) for (a, b), s in zip(keep, specs)]))
for (a, b), (I, J), s in zip(keep, pairs, specs):
    assert (b.cpu().numpy() == oracle.recon(I, J, s.conn)).all()
assert all(w["scan_rows"] == 0 for w in rc.recon_get_work(c, len(specs)))
clean("merging batch")
for H, W in ((1, 1), (1, 700), (700, 1), (31, 33), (64, 64), (300, 517), (33, 9001), (9000, 5)):
    for density in (0.5, 0.99, 0.9999, 1.0):
        B = (rng.random((H, W)) < density).astype(np.uint8)
        dB = dev(B)
        d2 = torch.empty((H, W), dtype=torch.int32, device="cuda"); site = torch.empty_like(d2)
        for s in (0, site.data_ptr()):
            rc.check(rc.recon_dt(c, dB.data_ptr(), d2.data_ptr(), s, H, W))
        ys, xs = np.nonzero(B == 0)
        si = site.cpu().numpy()
        if not len(ys):
            assert (si == -1).all() and (d2.cpu().numpy() == -1).all()
            continue
        y, x = np.mgrid[0:H, 0:W]
        assert (B.reshape(-1)[si] == 0).all()
        assert ((y - si // W) ** 2 + (x - si %% W) ** 2 == d2.cpu().numpy()).all()
    clean("distance transform %%d x %%d" %% (H, W))
rc.recon_free(c)
print("done")
'''


def test_no_failed_check_on_either_engine():
    import paper_1311_0378_gb300.build as b
    lib = b.build(checks=True)
    out = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT, "lib": lib}], capture_output=True, text=True,
                         timeout=900)
    assert out.returncode == 0 and out.stdout.splitlines()[-1] == "done", out.stderr[-2000:]
