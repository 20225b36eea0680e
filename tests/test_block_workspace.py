"""The workspace of contractions on the blocks whose reductions are cut into
parts: as large as the parts, and bounded for a whole batch (planner on the host)."""
import json
import os
import subprocess
import sys

from tests.conftest import ROOT

SCRIPT = r'''
import json
import paper_1203_2222_gb300 as P

def legs(q, m, k, n):
    return [(q, m, 1), (q, k, -1)], [(q, k, 1), (q, n, -1)]

def single(prec, *l):
    la, lb = legs(*l)
    return P.contract_plan(P.Structure(P.U1, la), P.Structure(P.U1, lb), [1], [0], prec).block_info()

def batch(prec, nb, *l):
    la, lb = legs(*l)
    A, B = P.Structure(P.U1, la), P.Structure(P.U1, lb)
    return P.contract_batch_plan([A] * nb, [B] * nb, [1], [0], prec).block_info()

dot = ([0, 1], [8, 2], [200000, 9], [8, 3])
wide = ([0], [200], [5000], [200])
print(json.dumps({"dot": [single(p, *dot) for p in (P.FP64, P.BF16X3)],
                  "wide": [single(p, *wide) for p in (P.FP64, P.BF16X3)],
                  "batch": [batch(p, n, *dot) for p in (P.FP64, P.BF16X3) for n in (4, 32, 200)]}))
'''


def test_workspace_of_cut_tiles():
    env = dict(os.environ, SYM_PLAN_DRYRUN="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, capture_output=True, text=True, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    d = json.loads(r.stdout)
    for info, size in zip(d["dot"], (8, 4)):
        # a part of a dot product adds up 128 values, not a slot of the largest tile
        assert info["cut"] == 1 and 0 < info["workspace"] <= info["tiles"]["dot"] * 128 * size
    for info in d["wide"] + d["batch"]:
        assert info["workspace"] <= 64 << 20
