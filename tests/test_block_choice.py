"""Which form the planner takes for contractions whose times differ clearly
(planner on the host; times in us on one GB300, forward and both gradients,
on the blocks / in matrix form)."""
import json
import os
import subprocess
import sys

from tests.conftest import ROOT

SCRIPT = r'''
import json
import paper_1203_2222_gb300 as P
from paper_1203_2222_gb300 import synthetic

def on_blocks(g, la, lb, pa, pb, prec):
    p = P.contract_plan(P.Structure(g, la), P.Structure(g, lb), pa, pb, prec)
    return sum(p.block_info()["tiles"].values()) > 0

def product(d, prec):
    legs = [([0, 2, 4], [d] * 3, 1), ([0, 2, 4], [d] * 3, -1)]
    return on_blocks(P.SU2, legs, legs, [1], [0], prec)

def recouple(d, j, prec=P.FP64):
    r = synthetic.su2_recouple(dmax=d, jmax2=j)
    return on_blocks(P.SU2, r["A"], r["B"], r["pairsA"], r["pairsB"], prec)

print(json.dumps({"f64": {d: product(d, P.FP64) for d in (128, 512, 1024)},
                  "f32": {d: product(d, P.BF16X3) for d in (128, 512, 1024)},
                  "recouple": {f"{d} {j}": recouple(d, j) for d, j in ((2, 4), (3, 3), (2, 7), (4, 6), (6, 6))},
                  "recouple32": {f"{d} {j}": recouple(d, j, P.BF16X3) for d, j in ((4, 5), (5, 5), (7, 4))}}))
'''


def test_form_of_clear_cases():
    env = dict(os.environ, SYM_PLAN_DRYRUN="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, capture_output=True, text=True, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    d = json.loads(r.stdout)
    # three sectors of d x d x d: FP64 193 / 318, 3000 / 2266, 19390 / 16460; FP32 (forward alone)
    # 27 / 31, 65 / 32 and the tensor cores far ahead
    assert d["f64"] == {"128": True, "512": False, "1024": False}
    assert d["f32"] == {"128": True, "512": False, "1024": False}
    # SU(2) recoupling: 190 / 235, 173 / 225; 412, 600 and 1000 in matrix form
    assert d["recouple"] == {"2 4": True, "3 3": True, "2 7": False, "4 6": False, "6 6": False}
    # FP32: 162 / 222, 150 / 209, 167 / 230
    assert d["recouple32"] == {"4 5": True, "5 5": True, "7 4": True}



CUT = r'''
import json
import paper_1203_2222_gb300 as P
from paper_1203_2222_gb300 import synthetic

# (L A) W by R of the fermion-parity step: four blocks of 80 x 80 by a reduction of 400, three of
# them with signs
r = synthetic.z2f_mps_heff(D=160)
S = {n: P.Structure(P.Z2F, r[n]) for n in "LAWR"}
T = P.contract_plan(S["L"], S["A"], [2], [0], P.FP64).out
T = P.contract_plan(T, S["W"], *map(list, r["steps"][0]), P.FP64).out
print(json.dumps(P.contract_plan(T, S["R"], *map(list, r["steps"][1]), P.FP64).block_info()))
'''


def test_tiles_of_one_size_are_cut_alike():
    env = dict(os.environ, SYM_PLAN_DRYRUN="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CUT], env=env, capture_output=True, text=True, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    assert json.loads(r.stdout)["cut"] in (0, 100)
