"""The parameters' lists of columns when they are shorter than the columns (slots that are constants,
columns that are always 0): the checking build tests every entry it loads against the lists' length, in
both precisions, and the results match the oracle."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import json, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import musr_inputs as mi
import oracle
from paper_1509_07685_gb300 import binding as B
B.LIB_PATH = sys.argv[2]
B.load()
out = {}
for nhist in (1, 7):  # one chunk: the lists go through shared memory
    rng = np.random.default_rng(nhist)
    counts = rng.poisson(30.0, size=(nhist, 900)).astype(np.float32)
    terms = [[("AMP", (2,)), ("EXP", (3,)), ("TFCOS", (4, 5))]]
    # fitted: N0 of each histogram and the shared rate; the rest constants
    rows = np.array([[j, -1, -2, nhist, -3, -4] for j in range(nhist)], np.int32)
    truth = np.array([30.0 + j for j in range(nhist)] + [0.4])
    p = mi.Problem(counts, np.zeros(nhist), 8.0, (0.0, 7.2), terms, rows, np.array([1.5, 0.06, 3.0, 17.0]), nhist + 1,
                   truth, [f"p{i}" for i in range(nhist + 1)])
    ref = oracle.cost(p, truth, 1)
    with B.Context(p) as ctx:
        for prec in (B.MUSR_SPLIT, B.MUSR_FP64):
            v, g, st = ctx.eval(truth, 1, prec)
            dst, word = B.musr_debug_word(ctx.ctx)
            out[f"{nhist} {prec}"] = [int(st), int(dst), int(word), abs(v - ref[0]) / abs(ref[0]),
                                      float(np.max(np.abs(g - ref[1]) / (ref[2] + 1e-300))), int(prec)]
print(json.dumps(out))
"""


def test_lists_shorter_than_the_columns(musr_lib):
    from paper_1509_07685_gb300 import build
    lib = build.build(debug=True)
    r = subprocess.run([sys.executable, "-c", SCRIPT, ROOT, lib], capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
    for name, (st, dst, word, err, gerr, prec) in json.loads(r.stdout.strip().splitlines()[-1]).items():
        tol = 1e-9 if prec == 0 else 2.0 ** -16  # as test_gpu_debug_checks.py
        assert (st, dst, word) == (0, 0, 0) and err <= tol and gerr <= tol, (name, word, err, gerr)
