"""Every slab height that the autotuner of the FP64 apply may choose and report
(bdu_stats.apply_variant) can be asked for (bdu_options.nb), odd ones among
them, and gives the oracle's results bit for bit."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle as O
from paper_2509_02840_gb300 import bdu, inputs as I

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("nb", [2, 4, 5, 7, 9, 11, 13, 63])
@pytest.mark.parametrize("m,n", [(5, 4), (66, 34), (131, 128), (260, 259)])
def test_heights(m, n, nb):
    Q, d, e, P = I.factorization(m, n, config=0, which=m + nb)
    B, C = I.dense_update(m, n, h=2, config=0)
    with bdu.Factorization(Q, d, e, P, precision=bdu.FP64, nb=nb) as F:
        F.update(B, C)
        got = F.read()
    for name, a, b in zip("QdeP", got, O.update(Q, d, e, P, B, C)):
        assert np.array_equal(a, b), name


@pytest.mark.parametrize("n", [150, 449, 600, 1030])
def test_tuned_height_can_be_asked_for(n):
    Q = np.eye(n)
    g = np.random.default_rng(n)
    d, e = g.uniform(1, 10, n), g.standard_normal(n - 1)
    b, c = g.standard_normal(n), g.standard_normal(n)
    with bdu.Factorization(Q, d, e, Q, precision=bdu.FP64) as F:
        F.update(b, c)
        tuned, got = F.stats()["apply_variant"], F.read()
    for nb in set(tuned):
        with bdu.Factorization(Q, d, e, Q, precision=bdu.FP64, nb=nb) as F:
            F.update(b, c)
            for name, x, y in zip("QdeP", got, F.read()):
                assert np.array_equal(x, y), name


def test_heights_timed_with_another_kernel_are_not_taken(tmp_path):
    """A BDU_TUNE_FILE of the time before FP64 keys named the kernel: its heights
    stay in the file and are not used."""
    path = tmp_path / "tune.json"
    old = {"%s|fp64|%d|0" % (torch.cuda.get_device_name(0), n): 64 for n in (157, 99)}
    path.write_text(json.dumps(old))
    code = ("import sys; sys.path.insert(0, %r)\n"
            "from paper_2509_02840_gb300 import bdu, inputs as I\n"
            "Q, d, e, P = I.factorization(157, 99, config=0, which=9)\n"
            "with bdu.Factorization(Q, d, e, P) as F:\n"
            "    F.update(*I.dense_update(157, 99, 0, config=0))\n"
            "    print(F.stats()['tunings'])\n" % ROOT)
    run = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, BDU_TUNE_FILE=str(path)),
                         capture_output=True, text=True, check=True)
    assert int(run.stdout) == 2
    table = json.loads(path.read_text())
    assert all(table[k] == v for k, v in old.items()) and len(table) == 4
