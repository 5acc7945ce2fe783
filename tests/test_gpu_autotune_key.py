"""Which boxes share an autotuned choice: the largest boxes that have the one-launch form, and the
somewhat larger ones that lack it, are tuned apart, in whichever order; choices written for another set of
kernels are not taken. In processes of their own: choices are kept per process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import sys, numpy as np
sys.path.insert(0, %r)
import paper_2602_16486_gb300 as fl
for lattice, dims in %r:
    lam = np.ones(9 if lattice == 0 else 27)
    lam[[4, 5] if lattice == 0 else [7, 8, 9]] = 1.6
    with fl.Lattice(lattice, dims, lam, 1e-4, 1.0, 3) as lat:
        print("CHOSEN", lat.autotune(4))
"""


def _tune(boxes, cache):
    res = subprocess.run([sys.executable, "-c", CODE % (ROOT, boxes)], capture_output=True, text=True,
                         env=dict(os.environ, FLBM_AUTOTUNE_CACHE=str(cache)))
    assert res.returncode == 0, res.stderr
    return [int(line.split()[1]) for line in res.stdout.splitlines() if line.startswith("CHOSEN")]


@pytest.mark.parametrize("boxes", [[(1, (18, 18, 18)), (1, (16, 16, 16))], [(1, (16, 16, 16)), (1, (18, 18, 18))],
                                   [(0, (64, 130, 1)), (0, (64, 128, 1))]])
def test_boxes_with_and_without_the_one_launch_form(tmp_path, boxes):
    cache = tmp_path / "tune.txt"
    chosen = _tune(boxes, cache)
    lines = [line.rsplit("\t", 1) for line in cache.read_text().splitlines()]
    assert len(lines) == 2 and lines[0][0] != lines[1][0]
    assert [int(v) for _, v in lines] == chosen
    assert _tune(boxes[::-1], cache) == chosen[::-1]  # read back
    assert len(cache.read_text().splitlines()) == 2


def test_choices_of_another_set_of_kernels_are_not_taken(tmp_path):
    import torch

    # A line as it was written when 8 was a kernel of its own: now it is never a candidate.
    name = torch.cuda.get_device_name(0)
    cache = tmp_path / "tune.txt"
    cache.write_text("%s|1|0|0|12|1|1|0|1\t8\n" % name)
    chosen, = _tune([(1, (16, 16, 16))], cache)
    assert chosen in (1, 2, 5, 7)
    lines = cache.read_text().splitlines()
    assert len(lines) == 2 and lines[0].endswith("\t8")
