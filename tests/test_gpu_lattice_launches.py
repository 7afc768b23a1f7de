"""Launches of the lattices beyond D2Q8: counted as they are queued, whichever
of single steps, captured steps and two-step launches a call takes."""
import numpy as np
import pytest

import paper_2010_01847_gb300 as plbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def launches(shape, steps, precision="fp32"):
    lattice = plbm.D3Q14 if len(shape) == 3 else plbm.D1Q2
    lat = plbm.LatticeND(lattice, shape, 0.9, 12.0, precision=precision)
    assert lat.kernel_launches == 0
    lat.init(np.ones(shape))
    lat.step(steps)
    n = lat.kernel_launches
    lat.init(np.ones(shape))
    assert lat.kernel_launches == 0
    lat.close()
    return n


@pytest.mark.parametrize("shape,precision", [((100,), "fp32"), ((20, 21, 22), "fp32"),
                                             ((130, 130, 130), "fp64")])
def test_one_launch_per_step(shape, precision):
    assert launches(shape, 130, precision) == 130      # two captured runs of 64 and two steps


@pytest.mark.parametrize("steps,want", [(1, 1), (2, 2), (3, 2), (7, 4), (8, 5)])
def test_pairs_of_steps(steps, want):
    assert launches((130, 130, 130), steps) == want    # the last one or two are single
