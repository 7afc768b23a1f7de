"""An autotuned choice given to a second lattice through the public settings."""
import pytest

import paper_2010_01847_gb300 as plbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("nx,ny", [(2048, 2048), (2050, 1999)])
def test_choice_carries_over(nx, ny):
    """At these sizes the strip march is several times faster than a launch
    per step, and the tuned lattice says so: the second lattice takes as many
    launches, and ends in the same bits."""
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    e = torch.rand((ny, nx), generator=g, dtype=torch.float64, device="cuda")
    e.sub_(0.5).mul_(1e-3).add_(1.0)
    z = torch.zeros_like(e)
    a, b = (plbm.Lattice(nx, ny, 0.9, 12.0) for _ in range(2))
    kernel, us = a.autotune(10)
    assert kernel == a.kernel == "wave" and us > 0
    b.set_kernel(kernel)
    b.set_wave_config(a.wave_config["steps"], a.wave_config["rows"])
    taken = []
    for lat in (a, b):
        lat.init(e, z, z)
        before = lat.kernel_launches
        lat.step(41)
        taken.append(lat.kernel_launches - before)
    assert taken[0] == taken[1] < 20
    for u, v in zip(a.moments_device(), b.moments_device()):
        assert torch.equal(u, v)
