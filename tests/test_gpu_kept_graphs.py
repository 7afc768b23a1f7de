"""Captured launches that outlive a call: a replay advances the lattice by the
steps it is counted for, whatever selected the kernel since the capture."""
import numpy as np
import pytest

import paper_2010_01847_gb300 as plbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


def start(nx, ny, seed, amplitude=1e-3):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    e = torch.rand((ny, nx), generator=g, dtype=torch.float64, device="cuda")
    e.sub_(0.5).mul_(amplitude).add_(1.0)
    return e, 0.01 * (e - 1.0), torch.zeros_like(e)


@pytest.mark.parametrize("precision,steps", [("fp32", 4), ("fp16", 2)])
@pytest.mark.parametrize("init_between", [True, False])
def test_selecting_the_default_again_after_other_steps_per_launch(precision, steps, init_between):
    """A graph of `steps`-step launches, then set_kernel("auto") on a lattice
    of 2^24 nodes: the same kernel with another number of steps per launch."""
    nx = ny = 4096
    f = start(nx, ny, 3)
    lat = plbm.Lattice(nx, ny, 0.9, 12.0, precision=precision)
    assert lat.kernel == "wave"
    lat.set_wave_config(steps, 128)
    lat.init(*f)
    lat.step(194)      # captures launches of `steps` steps; ends on the buffer it began on
    lat.set_kernel("auto")
    assert lat.kernel == "wave" and lat.wave_config["steps"] != steps
    plain = plbm.Lattice(nx, ny, 0.9, 12.0, precision=precision)
    plain.set_graph_chunk(0)                     # launch by launch
    plain.init(*f)
    if init_between:
        lat.init(*f)
    else:
        plain.set_wave_config(steps, 128)
        plain.step(194)
        plain.set_kernel("auto")
    lat.step(194)
    plain.step(194)
    assert lat.step_count == plain.step_count
    for a, b in zip(lat.moments_device(), plain.moments_device()):
        assert torch.equal(a, b)


@pytest.mark.parametrize("precision,rounding", [
    ("fp64", "nearest"), ("fp32", "nearest"), ("fp16", "nearest"), ("bf16", "stochastic")])
def test_second_state_on_kept_graphs(precision, rounding):
    """Single steps replayed from graphs of an earlier state: one of the same
    amplitude, then one that moves the scale of 16-bit storage, which the
    captured coefficients hold."""
    nx, ny = 96, 65
    make = lambda: plbm.Lattice(nx, ny, 0.9, 12.0, plbm.PERIODIC_GRADIENT, plbm.DIFFUSE_WALLS,
                                1e-3, precision=precision, rounding=rounding, kernel="vector")
    kept = make()
    scales = []
    for seed, amplitude in ((1, 1e-3), (2, 1e-3), (3, 0.25), (4, 0.25)):
        f = start(nx, ny, seed, amplitude)
        fresh = make()
        for lat in (kept, fresh):
            lat.init(*f)
            lat.step(195)
        assert kept.step_count == fresh.step_count == 195
        assert np.array_equal(kept.populations(), fresh.populations())
        scales.append(kept.storage_scale)
    assert (scales[1] != scales[2]) == (precision in ("fp16", "bf16"))


@pytest.mark.parametrize("lattice,shape,precision", [
    (plbm.D3Q14, (12, 9, 15), "fp64"), (plbm.D3Q14, (16, 16, 16), "fp32"),
    (plbm.D1Q2, (301,), "fp64")])
def test_second_state_on_kept_graphs_nd(lattice, shape, precision):
    rng = np.random.default_rng(5)
    kept = plbm.LatticeND(lattice, shape, 0.9, 12.0, precision=precision)
    for amplitude in (1e-3, 1e-3, 0.25):
        e = 1.0 + amplitude * (rng.random(shape) - 0.5)
        fresh = plbm.LatticeND(lattice, shape, 0.9, 12.0, precision=precision)
        got = []
        for lat in (kept, fresh):
            lat.init(e)
            lat.step(195)
            got.append(lat.moments())
        for a, b in zip(*got):
            assert np.array_equal(a, b)
