"""Multi-step launches of mid-size FP32 lattices (the tile kernel and the
strip march an untimed lattice picks by its size): bit-identical to one
launch per step for every boundary kind, odd and thin sizes, tile and strip
remainders, any split of the steps into calls, and nothing written outside
the population buffers."""
import numpy as np
import pytest

import paper_2010_01847_gb300 as plbm
from paper_2010_01847_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

P, G, D, S = plbm.PERIODIC, plbm.PERIODIC_GRADIENT, plbm.DIFFUSE_WALLS, plbm.SIDES
ISO, FLUX, DIFF = plbm.ISOTHERMAL, plbm.HEAT_FLUX, plbm.DIFFUSE
SQUARE = [(ISO, 1.0), (ISO, 1.0002), (ISO, 0.9999), (FLUX, 1e-4)]
X_OPEN = [(FLUX, 1e-4), (DIFF, 0.0), (None, 0), (None, 0)]
X_MIXED = [(ISO, 1.001), (FLUX, -1e-4), (None, 0), (None, 0)]
Y_OPEN = [(None, 0), (None, 0), (DIFF, 0.0), (FLUX, 1e-4)]

# (nx, ny, bc_x, bc_y, sides): one tile column and several, ragged last tiles,
# odd columns and rows, seams and walls at tile edges, rows fewer than a halo,
# lattices narrower than a tile, sides on either axis and both, and (the last
# three) strip-march sizes
CASES = [
    (128, 128, P, P, None), (130, 67, G, D, None), (131, 40, G, P, None), (57, 201, P, D, None),
    (5121, 1, P, P, None), (2600, 2, G, D, None), (2000, 3, P, P, None), (3, 2000, G, D, None),
    (64, 90, G, D, None), (65, 90, P, P, None), (101, 101, S, S, SQUARE), (64, 129, S, S, SQUARE),
    (97, 130, S, P, X_OPEN), (401, 33, S, P, X_MIXED), (90, 100, P, S, Y_OPEN),
    (91, 100, G, S, Y_OPEN), (100, 90, S, D, [(ISO, 1.0), (ISO, 1.001), (None, 0), (None, 0)]),
    (1024, 256, G, D, None), (777, 333, P, P, None),
    (1536, 1100, P, P, None), (2050, 1030, G, D, None), (4098, 700, G, P, None),
]


def lattice(case, kernel, **kw):
    nx, ny, bx, by, sides = case
    return plbm.Lattice(nx, ny, 0.9, 12.0, bx, by, 1e-3 if bx == G else 0.0, sides=sides,
                        kernel=kernel, **kw)


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c[0]}x{c[1]}_bc{c[2]}{c[3]}")
def test_bit_identical_to_single_steps(case):
    nx, ny = case[:2]
    f = inputs.random_state_fields(nx, ny, seed=nx + 3 * ny)
    out = []
    for kernel in ("auto", None):
        lat = lattice(case, "auto")
        single = lat.kernel
        assert single in ("vector", "scalar")
        if kernel is None:
            lat.set_kernel(single)          # one launch per step
        lat.init(*f)
        launches = lat.kernel_launches
        lat.step(31)
        launches = lat.kernel_launches - launches
        got = [lat.populations()]
        for n in (1, 2, 12, 13):
            lat.step(n)
        got.append(lat.step_residual(27))
        blob = lat.get_state()
        lat.step(9)
        got += [lat.populations(), *lat.moments(), lat.step_count]
        lat.set_state(blob)
        lat.step(9)
        got.append(lat.populations())
        out.append((launches, got))
        lat.close()
    (fast, a), (plain, b) = out
    assert plain == 31 and fast < 31
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("case", [CASES[0], CASES[5], CASES[11], CASES[13], CASES[19]],
                         ids=lambda c: f"{c[0]}x{c[1]}_bc{c[2]}{c[3]}")
def test_guard_bands_untouched(case):
    nx, ny = case[:2]
    nbytes = plbm.load_library().lbm_population_bytes(plbm.Grid(nx, ny), plbm.FP32)
    guard, nb = 1 << 16, (nbytes + 255) // 256 * 256
    raw = torch.full((3 * guard + 2 * nb,), 0xA5, dtype=torch.uint8, device="cuda")
    bufs = (raw[guard:guard + nb], raw[2 * guard + nb:2 * guard + 2 * nb])
    lat = lattice(case, "auto", buffers=bufs)
    lat.init(*inputs.random_state_fields(nx, ny, seed=5))
    lat.step(25)
    lat.step_residual(8)
    lat.sync()
    lat.close()
    for band in (raw[:guard], raw[guard + nbytes:2 * guard + nb], raw[2 * guard + nb + nbytes:]):
        assert bool((band == 0xA5).all())


def test_autotune_keeps_state_and_side_switches_take_effect():
    case = CASES[10]
    f = inputs.random_state_fields(*case[:2], seed=2)
    a, b = lattice(case, "auto"), lattice(case, "scalar")
    for lat in (a, b):
        lat.init(*f)
        lat.step(20)
    a.autotune(12)
    for lat in (a, b):
        lat.set_side(plbm.TOP, DIFF)
        lat.step(23)
    assert np.array_equal(a.populations(), b.populations())
