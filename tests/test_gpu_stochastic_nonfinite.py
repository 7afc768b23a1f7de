"""Stochastic rounding of a state that is not finite: NaN is stored as NaN, as
rounding to nearest stores it, so a diverged run is reported."""
import struct

import numpy as np
import pytest

import paper_2010_01847_gb300 as plbm
from paper_2010_01847_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

NX, NY = 256, 40


def poisoned(precision, rounding, kernel, word):
    """A lattice whose plane 2 holds `word` (16 bits) at one node."""
    lat = plbm.Lattice(NX, NY, 0.9, 12.0, precision=precision, rounding=rounding, kernel=kernel)
    lat.init(*inputs.random_state_fields(NX, NY, seed=11))
    blob = bytearray(lat.get_state())
    nbytes = plbm.load_library().lbm_population_bytes(plbm.Grid(NX, NY), lat.precision)
    head = len(blob) - 2 * nbytes
    node = 17 * NX + 101
    for buf in range(2):                       # plane 2 of both buffers
        struct.pack_into("<H", blob, head + buf * nbytes + 2 * (2 * NX * NY + node), word)
    lat.set_state(bytes(blob))
    return lat


@pytest.mark.parametrize("precision,word", [("bf16", 0x7fff), ("bf16", 0xffc0), ("fp16", 0x7e00),
                                            ("fp16", 0xffff), ("fp16", 0x7c00)])
@pytest.mark.parametrize("kernel", ["scalar", "vector", "wave"])
def test_nan_spreads_as_with_rounding_to_nearest(precision, word, kernel):
    bad = []
    for rounding in ("nearest", "stochastic"):
        lat = poisoned(precision, rounding, kernel, word)
        seen = []
        for n in (1, 1, 1, 5):
            lat.step(n)
            seen.append(~np.isfinite(lat.moments()[0]))
        with pytest.raises(plbm.LBMError) as ex:
            lat.step_residual(3)
        assert ex.value.status == plbm.ENONFINITE
        bad.append(seen)
    for a, b in zip(*bad):
        assert a.any() and np.array_equal(a, b)
