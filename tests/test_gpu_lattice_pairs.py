"""The two-step D3Q14 launches against single steps: the same bits, on sizes at
and off the edges of its tiles (30 x 8 own nodes) and with one to three planes
(periodic in z within the marched planes)."""
import numpy as np
import pytest

import paper_2010_01847_gb300 as plbm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.mark.parametrize("shape", [          # (nz, ny, nx), at least 2^19 nodes
    (1, 730, 731), (2, 513, 517), (3, 420, 450), (81, 81, 81), (97, 72, 90),
    (700, 25, 31), (6000, 3, 30), (2300, 240, 1), (9000, 1, 61)])
def test_pairs_equal_single_steps(shape):
    rng = np.random.default_rng(sum(shape))
    e = 1 + 1e-3 * rng.standard_normal(shape)
    q = 1e-3 * rng.standard_normal((3, *shape))
    out = []
    for chunks in ([7], [1] * 7, [2, 4, 1]):      # single calls of 1 or 2 steps take single steps
        lat = plbm.LatticeND(plbm.D3Q14, shape, 0.9, 12.0)
        lat.init(e, q)
        for n in chunks:
            lat.step(n)
        out.append(lat.moments())
        assert lat.step_count == 7
        lat.close()
    for e_n, q_n in out[1:]:
        np.testing.assert_array_equal(out[0][0], e_n)
        np.testing.assert_array_equal(out[0][1], q_n)


def test_init_reports_a_value_that_is_not_finite():
    shape = (5, 6, 7)
    lat = plbm.LatticeND(plbm.D3Q14, shape, 0.9, 12.0)
    e, q = np.ones(shape), np.zeros((3, *shape))
    lat.init(e, q)
    lat.step(3)
    before = lat.moments()
    for field, bad in ((0, np.nan), (1, np.inf)):
        fe, fq = e.copy(), q.copy()
        (fe, fq)[field].flat[-1] = bad
        with pytest.raises(plbm.LBMError) as ex:
            lat.init(fe, fq)
        assert ex.value.status == plbm.EINVAL
    assert lat.step_count == 3                     # the state is kept
    np.testing.assert_array_equal(lat.moments()[0], before[0])
