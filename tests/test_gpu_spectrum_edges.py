"""Spectrum decisions at their closest: bin edges on the binned quantities of
particles and one unit in the last place beside them, negative and zero edges,
region bounds on particle positions, and a box so far from the origin that a
position is rounded by a good part of a cell."""
import numpy as np
import pytest

import oracle as orc
from paper_1412_1087_gb300 import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1412_1087_gb300 import mhdpic as m  # noqa: E402


def _quantity(box, kind):   # the defined operations, in IEEE double
    v = box.p.astype(np.float64)
    v2 = (v[0] * v[0] + v[1] * v[1]) + v[2] * v[2]
    if kind == m.MHDPIC_SPEC_MOMENTUM:
        return np.sqrt(v2)
    return v2 / (np.sqrt(box.C * box.C + v2) / box.C + 1.0)


@pytest.mark.parametrize("kind", [m.MHDPIC_SPEC_ENERGY, m.MHDPIC_SPEC_MOMENTUM])
@pytest.mark.parametrize("prec,x0", [(m.MHDPIC_PREC_MIXED, 0.0), (m.MHDPIC_PREC_MIXED, 2.0 ** 51), (m.MHDPIC_PREC_FP64, 0.0)])
def test_edges_and_bounds_on_particles(kind, prec, x0):
    box = wl.bell_2d(seed=71, n=24, ppc=8)
    box.x0 = (x0, x0, 0.0)
    box.p[:, 5] = 0.0
    box.p[:, 6] = np.float32(1e-20)
    eng = m.Engine([box], precision=prec)
    q = np.sort(_quantity(box, kind))
    pick = q[:: max(1, q.size // 40)]
    edges = np.unique(np.concatenate([[-3.0, -0.0], pick, np.nextafter(pick, np.inf), np.nextafter(pick, 0.0)]))
    x = wl.absolute_positions(box)
    regions = [None, [x[0, 10], x[0, 11] + 9.0, x[1, 20], np.inf],
               [np.nextafter(x[0, 30], -np.inf), x[0, 31] + 3.0, -np.inf, x[1, 33]]]
    for region in regions:
        counts, sums = eng.spectrum(kind, edges, region, n_moment=5)
        oc, os_ = orc.spectrum(orc.grid_of(box), orc.params_of(box), x, box.p.astype(np.float64), kind, edges, region, 5)
        np.testing.assert_array_equal(counts[0], oc)
        np.testing.assert_allclose(sums[0], os_, rtol=1e-12)
    eng.close()
