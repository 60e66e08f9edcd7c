"""The FP64 push's integer deposits and refined reciprocals where they could go
wrong: units in which gamma^2 and |B|^2 leave single precision's range (the
reciprocals then divide), particles on cell faces and in corners (weights 0 and
1/2), and stencils that leave the tile."""
import numpy as np
import pytest

import oracle as orc
from paper_1412_1087_gb300 import workloads as wl
from tests._parity import momenta_of, periodic_diff, positions_of, rel_l2, sorted_oracle_state, tilt_B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1412_1087_gb300 import mhdpic as m  # noqa: E402


def _box(ndim, units, faces):
    if ndim == 3:
        box = wl.alfvenic_beam_3d(n=10, ppc=5, nmodes=6, seed=51)
    else:
        box = wl.periodic_thermal_2d(nx=21, ny=18, ppc=7, dv_amp=0.3, seed=52)
    tilt_B(box, 53)
    if units != 1.0:   # speeds in units of 1/units and fields in units of `units`
        box.p = (box.p.astype(np.float64) * units).astype(np.float32)
        box.C *= units
        box.dt /= units
        box.B /= units
        box.mom *= units
        box.qm_cr *= units * units
        box.m_cr /= units * units   # the charge as before
    if faces:
        box.off[:, ::3] = 0.0
        box.off[0, 1::3] = np.float32(1.0) - np.float32(2.0 ** -24)
        box.p[:, ::6] = 0.0   # stays on its corner
    return box


@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("units,faces,steps", [(1e16, False, 1), (1e-16, False, 1), (1.0, True, 1), (1.0, False, 9)])
def test_fp64_push_matches_oracle(ndim, units, faces, steps):
    box = _box(ndim, units, faces)
    eng = m.Engine([box], precision=m.MHDPIC_PREC_FP64, device="cuda:0")
    _, _, x, v = sorted_oracle_state(box)
    st = orc.State(box, x, v)
    corr = 0.0
    for _ in range(steps):   # the fields stay as staged; no sort, so particles leave their tiles
        c, md = st.push_only(box.dt)
        corr = corr + c
        eng.interp_push(box.dt, 1)
    gc, gm = eng.deposits(0).cpu().numpy(), eng.deposits(1).cpu().numpy()
    for q in range(4):
        assert rel_l2(gm[q], md[q]) < 1e-12, ("moments", q)
        # the corrector's scale is sized for its bound: sums over the steps
        assert rel_l2(gc[q], corr[q]) < 1e-12 * steps, ("corrector", q)
    xg, vg = positions_of(eng), momenta_of(eng)
    for d in range(box.ndim):
        assert np.abs(periodic_diff(xg[d], st.x[d], box.n[d] * box.dx[d])).max() < 1e-12 * steps * (1 + box.n[d])
    assert np.all(np.abs(vg - st.v) <= 1e-12 * steps * np.sqrt((st.v ** 2).sum(0)))
    assert eng.status() == 0
    eng.close()


@pytest.mark.parametrize("one_cell", [False, True])
@pytest.mark.parametrize("ndim,brick", [(3, (8, 8, 8)), (2, (36, 36, 1)), (2, (32, 32, 1)), (3, (4, 4, 2))])
def test_fp64_tile_words_give_the_same_integers(ndim, brick, one_cell):
    """Bricks too large for the 32-bit words (8^3, 36^2) take a 64-bit tile: the
    sums are integers, the same for every brick, tile and order; with every
    particle in one cell the words are as full as they get (2,646 particles in
    2-D and 5,000 in 3-D, more than an item takes)."""
    box = _box(ndim, 1.0, False)
    if one_cell:
        box.cell[:] = box.cell[0]
    got = []
    for b in ((0, 0, 0), brick):
        eng = m.Engine([box], precision=m.MHDPIC_PREC_FP64, device="cuda:0", brick=b)
        for _ in range(3):
            eng.interp_push(box.dt, 1)
        got.append([eng.deposits(i).clone() for i in (0, 1)])
        assert eng.status() == 0
        eng.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
