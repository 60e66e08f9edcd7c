"""The sort at the edges of its passes, bit for bit against the oracle's stable
sort: one, two and eight scan tiles of 4,096 keys and the two-launch scan
beyond, cells of up to 128, 1,024 and more particles side by side (registers,
a warp, a block), and a step after it (the work list)."""
import numpy as np
import pytest

import oracle as orc
from paper_1412_1087_gb300 import workloads as wl
from tests._parity import rel_l2, sorted_oracle_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1412_1087_gb300 import mhdpic as m  # noqa: E402


@pytest.mark.parametrize("prec", [m.MHDPIC_PREC_MIXED, m.MHDPIC_PREC_FP64])
@pytest.mark.parametrize("nx,ny,crowd", [(24, 16, (128, 129, 130)), (63, 64, (1, 2, 33)), (176, 184, (1024, 1025, 64)),
                                         (184, 184, (127, 600, 8300))])
def test_sort_and_step_match_oracle(prec, nx, ny, crowd):
    box = wl.periodic_thermal_2d(nx=nx, ny=ny, ppc=2, dv_amp=0.2, seed=81)
    rng = np.random.default_rng(82)
    cells = np.concatenate([np.full(n, nx * 3 + 5 + i) for i, n in enumerate(crowd)]).astype(np.int32)
    extra = cells.size
    box.cell = np.concatenate([box.cell, cells])
    order = rng.permutation(box.cell.size)
    box.cell = np.ascontiguousarray(box.cell[order])
    box.off = np.ascontiguousarray(np.concatenate([box.off, rng.random((2, extra), dtype=np.float32)], axis=1)[:, order])
    box.p = np.ascontiguousarray(np.concatenate([box.p, rng.choice(box.p, extra, axis=1)], axis=1)[:, order])
    perm, counts, x, v = sorted_oracle_state(box)
    eng = m.Engine([box], precision=prec, device="cuda:0")
    v0 = eng.velocities().cpu().numpy()
    assert np.array_equal(v0, v)                  # the order of the initial sort
    # a shuffle of the sorted particles, sorted again
    if prec == m.MHDPIC_PREC_MIXED:
        eng.set_particles(box.cell, box.off, box.p)
    else:
        eng.x.copy_(torch.from_numpy(wl.absolute_positions(box)))
        eng.p64.copy_(torch.from_numpy(box.p.astype(np.float64)))
    got, cnt = eng.sort(want_perm=True, want_counts=True)
    assert np.array_equal(got.cpu().numpy(), perm) and np.array_equal(cnt.cpu().numpy(), counts)
    st = orc.State(box, x, v)
    corr, md = st.push_only(box.dt)
    eng.interp_push(box.dt, 1)
    # FP64: the fixed-point unit of the current is at most 2 H 2^-62 of its bound
    # per particle, H = 9 (4 maxcount + 64) contributions, and a particle's
    # current is |u|/C = 1/10 of the bound: rounding errors of 0.29 units
    # against contributions of 0.2 / 10 of the bound (rms of weight and
    # direction) are 29 H 2^-62 in the 2-norm; twice that is allowed
    H = 9.0 * (4.0 * max(crowd) + 64.0)
    tol = max(1e-12, 2 * 29.0 * H * 2.0 ** -62) if prec == m.MHDPIC_PREC_FP64 else 1e-5
    gm = eng.deposits(1).cpu().numpy()
    for q in range(4):
        assert rel_l2(gm[q], md[q]) < tol, q
    assert eng.status() == 0
    eng.close()
