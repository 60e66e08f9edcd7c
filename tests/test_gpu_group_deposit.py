"""The warp-wide 64-bit deposit (12 lanes to a particle) at particle counts
around the warp and the block, in both precisions and dimensions, against the
oracle's deposit: no particles, one, a warp less and more one, a ragged tail."""
import ctypes

import numpy as np
import pytest

import oracle as orc
from paper_1412_1087_gb300 import workloads as wl
from tests._parity import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1412_1087_gb300 import mhdpic as m  # noqa: E402


@pytest.mark.parametrize("prec", [m.MHDPIC_PREC_MIXED, m.MHDPIC_PREC_FP64])
@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("count", [0, 1, 31, 33, 263])
def test_deposit_matches_oracle(prec, ndim, count):
    box = (wl.alfvenic_beam_3d(n=7, ppc=1, nmodes=2, seed=61) if ndim == 3
           else wl.periodic_thermal_2d(nx=19, ny=15, ppc=1, seed=62))
    x, v = wl.absolute_positions(box)[:, :count], box.p[:, :count].astype(np.float64)
    g, p = m.Grid(), m.Params()
    g.ndim = ndim
    for d in range(3):
        g.n[d], g.dx[d], g.x0[d], g.bc[d] = box.n[d], box.dx[d], box.x0[d], box.bc[d]
    p.qm_cr, p.qm_gas, p.C, p.m_cr, p.hall, p.shape = box.qm_cr, box.qm_gas, box.C, box.m_cr, 0, m.MHDPIC_SHAPE_TSC
    pos, vel = m.pack_records_arrays(box.cell[:count], box.off[:, :count], box.p[:, :count])
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (pos, vel, x, v)]
    out = torch.full((4, box.ncell), float("nan"), dtype=torch.float64, device="cuda")
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    q = [t.data_ptr() for t in dev]
    mixed = prec == m.MHDPIC_PREC_MIXED
    m.mhdpic_deposit_moments_noalloc(g, p, prec, count, pos=q[0] if mixed else 0, vel=q[1] if mixed else 0,
                                     x=0 if mixed else q[2], p64=0 if mixed else q[3], out=out.data_ptr(), stream=st)
    got = out.cpu().numpy()
    if count == 0:
        assert not got.any()
        return
    want = orc.deposit_moments(orc.grid_of(box), orc.params_of(box), np.ascontiguousarray(x), np.ascontiguousarray(v),
                               box.ncell)
    for k in range(4):
        assert rel_l2(got[k], want[k]) < 1e-12, k
