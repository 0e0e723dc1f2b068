"""Copies between the caller's layout and the padded one: wide, tall and small walls."""

import pytest
import torch

from oracle import fem
from synth import BOTTOM, LEFT, dirichlet_design

pytestmark = pytest.mark.gpu
EP = [1.0, 0.5, 0.25, 1e-9]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("nx,ny,nc", [(2, 2, 1), (30, 4, 1), (34, 2, 1), (254, 10, 1), (4160, 64, 6), (64, 4160, 6),
                                      (60, 1028, 2), (1000, 136, 3)])
def test_copies_of_any_shape(nx, ny, nc, prec):
    """The operator in place (through the padded vectors) equals the one between two arrays
    bit for bit; the moduli come back as the oracle forms them."""
    import paper_2301_07457_gb300 as mto
    m = mto.Mesh(nx, ny, n_coarsen=nc, precision=prec, fixed_edges=BOTTOM | LEFT)
    x = dirichlet_design(nx, ny, 4, seed=nx)
    m.set_design(torch.from_numpy(x).cuda(), EP, 3.0)
    v = torch.randn(*m.level_shape(nc), dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(1))
    y, w = m.apply_operator(nc, v), v.clone()
    assert m._lib.mto_apply_operator(m._h, nc, 0, w.data_ptr(), w.data_ptr()) == 0
    torch.cuda.synchronize()
    assert torch.equal(w, y) and torch.count_nonzero(y) > 0
    E = torch.from_numpy(fem.simp_moduli(x, EP, 3.0))
    assert torch.all((m.moduli().cpu() - E).abs() <= 1e-14 * E)
    m.close()
