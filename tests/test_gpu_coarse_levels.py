"""The coarse multigrid levels' kernels (cell-parallel applies and the one-launch coarse CG) against the
CPU FP64 oracle, at the sizes where their index arithmetic can go wrong."""
import numpy as np
import pytest

from oracle import operators as O
from oracle.mesh import ShellMesh
from oracle.multigrid import Hierarchy
from paper_2609_21633_gb300 import inputs
from tests.layout import LayoutMap, max_rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ORACLE_BC = {0: O.FREE, 1: O.NOSLIP}


# levels = 2 on (4, 9): the coarsest level has 3210 unique nodes, more than the CG cluster's 2048 threads;
# (2, 3): two node layers on the coarsest level; (2, 33): radial coarsening first; (3, 7): an odd cell count stops it
@pytest.mark.parametrize("level,n_r,levels,bc,kappa,quad", [
    (4, 9, 2, (0, 0), 0.0, 1), (4, 9, 2, (1, 1), 0.3, 1), (4, 9, 2, (1, 0), 0.0, 2), (2, 3, 0, (0, 0), 0.3, 1),
    (2, 33, 0, (0, 0), 0.0, 1), (3, 7, 0, (0, 0), 0.0, 2)])
def test_vcycle_coarse_levels(level, n_r, levels, bc, kappa, quad):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_21633_gb300 as tn
    om = ShellMesh(level, n_r, 0.55, 1.0)
    eta = inputs.lognormal_viscosity(om.n_wedges, 3, 0.5)
    m = tn.tn_mesh_create(level, n_r, 0.55, 1.0, bc[0], bc[1], hg_kappa=kappa, radial_quad_points=quad)
    mp = LayoutMap(tn.tn_mesh_info(m, 0), om)
    tn.tn_set_viscosity(m, torch.tensor(mp.wedges_to_layout(eta), device="cuda"))
    opts = tn.tn_mg_default_opts(coarse_rtol=0.0, coarse_max_iters=12, levels=levels)

    def dev(v, dtype=torch.float64):
        return [torch.tensor(mp.to_layout(v[c]), device="cuda", dtype=dtype) for c in range(3)]

    v0 = inputs.normal((3, om.n_nodes), 4)
    tn.tn_mg_setup(m, torch.float64, opts, dev(v0))
    H = Hierarchy(level, n_r, 0.55, 1.0, eta, bc=(ORACLE_BC[bc[0]], ORACLE_BC[bc[1]]), nlev=levels or None,
                  coarse_rtol=0.0, coarse_max_iters=12, kappa=kappa, quad=quad)
    H.setup(v0.ravel())
    r = O.project(O.boundary_projectors(om, H.bc), inputs.normal((3, om.n_nodes), 5))
    want = H.vcycle(r.ravel()).reshape(3, -1)
    z = [torch.zeros_like(t) for t in dev(r)]
    tn.tn_vcycle(m, dev(r), z)
    got = np.stack([mp.from_layout(t.cpu().numpy()) for t in z])
    assert max_rel(got, want) <= 1e-10
    # FP32: the bound of a V-cycle whose coarse CG runs a fixed number of steps in single precision
    tn.tn_mg_setup(m, torch.float32, opts, dev(v0, torch.float32))
    z32 = [torch.zeros_like(t) for t in dev(r, torch.float32)]
    tn.tn_vcycle(m, dev(r, torch.float32), z32)
    got = np.stack([mp.from_layout(t.double().cpu().numpy()) for t in z32])
    assert max_rel(got, want) <= 1e-3
    tn.tn_mesh_destroy(m)
