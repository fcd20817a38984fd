"""Heun steps through the assembled rows of the energy residual against the CPU FP64 oracle and against the
element-by-element residuals (which a captured first call takes)."""
import numpy as np
import pytest

from oracle import energy as OE
from oracle.mesh import ShellMesh
from paper_2609_21633_gb300 import inputs
from tests.layout import LayoutMap, max_rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# speed: cell Peclet numbers from below 1 to far above 4, where the upwind factor changes its formula
@pytest.mark.parametrize("level,n_r,speed,supg", [(1, 3, 1.0, True), (2, 5, 2000.0, True), (3, 9, 60.0, True),
                                                  (3, 9, 60.0, False), (4, 7, 0.0, True), (5, 5, 300.0, True)])
def test_heun_rows(level, n_r, speed, supg):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_21633_gb300 as tn
    om = ShellMesh(level, n_r, 0.55, 1.0)
    m = tn.tn_mesh_create(level, n_r, 0.55, 1.0)
    mp = LayoutMap(tn.tn_mesh_info(m, 0), om)
    T = inputs.temperature(om.node_xyz(), 0.55, 1.0) + 0.01 * inputs.normal(om.n_nodes, 3)
    u = speed * inputs.normal((3, om.n_nodes), 4)
    dt = 0.2 * tn.tn_energy_stable_dt(m) / (1.0 + speed)
    ud = [torch.tensor(mp.to_layout(u[c]), device="cuda") for c in range(3)]
    T0 = torch.tensor(mp.to_layout(T), device="cuda")
    # a captured call: no workspace can be allocated, so the residuals go element by element
    Tc = T0.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        tn.tn_energy_steps(m, Tc, ud, dt, 3, supg)
    g.replay()
    Td = T0.clone()
    tn.tn_energy_steps(m, Td, ud, dt, 3, supg)
    got, elem = mp.from_layout(Td.cpu().numpy()), mp.from_layout(Tc.cpu().numpy())
    want = OE.heun_steps(om, T, u, dt, 3, supg)
    assert max_rel(got, want) <= 1e-13
    assert max_rel(elem, want) <= 1e-13
    T2 = T0.clone()
    tn.tn_energy_steps(m, T2, ud, dt, 3, supg)
    assert torch.equal(Td, T2)
    tn.tn_mesh_destroy(m)
