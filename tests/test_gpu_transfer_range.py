"""Prolongation keeps the coarse values at coincident nodes bit for bit, up to the largest finite value."""
import numpy as np
import pytest

from oracle import operators as O
from oracle.mesh import ShellMesh
from tests.layout import LayoutMap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("ncomp", [1, 3])
def test_coincident_nodes(dtype, ncomp):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_21633_gb300 as tn
    td = torch.float64 if dtype == "f64" else torch.float32
    om = ShellMesh(3, 5, 0.55, 1.0)
    pm = O.pressure_mesh(om)
    m = tn.tn_mesh_create(3, 5, 0.55, 1.0)
    mp, pmap = LayoutMap(tn.tn_mesh_info(m, 0), om), LayoutMap(tn.tn_mesh_info(m, 1), pm)
    big, tiny = torch.finfo(td).max, torch.finfo(td).tiny * torch.finfo(td).eps  # largest and smallest magnitudes
    x = np.random.default_rng(1).standard_normal(pm.n_nodes)
    x[0::4], x[1::4], x[2::4] = big, -big, tiny
    c = [torch.tensor(pmap.to_layout(x), device="cuda").to(td) for _ in range(ncomp)]
    f = [torch.zeros(mp.n_layout, device="cuda", dtype=td) for _ in range(ncomp)]
    tn.tn_prolong(m, 0, c, f)
    Pt = O.prolongation(om, pm)
    rows = np.flatnonzero(np.diff(Pt.indptr) == 1)  # fine nodes that are coarse nodes
    cols = Pt.indices[Pt.indptr[rows]]
    want = pmap.from_layout(c[0].double().cpu().numpy())[cols]
    for t in f:
        got = np.full(om.n_nodes, np.nan)
        got[mp.node] = t.double().cpu().numpy()[mp.idx]
        assert np.array_equal(got[rows], want)
    tn.tn_mesh_destroy(m)
