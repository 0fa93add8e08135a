"""Cluster kernels of the mixed path (panels, triangular solves): what a cluster computes does not depend
on its number of CTAs, which follows the batch.  Batches of 64 systems and more take the same roundings
in the panels (up to 1536 rows), and every product and sum of the solves has one order, so solutions
are equal bit for bit whatever the batch size."""
import numpy as np
import pytest

from workloads import ico_sphere, octa_sphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh", ["66 nodes", "258 nodes", "642 nodes"])
def test_solutions_do_not_depend_on_the_batch(mesh):
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    m = {"66 nodes": octa_sphere(1), "258 nodes": octa_sphere(2), "642 nodes": ico_sphere(4)}[mesh]
    ks = 0.3 + 0.009 * np.arange(160)
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    out = {}
    for batch in (64, 80, 160):  # 4 and 2 CTAs a system in the solves, one above 152
        sol.set_option("mixed.batch", batch)
        out[batch] = sol.solve_frequencies(ks[:80 if batch == 80 else 160], B.BIE_MODE_MIXED)[0]
    full = out[160][:128]  # (the last, partial batch of 64 has 32 systems: other panels)
    assert torch.equal(out[64][:128], full)
    assert torch.equal(out[80], full[:80])
    sol.close()
