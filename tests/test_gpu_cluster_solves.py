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


def _batches(mesh, ks, batches):
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    sol = Solver(0)
    sol.set_geometry(mesh.nodes, mesh.elems, mesh.normals, mesh.bc)
    out = []
    for batch in batches:
        sol.set_option("mixed.batch", batch)
        surf, rep = sol.solve_frequencies(ks, B.BIE_MODE_MIXED)
        assert all(r.flags & B.BIE_FLAG_NOT_CONVERGED == 0 for r in rep)
        out.append(surf)
    sol.close()
    return out


def test_cluster_sizes_between_the_powers_of_two():
    """18 tall systems at once take clusters of 9, 7, 6 or 5 CTAs where 8 take two rounds and 4 do not hold a
    leaf; 6 at once take 16: the same leaves, the same bits."""
    import torch

    a, b = _batches(ico_sphere(13), 0.7 + 0.21 * np.arange(18), (18, 6))  # 6762 nodes
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))


def test_narrower_leaves():
    """40 systems of 5010 nodes take leaves of eight columns in one round of clusters, 8 at once sixteen: other
    roundings of the factor, solutions within the refinement's target (backward error 1e-11 on both
    sides, times a condition number of some hundred)."""
    import torch
    from workloads import merge_meshes, scale_translate

    mesh = merge_meshes([scale_translate(ico_sphere(5), 1.0, (2.5 * i, 0.3 * i, 0.0)) for i in range(5)])
    a, b = _batches(mesh, 0.55 + 0.043 * np.arange(40), (40, 8))
    for x, y in zip(a, b):
        assert torch.linalg.norm(x - y) <= 1e-8 * torch.linalg.norm(y)
