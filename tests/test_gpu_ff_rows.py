"""Float-float assembly where every element carries one boundary condition, against the FP64 bulk: hard
and soft elements, an odd number of quadrature points (the halves differ), k = 0, rows in shared memory
and (beyond 4600 nodes) in the matrix.  48-bit arithmetic: a phase up to k R = 62 is off by some
62 x 2^-48 = 2e-13 of its term, so entries agree to 1e-12 of the largest."""
import numpy as np
import pytest

from workloads import ico_sphere, merge_meshes, octa_sphere, scale_translate

pytestmark = pytest.mark.gpu


def _mesh(name):
    if name == "both":
        return merge_meshes([scale_translate(octa_sphere(1), 0.8, (0, 0, -1.0), bc=1),
                             scale_translate(ico_sphere(2), 1.1, (0.3, 0, 1.3))])
    return {"hard": octa_sphere(2), "soft": octa_sphere(1, bc=1), "4842 nodes": ico_sphere(11)}[name]


@pytest.mark.parametrize("mesh,ng,k", [("hard", (4, 6), 0.0), ("hard", (4, 6), 31.0), ("soft", (3, 5), 0.7),
                                       ("both", (3, 5), 15.0), ("both", (4, 6), 0.0), ("4842 nodes", (4, 6), 7.0)])
def test_float_float_rows_match_fp64(mesh, ng, k):
    import torch
    from paper_1706_07919_gb300 import Solver

    m = _mesh(mesh)
    sol = Solver(0)
    sol.set_quadrature(*ng)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    sol.set_incident_plane_wave(np.array([0.6, 0.0, 0.8]))
    sol.set_option("assemble.bulk_ff", 1)
    A, b = sol.assemble(k)
    sol.set_option("assemble.bulk_ff", 0)
    A64, b64 = sol.assemble(k)
    assert (A - A64).abs().max() <= 1e-12 * A64.abs().max()
    assert torch.linalg.norm(b - b64) <= 1e-12 * torch.linalg.norm(b64)
    sol.close()
