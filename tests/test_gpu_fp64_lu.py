"""The FP64 LU (cluster panels, trailing updates split into 8-bit digits on the tensor cores, blocked
solves): the solution's backward error against the assembled system.  Gaussian elimination with
partial pivoting has a backward error below about n eps times the growth (a few units on these
well-scaled systems): 8 n 2^-53 here.  A mesh of a unit hard body and a tiny soft one mixes rows and columns
whose entries differ by the bodies' sizes, which the digits' row and column scales take up."""
import numpy as np
import pytest

from workloads import ico_sphere, merge_meshes, octa_sphere, scale_translate

pytestmark = pytest.mark.gpu

MESHES = {
    "66": lambda: octa_sphere(1),
    "132 (a panel of four rows)": lambda: merge_meshes([scale_translate(octa_sphere(1), 1.0, (0, 0, z)) for z in (-1.3, 1.3)]),
    "258": lambda: octa_sphere(2),
    "362": lambda: ico_sphere(3),
    "642 soft": lambda: ico_sphere(4, bc=1),
    "hard and tiny soft": lambda: merge_meshes([ico_sphere(3), scale_translate(octa_sphere(1), 1e-5, (0, 0, 1.5), bc=1)]),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_backward_error(name):
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    m = MESHES[name]()
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    ks = [0.9, 1.7, 2.4]
    surf = sol.solve_frequencies(ks, B.BIE_MODE_FP64)[0].cpu().numpy()
    for i, k in enumerate(ks):
        A, b = (t.cpu().numpy() for t in sol.assemble(k))
        x = np.where(m.bc == 0, surf[i, 0], surf[i, 1])
        # unknowns of the tiny body are larger by its size: the error relative to each row's own terms
        scale = np.abs(A) @ np.abs(x) + np.abs(b)
        assert np.max(np.abs(b - A @ x) / scale) <= 8 * m.N * 2.0 ** -53
    sol.close()


@pytest.mark.parametrize("batch", [1, 3, 40])
def test_batches_give_the_same_solutions(batch):
    """A system's solution does not depend on the systems beside it (which decide the clusters)."""
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    m = octa_sphere(2)
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    ks = 0.6 + 0.05 * np.arange(batch)
    many = sol.solve_frequencies(ks, B.BIE_MODE_FP64)[0].cpu().numpy()
    one = sol.solve_frequencies(ks[-1:], B.BIE_MODE_FP64)[0].cpu().numpy()[0]
    assert np.linalg.norm(many[-1] - one) <= 1e-12 * np.linalg.norm(one)
    sol.close()
