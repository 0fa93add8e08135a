"""Closest surface points (nearest node found with FP32 distances and decided in FP64, then one Newton
search per element at that node) do not depend on how many points a CTA takes (1 to 32), through the
field: a wrong node or element changes it by the discretisation error (1e-4 and more).  With the same
surface points the field differs by the order of its sums: 1e-12 of it, per distance.  (Against the
oracle the points are checked in test_gpu_fp64.py; where two elements' distances agree to rounding the
oracle's search may end on the other one.)"""
import numpy as np
import pytest

from workloads import ico_sphere, octa_sphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,M", [("66 nodes", 1), ("66 nodes", 2), ("66 nodes", 33), ("66 nodes", 700),
                                    ("66 nodes", 5003), ("2562 nodes", 1), ("2562 nodes", 153), ("2562 nodes", 700)])
def test_closest_points_do_not_depend_on_the_batch(mesh, M):
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    m = octa_sphere(1) if mesh == "66 nodes" else ico_sphere(8)
    rng = np.random.default_rng(M)
    x = rng.standard_normal((M, 3))
    x /= np.linalg.norm(x, axis=1)[:, None]
    shell = np.arange(M) % 4
    x *= np.array([1.02, 1.5, 4.0, 30.0])[shell][:, None]
    k = 2.0
    P = np.exp(1j * k * m.nodes[:, 0])
    Pn = 1j * np.exp(1j * k * m.nodes[:, 1])
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    surf = torch.tensor(np.stack([P, Pn])[None], device="cuda")
    xd = torch.tensor(x, device="cuda")
    T = sol.eval_field(xd, np.array([k]), surf, B.BIE_MODE_FP64).cpu().numpy()[0]
    ref = np.concatenate([sol.eval_field(xd[j:j + 150], np.array([k]), surf, B.BIE_MODE_FP64).cpu().numpy()[0]
                          for j in range(0, M, 150)])  # one point a CTA
    for s in range(4):
        i = shell == s
        if i.any():
            assert np.linalg.norm(T[i] - ref[i]) <= 1e-12 * np.linalg.norm(ref[i])
    sol.close()


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
@pytest.mark.parametrize("variant", [0, 1, 2])
def test_points_that_are_not_finite(mode, variant):
    """A NaN or infinite observation point has no nearest element: its field is not finite, the other points'
    are their own."""
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B
    from workloads import octa_sphere, shell_points

    m = octa_sphere(1)
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    sol.set_option("field.variant", variant)
    md = B.BIE_MODE_MIXED if mode == "mixed" else B.BIE_MODE_FP64
    x = torch.tensor(shell_points(70, 1.2, 3.0, seed=4), device="cuda:0")
    k = 0.3 * np.arange(1, 21)
    g = torch.Generator("cuda:0").manual_seed(2)
    surf = torch.randn((20, 2, m.N), dtype=torch.complex128, device="cuda:0", generator=g)
    good = sol.eval_field(x, k, surf, md)
    bad = x.clone()
    bad[3, 1], bad[40, 0], bad[69] = float("nan"), float("inf"), float("nan")
    got = sol.eval_field(bad, k, surf, md)
    keep = torch.ones(70, dtype=torch.bool, device="cuda:0")
    keep[[3, 40, 69]] = False
    assert torch.equal(torch.view_as_real(got[:, keep]), torch.view_as_real(good[:, keep]))
    assert not torch.isfinite(torch.view_as_real(got[:, ~keep])).all(dim=2).any()
    sol.close()
