"""The FP64 kernels that take several wavenumbers at once (assembly: 4, 2 or 1 per thread; field:
groups of 16; equally spaced or not) against one wavenumber at a time and against the oracle.
Tolerances: the kernels differ from a one-wavenumber evaluation by a few ulps per phase (k R up to
about 30: 30 x 2^-53 = 3e-15) and per rotation (15 x 2^-53), far below 1e-12 of the largest value;
solutions carry the systems' condition numbers (below 1e2 here)."""
import numpy as np
import pytest

import oracle
from workloads import merge_meshes, octa_sphere, scale_translate, shell_points

pytestmark = pytest.mark.gpu


def _mesh():
    return merge_meshes([scale_translate(octa_sphere(1), 1.0, (0, 0, -1.4)),
                         scale_translate(octa_sphere(2), 0.7, (0, 0, 1.0), bc=1)])


def _ks(nk, uniform):
    k = 0.37 + 0.21 * np.arange(nk)
    return k if uniform else k + 0.05 * np.sin(3.0 * np.arange(nk))


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("nk", [2, 3, 5, 9])
def test_solves_in_groups_match_single_solves(nk, uniform):
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    m = _mesh()
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    ks = _ks(nk, uniform)
    if nk == 5:
        ks[0] = 0.0
    many = sol.solve_frequencies(ks, B.BIE_MODE_FP64)[0].cpu().numpy()
    for i, k in enumerate(ks):
        one = sol.solve_frequencies([k], B.BIE_MODE_FP64)[0].cpu().numpy()[0]
        assert np.linalg.norm(many[i] - one) <= 1e-11 * np.linalg.norm(one)
    P, Pn = oracle.solve_frequency(m, ks[-1], np.array([0.0, 0.0, 1.0]))
    for got, ref in ((many[-1, 0], P), (many[-1, 1], Pn)):
        assert np.linalg.norm(got - ref) <= 1e-10 * np.linalg.norm(ref)
    sol.close()


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("M", [1, 33, 700])
@pytest.mark.parametrize("nk", [1, 2, 3, 16, 19])
def test_fields_in_groups_match_single_fields(nk, M, uniform):
    """(The same closest surface points on both sides; against the oracle, whose own iteration ends a
    few ulps elsewhere, the FP64 field is checked in test_gpu_fp64.py.)"""
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    m = _mesh()
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    ks = _ks(nk, uniform)
    if nk == 3:
        ks[0] = 0.0
    rng = np.random.default_rng(5)
    surf = rng.standard_normal((nk, 2, m.N)) + 1j * rng.standard_normal((nk, 2, m.N))
    x = torch.tensor(shell_points(M, 2.6, 6.0, seed=M), device="cuda:0")
    s = torch.tensor(surf, device="cuda:0")
    got = sol.eval_field(x, ks, s, B.BIE_MODE_FP64).cpu().numpy()
    for i in {0, nk // 2, nk - 1}:
        ref = sol.eval_field(x, ks[i:i + 1], s[i:i + 1].contiguous(), B.BIE_MODE_FP64).cpu().numpy()[0]
        assert np.abs(got[i] - ref).max() <= 1e-12 * np.abs(ref).max() + 1e-12 * np.abs(surf).max()
    sol.close()


@pytest.mark.parametrize("mesh", ["66 nodes", "258 nodes", "1002 nodes"])
def test_fp64_field_of_a_point_is_its_own(mesh):
    """A point's FP64 values do not depend on the other points of the call, nor on further groups of 16
    wavenumbers: one order of the sums, whichever share of the quadrature points a CTA takes."""
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B
    from workloads import ico_sphere, octa_sphere

    m = {"66 nodes": octa_sphere(1), "258 nodes": octa_sphere(2), "1002 nodes": ico_sphere(5)}[mesh]
    sol = Solver(0)
    sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    g = torch.Generator("cuda:0").manual_seed(m.N)
    x = torch.randn((3001, 3), dtype=torch.float64, device="cuda:0", generator=g)
    x *= (1.05 + torch.rand((3001, 1), dtype=torch.float64, device="cuda:0", generator=g)) / x.norm(dim=1, keepdim=True)
    ks = 0.4 + 0.07 * np.arange(48)
    surf = torch.randn((48, 2, m.N), dtype=torch.complex128, device="cuda:0", generator=g)
    full = sol.eval_field(x, ks, surf, B.BIE_MODE_FP64)
    for M in (1, 2, 33, 500):
        for nk in (16, 48):
            part = sol.eval_field(x[:M].contiguous(), ks[:nk], surf[:nk].contiguous(), B.BIE_MODE_FP64)
            assert torch.equal(torch.view_as_real(part), torch.view_as_real(full[:nk, :M]))
    sol.close()
