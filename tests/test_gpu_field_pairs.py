"""The packed field kernel (two groups of 16 wavenumbers in the halves of packed FP32 registers)
against the one-group kernel: every half performs the one-group kernel's operations in its order, and
run sums are added in the order of the runs whatever the layout, so the values are equal bit for bit."""
import numpy as np
import pytest

from workloads import merge_meshes, octa_sphere, scale_translate, shell_points

pytestmark = pytest.mark.gpu


def _lists(nk):
    uni = 0.11 * np.arange(1, nk + 1)
    picked = np.concatenate([[0.0], np.cumsum(0.05 + 0.1 * np.random.default_rng(nk).random(nk))])[:nk]
    runs = np.concatenate([uni, [uni[-1] + 0.03, uni[-1] + 0.07], uni[-1] + 1.0 + 0.25 * np.arange(5)])
    return {"uniform": uni, "from zero": 0.11 * np.arange(nk), "picked": picked, "runs": runs}


@pytest.mark.parametrize("ng", [1, 4])
@pytest.mark.parametrize("M", [1, 2, 9, 31, 33, 200, 5000])
@pytest.mark.parametrize("nk", [1, 5, 16, 17, 32, 49])
def test_packed_pairs_match_one_group_kernel(nk, M, ng):
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    # one rule per element (Q = 1) leaves a ragged last run of quadrature points
    mesh = merge_meshes([scale_translate(octa_sphere(1), 1.0, (0, 0, -1.4)),
                         scale_translate(octa_sphere(1), 0.7, (0, 0, 1.0), bc=1)])
    sol = Solver(0)
    sol.set_quadrature(ng, 6)
    sol.set_geometry(mesh.nodes, mesh.elems, mesh.normals, mesh.bc)
    x = torch.tensor(shell_points(M, 2.6, 6.0, seed=M), dtype=torch.float64, device="cuda:0")
    for name, k in _lists(nk).items():
        rng = np.random.default_rng(7)
        surf = torch.tensor(rng.standard_normal((len(k), 2, mesh.N)) + 1j * rng.standard_normal((len(k), 2, mesh.N)),
                            device="cuda:0")
        T = {}
        for v in (1, 2):
            sol.set_option("field.variant", v)
            T[v] = sol.eval_field(x, k, surf, B.BIE_MODE_MIXED)
        assert torch.equal(T[1], T[2]), name
    sol.close()


def test_one_group_tail_at_many_points():
    """A last group of 16 at many points takes the one-group kernel: same values either way."""
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    mesh = octa_sphere(1)
    sol = Solver(0)
    sol.set_geometry(mesh.nodes, mesh.elems, mesh.normals, mesh.bc)
    for M, nk in ((15300, 45), (40000, 33)):
        x = torch.tensor(shell_points(M, 1.1, 3.0, seed=1), dtype=torch.float64, device="cuda:0")
        k = 0.2 * np.arange(1, nk + 1)
        surf = torch.tensor(np.random.default_rng(3).standard_normal((nk, 2, mesh.N)) + 0j, device="cuda:0")
        sol.set_option("field.variant", 1)
        a = sol.eval_field(x, k, surf, B.BIE_MODE_MIXED)
        sol.set_option("field.variant", 2)
        assert torch.equal(a, sol.eval_field(x, k, surf, B.BIE_MODE_MIXED))
    sol.close()


def test_many_short_runs_take_bounded_scratch():
    """128 equally spaced runs of 4 wavenumbers: the scratch stays that of other lists of 512 (32 bytes a
    wavenumber and quadrature point, and the rest below 64 MB), and the values are the one-group kernel's."""
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B
    from workloads import ico_sphere

    mesh = ico_sphere(8)  # 20 480 quadrature points
    k = np.concatenate([i + 0.1 * np.arange(1, 5) for i in range(128)]) / 16
    x = torch.tensor(shell_points(40, 1.3, 3.0, seed=2), dtype=torch.float64, device="cuda:0")
    g = torch.Generator("cuda:0").manual_seed(1)
    surf = torch.randn((len(k), 2, mesh.N), dtype=torch.complex128, device="cuda:0", generator=g)
    out = torch.empty((len(k), 40), dtype=torch.complex128, device="cuda:0")
    sol = Solver(0)
    sol.set_geometry(mesh.nodes, mesh.elems, mesh.normals, mesh.bc)
    sol.eval_field(x, k[:4], surf[:4], B.BIE_MODE_MIXED)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sol.eval_field(x, k, surf, B.BIE_MODE_MIXED, out=out)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 32 * len(k) * 16 * mesh.elems.shape[0] + (64 << 20)
    sol.set_option("field.variant", 1)
    assert torch.equal(out, sol.eval_field(x, k, surf, B.BIE_MODE_MIXED))
    sol.close()
