"""FP64 factorisation whose bounded waits give up: every call on it returns BIE_ERR_TIMEOUT, with and without
reports, and the context solves as before once the waits have their limit again.  The waits are made to
give up on the host's word (a limit of no polls): the kernel then ends by its own error path."""
import numpy as np
import pytest

from workloads import ico_sphere, linear_from_quadratic, octa_sphere

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["solve", "multi", "linear"])
@pytest.mark.parametrize("reports", [True, False])
def test_a_wait_that_gives_up_is_an_error(call, reports):
    import torch
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    sol = Solver(0)
    if call == "linear":
        m = linear_from_quadratic(ico_sphere(5))  # 252 vertices
        sol.set_geometry_linear(m.nodes, m.elems, m.normals, m.bc)
    else:
        m = octa_sphere(2)
        sol.set_geometry(m.nodes, m.elems, m.normals, m.bc)
    ks = np.array([0.7, 1.1, 1.9])
    dirs = np.array([[0.0, 0.0, 1.0], [1.0, 0.0, 0.0]])
    nd = 2 if call == "multi" else 1
    surf = torch.zeros((len(ks), nd, 2, sol.N), dtype=torch.complex128, device="cuda:0")

    def go():
        if call == "multi":
            B.bie_solve_frequencies_multi(sol.ctx, ks, dirs, B.BIE_MODE_FP64, surf, reports=reports)
        else:
            B.bie_solve_frequencies(sol.ctx, ks, B.BIE_MODE_FP64, surf, reports=reports)
        return surf.clone()

    good = go()
    sol.set_option("fp64.wait_polls", 0)
    for _ in range(2):
        with pytest.raises(B.BieError) as e:
            go()
        assert e.value.code == B.BIE_ERR_TIMEOUT
    sol.set_option("fp64.wait_polls", 2 ** 22)
    assert torch.equal(go(), good)
    sol.close()


def test_limit_is_checked():
    from paper_1706_07919_gb300 import Solver
    from paper_1706_07919_gb300 import binding as B

    sol = Solver(0)
    for v in (-1, 2 ** 31):
        with pytest.raises(B.BieError) as e:
            sol.set_option("fp64.wait_polls", v)
        assert e.value.code == B.BIE_ERR_INVALID_ARG
    sol.close()
