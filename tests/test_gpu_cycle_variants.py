"""V-cycle kernels on both sides of the rule that lets them load ahead of their wait: one
batch of every direction (large launches, plain kernels) and one direction to a batch
(small launches, loads ahead) solve the same problem."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1910_11463_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pair():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1910_11463_gb300 import pair as P
    return P


# every solve ends at ||b - A psi|| <= inner_tol ||b||, so two of them differ by a small
# multiple of inner_tol however their sums are ordered
@pytest.mark.parametrize("mesh,n", [("hex", 20), ("tet", 12)])
@pytest.mark.parametrize("precision,inner_tol,tol", [(0, 1e-12, 1e-10), (1, 1e-10, 1e-8), (2, 1e-10, 1e-8)])
def test_batch_size_does_not_change_the_flux(pair, mesh, n, precision, inner_tol, tol):
    prob = I.small_hex(n, order=4, seed=3) if mesh == "hex" else I.small_tet(n, order=4, seed=3)
    air = pair.default_air_params(precision=precision, distance=1 if mesh == "hex" else 2, theta=0.5, phi_A=0.05)
    out = []
    for concurrent, batch in ((1, 0), (1, 1)):
        si = pair.default_si_params(max_iters=3, fixed_iters=1, inner_tol=inner_tol, concurrent=concurrent, batch=batch)
        phi, _, info = pair.si_solve_problem(prob, air=air, si=si)
        assert info["batches"] == (1 if batch == 0 else prob.M)
        out.append(phi.cpu().numpy())
    assert np.linalg.norm(out[0] - out[1]) <= tol * np.linalg.norm(out[0])
