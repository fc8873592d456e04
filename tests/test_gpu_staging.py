"""The hyper-power Horner steps of the tensor-core preconditioners, which write the next fast
diagonalisation's staging copy (csrc/k_mma.cu, k_pad_rows), against the FP64 recursion."""
import numpy as np
import pytest

from paper_2311_06926_gb300 import Stokes, synthetic

from gpu_common import dev, host, reduced_tol, relerr

pytestmark = pytest.mark.gpu


# rows of 31..33 and of 160..162 entries (a lane's last and first entry of a step), of 2; orders
# whose last step is the first, second and third; several items per launch
@pytest.mark.parametrize("prec", ["tf32", "bf16"])
@pytest.mark.parametrize("n,p,q,s,nrhs", [(2, 1, 2, 1, 1), (30, 2, 2, 1, 1), (31, 2, 3, 1, 3),
                                          (32, 1, 4, 1, 1), (13, 3, 2, 2, 2), (13, 3, 3, 2, 1),
                                          (159, 2, 3, 1, 1), (161, 1, 2, 1, 1)])
def test_staged_horner_steps(prec, n, p, q, s, nrhs):
    """Bound: reduced_tol, for the velocities and the pressure each."""
    if prec == "bf16" and n > 150:
        pytest.skip("rows of this length are covered by tf32")
    G64 = Stokes(n, p, max_order=q, max_steps=s, autotune=False)
    X = np.concatenate([synthetic.random_vector(G64.size, 30 + n + k) for k in range(nrhs)])
    ref = [host(G64.apply_hyperpower(q, s, dev(x))) for x in np.split(X, nrhs)]
    nv = G64.n_vel
    G64.close()
    G = Stokes(n, p, precision=prec, nrhs=nrhs, max_order=q, max_steps=s, autotune=False)
    got = np.split(host(G.apply_hyperpower(q, s, dev(X))), nrhs)
    tol = reduced_tol(prec, s, n + p, order=q)
    for g, r in zip(got, ref):
        assert relerr(g[:nv], r[:nv]) < tol
        assert relerr(g[nv:], r[nv:]) < tol
    G.close()
