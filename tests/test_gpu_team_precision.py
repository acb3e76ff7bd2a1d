"""Error of the tensor-core dense apply against the FP64 oracle where an input is
short.  The tensor core's additions do not round to nearest, so the error grows with the
number of products that go into one accumulator; an input of few 16-entry steps must not
go into few accumulators.

Tolerance: the error that an apply had on the same inputs with every input split into
eight partial sums, joined in rounded FP32 (measured, see each case)."""
import numpy as np
import pytest

from oracle.operator import Grid
from oracle.sweep import SweepPreconditioner
from paper_1502_07266_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.fixture(scope="module")
def helm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1502_07266_gb300 import helm as H
    return H


@pytest.mark.parametrize("n,b,d,b_aux,schedule,nrhs,bound", [
    (33, 4, 1, 1, "two_front", 9, 5.7e-6),            # inputs of 6 steps: measured 5.69e-6
    (27, 6, 1, 1, "two_front", 16, 5.3e-6),           # 5: 5.25e-6
    (20, 5, 1, 5, "one_front", 9, 3.75e-6),           # 12: 3.71e-6
])
def test_error_of_short_inputs(helm, n, b, d, b_aux, schedule, nrhs, bound):
    om = W.omega_for(n)
    c32 = W.velocity_random(n, b, seed=n).astype(np.float32)
    f = W.random_rhs(nrhs, n, b, seed=nrhs + n).astype(np.complex64)
    S = helm.Solver(torch.from_numpy(c32).cuda(), om, n, b, d, b_aux=b_aux, precision="split_fp16", apply_form="dense",
                    schedule=schedule)
    z = S.apply(torch.from_numpy(f).cuda()).cpu().numpy()
    assert S.status() == helm.HELM_OK
    S.close()
    P = SweepPreconditioner(c32.astype(np.float64), Grid(n, b, om), d=d, b_aux=b_aux, schedule=schedule)
    zo = P.apply(f.astype(np.complex128))
    err = np.linalg.norm(z - zo) / np.linalg.norm(zo)
    assert err <= bound, err
