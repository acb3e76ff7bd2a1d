"""Team apply with blocks of several lines and with several tiles a rank, against the
FP64 oracle, at the edges of its paths: 2 and 4 lines keep a column's lines in one
group of 8 rows, 3 and 5 do not; a centre block (one front: the last one) of as many lines
as the others, of fewer, and of more; one CTA a team (dense_clusters 1 leaves 8 CTAs:
several tiles a rank); 1, 8, 9 and 33 right-hand sides.

Tolerance: 1e-5 per right-hand side for split FP16, 3e-3 for FP16 operators, the bounds
every dense apply of this size meets; ten repeats give the same bits."""
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


@pytest.mark.parametrize("n,b,d,b_aux,schedule,nrhs,clusters,precision", [
    (16, 3, 2, 1, "two_front", 1, 0, "split_fp16"),
    (15, 2, 2, 2, "two_front", 33, 0, "fp16"),
    (14, 3, 2, 3, "one_front", 8, 0, "split_fp16"),     # the last block of one line
    (15, 4, 2, 3, "one_front", 9, 0, "split_fp16"),     # of two, like the others
    (20, 2, 4, 1, "two_front", 9, 0, "split_fp16"),
    (18, 2, 4, 2, "one_front", 5, 0, "split_fp16"),
    (31, 2, 5, 1, "two_front", 3, 0, "split_fp16"),
    (16, 3, 3, 2, "two_front", 9, 0, "split_fp16"),
    (22, 4, 2, 4, "one_front", 17, 1, "split_fp16"),    # several tiles and several gathers
    (22, 4, 2, 4, "one_front", 4, 1, "fp16"),
    (24, 3, 1, 3, "one_front", 33, 1, "split_fp16"),    # one line, several tiles
    (21, 3, 1, 2, "two_front", 6, 1, "fp16"),
])
def test_blocks(helm, n, b, d, b_aux, schedule, nrhs, clusters, precision):
    om = W.omega_for(n)
    c32 = W.velocity_random(n, b, seed=n).astype(np.float32)
    f = W.random_rhs(nrhs, n, b, seed=nrhs + n).astype(np.complex64)
    S = helm.Solver(torch.from_numpy(c32).cuda(), om, n, b, d, b_aux=b_aux, precision=precision, apply_form="dense",
                    schedule=schedule, dense_clusters=clusters)
    ft = torch.from_numpy(f).cuda()
    z = S.apply(ft).clone()
    for _ in range(10):
        assert torch.equal(S.apply(ft), z)
    assert S.status() == helm.HELM_OK
    S.close()
    P = SweepPreconditioner(c32.astype(np.float64), Grid(n, b, om), d=d, b_aux=b_aux, schedule=schedule)
    zo = P.apply(f.astype(np.complex128))
    z = z.cpu().numpy()
    errs = [np.linalg.norm(z[r] - zo[r]) / np.linalg.norm(zo[r]) for r in range(nrhs)]
    assert max(errs) <= (1e-5 if precision == "split_fp16" else 3e-3), errs
