"""FP16 form of the dense apply: rows that its tiles of 64 + 1 or 2 rows hold beyond 64
are kept to 22 bits, not 11.  With one cluster an operator of 65 or 66 rows is one such
tile.

Tolerance: hi + lo parts carry a value to 2^-22 of the row's scale (the lo part is
rounded to 11 bits of a remainder below 2^-11; the scale puts the row's largest entry
within a factor of two of it): 2^-20 of the row's largest real or imaginary part.  The
hi parts alone are within 2^-11 of an entry.  The apply keeps the form's 3e-3.
"""
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


@pytest.mark.parametrize("n,b,b_aux,rows", [(9, 2, 4, 65), (7, 2, 5, 66)])
def test_extra_rows_keep_their_bits(helm, n, b, b_aux, rows):
    om = W.omega_for(n)
    c = torch.from_numpy(W.velocity_random(n, b, seed=n).astype(np.float32)).cuda()
    N = n + 2 * b
    M = N - b - 1                                     # a block well inside, its window not cut
    G = {}
    for precision in ("fp16", "fp32"):
        S = helm.Solver(c, om, n, b, 1, b_aux=b_aux, precision=precision, apply_form="dense", dense_clusters=1)
        G[precision] = S.dense_operator(M, M)[0].to(torch.complex128)
        if precision == "fp16":
            f = W.random_rhs(9, n, b, seed=3).astype(np.complex64)
            z = S.apply(torch.from_numpy(f).cuda()).cpu().numpy()
            assert S.status() == helm.HELM_OK
        S.close()
    assert G["fp32"].shape[0] == rows
    w = torch.view_as_real(G["fp32"])
    d = torch.view_as_real(G["fp16"]) - w
    rel = d.abs().amax(1) / w.abs().amax(1)           # per row, real and imaginary part
    assert float(rel[64:].max()) <= 2.0 ** -20
    assert 2.0 ** -16 < float(rel[:64].max()) <= 2.0 ** -11
    P = SweepPreconditioner(c.double().cpu().numpy(), Grid(n, b, om), d=1, b_aux=b_aux)
    zo = P.apply(f.astype(np.complex128))
    err = np.linalg.norm((z - zo).reshape(9, -1), axis=1) / np.linalg.norm(zo.reshape(9, -1), axis=1)
    assert err.max() <= 3e-3, err
