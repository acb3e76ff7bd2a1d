"""Inputs that outgrow the scale predicted for them, for 1 to 8 and for more right-hand
sides.  The prediction takes the largest entry of the team's input before and of the
right-hand side on the next lines, with room for a growth by 2^7.  With large sources in
the upper front alone, the centre's input grows past that out of the upper front's
coupling: its entries take scales of their own, which the gather evens out.  The growth is
computed here from the oracle's own right-hand sides, so that the case is known to be one.

Tolerance: 1e-5 per right-hand side, the bound of every split FP16 apply of this size."""
import numpy as np
import pytest

from oracle.operator import Grid
from oracle.sweep import SweepPreconditioner
from paper_1502_07266_gb300 import workloads as W

torch = pytest.importorskip("torch")
N_, B_, AUX = 12, 3, 2


def problem(nrhs):
    c32 = W.velocity_random(N_, B_, seed=N_).astype(np.float32)
    f = W.random_rhs(nrhs, N_, B_, seed=nrhs + N_).astype(np.complex64)
    a = np.full((nrhs,) + f.shape[1:], 1e-6, np.float32)
    n = f.shape[1]
    for r in range(nrhs):                             # [right-hand side, layer, line, x]
        a[r, (2 + 3 * r) % n, n - 3 - r % 3, (1 + 5 * r) % n] = 1e3
    P = SweepPreconditioner(c32.astype(np.float64), Grid(N_, B_, W.omega_for(N_)), d=1, b_aux=AUX, schedule="two_front")
    return c32, f * a, P


def largest_growth(P, f):
    """Per right-hand side the largest factor by which an input exceeds what its scale is predicted from."""
    worst = np.zeros(f.shape[0])

    def biggest(v):
        return np.maximum(np.abs(v.real), np.abs(v.imag)).reshape(v.shape[0], -1).max(axis=1)

    def inner(M, g):
        probs, last, seen = P.slab_problems(M), {}, set()

        def solve(Mp, rhs):
            team = Mp > P.centre
            if team in last:
                m, e = P.blocks[Mp]
                base = last[team] if Mp in seen else np.maximum(last[team], biggest(g[:, :, m:e]))
                np.maximum(worst, biggest(rhs) / np.maximum(base, 1e-300), out=worst)
            last[team] = biggest(rhs)
            seen.add(Mp)
            return probs[Mp].restricted_apply(rhs)
        return P.sweep(solve, g, axis=2)
    P.inner_sweep = inner
    z = P.apply(f.astype(np.complex128))
    return worst, z


@pytest.mark.parametrize("nrhs", [5, 11])
def test_the_cases_grow(nrhs):
    _, f, P = problem(nrhs)
    assert largest_growth(P, f)[0].min() > 2.0 ** 9


@pytest.mark.gpu
@pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
@pytest.mark.parametrize("nrhs", [5, 11])
def test_growth(nrhs):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1502_07266_gb300 import helm
    c32, f, P = problem(nrhs)
    S = helm.Solver(torch.from_numpy(c32).cuda(), W.omega_for(N_), N_, B_, 1, b_aux=AUX, precision="split_fp16",
                    apply_form="dense", schedule="two_front")
    z = S.apply(torch.from_numpy(f).cuda()).cpu().numpy()
    assert S.status() == helm.HELM_OK
    S.close()
    growth, zo = largest_growth(P, f)
    assert growth.min() > 2.0 ** 9
    errs = [np.linalg.norm(z[r] - zo[r]) / np.linalg.norm(zo[r]) for r in range(nrhs)]
    assert max(errs) <= 1e-5, errs
