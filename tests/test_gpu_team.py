"""Team kernel of the dense form (tensor-core precisions) at the edges of its
layout, against the FP64 oracle's apply.

A group takes 8 right-hand sides, or 16 each when there are more than 8; a rank owns
groups of 8 columns and multiplies them in tiles of 4 or 8 groups; an input is
padded to a multiple of 16 entries.  The sizes below cross each edge: right-hand
sides 1, 8 | 9, 16 | 17, 33; few CTAs (several tiles a rank, several groups side by
side on one team's CTAs) and as many as the chip holds (some ranks own one group);
blocks of 1 and 2 lines; inputs that are and are not multiples of 16.

Tolerance: 1e-5 relative per right-hand side for split FP16 (operands of 22 bits,
relative rounding 2^-22 a product, sums in FP32 over the sweep's depth), 3e-3 for
FP16 operators (11 bits); the bounds every dense apply of this size meets.
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


def _errs(helm, n, b, d, schedule, nrhs, clusters, precision, shape=None):
    om = W.omega_for(n)
    c32 = W.velocity_random(n, b, seed=n).astype(np.float32)
    f = W.random_rhs(nrhs, n, b, seed=nrhs + n).astype(np.complex64)
    if shape is not None:
        f *= shape(f.shape[1])
    aux = {"b_aux": 2} if schedule == "two_front" else {}
    S = helm.Solver(torch.from_numpy(c32).cuda(), om, n, b, d, **aux, precision=precision, apply_form="dense",
                    schedule=schedule, dense_clusters=clusters)
    z = S.apply(torch.from_numpy(f).cuda()).cpu().numpy()
    assert S.status() == helm.HELM_OK
    S.close()
    P = SweepPreconditioner(c32.astype(np.float64), Grid(n, b, om), d=d, **aux, schedule=schedule)
    zo = P.apply(f.astype(np.complex128))
    return [np.linalg.norm(z[r] - zo[r]) / np.linalg.norm(zo[r]) for r in range(nrhs)]


@pytest.mark.parametrize("n,b,d,schedule,nrhs,clusters,precision", [
    (13, 3, 1, "two_front", 8, 0, "split_fp16"),
    (13, 3, 1, "two_front", 9, 0, "split_fp16"),
    (12, 2, 2, "two_front", 16, 1, "split_fp16"),
    (11, 3, 2, "two_front", 17, 2, "fp16"),
    (14, 4, 1, "one_front", 33, 1, "split_fp16"),
    (14, 2, 1, "one_front", 1, 1, "fp16"),
    (10, 2, 2, "one_front", 16, 0, "split_fp16"),
    (4, 2, 1, "two_front", 1, 0, "split_fp16"),
])
def test_edges(helm, n, b, d, schedule, nrhs, clusters, precision):
    errs = _errs(helm, n, b, d, schedule, nrhs, clusters, precision)
    assert max(errs) <= (1e-5 if precision == "split_fp16" else 3e-3), errs


@pytest.mark.parametrize("schedule,nrhs", [("one_front", 3), ("two_front", 9)])
def test_growth_past_the_predicted_scale(helm, schedule, nrhs):
    """The scale of an input is predicted from the one before with room for a growth by
    2^7.  Entries that grow by 1e9 from one column to the next, at another place for
    every right-hand side, take scales of their own, and the gather evens them out."""
    def shape(N):
        a = np.full((nrhs, N, N, N), 1e-6, np.float32)
        for r in range(nrhs):
            a[r, (2 + 3 * r) % N, (5 + 2 * r) % N, (1 + 5 * r) % N] = 1e3
        return a
    errs = _errs(helm, 12, 3, 1, schedule, nrhs, 0, "split_fp16", shape)
    assert max(errs) <= 1e-5, errs


def test_infinities_and_nans_stay_in_their_column(helm):
    """A right-hand side with an infinity and one with a NaN end, and leave the other
    columns of their group as they are without them."""
    n, b = 9, 3
    om = W.omega_for(n)
    c32 = W.velocity_random(n, b, seed=n).astype(np.float32)
    f = W.random_rhs(5, n, b, seed=5).astype(np.complex64)
    g = f.copy()
    g[1, 4, 5, 6] = np.inf
    g[3, 6, 5, 4] = np.nan
    S = helm.Solver(torch.from_numpy(c32).cuda(), om, n, b, 1, b_aux=2, precision="split_fp16", apply_form="dense",
                    schedule="two_front")
    z = S.apply(torch.from_numpy(f).cuda()).cpu().numpy()
    w = S.apply(torch.from_numpy(g).cuda()).cpu().numpy()
    assert S.status() == helm.HELM_OK
    S.close()
    for r in (0, 2, 4):
        assert np.array_equal(z[r], w[r])
    assert not np.isfinite(w[1]).all() and not np.isfinite(w[3]).all()


def test_repeated_applies_are_the_same_bits(helm):
    """Nothing in an apply depends on which rank or front is ahead: with sources of
    unequal size (the centre, the lower and the upper front see different scales) 40
    applies give the same bits."""
    n, b = 14, 3
    om = W.omega_for(n)
    c32 = W.velocity_random(n, b, seed=n).astype(np.float32)
    f = W.random_rhs(33, n, b, seed=8).astype(np.complex64)
    f *= np.exp(np.linspace(-9.0, 9.0, f.shape[2], dtype=np.float32))[None, None, :, None]
    S = helm.Solver(torch.from_numpy(c32).cuda(), om, n, b, 1, b_aux=2, precision="split_fp16", apply_form="dense",
                    schedule="two_front")
    ft = torch.from_numpy(f).cuda()
    z = S.apply(ft).clone()
    for _ in range(39):
        assert torch.equal(S.apply(ft), z)
    assert S.status() == helm.HELM_OK
    S.close()


@pytest.mark.parametrize("n,b,d,b_aux,schedule,nrhs,clusters,precision", [
    (14, 3, 2, 2, "two_front", 33, 0, "split_fp16"),    # two lines a block
    (13, 4, 2, 3, "one_front", 9, 0, "fp16"),
    (15, 4, 3, 2, "two_front", 5, 0, "split_fp16"),     # three, of which 8 is no multiple
    (33, 6, 2, 6, "one_front", 17, 1, "split_fp16"),    # inputs of several gathers, several tiles a rank
    (33, 6, 2, 6, "one_front", 3, 2, "fp16"),
    (16, 3, 1, 2, "two_front", 9, 1, "split_fp16"),     # one line a block, several tiles a rank
])
def test_every_path_repeats_its_bits(helm, n, b, d, b_aux, schedule, nrhs, clusters, precision):
    """20 applies of unequal sources give the same bits, and they are those of the FP32
    form up to the two forms' bounds (1e-5 each; 3e-3 with FP16 operators)."""
    om = W.omega_for(n)
    c = torch.from_numpy(W.velocity_random(n, b, seed=n).astype(np.float32)).cuda()
    f = W.random_rhs(nrhs, n, b, seed=8).astype(np.complex64)
    f *= np.exp(np.linspace(-4.0, 4.0, f.shape[2], dtype=np.float32))[None, None, :, None]
    ft = torch.from_numpy(f).cuda()
    S = helm.Solver(c, om, n, b, d, b_aux=b_aux, precision=precision, apply_form="dense", schedule=schedule,
                    dense_clusters=clusters)
    z = S.apply(ft).clone()
    for _ in range(19):
        assert torch.equal(S.apply(ft), z)
    assert S.status() == helm.HELM_OK
    S.close()
    S = helm.Solver(c, om, n, b, d, b_aux=b_aux, precision="fp32", apply_form="dense", schedule=schedule)
    w = S.apply(ft)
    S.close()
    err = torch.linalg.vector_norm((z - w).reshape(nrhs, -1), dim=1) / torch.linalg.vector_norm(w.reshape(nrhs, -1), dim=1)
    assert float(err.max()) <= (2e-5 if precision == "split_fp16" else 3e-3 + 1e-5), err
