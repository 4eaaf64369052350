"""GPU parity at the edges of the tiles and work splits of the hot path's kernels.

Each case sits where a tile, a column block or a dispatch rule changes: sizes one below, at and
one above the edge, and the smallest and largest of the range.  References and tolerances are
those of ``test_gpu_kernels.py``: the FP64 oracle on the same factors, 1e-5 for the FP32 kernels
and the Tucker tolerance 1e-6 for the three-term tensor-core chain, per output vector in l2 and
element-wise.
"""
import numpy as np
import pytest

from oracle import apply, hosvd
from paper_2103_05822_gb300.inputs import complex_gaussian, synthetic_tucker

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _problem(seed, nt, npf, nbetas, ranks, R, engine):
    from paper_2103_05822_gb300 import tfmm
    rng = np.random.default_rng(seed)
    syn = synthetic_tucker(nt, npf, nbetas, ranks, seed)
    n = sum(nbetas)
    members = np.split(rng.permutation(n), np.cumsum(nbetas)[:-1])  # members in no order
    T = [[hosvd.Tucker(s.U_theta, s.U_phi, s.U_beta, s.core) for s in per] for per in syn]
    factors = [[(t.U_theta, t.U_phi, t.U_beta, t.core) for t in per] for per in T]
    w = rng.uniform(0.05, 1.0, nt * npf)
    plan = tfmm.tfmm_plan_from_tucker(n, nt, npf, members, factors, weights=w, max_rhs=R, mrhs_precision=engine)
    return tfmm, plan, n, members, T, w


def _worst(got, ref):
    d = np.abs(got - ref)
    return max(np.linalg.norm(d) / np.linalg.norm(ref), d.max() / np.abs(ref).max())


def _check(seed, nt, npf, nbetas, ranks, R, engine, tol, pad=0, betas=(0.0, 0.5 - 0.25j)):
    """Aggregation, then disaggregation of other spectra into a y with `pad` untouched rows."""
    tfmm, plan, n, members, T, w = _problem(seed, nt, npf, nbetas, ranks, R, engine)
    G, nd, ld = len(nbetas), nt * npf, n + pad
    X = complex_gaussian((R, ld), seed + 1).astype(np.complex64)
    spec = torch.full((R, G, 2, nd), float("nan"), dtype=torch.complex64, device="cuda")
    tfmm.tfmm_aggregate(plan, torch.from_numpy(X).cuda(), spec, R=R, ldx=ld)
    S = spec.cpu().numpy()
    g_in = complex_gaussian((R, G, 2, nd), seed + 2).astype(np.complex64)
    for beta in betas:
        y0 = complex_gaussian((R, ld), seed + 3).astype(np.complex64)
        if beta == 0:
            y0[:, :n] = np.nan  # beta = 0 overwrites
        y = torch.from_numpy(y0).cuda()
        tfmm.tfmm_disaggregate(plan, torch.from_numpy(g_in).cuda(), y, R=R, ldy=ld, beta=beta)
        Y = y.cpu().numpy()
        assert np.array_equal(Y[:, n:], y0[:, n:])
        for r in range(R):
            ref = apply.disaggregate_all(T, members, g_in[r].astype(np.complex128), n, w, beta=beta,
                                         y0=y0[r, :n].astype(np.complex128) if beta else None)
            for ids in members:
                assert _worst(Y[r, ids], ref[ids]) <= tol, (r, beta, len(ids))
    for r in range(R):
        ref = apply.aggregate_all(T, members, X[r, :n].astype(np.complex128))
        for g in range(G):
            for a in range(2):
                assert _worst(S[r, g, a], ref[g, a]) <= tol, (r, g, a)
    tfmm.tfmm_sync(plan)


@pytest.mark.parametrize("R", [2, 4, 5])
def test_gather_and_order_kernels_at_their_tile_edges(R):
    """512 members and 4 columns per block: groups of 511, 512, 513 and 1025, R around 4."""
    nbetas = [9, 511, 512, 513, 1025]
    ranks = [[(5, 6, min(nb, 20))] * 2 for nb in nbetas]
    _check(2100 + R, 9, 18, nbetas, ranks, R, 3, 1e-6, pad=3)
