"""GPU parity at the edges of the tiles and work splits of the hot path's kernels.

Each case sits where a tile, a column block or a dispatch rule changes: sizes one below, at and
one above the edge, and the smallest and largest of the range.  References and tolerances are
those of ``test_gpu_kernels.py``: the FP64 oracle on the same factors, 1e-5 for the FP32 kernels
and the Tucker tolerance 1e-6 for the three-term tensor-core chain, per output vector in l2 and
element-wise.
"""
import math

import numpy as np
import pytest

import oracle
from oracle import apply, hosvd, translation
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


# box counts (K_x, K_y, K_z): 2K - 1 below, at and above the sides the one-CTA transforms take
# (4 ... 36), cubes that are not full, a plate and a side past the last (cuFFT)
@pytest.mark.parametrize("K", [(1, 1, 1), (2, 2, 2), (3, 3, 3), (4, 4, 4), (5, 4, 5), (6, 6, 6), (8, 8, 8), (9, 8, 7),
                               (9, 9, 9), (10, 10, 10), (12, 12, 12), (13, 13, 13), (15, 15, 15), (16, 15, 14),
                               (18, 18, 18), (12, 12, 1), (19, 19, 19)])
def test_translation_over_box_grids(K):
    """Incoming spectra against the oracle's direct sums, one small patch (one RWG) per occupied box."""
    from paper_2103_05822_gb300 import tfmm
    box, rng = 0.5, np.random.default_rng(sum(K))
    cells = np.unique(np.vstack([[0, 0, 0], np.array(K) - 1, rng.integers(0, K, (12, 3))]), axis=0)
    mid = box * (cells + 0.25 + 0.5 * rng.uniform(0.1, 1.0, (len(cells), 3)))
    mid[0] = 0.25 * box  # the lowest corner anchors the grid
    v, f = [], []
    for m in mid:
        f += [[len(v), len(v) + 1, len(v) + 2], [len(v) + 1, len(v), len(v) + 3]]
        v += [m - [0.02, 0, 0], m + [0.02, 0, 0], m + [0, 0.03, 0], m + [0, -0.02, 0.02]]
    v, f = np.array(v), np.array(f)
    P = oracle.problem.build(v, f, k=2 * math.pi, box=box, digits=1, tol=1e-2, compress=False)
    prm = tfmm.tfmm_params_default(box=box, digits=1.0, tol=1e-2, max_rhs=2)
    plan = tfmm.tfmm_plan_create(tfmm.tfmm_mesh_create(v, f), prm)
    assert plan.info["K"] == list(K) and plan.info["n_groups"] == len(cells) == P.groups.n_groups
    G, nd = len(cells), P.grid.n_dir
    F = complex_gaussian((2, G, 2, nd), 5).astype(np.complex64)
    out = torch.full((2, G, 2, nd), float("nan"), dtype=torch.complex64, device="cuda")
    tfmm.tfmm_translate(plan, torch.from_numpy(F).cuda(), out)
    got = out.cpu().numpy()
    for r in range(2):
        ref = translation.translate(F[r].astype(np.complex128), P.groups, P.grid, P.k)
        top = np.abs(ref).max()
        if max(K) < 3:
            assert top == 0 and np.abs(got[r]).max() <= 1e-6 * np.abs(F[r]).max()  # touching boxes only
        else:
            assert np.linalg.norm(got[r] - ref) <= 1e-5 * np.linalg.norm(ref)
            assert np.abs(got[r] - ref).max() <= 1e-5 * top


@pytest.mark.parametrize("order", [1, 2, 5, 10])
@pytest.mark.parametrize("nu,R", [(2, 65), (3, 64), (4, 1), (7, 130)])
def test_planewave_expansion_and_its_limit(nu, R, order):
    """V against the same rule point by point in FP64: meshes whose triangles all, partly or never
    spread the phase past the expansion's limit, low and high rules, R around the 64 incidences of a
    block.  Bound: rounding V to FP32 (6e-8 an entry) and half as much again for the expansion."""
    from paper_2103_05822_gb300 import tfmm
    from paper_2103_05822_gb300.inputs import icosphere
    v, f = icosphere(1.0, nu, center=(3.0, -2.0, 11.0))
    mesh = tfmm.tfmm_mesh_create(v, f)
    plan = tfmm.tfmm_plan_create(mesh, tfmm.tfmm_params_default(box=0.5, digits=1.0, tol=1e-2, quad_order=order))
    edge, _, free = tfmm.tfmm_mesh_rwg(mesh)
    rng = np.random.default_rng(order)
    kh = rng.standard_normal((R, 3))
    kh /= np.linalg.norm(kh, axis=1)[:, None]
    pol = np.cross(kh, rng.standard_normal((R, 3)))
    V = torch.full((R, len(edge)), float("nan"), dtype=torch.complex64, device="cuda")
    tfmm.tfmm_planewave(plan, kh, pol, V)
    x, w = np.polynomial.legendre.leggauss(order)
    u, w = 0.5 * (x + 1), 0.5 * w
    q1, q2 = v[edge[:, 0]], v[edge[:, 1]]
    length = np.linalg.norm(q1 - q2, axis=1)
    ref = np.zeros((R, len(edge)), complex)
    for side, sign in ((0, 1.0), (1, -1.0)):
        p = v[free[:, side]]
        for a in range(order):
            for b in range(order):
                rho = u[a] * (q1 - p) + u[b] * (1 - u[a]) * (q2 - p)
                amp = sign * w[a] * w[b] * (1 - u[a]) * length[:, None] * rho
                ref -= (pol @ amp.T) * np.exp(-2j * math.pi * (kh @ (p + rho).T))
    got = V.cpu().numpy()
    assert np.linalg.norm(got - ref) <= 9e-8 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 9e-8 * np.abs(ref).max()


def _small_ranks(rng, nt, npf, nb, top):
    return [(int(rng.integers(1, nt + 1)), int(rng.integers(1, npf + 1)), int(rng.integers(1, min(nb, top) + 1)))
            for _ in range(2)]


@pytest.mark.parametrize("R", [1, 2, 5, 16, 17, 33])
@pytest.mark.parametrize("nt,npf", [(5, 10), (8, 15), (14, 28)])
def test_small_groups_in_shared_memory(nt, npf, R):
    """Everything of a group in one CTA: column blocks of 1, 4, 8 and 16 and what is left of them, full and
    rank-1 factors, odd and even sizes, the bank padding's steps."""
    rng = np.random.default_rng(31 * nt + R)
    nbetas = [2, 3, 8, 15, 16, 31, 64, 65, 100]
    ranks = [_small_ranks(rng, nt, npf, nb, 30) for nb in nbetas]
    ranks[1], ranks[3] = [(1, 1, 1), (nt, 1, 2)], [(nt, npf, 15), (1, npf, 1)]
    _check(3000 + 40 * nt + R, nt, npf, nbetas, ranks, R, 0, 1e-5, pad=2)


@pytest.mark.parametrize("R", [1, 6])
def test_small_groups_by_size_class(R):
    """Enough groups for several launches by size (four per SM)."""
    rng = np.random.default_rng(77)
    G = 4 * torch.cuda.get_device_properties(0).multi_processor_count + 3
    nbetas = [int(n) for n in rng.integers(2, 40, G)]
    ranks = [_small_ranks(rng, 4, 8, nb, 12) for nb in nbetas]
    _check(3700 + R, 4, 8, nbetas, ranks, R, 0, 1e-5, betas=(0.5 - 0.25j,))


@pytest.mark.parametrize("R", [16, 17, 40, 48, 80, 81, 129])
def test_stage_kernel_forms(R):
    """Stacked products with two accumulator copies, one, and products one by one; a second column tile;
    K of one step, one and two k-tiles, odd r_phi, rows around 128."""
    nbetas = [15, 33, 64, 127, 129, 300]
    ranks = [[(5, 7, 15), (3, 5, 14)], [(8, 16, 33), (1, 1, 1)], [(9, 13, 64), (6, 3, 31)],
             [(12, 11, 127), (12, 10, 96)], [(12, 22, 129), (2, 2, 4)], [(11, 19, 200), (10, 20, 128)]]
    _check(4000 + R, 12, 24, nbetas, ranks, R, 3, 1e-6, betas=(0.5 - 0.25j,))


@pytest.mark.parametrize("R", [2, 9])
@pytest.mark.parametrize("nt,npf,top", [(16, 31, (16, 31)), (17, 32, (17, 30)), (32, 64, (32, 48)), (33, 48, (32, 40)),
                                        (33, 66, (33, 49)), (40, 75, (9, 49))])
def test_disaggregation_first_step_forms(nt, npf, top, R):
    """Tiles of 16 and 32 directions and ranks past both (the separate kernels), n_theta odd, below and above
    a slab's 16, n_phi off the tiles, r_phi around the 32 columns held in registers and 48."""
    rt, rp = top
    nbetas = [40, 120, 90]
    ranks = [[(rt, rp, 24), (max(1, rt - 1), max(1, rp - 1), 20)], [(rt, min(rp, 33), 100), (max(1, rt // 2), rp, 9)],
             [(max(1, rt - 3), min(rp, 8), 64), (rt, max(1, rp // 2), 90)]]
    _check(5000 + 10 * nt + R, nt, npf, nbetas, ranks, R, 3, 1e-6, betas=(0.5 - 0.25j,))


@pytest.mark.parametrize("threads", [64, 256, 512])
def test_persistent_row_groups(threads, monkeypatch):
    """Rows taken four, two and one at a time by 2, 8 and 16 warps, row lengths around 64 and 128
    complex numbers, core columns split into slices and not."""
    from paper_2103_05822_gb300 import tfmm
    made = tfmm.tfmm_plan_from_tucker

    def persistent(*args, **kw):
        plan = made(*args, **kw)
        tfmm.tfmm_plan_tuning_set(plan, agg_threads=threads, dis_threads=threads, single_rhs_split=2)
        return plan

    monkeypatch.setattr(tfmm, "tfmm_plan_from_tucker", persistent)
    nbetas = [8, 63, 64, 66, 127, 130, 260, 515]
    rb = [2, 15, 16, 17, 47, 64, 65, 130]
    ranks = [[(5, 4, r), (7, 13, max(2, r - 1))] for r in rb]
    _check(6000 + threads, 10, 20, nbetas, ranks, 1, 0, 1e-5, pad=1)


@pytest.mark.parametrize("split", [0, 1])
def test_split_path_blocks(split):
    """Blocks of phi directions and of U_phi's columns with remainders; with `split` 0 the items are too
    large for the persistent kernels' shared memory, so that the split path takes them by itself."""
    from paper_2103_05822_gb300 import tfmm
    nbetas = [9, 700, 12000] if split == 0 else [9, 33, 700]
    nt, npf = (66, 131) if split == 0 else (11, 23)
    top = [(5, 7, 9), (20, 41, 30), (11, 40, 17)] if split == 0 else [(3, 5, 9), (11, 23, 33), (7, 10, 65)]
    ranks = [[r, (max(1, r[0] - 2), max(1, r[1] - 3), r[2])] for r in top]
    made, seen = tfmm.tfmm_plan_from_tucker, []

    def tuned(*args, **kw):
        plan = made(*args, **kw)
        if split:
            tfmm.tfmm_plan_tuning_set(plan, single_rhs_split=1)
        seen.append(tfmm.tfmm_plan_tuning_get(plan)["dis_blocks"])
        return plan

    tfmm.tfmm_plan_from_tucker = tuned
    try:
        _check(7000 + split, nt, npf, nbetas, ranks, 1, 0, 1e-5, pad=1)
    finally:
        tfmm.tfmm_plan_from_tucker = made
    assert (seen[0] == 0) == (split == 0)


@pytest.mark.parametrize("R", [2, 4, 5, 16, 17, 32, 33, 64, 65])
def test_fp32_chain_tile_shapes_and_few_columns(R):
    """FP32 engine on groups too large for one CTA's shared memory: the columns' single-RHS kernels up to
    four right-hand sides, then the chain with 64- and 32-row tiles of 64, 32 and 16 columns."""
    nbetas = [63, 520, 130, 31]
    ranks = [[(5, 4, 15), (16, 24, 16)], [(16, 24, 150), (17, 33, 65)], [(9, 17, 33), (3, 2, 64)], [(4, 8, 17), (2, 3, 6)]]
    _check(8000 + R, 24, 48, nbetas, ranks, R, 0, 1e-5, pad=1)


@pytest.mark.parametrize("R", [2, 5, 19])
@pytest.mark.parametrize("nt,npf,top", [(13, 25, (13, 14)), (13, 26, (12, 16)), (16, 32, (15, 18)), (20, 33, (16, 17)),
                                        (24, 48, (17, 33)), (26, 52, (18, 30)), (40, 80, (33, 15)), (64, 128, (20, 15))])
def test_aggregation_last_steps_forms(nt, npf, top, R):
    """Odd and even N_theta by the powers of two in it (the order in which rows are staged), spectra of odd and
    even length, one and two staging buffers, K steps that only the larger item has, the most lanes."""
    rt, rp = top
    nbetas = [140, 60]
    ranks = [[(rt, rp, 70), (rt - 1, rp - 5, 40)], [(5, 7, 30), (rt, 4, 25)]]
    _check(9000 + nt + R, nt, npf, nbetas, ranks, R, 3, 1e-6, pad=1)


@pytest.mark.parametrize("rb", [60, 100, 160])
def test_split_by_stage(rb):
    """Largest items of 0.4, 0.7 and 1.1 MB: no stage split, the disaggregation only, both."""
    _check(9500 + rb, 20, 40, [600, 333], [[(14, 16, rb), (9, 11, 50)], [(12, 13, rb - 1), (5, 6, 25)]], 1, 0, 1e-5, pad=1)


@pytest.mark.parametrize("per_sm", [(1, 2), (2, 3), (1, 1), (1, 1, 1)])
def test_split_path_parts_by_item_count(per_sm, monkeypatch):
    """Items for four, three, two and one part of the theta / phi steps (one: whole items, larger register
    tiles), column tiles of the second step up to and past three to an SM (four and two loads in flight)."""
    from paper_2103_05822_gb300 import tfmm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    items = {(1, 2): sms // 2, (2, 3): 2 * sms // 3, (1, 1): sms, (1, 1, 1): sms + 2}[per_sm]
    made = tfmm.tfmm_plan_from_tucker

    def split(*args, **kw):
        plan = made(*args, **kw)
        tfmm.tfmm_plan_tuning_set(plan, single_rhs_split=1)
        return plan

    monkeypatch.setattr(tfmm, "tfmm_plan_from_tucker", split)
    rng = np.random.default_rng(items)
    nbetas = [int(n) for n in rng.integers(18, 60, items // 2)]
    ranks = [[(12, 23, int(rng.integers(1, 18))), (12, int(rng.integers(22, 24)), 17)] for _ in nbetas]
    _check(9700 + items, 13, 26, nbetas, ranks, 1, 0, 1e-5, pad=1)


@pytest.mark.parametrize("threads", [0, 512])
def test_between_two_and_three_groups_per_sm(threads, monkeypatch):
    """All groups at once on three CTAs an SM: of 320 threads (the default for small items), and of 512 in the
    form with fewer registers."""
    from paper_2103_05822_gb300 import tfmm
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    made = tfmm.tfmm_plan_from_tucker

    def persistent(*args, **kw):
        plan = made(*args, **kw)
        tfmm.tfmm_plan_tuning_set(plan, single_rhs_split=2, **({"dis_threads": threads} if threads else {}))
        t = tfmm.tfmm_plan_tuning_get(plan)
        assert t["dis_threads"] == (threads or 320) and t["dis_blocks"] == 2 * sms + 6
        return plan

    monkeypatch.setattr(tfmm, "tfmm_plan_from_tucker", persistent)
    rng = np.random.default_rng(41)
    nbetas = [int(n) for n in rng.integers(60, 68, 2 * sms + 6)]  # even enough for three (uneven groups run on two)
    ranks = [[(9, 17 + i % 2, 57 + i % 3), (8 + i % 2, 18, 59)] for i in range(len(nbetas))]
    _check(9800 + threads, 9, 18, nbetas, ranks, 1, 0, 1e-5, pad=1)
