"""What one call, one plan or one refused request leaves behind for the next, on the GPU.

Scratch planes, launch limits and launch shapes outlive a call: each test makes a call that could
disturb them and compares what follows with the same call on its own, bit for bit where the same
kernels run.  Oracle bounds are those of ``test_gpu_kernels.py``.
"""
import numpy as np
import pytest

from oracle import apply
from paper_2103_05822_gb300.inputs import complex_gaussian
from test_gpu_edges import _problem, _worst

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _inputs(plan, R, seed):
    i = plan.info
    x = torch.from_numpy(complex_gaussian((R, i["n_rwg"]), seed).astype(np.complex64)).cuda()
    g = torch.from_numpy(complex_gaussian((R, i["n_groups"], 2, i["n_dir"]), seed + 1).astype(np.complex64)).cuda()
    return x, g


def _agg(tfmm, plan, x):
    i = plan.info
    spec = torch.full((len(x), i["n_groups"], 2, i["n_dir"]), float("nan"), dtype=torch.complex64, device="cuda")
    tfmm.tfmm_aggregate(plan, x, spec, R=len(x))
    return spec


def _dis(tfmm, plan, g):
    y = torch.full((len(g), plan.info["n_rwg"]), float("nan"), dtype=torch.complex64, device="cuda")
    tfmm.tfmm_disaggregate(plan, g, y, R=len(g))
    return y


# (n_theta, n_phi, rank): fused AG3 + AG4 and DG1a + DG1b; n_phi past the fused AG3 + AG4's lanes; r_theta past
# the fused DG1 and n_phi past the stacked DG1b; the stacked DG1b with odd n_phi
@pytest.mark.parametrize("nt,npf,rank", [(12, 25, (5, 9, 20)), (66, 131, (5, 9, 20)), (66, 131, (33, 9, 20)),
                                         (40, 75, (33, 17, 30))])
@pytest.mark.parametrize("terms", [2, 3])
def test_non_finite_data_does_not_outlive_its_call(nt, npf, rank, terms):
    """The planes of the two stages share buffers in different layouts, so that one stage's values lie in the
    padding of the other's: after a call on NaN, calls on finite data give what they gave before."""
    nbetas = [40, 33]
    tfmm, plan, *_ = _problem(41, nt, npf, nbetas, [[rank, (3, 5, 9)], [(2, 3, 7), rank]], 3, terms)
    x, g = _inputs(plan, 3, 42)
    spec, y = _agg(tfmm, plan, x), _dis(tfmm, plan, g)
    assert torch.isfinite(torch.view_as_real(spec)).all() and torch.isfinite(torch.view_as_real(y)).all()
    _dis(tfmm, plan, torch.full_like(g, float("nan")))
    assert torch.equal(_agg(tfmm, plan, x), spec)
    _agg(tfmm, plan, torch.full_like(x, float("nan")))
    assert torch.equal(_dis(tfmm, plan, g), y)
    tfmm.tfmm_sync(plan)


@pytest.mark.parametrize("split", [1, 2])
def test_a_smaller_plan_leaves_a_larger_ones_launches_alone(split):
    """A kernel's shared-memory limit is one for all plans: one of 136 KB runs on after one of 72 KB was made."""
    def make(nb, seed):
        tfmm, plan, n, members, T, w = _problem(seed, 6, 12, [nb, 40], [[(3, 4, 9)] * 2] * 2, 1, 0)
        tfmm.tfmm_plan_tuning_set(plan, single_rhs_split=split)
        return tfmm, plan, n, members, T, w

    tfmm, large, n, members, T, w = make(16000, 51)
    small = make(8000, 53)[1]
    x, g = _inputs(large, 1, 54)
    spec, y = _agg(tfmm, large, x).cpu().numpy()[0], _dis(tfmm, large, g).cpu().numpy()[0]
    ref = apply.aggregate_all(T, members, x.cpu().numpy()[0].astype(np.complex128))
    for i in range(2):
        for a in range(2):
            assert _worst(spec[i, a], ref[i, a]) <= 1e-5
    assert _worst(y, apply.disaggregate_all(T, members, g.cpu().numpy()[0].astype(np.complex128), n, w)) <= 1e-5
    del small


def test_more_columns_than_one_launch_of_the_gather_takes():
    """262,148 columns on the tensor cores: past 65,535 blocks of four."""
    R = 4 * 65535 + 8
    tfmm, plan, n, members, T, w = _problem(61, 3, 5, [6], [[(2, 3, 4), (3, 2, 5)]], R, 3)
    i = plan.info
    few = complex_gaussian((7, n), 62).astype(np.complex64)
    g7 = complex_gaussian((7, 1, 2, i["n_dir"]), 63).astype(np.complex64)
    spec = _agg(tfmm, plan, torch.from_numpy(np.resize(few, (R, n))).cuda()).cpu().numpy()
    y = _dis(tfmm, plan, torch.from_numpy(np.resize(g7, (R, 1, 2, i["n_dir"]))).cuda()).cpu().numpy()
    for r in range(7):
        ref = apply.aggregate_all(T, members, few[r].astype(np.complex128))
        assert max(_worst(spec[r, 0, a], ref[0, a]) for a in range(2)) <= 1e-6
        assert _worst(y[r], apply.disaggregate_all(T, members, g7[r].astype(np.complex128), n, w)) <= 1e-6
        assert (spec[r::7] == spec[r]).all() and (y[r::7] == y[r]).all()


def _large_item_plan(threads=64):
    """One group whose items fit the persistent kernels with 64 threads a CTA and not with 512 (their scratch),
    and of less bytes than the automatic choice splits."""
    tfmm, plan, *_ = _problem(71, 3, 6, [28500], [[(1, 1, 1)] * 2], 1, 0)
    assert tfmm.tfmm_plan_tuning_get(plan)["dis_blocks"] == 0
    tfmm.tfmm_plan_tuning_set(plan, agg_threads=threads, dis_threads=threads, single_rhs_split=0)
    assert tfmm.tfmm_plan_tuning_get(plan)["dis_blocks"] > 0
    return tfmm, plan


@pytest.mark.parametrize("change", [{"agg_threads": 512}, {"dis_threads": 512}, {"single_rhs_split": 1},
                                    {"single_rhs_split": 1, "mrhs_precision": 3},
                                    {"agg_threads": 96, "tc_dg1a_pairs": 64}])
@pytest.mark.parametrize("graph", [True, False])
def test_a_refused_tuning_changes_nothing(change, graph):
    tfmm, plan = _large_item_plan()
    x, g = _inputs(plan, 1, 72)
    spec, y = _agg(tfmm, plan, x), _dis(tfmm, plan, g)
    before = tfmm.tfmm_plan_tuning_get(plan)
    if graph:
        out = torch.zeros_like(spec)
        held = tfmm.tfmm_graph_capture(plan, 1, out, x=x)
    elif 512 not in change.values():
        return  # only a graph that is still held forbids the others
    with pytest.raises(tfmm.TfmmError) as e:
        tfmm.tfmm_plan_tuning_set(plan, **change)
    assert e.value.status == tfmm.INVALID_ARG
    assert tfmm.tfmm_plan_tuning_get(plan) == before
    assert torch.equal(_agg(tfmm, plan, x), spec) and torch.equal(_dis(tfmm, plan, g), y)
    if graph:
        out.zero_()
        held.launch()
        torch.cuda.synchronize()
        assert torch.equal(out, spec)
        tfmm.tfmm_graph_destroy(held)


def test_autotuning_beside_a_graph_skips_shapes_without_room():
    tfmm, plan = _large_item_plan()
    x, g = _inputs(plan, 1, 73)
    spec = _agg(tfmm, plan, x)
    out = torch.zeros_like(spec)
    held = tfmm.tfmm_graph_capture(plan, 1, out, x=x)
    t = tfmm.tfmm_autotune(plan, R=1, budget_ms=500.0)
    assert t["agg_blocks"] > 0 and t["dis_blocks"] > 0 and t["single_rhs_split"] == 0
    _agg(tfmm, plan, x), _dis(tfmm, plan, g)
    held.launch()
    torch.cuda.synchronize()
    assert torch.equal(out, spec)
    tfmm.tfmm_graph_destroy(held)


@pytest.mark.parametrize("G,nb", [(3, 60), (400, 24), (3, 2500)])
def test_one_column_after_another_gives_the_bits_of_one_column_calls(G, nb):
    """mrhs_precision 1 on groups that fit one CTA's shared memory, few (one launch a column there) and many
    (the persistent kernels), and on groups that do not."""
    rng = np.random.default_rng(81)
    ranks = [[(5, 7, min(nb, 20)), (4, 9, min(nb, 17))] for _ in range(G)]
    nbetas = [int(v) for v in rng.integers(max(1, nb - 3), nb + 1, G)]
    ranks = [[(a, b, min(c, n)) for a, b, c in r] for r, n in zip(ranks, nbetas)]
    tfmm, plan, *_ = _problem(82, 10, 21, nbetas, ranks, 5, 1)
    x, g = _inputs(plan, 5, 83)
    spec, y = _agg(tfmm, plan, x), _dis(tfmm, plan, g)
    for r in range(5):
        assert torch.equal(spec[r], _agg(tfmm, plan, x[r:r + 1])[0])
        assert torch.equal(y[r], _dis(tfmm, plan, g[r:r + 1])[0])


@pytest.mark.parametrize("nt,npf,nbetas,rank,R,stages", [
    (17, 34, [70, 70, 66], (14, 19, 66), 6, "d"),    # one column a pass in the disaggregation: the chain
    (17, 34, [70, 70, 66], (14, 19, 66), 3, "d"),    # the same, few columns: the persistent kernels
    (14, 28, [60, 55, 31], (9, 13, 31), 64, "ad"),   # many columns for three groups' CTAs: the chain
])
def test_small_groups_leave_what_others_do_faster(nt, npf, nbetas, rank, R, stages):
    """The stages that take the kernels of single_rhs_split 2 (never the small-group ones) have their bits."""
    tfmm, plan, *_ = _problem(91, nt, npf, nbetas, [[rank, (3, 5, 9)]] * 3, R, 0)
    x, g = _inputs(plan, R, 92)
    spec, y = _agg(tfmm, plan, x), _dis(tfmm, plan, g)
    tfmm.tfmm_plan_tuning_set(plan, single_rhs_split=2)
    assert torch.equal(_agg(tfmm, plan, x), spec) == ("a" in stages)
    assert torch.equal(_dis(tfmm, plan, g), y) == ("d" in stages)


@pytest.mark.parametrize("kernels", ["small", "split"])
def test_autotuning_leaves_a_launch_shape_alone_that_does_not_run(kernels):
    """One column on the small-group kernels or the split path: their time is reported and the persistent
    kernels' shape, which nothing was measured with, stays."""
    nbetas = [60, 50] if kernels == "small" else [2500, 900]
    rank = (5, 7, 20) if kernels == "small" else (20, 30, 120)
    tfmm, plan, *_ = _problem(95, 21, 42, nbetas, [[rank, rank]] * 2, 1, 0)
    shape = ("agg_threads", "agg_ctas_per_sm", "agg_order", "dis_threads", "dis_ctas_per_sm", "dis_order")
    for threads in (96, 448):
        tfmm.tfmm_plan_tuning_set(plan, agg_threads=threads, dis_threads=threads)
        before = tfmm.tfmm_plan_tuning_get(plan)
        t = tfmm.tfmm_autotune(plan, R=1, budget_ms=300.0)
        assert [t[k] for k in shape] == [before[k] for k in shape]
        assert 0 < t["agg_ms"] < 10 and 0 < t["dis_ms"] < 10


def test_planewave_call_does_not_pay_for_the_rules_moments():
    """The allocation-free entry point only queues work: its host time at 100 points a triangle is that at one
    point and the rule itself (7 us; the moments, if computed in the call, take 250)."""
    import time
    from paper_2103_05822_gb300 import tfmm
    from paper_2103_05822_gb300.inputs import icosphere
    v, f = icosphere(1.0, 6)
    mesh = tfmm.tfmm_mesh_create(v, f)
    kh, pol = np.array([[0.0, 0.0, 1.0]]), np.array([[1.0, 0.0, 0.0]])

    def host_us(order):
        plan = tfmm.tfmm_plan_create(mesh, tfmm.tfmm_params_default(box=0.5, digits=1.0, tol=1e-1, quad_order=order))
        V = torch.empty((1, plan.info["n_rwg"]), dtype=torch.complex64, device="cuda")
        best = 1e9
        for _ in range(30):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(4):
                tfmm.tfmm_planewave_noalloc(plan, kh, pol, V)
            best = min(best, (time.perf_counter() - t0) / 4 * 1e6)
        return best

    one = host_us(1)
    assert host_us(10) <= one + 80


@pytest.mark.parametrize("nt,npf,rt,rp", [(64, 128, 16, 64), (58, 116, 16, 41), (48, 96, 32, 48)])
def test_first_step_of_the_disaggregation_keeps_its_precision_on_fine_grids(nt, npf, rt, rp):
    """Past 64 directions of phi the DG1b accumulator restarts; no form that is chosen may be less precise than
    the separate kernels (a pair count set by the tuning).  Errors are means over 24 columns, whose own
    scatter of 7 % each leaves 2 %; one accumulator over all directions reads 15 to 22 % more."""
    total = {0: 0.0, 64: 0.0}
    for seed in (1, 2, 3):
        tfmm, plan, n, members, T, w = _problem(seed, nt, npf, [150, 130], [[(rt, rp, 120)] * 2] * 2, 8, 3)
        _, g = _inputs(plan, 8, seed + 9)
        host = g.cpu().numpy().astype(np.complex128)
        ref = [apply.disaggregate_all(T, members, host[r], n, w) for r in range(8)]
        for pairs in total:
            tfmm.tfmm_plan_tuning_set(plan, tc_dg1a_pairs=pairs)
            y = _dis(tfmm, plan, g).cpu().numpy()
            total[pairs] += sum(np.linalg.norm(y[r] - ref[r]) / np.linalg.norm(ref[r]) for r in range(8))
    assert total[0] <= 1.1 * total[64]


def test_fused_tensor_core_kernels_take_no_planes_for_what_they_keep_on_chip():
    """V'' and P'' of 128 columns would be 153 MB here; X, T, M', y and the factor planes are about 70 MB, and
    allocations come in steps of 2 MB.  A tile preference that turns the fused kernels off brings them back."""
    nt, npf, rank, R, G = 26, 52, (12, 14, 30), 128, 60
    planes = 2 * G * 12 * npf * R * 16  # 2 x 3 terms of 2 bytes, r_theta rounded up to 8
    tfmm, first, *_ = _problem(101, nt, npf, [40, 40], [[rank, rank]] * 2, R, 3)
    x, g = _inputs(first, R, 102)
    _agg(tfmm, first, x), _dis(tfmm, first, g)  # the kernels are loaded
    tfmm, plan, *_ = _problem(103, nt, npf, [40] * G, [[rank, rank]] * G, R, 3)
    x, g = _inputs(plan, R, 104)
    spec, y = torch.empty_like(g), torch.empty_like(x)

    def call():
        tfmm.tfmm_aggregate(plan, x, spec)
        tfmm.tfmm_disaggregate(plan, g, y)
        torch.cuda.synchronize()

    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    call()
    assert free - torch.cuda.mem_get_info()[0] < 0.75 * planes
    fused = y.clone()
    tfmm.tfmm_plan_tuning_set(plan, tc_dg1a_pairs=64)
    call()
    assert free - torch.cuda.mem_get_info()[0] > planes
    assert torch.linalg.vector_norm(y - fused) <= 2e-6 * torch.linalg.vector_norm(fused)
    tfmm.tfmm_plan_tuning_set(plan, tc_dg1a_pairs=0)
    call()
    assert torch.equal(y, fused)
