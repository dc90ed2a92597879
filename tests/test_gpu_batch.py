"""Parity of the CUDA batched path (neighbour build, E/F/W, fitness) with the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1909_11474_gb300 import inputs as I

from ._util import (TOL32, TOL64, energy_rel_err, fitness_bounds, force_err, targets_to_device, to_device,
                    virial_rel_err)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1909_11474_gb300 import binding
    return binding.Context(0)


def _build(ctx, cs, R1=2.8, R2=3.2, M=16):
    pos, box = to_device(cs)
    ctx.build_neighbors(cs.atom_off, pos, box, R1, R2, M)
    return pos, box


def _oracle_lists(cs, R2=3.2):
    out = []
    for c in range(cs.C):
        nl = oracle.neighbor_list(*cs.config(c), R2)
        a = int(cs.atom_off[c])
        for i in range(cs.natoms[c]):
            e = slice(nl["off"][i], nl["off"][i + 1])
            out.append((nl["j"][e] + a, nl["n"][e]))
    return out


def _mixed_set(seed=5, C=10):
    rng = np.random.default_rng(seed)
    sizes = [(1, 1, 1), (2, 2, 2), (1, 2, 3), (3, 2, 2), (2, 1, 1)]
    return I.make_cells(rng, C, lambda: sizes[rng.integers(0, len(sizes))],
                        lambda: I.random_strain(rng, 0.03), lambda: float(rng.uniform(0.05, 0.2)),
                        lambda: int(rng.integers(0, 3)))


def _special_set():
    """Edge cases: a lone atom (no neighbours), a dimer (zeta = 0), one atom whose only neighbours are
    its own images, a compressed 8-atom cell with several images of the same j."""
    pos_list, box_list = [], []
    pos_list.append(np.array([[1.0, 2.0, 3.0]])); box_list.append(np.eye(3) * 12.0)
    pos_list.append(np.array([[0.0, 0.0, 0.0], [2.3, 0.1, 0.0]])); box_list.append(np.eye(3) * 15.0)
    pos_list.append(np.array([[0.1, 0.2, 0.3]])); box_list.append(np.eye(3) * 2.5)
    p, b = I.diamond_supercell((1, 1, 1), a=4.6)
    pos_list.append(p + np.random.default_rng(3).normal(0, 0.05, p.shape)); box_list.append(b)
    return I.pack_configs(pos_list, box_list)


@pytest.mark.parametrize("which", ["single", "ga", "mixed", "special"])
def test_neighbor_lists_bit_exact(ctx, which):
    cs = {"single": lambda: I.workload_single_cell()["configs"],
          "ga": lambda: I.workload_ga_batch(P=2, C=20)["configs"],
          "mixed": _mixed_set, "special": _special_set}[which]()
    _build(ctx, cs)
    cnt, nbr, shift = ctx.export_neighbors()
    ref = _oracle_lists(cs)
    assert len(ref) == cs.Ntot
    for i, (j, n) in enumerate(ref):
        assert cnt[i] == len(j), i
        assert np.array_equal(nbr[i, :cnt[i]], j), i
        assert np.array_equal(shift[i, :cnt[i]], n), i
        assert (nbr[i, cnt[i]:] == -1).all()


def _compare_eval(ctx, cs, params, precision, tol):
    P = len(params)
    pt = torch.tensor(params, dtype=torch.float64, device="cuda")
    E, F, W = ctx.eval(pt, precision=precision)
    torch.cuda.synchronize()
    assert ctx.get_status() == 0
    Er, Wr, Fr, ES, WS, FS = oracle.evaluate_batch(cs, params, scales=True, force_scales=True)
    E, F, W = E.cpu().numpy(), F.cpu().double().numpy(), W.cpu().numpy()
    eE = energy_rel_err(E, Er, ES).max()
    eW = virial_rel_err(W, Wr, WS).max()
    eF = force_err(F, Fr, FS)
    assert eE < tol["E"], eE
    assert eW < tol["W"], eW
    assert eF < tol["F"], eF
    return eE, eW, eF


@pytest.mark.parametrize("precision", [32, 64])
def test_single_cell_eval(ctx, precision):
    w = I.workload_single_cell()
    _build(ctx, w["configs"])
    _compare_eval(ctx, w["configs"], w["params"], precision, TOL32 if precision == 32 else TOL64)


def test_physical_forces_strict_absolute_bar(ctx):
    """Table 2 parameters on strained, displaced 64-atom cells: |dF| < 1e-4 eV/A with no scaling."""
    w = I.workload_ga_batch(P=2, C=8)
    _build(ctx, w["configs"])
    params = np.stack([w["hidden"], w["hidden"] * np.array([1.02, 0.99, 1.0, 1.05, 0.97, 1.03])])
    E, F, W = ctx.eval(torch.tensor(params, device="cuda"), precision=32)
    _, _, Fr = oracle.evaluate_batch(w["configs"], params)
    assert np.abs(F.cpu().double().numpy() - Fr).max() < 1e-4


@pytest.mark.parametrize("precision", [32, 64])
def test_ga_batch_eval_ragged_tiles(ctx, precision):
    """P = 37 spans three parameter tiles of 16 with a ragged tail; 64-atom strained cells."""
    w = I.workload_ga_batch(P=37, C=6)
    _build(ctx, w["configs"])
    _compare_eval(ctx, w["configs"], w["params"], precision, TOL32 if precision == 32 else TOL64)


@pytest.mark.parametrize("precision", [32, 64])
def test_mixed_sizes_eval(ctx, precision):
    """8..96-atom cells with vacancies, strain and pairs inside the switching region."""
    cs = _mixed_set()
    _build(ctx, cs)
    params = I.population(np.random.default_rng(8), 5)[0]
    _compare_eval(ctx, cs, params, precision, TOL32 if precision == 32 else TOL64)


@pytest.mark.parametrize("precision", [32, 64])
def test_special_cases_eval(ctx, precision):
    cs = _special_set()
    _build(ctx, cs)
    _compare_eval(ctx, cs, I.TABLE2_PARAMS[None, :], precision, TOL32 if precision == 32 else TOL64)


@pytest.mark.parametrize("precision", [32, 64])
def test_fitness_matches_oracle(ctx, precision):
    w = I.workload_ga_batch(P=21, C=5)
    cs = w["configs"]
    Eh, Wh, Fh = oracle.evaluate_batch(cs, w["hidden"][None, :])
    t = I.with_targets(w, Eh[0] / cs.natoms, Wh[0] / cs.natoms[:, None], Fh[0],
                       mask=np.array([7, 3, 5, 6, 1], np.uint8))
    wts = (1.0, 0.7, 0.3)
    E, W, F, ES, WS, FS = oracle.evaluate_batch(cs, w["params"], scales=True, force_scales=True)
    ref = oracle.fitness_from_predictions(cs, t, E, W, F, w=wts)
    _build(ctx, cs)
    Z, Zq, S = ctx.fitness(torch.tensor(w["params"], device="cuda"), targets_to_device(t),
                           w=wts, precision=precision)
    Z, Zq, S = Z.cpu().numpy(), Zq.cpu().numpy(), S.cpu().numpy()
    B = fitness_bounds(cs, t, E, W, F, ES, WS, TOL32 if precision == 32 else TOL64, FS=FS)
    D = ref["D"]
    assert (np.abs(np.sqrt(S) - np.sqrt(ref["S"])) <= B).all()
    assert (np.abs(Zq - ref["Zq"]) <= B / np.sqrt(D)[None, :]).all()
    assert (np.abs(Z - ref["Z"]) <= (np.asarray(wts)[None, :] * B / np.sqrt(D)[None, :]).sum(-1)).all()


def test_fitness_nonfinite_parameters_rank_last(ctx):
    w = I.workload_ga_batch(P=3, C=2)
    cs = w["configs"]
    _build(ctx, cs)
    params = w["params"].copy()
    params[1, 0] = np.nan
    t = {"E": np.full(cs.C, -4.6), "W": np.zeros((cs.C, 6)), "F": np.zeros((cs.Ntot, 3)),
         "mask": np.full(cs.C, 7, np.uint8)}
    Z, _, _ = ctx.fitness(torch.tensor(params, device="cuda"), targets_to_device(t))
    Z = Z.cpu().numpy()
    assert np.isinf(Z[1]) and np.isfinite(Z[0]) and np.isfinite(Z[2])


@pytest.mark.parametrize("which", ["ga", "mixed", "special"])
def test_plain_fp64_path(ctx, which):
    """The plain one-launch-per-(p, c) FP64 path against the oracle and the batched FP64 path."""
    if which == "ga":
        w = I.workload_ga_batch(P=3, C=4)
        cs, params = w["configs"], w["params"]
    elif which == "mixed":
        cs, params = _mixed_set(C=6), I.population(np.random.default_rng(9), 2)[0]
    else:
        cs, params = _special_set(), I.TABLE2_PARAMS[None, :]
    _build(ctx, cs)
    pt = torch.tensor(params, device="cuda")
    E, F, W = ctx.eval_plain(pt)
    Eb, Fb, Wb = ctx.eval(pt, precision=64)
    torch.cuda.synchronize()
    assert ctx.get_status() == 0
    Er, Wr, Fr, ES, WS, FS = oracle.evaluate_batch(cs, params, scales=True, force_scales=True)
    E, F, W = E.cpu().numpy(), F.cpu().numpy(), W.cpu().numpy()
    assert energy_rel_err(E, Er, ES).max() < TOL64["E"]
    assert virial_rel_err(W, Wr, WS).max() < TOL64["W"]
    assert force_err(F, Fr, FS) < TOL64["F"]
    assert np.allclose(E, Eb.cpu().numpy(), rtol=1e-12, atol=1e-12)
    assert np.allclose(F, Fb.cpu().numpy(), rtol=1e-10, atol=1e-11)


def test_kernel_timer_and_launch_count(ctx):
    """The measurement hooks: one timed batched-kernel sequence per fitness call while enabled, none
    after disabling, and a launch count that grows by the same amount for identical calls."""
    w = I.workload_ga_batch(P=40, C=6)
    cs = w["configs"]
    _build(ctx, cs)
    t = {"E": np.full(cs.C, -4.6), "W": np.zeros((cs.C, 6)), "F": np.zeros((cs.Ntot, 3)),
         "mask": np.full(cs.C, 7, np.uint8)}
    params, tg = torch.tensor(w["params"], device="cuda"), targets_to_device(t)
    ctx.profile(True)
    n0 = ctx.kernel_launches()
    ctx.fitness(params, tg)
    n1 = ctx.kernel_launches()
    ctx.fitness(params, tg)
    ctx.fitness(params, tg)
    n3 = ctx.kernel_launches()
    count, ms = ctx.profile_read()
    assert count == 3 and ms > 0.0
    assert n1 - n0 >= 3 and n3 - n1 == 2 * (n1 - n0)   # prep + batched kernel(s) + finalize per call
    ctx.profile(False)
    ctx.fitness(params, tg)
    assert ctx.profile_read() == (0, 0.0)
    assert ctx.get_status() == 0


def test_fitness_graph_replay_matches_direct_launches(ctx):
    """The fitness call replayed from its captured CUDA graph (with programmatic dependent launch)
    gives the results of plain direct launches, and a change of arguments (targets, weights, P) or of
    the neighbour build re-captures."""
    w = I.workload_ga_batch(P=45, C=7)
    cs = w["configs"]
    _build(ctx, cs)
    rng = np.random.default_rng(11)
    t1 = {"E": np.full(cs.C, -4.6), "W": rng.normal(0, 0.01, (cs.C, 6)), "F": rng.normal(0, 0.3, (cs.Ntot, 3)),
          "mask": np.array([7, 1, 2, 4, 7, 3, 6], np.uint8)}
    t2 = dict(t1, E=np.full(cs.C, -4.5))
    params = torch.tensor(w["params"], device="cuda")
    tg1, tg2 = targets_to_device(t1), targets_to_device(t2)

    def run(graphs, tg, wts, P=None):
        ctx.set_launch_mode(graphs=graphs, pdl=graphs)
        Z, Zq, S = ctx.fitness(params[:P], tg, w=wts)
        return torch.cat([Z[:, None], Zq, S], 1).cpu().numpy()

    for tg, wts in [(tg1, (1.0, 1.0, 1.0)), (tg2, (1.0, 1.0, 1.0)), (tg2, (0.5, 2.0, 1.0)), (tg1, (1.0, 1.0, 1.0))]:
        direct = run(False, tg, wts)
        first = run(True, tg, wts)       # captures
        again = run(True, tg, wts)       # replays
        assert np.array_equal(direct, first) and np.array_equal(direct, again)
    assert np.array_equal(run(False, tg1, (1, 1, 1), P=33), run(True, tg1, (1, 1, 1), P=33))
    # a new neighbour build of other configurations: the replay must not reuse the old schedule
    w2 = I.workload_ga_batch(P=45, C=4)
    cs2 = w2["configs"]
    _build(ctx, cs2)
    t3 = targets_to_device({"E": np.full(cs2.C, -4.6), "W": np.zeros((cs2.C, 6)),
                            "F": np.zeros((cs2.Ntot, 3)), "mask": np.full(cs2.C, 7, np.uint8)})
    assert np.array_equal(run(False, t3, (1, 1, 1)), run(True, t3, (1, 1, 1)))
    ctx.set_launch_mode()
    assert ctx.get_status() == 0


def test_build_errors_reported_by_next_call(ctx):
    """The neighbour build is queued and checked by the next call that uses it: a list overflow and
    non-finite positions come back from that call, and a valid rebuild afterwards works."""
    from paper_1909_11474_gb300 import binding
    cs = I.workload_single_cell()["configs"]
    params = torch.tensor(I.TABLE2_PARAMS[None, :], device="cuda")
    _build(ctx, cs, M=2)                      # diamond has 4 neighbours per atom
    with pytest.raises(binding.TersoffError) as ei:
        ctx.eval(params)
    assert ei.value.code == binding.E_NBR_OVERFLOW
    pos, box = to_device(cs)
    pos[5, 1] = float("nan")
    ctx.build_neighbors(cs.atom_off, pos, box, 2.8, 3.2, 16)
    with pytest.raises(binding.TersoffError) as ei:
        ctx.build_info()
    assert ei.value.code == binding.E_NONFINITE
    ctx.get_status()                           # clear the status bits of the failed builds
    _build(ctx, cs)
    E, F, W = ctx.eval(params, precision=64)
    r = oracle.evaluate(*cs.config(0), I.TABLE2_PARAMS)
    assert abs(float(E[0, 0]) - r["E"]) < 1e-9 * abs(r["E"])
    assert ctx.get_status() == 0


def test_autotune_keeps_results_within_the_bars(ctx):
    """The schedule autotuner times its candidates, keeps the fastest, and the tuned fitness still
    meets the oracle bounds (a partly filled last tile here: P = 45 = 32 + 13)."""
    w = I.workload_ga_batch(P=45, C=5)
    cs = w["configs"]
    Eh, Wh, Fh = oracle.evaluate_batch(cs, w["hidden"][None, :])
    t = I.with_targets(w, Eh[0] / cs.natoms, Wh[0] / cs.natoms[:, None], Fh[0])
    E, W, F, ES, WS, FS = oracle.evaluate_batch(cs, w["params"], scales=True, force_scales=True)
    ref = oracle.fitness_from_predictions(cs, t, E, W, F)
    B = fitness_bounds(cs, t, E, W, F, ES, WS, TOL32, FS=FS)
    _build(ctx, cs)
    params, tg = torch.tensor(w["params"], device="cuda"), targets_to_device(t)
    ms, tried = ctx.autotune(params, tg, reps=2)
    assert ms > 0.0 and tried >= 4             # chunkings 1, 2 x narrow last tile on / off
    Z, Zq, S = ctx.fitness(params, tg)
    S = S.cpu().numpy()
    assert (np.abs(np.sqrt(S) - np.sqrt(ref["S"])) <= B).all()
    assert ctx.get_status() == 0


@pytest.mark.parametrize("P", [45, 40, 7])
@pytest.mark.parametrize("tile,warps,items,narrow", [(32, 8, 1, 1), (32, 8, 3, 0), (16, 8, 1, 1), (16, 8, 2, 0),
                                                     (16, 8, 5, 1), (32, 12, 1, 1), (32, 12, 2, 0)])
def test_every_schedule_meets_the_oracle_bars(ctx, P, tile, warps, items, narrow):
    """Each schedule the autotuner can choose (tile width, work items per configuration, narrow last
    tile) gives a fitness within the oracle bounds, for full, half and small last tiles."""
    w = I.workload_ga_batch(P=P, C=5)
    cs = w["configs"]
    Eh, Wh, Fh = oracle.evaluate_batch(cs, w["hidden"][None, :])
    t = I.with_targets(w, Eh[0] / cs.natoms, Wh[0] / cs.natoms[:, None], Fh[0])
    E, W, F, ES, WS, FS = oracle.evaluate_batch(cs, w["params"], scales=True, force_scales=True)
    ref = oracle.fitness_from_predictions(cs, t, E, W, F)
    B = fitness_bounds(cs, t, E, W, F, ES, WS, TOL32, FS=FS)
    _build(ctx, cs)
    ctx.set_schedule(P, tile=tile, items_per_config=items, narrow=bool(narrow), warps=warps)
    Z, Zq, S = ctx.fitness(torch.tensor(w["params"], device="cuda"), targets_to_device(t))
    S = S.cpu().numpy()
    assert (np.abs(np.sqrt(S) - np.sqrt(ref["S"])) <= B).all()
    assert ctx.get_status() == 0


@pytest.mark.parametrize("change_counts", [False, True])
def test_fitness_queued_before_rebuild_check(ctx, change_counts):
    """A fitness call right after a rebuild of the same layout is queued before the host has checked
    the new neighbour counts. Whether the counts stayed or changed, its results equal those of a fresh
    context built once on the new positions."""
    from paper_1909_11474_gb300 import binding
    w = I.workload_ga_batch(P=37, C=6)
    cs = w["configs"]
    t = {"E": np.full(cs.C, -4.6), "W": np.zeros((cs.C, 6)), "F": np.zeros((cs.Ntot, 3)),
         "mask": np.full(cs.C, 7, np.uint8)}
    params, tg = torch.tensor(w["params"], device="cuda"), targets_to_device(t)
    ctx.set_launch_mode()
    _build(ctx, cs)
    ctx.fitness(params, tg)
    pos2 = cs.pos.copy() + np.random.default_rng(4).normal(0, 0.01, cs.pos.shape)
    box2 = cs.box.copy()
    if change_counts:   # move one atom of configuration 2 by 0.7 A along <110>: it gains second-shell bonds
        a0 = cs.atom_off[2]
        pos2[a0] += 0.7 * np.array([1.0, 1.0, 0.0]) / np.sqrt(2.0)
    p2, b2 = torch.tensor(pos2, device="cuda"), torch.tensor(box2, device="cuda")
    n_before = ctx.export_neighbors()[0].copy()
    ctx.build_neighbors(cs.atom_off, p2, b2, 2.8, 3.2, 16)
    Z, Zq, S = ctx.fitness(params, tg)
    got = torch.cat([Z[:, None], Zq, S], 1).cpu().numpy()
    assert ctx.get_status() == 0
    n_after = ctx.export_neighbors()[0]
    assert (not np.array_equal(n_before, n_after)) == change_counts
    fresh = binding.Context(0)
    fresh.build_neighbors(cs.atom_off, p2, b2, 2.8, 3.2, 16)
    Z2, Zq2, S2 = fresh.fitness(params, tg)
    ref = torch.cat([Z2[:, None], Zq2, S2], 1).cpu().numpy()
    assert np.array_equal(got, ref)


@pytest.mark.parametrize("precision", [32, 64])
def test_large_cells_in_clusters_eval(ctx, precision):
    """Cells of up to 512 atoms with up to 6 neighbours per atom (the uneven workload's largest): the
    schedule spreads each over a thread-block cluster of up to 16 CTAs; E/F/W against the oracle."""
    w = I.workload_uneven(P=2, C=24)
    cs = w["configs"]
    big = np.argsort(cs.natoms)[-6:]
    pos_list = [cs.config(int(c))[0] for c in big]
    box_list = [cs.config(int(c))[1] for c in big]
    sub = I.pack_configs(pos_list, box_list)
    assert sub.natoms.max() >= 380
    _build(ctx, sub)
    _compare_eval(ctx, sub, w["params"][:2], precision, TOL32 if precision == 32 else TOL64)
    clusters = sorted({b["cluster"] for b in ctx.schedule_info(precision)})
    print("cluster sizes", clusters)
    assert max(clusters) >= 8


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("reps,vac,sigma", [((3, 2, 2), 1, 0.30), ((4, 4, 2), 3, 0.22), ((4, 4, 4), 5, 0.27)])
def test_cluster_gather_on_disordered_cells(precision, reps, vac, sigma):
    """Cells spread over a cluster, whose lists of up to 8 bonds take both words of reverse-row addresses, with
    atom counts that leave the last rank a shorter slice: E/F/W against the oracle."""
    from paper_1909_11474_gb300 import binding
    rng = np.random.default_rng(int(np.prod(reps)))
    pos, box = I.diamond_supercell(reps)
    pos = pos[np.sort(rng.choice(len(pos), len(pos) - vac, replace=False))]
    cs = I.pack_configs([pos + rng.normal(0, sigma, pos.shape)], [box])
    params = I.population(rng, 3)[0]
    ctx = binding.Context(0)
    p, b = to_device(cs)
    ctx.build_neighbors(cs.atom_off, p, b, 2.8, 3.2, 16)
    assert 4 < ctx.build_info()[2] <= 8
    assert precision == 64 or ctx.schedule_info(precision)[0]["cluster"] > 1
    E, F, W = ctx.eval(torch.tensor(params, device="cuda"), precision=precision)
    torch.cuda.synchronize()
    assert ctx.get_status() == 0
    Er, Wr, Fr, ES, WS, FS = oracle.evaluate_batch(cs, params, scales=True, force_scales=True)
    tol = TOL32 if precision == 32 else TOL64
    assert energy_rel_err(E.cpu().numpy(), Er, ES).max() < tol["E"]
    assert virial_rel_err(W.cpu().numpy(), Wr, WS).max() < tol["W"]
    assert force_err(F.cpu().double().numpy(), Fr, FS) < tol["F"]


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("P", [1, 7, 8, 9, 17])
def test_fp64_tiles_and_parameter_ranges(P, form):
    """The FP64 kernel's tiles of eight sets, full and partly filled, over ragged cells (several atoms of different
    list lengths in a warp; lone atoms and dimers), with parameter sets inside and outside the ranges of its
    fixed-point functions (n beyond [1/64, 4), prefactors that are negative, tiny or huge, r0 beyond 16): E, F and W
    of every set equal those of the set evaluated alone, and for the minimal form those of the plain FP64 path (but for
    where zeta <= 0, the dimer and a negative beta, which the batched kernels clamp to 1e-30 and the plain path takes
    as b = 1, b' = 0)."""
    from paper_1909_11474_gb300 import binding
    rng = np.random.default_rng(17)
    parts = [(np.array([[0.5, 0.5, 0.5]]), np.eye(3) * 9.0), (np.array([[0.0, 0, 0], [2.3, 0.2, 0]]), np.eye(3) * 12.0)]
    for reps, sigma, vac in (((1, 1, 1), 0.1, 1), ((2, 2, 2), 0.25, 2), ((2, 3, 2), 0.2, 5)):
        pos, box = I.diamond_supercell(reps)
        pos = pos[np.sort(rng.choice(len(pos), len(pos) - vac, replace=False))]
        parts.append((pos + rng.normal(0, sigma, pos.shape), box))
    cs = I.pack_configs(*zip(*parts))
    x0 = I.TABLE2_PARAMS if form == 0 else np.array([3.2, 1.45, 2.25, 1.9, 0.65, -0.6, 0.06, 20.0, 3.0])
    x = x0[None, :] * (1 + 0.1 * rng.uniform(-1, 1, size=(17, len(x0))))
    iB = 3 if form == 0 else 6
    for k, (q, v) in enumerate([(4, 5.0), (4, 0.01), (0, -1.5), (iB, -0.2), (0, 1e-70), (0, 1e80), (2, 17.0), (1, 20.0),
                                (iB, 1e-65)]):
        x[(2 * k + 3) % 17, q] = v
    x[:P] = np.roll(x, -3, axis=0)[:P]
    ctx = binding.Context(0)
    ctx.set_form(form)
    p, b = to_device(cs)
    ctx.build_neighbors(cs.atom_off, p, b, 2.8, 3.2, 16)
    xt = torch.tensor(x[:P].copy(), device="cuda")
    E, F, W = ctx.eval(xt, precision=64)
    for k in range(P):
        E1, F1, W1 = ctx.eval(xt[k:k + 1].contiguous(), precision=64)
        assert torch.equal(E1[0], E[k]) and torch.equal(F1[0], F[k]) and torch.equal(W1[0], W[k])
    if form == 0:
        Ep, Fp, Wp = ctx.eval_plain(xt)
        for got, ref in ((E[:, 2:], Ep[:, 2:]), (F[:, 3:], Fp[:, 3:]), (W[:, 2:], Wp[:, 2:])):
            for k in np.flatnonzero(x[:P, 3] > 0):
                assert (got[k] - ref[k]).abs().max() <= 1e-10 * ref[k].abs().max(), (k, x[k])
    assert ctx.get_status() == 0


@pytest.mark.parametrize("k,tol", [(-105, 1e-10), (-90, 1e-13), (100, 1e-13), (118, 1e-13)])
def test_fp32_results_scale_with_a_power_of_two(ctx, k, tol):
    """D0 times 2^k multiplies every FP32 quantity of the energies, forces and virials by 2^k exactly, so the results are
    those of k = 0 times 2^k. The partial sums of a tile are added in FP32 splits for exponents from -95 to 123 and in
    64-bit integers outside; the FP64 results then differ by their last rounding, and for k = -105 by FP32 subnormals
    (2^-149 an operation against sums above 2^-105: 2^-44 each). Cells without bonds sum zeros in both."""
    pos, box = [], []
    for s in (I.workload_ga_batch(P=1, C=3)["configs"], _special_set()):
        for c in range(s.C):
            pos.append(s.config(c)[0])
            box.append(s.config(c)[1])
    cs = I.pack_configs(pos, box)
    _build(ctx, cs)
    params = np.tile(I.TABLE2_PARAMS, (9, 1)) * np.linspace(0.97, 1.03, 9)[:, None]
    scaled = params.copy()
    scaled[:, 0] *= 2.0 ** k
    out = []
    for x in (params, scaled):
        E, F, W = ctx.eval(torch.tensor(x, dtype=torch.float64, device="cuda"), precision=32)
        torch.cuda.synchronize()
        out.append((E.cpu().numpy(), F.cpu().double().numpy(), W.cpu().numpy()))
    assert ctx.get_status() == 0
    for a, b, t in zip(out[0], out[1], (tol, 1e-6, tol)):
        assert np.abs(b * 2.0 ** -k - a).max() <= t * np.abs(a).max()


@pytest.mark.parametrize("change", ["none", "counts", "overflow", "nonfinite"])
@pytest.mark.parametrize("C", [1, 6])
def test_eval_queued_before_rebuild_check(change, C):
    """An FP32 evaluation right after a rebuild of the same layout is queued before the host has read the counts and
    error flags that the build kernel leaves in pinned memory. Its results equal those of a fresh context built once on
    the new positions, and the build's errors come back from it."""
    from paper_1909_11474_gb300 import binding
    w = I.workload_ga_batch(P=9, C=C)
    cs = w["configs"]
    params = torch.tensor(w["params"], device="cuda")
    c = binding.Context(0)
    _build(c, cs)
    c.eval(params)
    pos2 = cs.pos.copy() + np.random.default_rng(4).normal(0, 0.01, cs.pos.shape)
    a0 = cs.atom_off[C - 1]
    if change == "counts":
        pos2[a0] += 0.7 * np.array([1.0, 1.0, 0.0]) / np.sqrt(2.0)
    if change == "overflow":                  # 33 atoms within a sphere of radius 0.8
        d = np.random.default_rng(1).normal(size=(33, 3))
        pos2[a0:a0 + 33] = pos2[a0] + 0.8 * d / np.linalg.norm(d, axis=1)[:, None]
    if change == "nonfinite":
        pos2[a0, 1] = np.nan
    p2, b2 = torch.tensor(pos2, device="cuda"), torch.tensor(cs.box, device="cuda")
    c.build_neighbors(cs.atom_off, p2, b2, 2.8, 3.2, 16)
    if change in ("overflow", "nonfinite"):
        with pytest.raises(binding.TersoffError) as ei:
            c.eval(params)
        assert ei.value.code == (binding.E_NBR_OVERFLOW if change == "overflow" else binding.E_NONFINITE)
        return
    got = c.eval(params)
    torch.cuda.synchronize()
    assert c.get_status() == 0
    fresh = binding.Context(0)
    fresh.build_neighbors(cs.atom_off, p2, b2, 2.8, 3.2, 16)
    for a, b in zip(got, fresh.eval(params)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("call", ["eval", "fitness"])
@pytest.mark.parametrize("C,reps", [(700, (1, 1, 1)), (120, (4, 4, 3))])
def test_stale_items_are_skipped_in_runs(call, C, reps):
    """A rebuild that changes the counts of nearly every configuration: the call queued ahead of the check skips one item
    after another (on single CTAs and on clusters, several items each), and its results are those of a fresh context."""
    from paper_1909_11474_gb300 import binding
    rng = np.random.default_rng(8)
    cs = I.make_cells(rng, C, lambda: reps, lambda: I.random_strain(rng, 0.01), lambda: 0.05, lambda: 0)
    pos2 = cs.pos.copy()
    for k in range(C):
        if k % 16:                            # one atom moved by 0.7 A along <110> gains second-shell bonds
            pos2[cs.atom_off[k]] += 0.7 * np.array([1.0, 1.0, 0.0]) / np.sqrt(2.0)
    t = {"E": np.full(cs.C, -4.6), "W": np.zeros((cs.C, 6)), "F": np.zeros((cs.Ntot, 3)),
         "mask": np.full(cs.C, 7, np.uint8)}
    params, tg = torch.tensor(I.population(rng, 37)[0], device="cuda"), targets_to_device(t)
    run = (lambda c: c.eval(params)) if call == "eval" else (lambda c: c.fitness(params, tg))
    pos, box = to_device(cs)
    new = torch.tensor(pos2, device="cuda")
    c = binding.Context(0)
    for x in (pos, new, pos):
        c.build_neighbors(cs.atom_off, x, box, 2.8, 3.2, 16)
        got = run(c)
        assert c.get_status() == 0
        fresh = binding.Context(0)
        fresh.build_neighbors(cs.atom_off, x, box, 2.8, 3.2, 16)
        for u, v in zip(got, run(fresh)):
            assert torch.equal(u, v)
        counts = c.export_neighbors()[0]
        assert x is not new or (np.add.reduceat(counts, cs.atom_off[:-1]) != before).sum() > 0.5 * C
        before = np.add.reduceat(counts, cs.atom_off[:-1])


@pytest.mark.parametrize("call", ["eval", "fitness"])
@pytest.mark.parametrize("change_counts", [False, True])
def test_rebuild_on_one_stream_and_call_on_another(call, change_counts):
    """A rebuild queued on one stream behind 20 ms of other work, and the FP32 call that uses it on another stream: the
    call's results are those of a fresh context built on the new positions, not of the old or a half-written geometry."""
    from paper_1909_11474_gb300 import binding
    w = I.workload_ga_batch(P=37, C=40)
    cs = w["configs"]
    t = {"E": np.full(cs.C, -4.6), "W": np.zeros((cs.C, 6)), "F": np.zeros((cs.Ntot, 3)),
         "mask": np.full(cs.C, 7, np.uint8)}
    params, tg = torch.tensor(w["params"], device="cuda"), targets_to_device(t)
    c = binding.Context(0)
    run = (lambda c: c.eval(params)) if call == "eval" else (lambda c: c.fitness(params, tg))
    pos, box = to_device(cs)
    pos2 = cs.pos + np.random.default_rng(4).normal(0, 0.01, cs.pos.shape)
    if change_counts:
        pos2[cs.atom_off[3]] += 0.7 * np.array([1.0, 1.0, 0.0]) / np.sqrt(2.0)
    new = torch.tensor(pos2, device="cuda")
    fresh = binding.Context(0)
    fresh.build_neighbors(cs.atom_off, new, box, 2.8, 3.2, 16)
    want = run(fresh)
    c.build_neighbors(cs.atom_off, pos, box, 2.8, 3.2, 16)
    run(c)
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):
        torch.cuda._sleep(int(0.02 * 2e9))
        c.build_neighbors(cs.atom_off, new, box, 2.8, 3.2, 16)
    with torch.cuda.stream(b):
        got = run(c)
    torch.cuda.synchronize()
    assert c.get_status() == 0
    for x, y in zip(got, want):
        assert torch.equal(x, y)


def test_evaluation_captured_right_after_a_rebuild():
    """A stream under capture cannot be ordered after the build on a stream outside: the host waits first, and the graph
    holds the evaluation of the new positions."""
    from paper_1909_11474_gb300 import binding
    cs = I.workload_ga_batch(P=1, C=3)["configs"]
    params = torch.tensor(I.population(np.random.default_rng(2), 9)[0], device="cuda")
    c = binding.Context(0)
    pos, box = to_device(cs)
    c.build_neighbors(cs.atom_off, pos, box, 2.8, 3.2, 16)
    c.eval(params)
    new = pos + 0.01 * torch.randn(pos.shape, dtype=torch.float64, device="cuda",
                                   generator=torch.Generator(device="cuda").manual_seed(3))
    c.build_neighbors(cs.atom_off, new, box, 2.8, 3.2, 16)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        got = c.eval(params)
    g.replay()
    torch.cuda.synchronize()
    fresh = binding.Context(0)
    fresh.build_neighbors(cs.atom_off, new, box, 2.8, 3.2, 16)
    for x, y in zip(got, fresh.eval(params)):
        assert torch.equal(x, y)


@pytest.mark.parametrize("tile,P", [(16, 16), (16, 21), (16, 5), (32, 5), (32, 40)])
def test_rebuild_with_a_long_list_and_equal_totals(tile, P):
    """Three triangles and a lone atom become a star of nine bonds: bonds and pair slots of the cell stay 18 and 36, so
    that its schedule record still matches and the fitness queued ahead of the check runs on lists longer than its
    kernel's. It reads nothing out of range, and the call returns TERSOFF_E_UNSUPPORTED."""
    from paper_1909_11474_gb300 import binding
    g = (1 + 5 ** 0.5) / 2
    ico = np.array([[0, s, t * g] for s in (1, -1) for t in (1, -1)])
    ico = np.concatenate([ico, ico[:, [2, 0, 1]], ico[:, [1, 2, 0]]]) / np.sqrt(1 + g * g)
    star = 20.0 + np.concatenate([3.1 * ico[:9], np.zeros((1, 3))])        # leaves 3.26 apart; the centre last
    tri = 2.4 * np.array([[0, 0, 0], [1, 0, 0], [0.5, 0.75 ** 0.5, 0]])
    rings = np.concatenate([tri, tri + 10.0, tri + 20.0, [[30.0, 5.0, 5.0]]])
    box = np.eye(3) * 40.0
    old, new = I.pack_configs([rings] * 3, [box] * 3), I.pack_configs([rings, star, rings], [box] * 3)
    slots = lambda m: ((m * (m - 1) // 2 + 3) // 4 * 4).sum()              # noqa: E731
    for cs, top in ((old, 2), (new, 9)):
        m = np.diff(oracle.neighbor_list(*cs.config(1), 3.2)["off"])
        assert (m.max(), m.sum(), slots(m)) == (top, 18, 36)
    t = targets_to_device({"E": np.full(3, -1.0), "W": np.zeros((3, 6)), "F": np.zeros((30, 3)),
                           "mask": np.full(3, 7, np.uint8)})
    params = torch.tensor(I.population(np.random.default_rng(1), P)[0], device="cuda")
    c = binding.Context(0)
    _build(c, old)
    c.set_schedule(P, tile=tile)
    want = [x.cpu() for x in c.fitness(params, t)]
    _build(c, new)
    with pytest.raises(binding.TersoffError) as ei:
        c.fitness(params, t)
    assert ei.value.code == binding.E_UNSUPPORTED
    torch.cuda.synchronize()
    c.get_status()
    _build(c, old)
    for x, y in zip(c.fitness(params, t), want):
        assert np.allclose(x.cpu(), y, rtol=1e-6)
    assert c.get_status() == 0


@pytest.mark.parametrize("change", ["overflow", "nonfinite"])
@pytest.mark.parametrize("C,reps", [(1, (2, 2, 2)), (6, (2, 2, 2)), (3, (4, 4, 2))])
def test_failed_rebuild_leaves_the_outputs_of_an_evaluation(change, C, reps):
    """The evaluation that returns a rebuild's error writes nothing: E, F and W keep what they held."""
    from paper_1909_11474_gb300 import binding
    rng = np.random.default_rng(3)
    cs = I.make_cells(rng, C, lambda: reps, lambda: I.random_strain(rng, 0.01), lambda: 0.05, lambda: 0)
    P = 9
    params = torch.tensor(I.population(rng, P)[0], device="cuda")
    c = binding.Context(0)
    _build(c, cs)
    c.eval(params)
    pos2 = cs.pos.copy()
    a0 = cs.atom_off[C - 1]
    if change == "overflow":                  # 33 atoms within a sphere of radius 0.8
        d = np.random.default_rng(1).normal(size=(33, 3))
        pos2[a0:a0 + 33] = pos2[a0] + 0.8 * d / np.linalg.norm(d, axis=1)[:, None]
    else:
        pos2[a0, 1] = np.nan
    p2, b2 = torch.tensor(pos2, device="cuda"), torch.tensor(cs.box, device="cuda")
    out = [torch.full(s, 7.0, dtype=t, device="cuda") for s, t in
           (((P, C), torch.float64), ((P, cs.Ntot, 3), torch.float32), ((P, C, 6), torch.float64))]
    c.build_neighbors(cs.atom_off, p2, b2, 2.8, 3.2, 16)
    rc = c.lib.tersoff_eval(c.h, params.data_ptr(), P, 32, *(x.data_ptr() for x in out), binding._stream(None))
    torch.cuda.synchronize()
    assert rc == (binding.E_NBR_OVERFLOW if change == "overflow" else binding.E_NONFINITE)
    for x in out:
        assert (x == 7.0).all()
    c.get_status()
    _build(c, cs)                             # and a valid rebuild evaluates again
    fresh = binding.Context(0)
    _build(fresh, cs)
    for x, y in zip(c.eval(params), fresh.eval(params)):
        assert torch.equal(x, y)
    assert c.get_status() == 0


PRELOAD = """
import numpy as np, torch
from paper_1909_11474_gb300 import binding, inputs as I
rng = np.random.default_rng(3)
cs = I.make_cells(rng, 4, lambda: (2, 2, 2), lambda: I.random_strain(rng, 0.02), lambda: 0.1, lambda: 0)
ctx = binding.Context(0)
pos, box = torch.tensor(cs.pos, device="cuda"), torch.tensor(cs.box, device="cuda")
params = torch.tensor(I.population(rng, 21)[0], device="cuda")
t = {"E": torch.full((4,), -4.6), "W": torch.zeros((4, 6)), "F": torch.zeros((cs.Ntot, 3))}
t = {k: v.double().cuda() for k, v in t.items()} | {"mask": torch.full((4,), 7, dtype=torch.uint8, device="cuda")}
out = [torch.empty(s, dtype=d, device="cuda") for s, d in
       (((21, 4), torch.float64), ((21, cs.Ntot, 3), torch.float64), ((21, 4, 6), torch.float64))]
ctx.build_neighbors(cs.atom_off, pos, box, 2.8, 3.2, 16)
for precision in (32, 64):
    ctx.fitness(params, t, precision=precision)       # the workspaces that fitness and evaluation share
torch.cuda.synchronize()
free = [torch.cuda.mem_get_info()[0]]
for precision in (32, 64):
    rc = ctx.lib.tersoff_eval(ctx.h, params.data_ptr(), 21, precision, *(x.data_ptr() for x in out), binding._stream(None))
    torch.cuda.synchronize()
    free.append(torch.cuda.mem_get_info()[0])
    assert rc == 0
print(*free)
"""


def test_first_evaluation_after_a_build_loads_no_code():
    """The build loads the evaluation kernels of both precisions too: free device memory does not change across a process's
    first evaluations. (In a process of its own, where no other test has loaded them.)"""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PRELOAD], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    free = r.stdout.split()[-3:]
    assert free[0] == free[1] == free[2], free


@pytest.mark.parametrize("precision", [32, 64])
def test_schedule_read_back_can_be_set(ctx, precision):
    """What schedule_info reports of a tuned schedule is what set_schedule takes (a program that keeps the schedules it has
    tuned), and the results are the tuned ones."""
    w = I.workload_ga_batch(P=45, C=5)
    cs = w["configs"]
    t = {"E": np.full(cs.C, -4.6), "W": np.zeros((cs.C, 6)), "F": np.zeros((cs.Ntot, 3)),
         "mask": np.full(cs.C, 7, np.uint8)}
    params, tg = torch.tensor(w["params"], device="cuda"), targets_to_device(t)
    _build(ctx, cs)
    ctx.autotune(params, tg, precision=precision, reps=1)
    want = ctx.fitness(params, tg, precision=precision)
    info = ctx.schedule_info(precision)
    _build(ctx, I.workload_ga_batch(P=45, C=4)["configs"])
    _build(ctx, cs)
    b = info[0]
    ctx.set_schedule(b["tuned_P"], tile=b["tile"], items_per_config=b["items_per_config"], narrow=bool(b["narrow"]),
                     precision=precision, warps=b["warps"])
    assert ctx.schedule_info(precision) == info
    for x, y in zip(ctx.fitness(params, tg, precision=precision), want):
        assert torch.equal(x, y)
    assert ctx.get_status() == 0


def test_a_failed_allocation_is_reported_once(ctx):
    """A fitness whose residual terms would take 15 TB fails to allocate them and says so; the calls after it, which check
    their own launches, succeed."""
    import ctypes

    from paper_1909_11474_gb300 import binding
    w = I.workload_ga_batch(P=5, C=300)
    cs = w["configs"]
    t = targets_to_device({"E": np.full(cs.C, -4.6), "W": np.zeros((cs.C, 6)), "F": np.zeros((cs.Ntot, 3)),
                           "mask": np.full(cs.C, 7, np.uint8)})
    params = torch.tensor(w["params"], device="cuda")
    pos, box = _build(ctx, cs)
    want = [x.cpu() for x in ctx.fitness(params, t)]
    Z = torch.empty(5, dtype=torch.float64, device="cuda")
    tg, wv = ctx._targets(t), (ctypes.c_double * 3)(1, 1, 1)
    rc = ctx.lib.tersoff_fitness(ctx.h, params.data_ptr(), 2 ** 31 - 1, ctypes.byref(tg), ctypes.addressof(wv), 32,
                                 Z.data_ptr(), None, None, binding._stream(None))
    assert rc == binding.E_CUDA and b"memory" in ctx.lib.tersoff_last_error(ctx.h)
    ctx.build_neighbors(cs.atom_off, pos, box, 2.8, 3.2, 16)
    for x, y in zip(ctx.fitness(params, t), want):
        assert torch.equal(x.cpu(), y)
    assert ctx.get_status() == 0
