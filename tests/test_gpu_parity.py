"""GPU path (through the C ABI) against the CPU oracle on identical Philox streams.

Bit-exact: lattices, cumulative activities K, interval activities dK and [eq]
ancestors, every interval.  psi_hat within 1e-12 relative (the psi terms use CUDA's
FP64 exp/expm1/log1p against glibc's; every other quantity is an integer).
Cases span several 1024-slot tiles with ragged tails, both lattice widths
(L <= 64 and 64 < L <= 128), both signs of s, s = 0, empty and full rings, one
clone, and a batch of uneven populations.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

PSI_RTOL = 1e-12


@pytest.fixture(scope="module")
def pg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1711_05095_gb300 import build
    build.build()
    import paper_1711_05095_gb300 as pg
    return pg


def oracle_pops(pops):
    return [oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"],
                              modified=q.get("weight_mode", 0) == 1, iid=q.get("selection", 0) == 1)
            for q in pops]


def assert_state_equal(gpu, orc, W, what):
    words = oracle.sites_to_words(orc.sites, W)
    assert np.array_equal(gpu["lattice"], words), what + ": lattice"
    assert np.array_equal(gpu["K"], orc.K), what + ": K"


def run_parity(pg, pops, s, dt, M):
    batch = pg.PopulationBatch(pops)
    orcs = oracle_pops(pops)
    W = batch.W
    for p, o in enumerate(orcs):
        assert_state_equal(batch.copy_state(p), o, W, "init pop %d" % p)
    for beta in range(1, M + 1):
        batch.evolve(dt, s)
        for p, o in enumerate(orcs):
            o.evolve(dt, s[p])
            g = batch.copy_state(p)
            assert_state_equal(g, o, W, "evolve beta=%d pop %d" % (beta, p))
            assert np.array_equal(g["dK"], o.dK), "dK beta=%d pop %d" % (beta, p)
        batch.resample()
        for p, o in enumerate(orcs):
            o.resample(s[p])
            g = batch.copy_state(p)
            assert np.array_equal(g["anc"], o.anc), "anc beta=%d pop %d" % (beta, p)
            assert_state_equal(g, o, W, "resample beta=%d pop %d" % (beta, p))
    psi, kh, t_obs = batch.estimate_psi()
    ev = batch.events()
    for p, o in enumerate(orcs):
        ps, ks = o.estimates()
        np.testing.assert_allclose(psi[p], ps, rtol=PSI_RTOL, atol=0.0)
        np.testing.assert_allclose(kh[p], ks, rtol=1e-15, atol=0.0)
        assert int(ev[p]) == o.events
    return batch, orcs


@pytest.mark.parametrize("L,N,nc,s", [
    (20, 10, 1000, 0.05),      # one tile, ragged
    (20, 10, 2500, -0.3),      # three tiles, negative bias
    (50, 25, 3072, 0.3),       # exact tiles
    (64, 31, 1500, 0.8),       # widest one-word ring
    (65, 30, 1100, 0.2),       # narrowest two-word ring
    (100, 50, 2049, -0.05),
    (128, 64, 4100, 0.01),     # widest ring
    (3, 1, 777, 0.4),          # smallest ring
    (37, 5, 1, 0.5),           # one clone
    (20, 10, 1234, 0.0),       # no bias: identity ancestry
    (12, 0, 300, 0.3),         # empty ring: no hops
    (12, 12, 300, -0.3),       # full ring: no hops
    (40, 20, 3000, 2.5),       # strong bias: many deletions
])
def test_parity_single(pg, L, N, nc, s):
    pops = [dict(L=L, N=N, n_clones=nc, seed=1234 + L)]
    batch, orcs = run_parity(pg, pops, [s], 0.1 if L < 100 else 0.05, 6)
    if s == 0.0:
        g = batch.copy_state(0)
        assert np.array_equal(g["anc"], np.arange(nc))
        assert batch.estimate_psi()[0][0] == 0.0


def test_parity_uneven_batch(pg):
    rng = np.random.default_rng(5)
    pops, s = [], []
    for i, L in enumerate([32, 64, 100, 128, 20, 77]):
        pops.append(dict(L=L, N=L // 2 - i, n_clones=int(rng.integers(900, 3000)), seed=99 + i))
        s.append(float(rng.uniform(-10, 30)) / L**2)
    run_parity(pg, pops, s, 0.1, 5)


def test_parity_long_dt(pg):
    # many hops per interval (dt = 2 at L = 50: ~50 hops per clone)
    run_parity(pg, [dict(L=50, N=25, n_clones=1500, seed=3)], [0.02], 2.0, 3)


RUN_CASES = {
    # two-word lattices: fused run, two captured graphs of 32 intervals plus direct ones
    "w2_plain": ([dict(L=50, N=25, n_clones=2000, seed=7), dict(L=100, N=40, n_clones=1300, seed=8)],
                 [0.01, -0.004], [70]),
    # one-word lattices, MODIFIED next to plain, a ragged multi-tile population
    "w1_mixed_weights": ([dict(L=20, N=10, n_clones=2500, seed=11, weight_mode=1),
                          dict(L=64, N=31, n_clones=1100, seed=12)], [0.3, -0.2], [37]),
    # two-word MODIFIED, strong bias (many deletions), runs split across calls
    "w2_modified_split": ([dict(L=100, N=50, n_clones=1500, seed=13, weight_mode=1),
                           dict(L=33, N=16, n_clones=700, seed=14)], [0.05, 2.5], [1, 33, 2]),
    # an [iid] population: every interval through the separate kernels
    "iid_unfused": ([dict(L=30, N=15, n_clones=1200, seed=15, selection=1),
                     dict(L=50, N=25, n_clones=900, seed=16, weight_mode=1)], [0.1, -0.05], [35]),
    # a single interval: the fused run's first and last stages only
    "one_interval": ([dict(L=40, N=20, n_clones=3000, seed=17)], [0.2], [1]),
    # runs of 1, 2, 3 and 40 intervals; a population of 64 full tiles beside one of a
    # single ragged tile; s < 0
    "many_splits": ([dict(L=50, N=25, n_clones=64 * 1024, seed=18), dict(L=20, N=10, n_clones=700, seed=19)],
                    [0.01, -0.3], [1, 2, 3, 40]),
    # one population of 65 tiles and a ragged last tile
    "tiles_65": ([dict(L=30, N=15, n_clones=65 * 1024 + 5, seed=20)], [0.05], [35]),
    # five populations of 1, 4, 2, 3 and 2 tiles: pop_run runs three chains of 5, 2 and
    # 5 tiles; a graph replay, then direct launches of the chains
    "halves_of_five": ([dict(L=30, N=15, n_clones=1000, seed=30), dict(L=50, N=25, n_clones=4000, seed=31),
                        dict(L=70, N=30, n_clones=1900, seed=32, weight_mode=1),
                        dict(L=128, N=64, n_clones=3072, seed=33), dict(L=9, N=4, n_clones=1500, seed=34)],
                       [0.2, -0.01, 0.1, 0.004, -0.5], [33, 5]),
    # strong bias: a wide activity range and tiles whose old clones leave no copies
    "strong_bias": ([dict(L=64, N=32, n_clones=5000, seed=21), dict(L=128, N=64, n_clones=3000, seed=22)],
                    [2.0, 0.5], [34]),
    # rings that fill the lattice words (L = 64 W: the fused kernel rotates the words
    # without a closing bit), one and two words
    "w1_full_ring": ([dict(L=64, N=20, n_clones=3000, seed=23), dict(L=64, N=40, n_clones=2100, seed=24)],
                     [0.02, -0.05], [36]),
    "w2_full_ring": ([dict(L=128, N=64, n_clones=3000, seed=25), dict(L=128, N=50, n_clones=2100, seed=26)],
                     [0.01, -0.02], [35]),
}


def test_run_chains(pg):
    # the split rule: population starts nearest k/K of the tiles, every chain at least
    # half its share; up to 8 chains within two waves of the fused kernel, else 2
    five = pg.PopulationBatch(RUN_CASES["halves_of_five"][0])
    assert five.run_chains() == [0, 5, 7, 12]
    w = workloads.s_sweep()
    sweep = pg.PopulationBatch(w["pops"])                 # 64 x 16 tiles
    assert sweep.run_chains() == [128 * c for c in range(9)]
    sweep.close()
    big = pg.PopulationBatch([dict(L=50, N=25, n_clones=4096 * 1024, seed=40 + i) for i in range(3)])
    assert big.run_chains() == [0, 4096, 12288]            # 3 x 4096 tiles: two chains
    big.close()
    # batches that do not fuse run one sequence
    assert pg.PopulationBatch([dict(L=30, N=15, n_clones=1200, seed=15, selection=1),
                               dict(L=30, N=15, n_clones=1200, seed=16)]).run_chains() == []
    assert pg.PopulationBatch([dict(L=200, N=100, n_clones=1200, seed=17),
                               dict(L=30, N=15, n_clones=1200, seed=18)]).run_chains() == []


@pytest.mark.parametrize("case", sorted(RUN_CASES))
def test_run_equals_steps(pg, case):
    pops, s, splits = RUN_CASES[case]
    a = pg.PopulationBatch(pops)
    b = pg.PopulationBatch(pops)
    for n in splits:
        a.run(0.1, s, n)
    for _ in range(sum(splits)):
        b.evolve(0.1, s)
        b.resample()
    P = len(pops)
    for p in range(P):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), key
    pa, ka, ta = a.estimate_psi()
    pb, kb, tb = b.estimate_psi()
    # same device arithmetic; only t_obs differs in rounding (n*dt against a sum of dt)
    np.testing.assert_allclose(pa * ta, pb * tb, rtol=1e-15)
    np.testing.assert_allclose(pa, pb, rtol=1e-14)
    np.testing.assert_allclose(ka, kb, rtol=1e-14)
    np.testing.assert_allclose(ta, tb, rtol=1e-13)
    np.testing.assert_array_equal(a.events(), b.events())


def test_full_size_s_sweep_sampled(pg):
    # the 64-population s-sweep at full size (2^20 clones) in the bench's launch
    # configuration (pop_run); three sampled populations checked bit for bit
    w = workloads.s_sweep()
    M = 4
    batch = pg.PopulationBatch(w["pops"])
    batch.run(w["dt"], w["s"], M)
    psi, _, _ = batch.estimate_psi()
    for p in (0, 31, 63):
        q = w["pops"][p]
        o = oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"])
        for _ in range(M):
            o.evolve(w["dt"])
            o.resample(w["s"][p])
        g = batch.copy_state(p)
        assert np.array_equal(g["anc"], o.anc)
        assert_state_equal(g, o, batch.W, "s-sweep pop %d" % p)
        np.testing.assert_allclose(psi[p], o.estimates()[0], rtol=PSI_RTOL)
    # properties at every population: N conserved, ancestors monotone and in range
    for p in range(0, 64, 9):
        g = batch.copy_state(p)
        counts = sum(np.vectorize(lambda v: bin(int(v)).count("1"))(g["lattice"][:, q])
                     for q in range(batch.W))
        assert np.all(counts == w["pops"][p]["N"])
        assert np.all(np.diff(g["anc"]) >= 0)
        assert g["anc"].min() >= 0 and g["anc"].max() < w["pops"][p]["n_clones"]


def test_full_size_large_population_run(pg):
    # the bench's population shape (L = 128, N_c = 2^20) through pop_run: the fused
    # kernel for rings that fill the words, with the per-tile activity counts, over
    # three intervals, against the oracle
    q = dict(L=128, N=64, n_clones=2**20, seed=2001)
    s = 15.0 / 128**2
    batch = pg.PopulationBatch([q])
    assert batch.get_tuning()["hist_mode"] == -1
    batch.run(0.05, [s], 3)
    o = oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"])
    for _ in range(3):
        o.evolve(0.05)
        o.resample(s)
    g = batch.copy_state(0)
    assert np.array_equal(g["anc"], o.anc)
    assert_state_equal(g, o, batch.W, "large population run")
    np.testing.assert_allclose(batch.estimate_psi()[0][0], o.estimates()[0], rtol=PSI_RTOL)


def test_full_size_large_population_one_interval(pg):
    # one population at the largest size (L = 128, N_c = 2^20), one interval
    q = dict(L=128, N=64, n_clones=2**20, seed=2000)
    s = 15.0 / 128**2
    batch = pg.PopulationBatch([q])
    batch.evolve(0.05, [s])
    batch.resample()
    o = oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"])
    o.evolve(0.05)
    o.resample(s)
    g = batch.copy_state(0)
    assert np.array_equal(g["anc"], o.anc)
    assert np.array_equal(g["dK"], o.dK)
    assert_state_equal(g, o, batch.W, "large population")
    np.testing.assert_allclose(batch.estimate_psi()[0][0], o.estimates()[0], rtol=PSI_RTOL)


def test_set_state_from_host(pg):
    q = dict(L=70, N=33, n_clones=1500, seed=42)
    words = workloads.random_subsets(q["L"], q["N"], q["n_clones"], seed=9)
    K0 = np.arange(q["n_clones"], dtype=np.int32)
    batch = pg.PopulationBatch([q])
    batch.set_state(0, words, K0)
    g = batch.copy_state(0)
    assert np.array_equal(g["lattice"], words) and np.array_equal(g["K"], K0)
    sites = np.zeros((q["n_clones"], q["L"]), dtype=np.uint8)
    for i in range(q["L"]):
        sites[:, i] = (words[:, i // 64] >> np.uint64(i % 64)) & np.uint64(1)
    out, K, dK = oracle.evolve_sites(q["L"], sites, 0.1, beta=1, seed=q["seed"], K=K0)
    batch.evolve(0.1, [0.1])
    g = batch.copy_state(0)
    assert np.array_equal(g["lattice"], oracle.sites_to_words(out, batch.W))
    assert np.array_equal(g["K"], K) and np.array_equal(g["dK"], dK)
    with pytest.raises(pg.PopError):
        bad = words.copy()
        bad[0, 0] ^= np.uint64(1)   # wrong particle number
        pg.PopulationBatch([q]).set_state(0, bad)


def test_call_order_and_bias_errors(pg):
    batch = pg.PopulationBatch([dict(L=20, N=10, n_clones=100, seed=1)])
    with pytest.raises(pg.PopError) as e:
        batch.resample()
    assert e.value.status == pg.POP_ERR_STATE
    with pytest.raises(pg.PopError) as e:
        batch.estimate_psi()
    assert e.value.status == pg.POP_ERR_STATE
    batch.evolve(0.1, [0.2])
    with pytest.raises(pg.PopError) as e:
        batch.evolve(0.1, [0.2])
    assert e.value.status == pg.POP_ERR_STATE
    batch.resample()
    with pytest.raises(pg.PopError) as e:
        batch.evolve(0.1, [0.3])
    assert e.value.status == pg.POP_ERR_STATE
    with pytest.raises(pg.PopError) as e:
        batch.evolve(-0.1, [0.2])
    assert e.value.status == pg.POP_ERR_ARG


@pytest.mark.parametrize("L,N,nc,s,dt", [
    (129, 64, 1100, 0.01, 0.05),     # narrowest ring of the one-clone-per-warp evolve
    (200, 37, 2100, -0.02, 0.05),
    (256, 128, 1025, 0.003, 0.05),   # exactly two lanes of sites
    (1000, 500, 700, 0.001, 0.01),
    (4096, 2048, 300, 0.0001, 0.005),  # widest ring: all 32 lanes, closing bond in lane 31
    (3000, 1, 500, 0.5, 0.2),        # one particle on a long ring
])
def test_parity_wide_rings(pg, L, N, nc, s, dt):
    run_parity(pg, [dict(L=L, N=N, n_clones=nc, seed=77 + L)], [s], dt, 3)


def test_parity_mixed_batch_wide(pg):
    # one ring above 128 sites puts every population of the batch on the wide path
    pops = [dict(L=50, N=25, n_clones=1500, seed=1), dict(L=300, N=150, n_clones=1100, seed=2),
            dict(L=7, N=3, n_clones=900, seed=3)]
    run_parity(pg, pops, [0.02, 0.004, -0.3], 0.05, 3)


MOD, IID = 1, 1


@pytest.mark.parametrize("L,N,nc,s,mode,sel", [
    (20, 10, 1500, 0.3, MOD, 0),
    (50, 25, 2100, -0.2, MOD, 0),
    (100, 40, 1100, 0.05, MOD, 0),       # two-word lattices
    (300, 150, 600, 0.01, MOD, 0),       # one clone per warp
    (37, 5, 1, 0.5, MOD, 0),             # one clone
    (20, 10, 1500, 0.3, 0, IID),
    (64, 31, 1300, -0.1, MOD, IID),
    (200, 100, 800, 0.02, 0, IID),       # one clone per warp
    (12, 0, 300, 0.3, MOD, 0),           # empty ring: A = 0, equal weights
])
def test_parity_modified_and_iid(pg, L, N, nc, s, mode, sel):
    pops = [dict(L=L, N=N, n_clones=nc, seed=555 + L, weight_mode=mode, selection=sel)]
    run_parity(pg, pops, [s], 0.1 if L < 100 else 0.05, 5)


def test_parity_mixed_modes_batch(pg):
    pops = [dict(L=30, N=15, n_clones=1200, seed=1),
            dict(L=40, N=20, n_clones=2100, seed=2, weight_mode=MOD),
            dict(L=50, N=25, n_clones=900, seed=3, selection=IID),
            dict(L=60, N=20, n_clones=1500, seed=4, weight_mode=MOD, selection=IID)]
    run_parity(pg, pops, [0.1, -0.05, 0.02, 0.3], 0.1, 4)


def test_parity_iid_beyond_the_staged_tile_prefixes(pg):
    # [iid] selection searches the tile prefixes first: from shared memory for up to
    # 2048 tiles, from global memory beyond (here 2101 tiles with a ragged last one)
    # next to a population of 3 tiles
    pops = [dict(L=20, N=10, n_clones=2100 * 1024 + 5, seed=91, selection=IID),
            dict(L=30, N=12, n_clones=2500, seed=92, selection=IID)]
    run_parity(pg, pops, [0.05, -0.1], 0.1, 2)


@pytest.mark.parametrize("L,dt", [(20, 10.0), (50, 1.0), (50, 10.0)])
def test_selection_study_state_point_matches_oracle(pg, L, dt):
    # the cloning-interval and selection study's configuration (lambda = 28, [eq] and
    # [iid], plain and MODIFIED weights in one batch, long intervals with wide activity
    # spreads), truncated to a few intervals: bit for bit against the oracle
    s = 28.0 / L ** 2
    pops = [dict(L=L, N=L // 2, n_clones=2100, seed=70 + 10 * m + e, weight_mode=m, selection=e)
            for m in (0, MOD) for e in (0, IID)]
    run_parity(pg, pops, [s] * 4, dt, 3)


@pytest.mark.parametrize("L,N,nc,W_case", [(50, 25, 2500, 1), (100, 50, 1300, 2), (300, 90, 700, 0)])
def test_density_mode_matches_oracle(pg, L, N, nc, W_case):
    q = dict(L=L, N=N, n_clones=nc, seed=31 + L)
    s = 20.0 / L**2
    batch = pg.PopulationBatch([q])
    o = oracle.Population(L, N, nc, q["seed"])
    for _ in range(4):
        batch.evolve(0.1, [s]); batch.resample()
        o.evolve(0.1); o.resample(s)
    for n in (0, 1, 3):
        got = batch.density_mode(n)[0]
        np.testing.assert_allclose(got, oracle.density_mode(o.sites, n), rtol=1e-12)


def test_full_size_uneven_batch_sampled(pg):
    # 256 populations of uneven L (32..128), N_c (2^10..2^18) and s, one batch, in
    # the captured-graph launch (pop_run); three small populations checked bit for
    # bit, invariants everywhere
    w = workloads.uneven_batch()
    M = 3
    batch = pg.PopulationBatch(w["pops"])
    batch.run(w["dt"], w["s"], M)
    psi, _, _ = batch.estimate_psi()
    ncs = np.array([q["n_clones"] for q in w["pops"]])
    for p in np.argsort(ncs)[:3]:
        q = w["pops"][p]
        o = oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"])
        for _ in range(M):
            o.evolve(w["dt"])
            o.resample(w["s"][p])
        g = batch.copy_state(int(p))
        assert np.array_equal(g["anc"], o.anc)
        assert_state_equal(g, o, batch.W, "uneven pop %d" % p)
        np.testing.assert_allclose(psi[p], o.estimates()[0], rtol=PSI_RTOL)
    for p in range(0, 256, 17):
        g = batch.copy_state(p)
        assert np.all(np.diff(g["anc"]) >= 0)
        assert g["anc"].max() < w["pops"][p]["n_clones"]
        assert np.all(np.isfinite(psi))


@pytest.mark.parametrize("case", ["one_word", "two_words_modified"])
def test_cloning_stage_beyond_4096_tiles(pg, case):
    # batches of more than 4096 tiles take the 256-thread cloning stage, and
    # populations of more than 64 tiles take their tile prefixes from k_tile_scan
    # (here over several 1024-tile chunks): every population checked bit for bit
    # against the oracle each interval, and in the large ones every new clone is its
    # ancestor's evolved clone with [eq] ancestors non-decreasing
    if case == "one_word":
        pops = [dict(L=20, N=10, n_clones=1500, seed=41), dict(L=30, N=15, n_clones=2100 * 1024, seed=42),
                dict(L=64, N=31, n_clones=777, seed=43, selection=1), dict(L=50, N=25, n_clones=2048 * 1024, seed=44),
                dict(L=40, N=20, n_clones=3000, seed=45, weight_mode=1)]
        s = [0.05, 0.01, -0.2, 0.02, 0.3]
    else:
        pops = [dict(L=100, N=50, n_clones=1100, seed=46, weight_mode=1),
                dict(L=128, N=64, n_clones=4096 * 1024, seed=47),
                dict(L=65, N=30, n_clones=2500, seed=48, weight_mode=1)]
        s = [0.1, 0.003, -0.1]
    batch = pg.PopulationBatch(pops)
    assert batch.slots // 1024 > 4096
    big = [p for p, q in enumerate(pops) if q["n_clones"] > 64 * 1024]
    orcs = oracle_pops(pops)
    for beta in range(1, 3):
        batch.evolve(0.1, s)
        evolved = {p: batch.copy_state(p) for p in big}
        batch.resample()
        for p, o in enumerate(orcs):
            o.evolve(0.1, s[p])
            o.resample(s[p])
            g = batch.copy_state(p)
            assert np.array_equal(g["anc"], o.anc), "anc beta=%d pop %d" % (beta, p)
            assert_state_equal(g, o, batch.W, "beta=%d pop %d" % (beta, p))
        for p in big:
            g, e = batch.copy_state(p), evolved[p]
            anc = g["anc"]
            assert np.all(np.diff(anc) >= 0)
            assert np.array_equal(g["lattice"], e["lattice"][anc]), "lattice beta=%d pop %d" % (beta, p)
            assert np.array_equal(g["K"], e["K"][anc]), "K beta=%d pop %d" % (beta, p)
    psi, _, _ = batch.estimate_psi()
    for p, o in enumerate(orcs):
        np.testing.assert_allclose(psi[p], o.estimates()[0], rtol=PSI_RTOL, atol=0.0)


def test_autotune_changes_no_result(pg):
    pops = [dict(L=50, N=25, n_clones=5000, seed=9), dict(L=128, N=64, n_clones=3000, seed=10)]
    s = [0.01, -0.002]
    a = pg.PopulationBatch(pops)
    tuned = a.autotune(0.1, s, trials=3)
    assert tuned["evolve_grid"] > 0 and tuned["tuned_us_per_interval"] > 0
    assert tuned["tuned_us_per_interval"] <= tuned["default_us_per_interval"]
    b = pg.PopulationBatch(pops)
    a.run(0.1, s, 40)
    b.run(0.1, s, 40)
    for p in range(2):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), key
    np.testing.assert_array_equal(a.estimate_psi()[0], b.estimate_psi()[0])
    np.testing.assert_array_equal(a.events(), b.events())
    with pytest.raises(pg.PopError):
        a.autotune(0.1, s)   # only before the first interval


@pytest.mark.parametrize("cfg", [
    dict(fuse_threads=128, fuse_clones=1, chains=1), dict(fuse_threads=128, fuse_clones=2, chains=1),
    dict(fuse_threads=256, fuse_clones=1, chains=1), dict(fuse_threads=128, fuse_clones=1, chains=2),
    dict(fuse_threads=128, fuse_clones=2, chains=4), dict(fuse_threads=256, fuse_clones=1, chains=8),
    dict(evolve_grid=7, chains=3), dict(gather_threads=256), dict(gather_threads=128),
    dict(hist_mode=0), dict(hist_mode=1, chains=4), dict(hist_mode=0, fuse_clones=2, chains=2)])
def test_every_tuned_parameter_changes_no_result(pg, cfg):
    # every value of every tuned parameter gives the same lattices, activities,
    # ancestors and psi as the configuration pop_init chose (a fused batch of five
    # populations, mixed L and tile counts, both signs of s)
    pops = [dict(L=50, N=25, n_clones=5000, seed=31), dict(L=128, N=64, n_clones=3000, seed=32),
            dict(L=100, N=40, n_clones=1100, seed=33), dict(L=70, N=35, n_clones=2500, seed=34),
            dict(L=128, N=60, n_clones=4100, seed=35)]
    s = [0.01, -0.002, 0.004, 0.0, 0.02]
    a = pg.PopulationBatch(pops)
    a.set_tuning(**cfg)
    got = a.get_tuning()
    for k, v in cfg.items():
        assert got[k] == v or (k == "chains" and 1 <= got[k] <= v), (k, got[k], v)
    b = pg.PopulationBatch(pops)
    a.run(0.1, s, 37)
    b.run(0.1, s, 37)
    for p in range(len(pops)):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), (p, key)
    np.testing.assert_array_equal(a.estimate_psi()[0], b.estimate_psi()[0])
    np.testing.assert_array_equal(a.events(), b.events())


def test_gather_tuning_of_a_batch_that_does_not_fuse_changes_no_result(pg):
    # an [iid] population keeps the separate cloning stage, whose block size the tuner
    # times on trials that write the population (kept aside and put back)
    pops = [dict(L=50, N=25, n_clones=6000, seed=41, selection=pg.POP_IID),
            dict(L=128, N=64, n_clones=5000, seed=42)]
    s = [0.01, 0.003]
    a = pg.PopulationBatch(pops)
    tuned = a.autotune(0.1, s, trials=2)
    assert tuned["gather_threads"] in (0, 128, 256)
    b = pg.PopulationBatch(pops)
    a.run(0.1, s, 20)
    b.run(0.1, s, 20)
    for p in range(2):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), (p, key)
    np.testing.assert_array_equal(a.estimate_psi()[0], b.estimate_psi()[0])


def test_set_tuning_rejects_out_of_range(pg):
    a = pg.PopulationBatch([dict(L=50, N=25, n_clones=2000, seed=1)])
    for bad in (dict(fuse_threads=64), dict(fuse_clones=3), dict(fuse_threads=256, fuse_clones=2),
                dict(chains=0), dict(chains=9), dict(gather_threads=512), dict(evolve_grid=0),
                dict(hist_mode=2), dict(hist_mode=-2)):
        with pytest.raises(pg.PopError):
            a.set_tuning(**bad)


def test_kernel_times_equals_run_and_counts(pg):
    # pop_kernel_times launches what pop_run launches (results identical); the
    # launch counters follow the fused sequence: one dynamical stage, then
    # (n - 1) x [weights, fused stage] per chain, then weights and the cloning stage.
    # With populations of more than 64 tiles (below) the fused stages count activities
    # per tile and, after the first fused interval, the tile scan takes k_weights' place
    # (a launch of the "weights" kind that also scans)
    pops = [dict(L=50, N=25, n_clones=3000, seed=21), dict(L=90, N=45, n_clones=2000, seed=22)]
    s = [0.02, -0.003]
    n = 40
    a = pg.PopulationBatch(pops)
    b = pg.PopulationBatch(pops)
    a.run(0.1, s, n)
    kt = b.kernel_times(0.1, s, n)
    for p in range(len(pops)):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), key
    np.testing.assert_array_equal(a.events(), b.events())
    # two chains (below): each fused interval is two launches of each kind, and the
    # reported time is the time during which either runs, per interval
    assert kt["evolve"][1] == 1 and kt["gather_evolve"][1] == 2 * (n - 1)
    assert kt["weights"][1] == 2 * (n - 1) + 1 and kt["gather"][1] == 1
    assert kt["evolve"][2] + kt["gather_evolve"][2] == int(b.events().sum())
    for name in ("evolve", "weights", "gather", "gather_evolve"):
        assert kt[name][0] > 0.0
    # pop_run splits this batch (3 + 2 tiles, each at least a quarter) into two chains,
    # each with its own [weights, fused stage] per interval, and kernel_times launches
    # the same chains
    assert a.run_chains() == [0, 3, 5] and b.run_chains() == [0, 3, 5]
    for batch, chains in ((a, 2), (b, 2)):
        c = batch.launch_count()
        assert c["evolve"] == 1 and c["gather_evolve"] == chains * (n - 1)
        assert c["weights"] == chains * (n - 1) + 1
        # the initial state, and the tile scan before the one separate cloning stage
        # (the fused stages of these 2- and 3-tile populations sum their tile sums)
        assert c["gather"] == 1 and c["other"] == 2
    # one population, or a split that would leave less than a quarter: one chain
    for pops1 in ([dict(L=50, N=25, n_clones=3000, seed=24)],
                  [dict(L=50, N=25, n_clones=9000, seed=25), dict(L=40, N=20, n_clones=2000, seed=26)]):
        d = pg.PopulationBatch(pops1)
        assert d.run_chains() == [0, d.slots // 1024]
        d.run(0.1, [0.02] * len(pops1), n)
        c = d.launch_count()
        assert c["gather_evolve"] == n - 1 and c["weights"] == n, pops1
    # [iid] batches keep the three separate kernels (and the [iid] selection) per interval
    c = pg.PopulationBatch([dict(L=30, N=15, n_clones=1500, seed=23, selection=1)])
    c.run(0.1, [0.1], 35)
    cnt = c.launch_count()
    assert cnt["evolve"] == 35 and cnt["weights"] == 35 and cnt["gather"] == 70
    assert cnt["gather_evolve"] == 0 and cnt["other"] == 1 + 35
    # populations of more than 64 tiles: the fused stage after k_weights takes the tile
    # scan too (once per chain, in the first fused interval); without the tile
    # histograms, in every interval
    big = [dict(L=50, N=25, n_clones=65 * 1024, seed=60 + i) for i in range(2)]
    d = pg.PopulationBatch(big)
    d.run(0.1, [0.02, 0.03], n)
    cnt = d.launch_count()
    chains = len(d.run_chains()) - 1
    assert cnt["gather_evolve"] == chains * (n - 1) and cnt["other"] == 1 + chains
    assert cnt["weights"] == chains * (n - 1) + 1
    d = pg.PopulationBatch(big)
    d.set_tuning(hist_mode=0)
    d.run(0.1, [0.02, 0.03], n)
    cnt = d.launch_count()
    assert cnt["gather_evolve"] == chains * (n - 1) and cnt["other"] == 1 + chains * (n - 1) + 1


@pytest.mark.parametrize("dt", [0.1, 1.5])
def test_tile_histograms_change_no_result(pg, dt):
    # the fused stage's per-tile activity counts (hist_mode 1) against k_weights'
    # pass over every clone (hist_mode 0): the same lattices, activities, ancestors and
    # psi bit for bit, over two chains and populations of one and many tiles.  At
    # dt = 1.5 the L = 128 populations hop about 100 times an interval, beyond the 64
    # counted activities, so their tile sums come from the slower pass over the clones
    # while the L = 20 population's still come from the counts
    pops = [dict(L=20, N=10, n_clones=5000, seed=71), dict(L=128, N=64, n_clones=70 * 1024, seed=72),
            dict(L=128, N=40, n_clones=3000, seed=73), dict(L=100, N=50, n_clones=66 * 1024, seed=74)]
    s = [0.05, 0.002, -0.01, 0.0]
    runs = []
    for mode in (1, 0):
        b = pg.PopulationBatch(pops)
        b.set_tuning(hist_mode=mode, chains=2)
        b.run(dt, s, 7)
        b.run(dt, s, 5)   # a second call: the counts of the first were all consumed
        runs.append(b)
    a, b = runs
    assert a.run_chains() == b.run_chains() and len(a.run_chains()) == 3
    for p in range(len(pops)):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), (p, key)
    np.testing.assert_array_equal(a.estimate_psi()[0], b.estimate_psi()[0])
    np.testing.assert_array_equal(a.events(), b.events())
    if dt > 1.0:
        assert int(b.copy_state(1)["dK"].max()) >= 64


def test_activity_spread_beyond_the_weight_table_is_reported(pg):
    # one particle on 128 sites, dt = 2.5e5: about 5e5 hops per clone with a spread of
    # ~5000 across 4000 clones, beyond the 4096-entry weight table: the cloning stage
    # reports POP_ERR_RANGE instead of indexing past the table
    b = pg.PopulationBatch([dict(L=128, N=1, n_clones=4000, seed=3)])
    b.evolve(2.5e5, [0.001])
    b.resample()
    with pytest.raises(pg.PopError) as e:
        b.events()
    assert e.value.status == pg.POP_ERR_RANGE
    b.close()
    # the device stays usable
    ok = pg.PopulationBatch([dict(L=20, N=10, n_clones=100, seed=4)])
    ok.run(0.1, [0.1], 3)
    assert np.isfinite(ok.estimate_psi()[0][0])


def test_an_interval_that_cannot_end_stops_at_the_step_limit(pg):
    # dt = 1e7 in FP32: once t is near 1e7 a waiting time of ~0.5 no longer changes t,
    # so only the per-interval step limit (2^24 steps) ends the clone's loop; the
    # kernel reports POP_ERR_RANGE and returns instead of spinning
    b = pg.PopulationBatch([dict(L=128, N=1, n_clones=1, seed=5)])
    b.evolve(1e7, [0.0])
    with pytest.raises(pg.PopError) as e:
        b.events()
    assert e.value.status == pg.POP_ERR_RANGE
    b.close()
    # the same through pop_run: the fused cloning + dynamical stage of the second
    # interval stops at the limit too
    b = pg.PopulationBatch([dict(L=128, N=1, n_clones=1, seed=6)])
    b.run(1e7, [0.0], 2)
    with pytest.raises(pg.PopError) as e:
        b.events()
    assert e.value.status == pg.POP_ERR_RANGE
    b.close()


@pytest.mark.parametrize("L,nc,mode,sel", [
    (255, 33, 0, 0), (256, 1025, MOD, IID),      # one lane per clone
    (257, 1500, MOD, 0), (512, 65, 0, IID),      # two lanes: one site in the second, both full
    (513, 70, 0, 0), (1024, 40, MOD, 0),         # four
    (1025, 31, MOD, IID), (2048, 17, 0, 0),      # eight
    (2049, 9, 0, 0),                             # sixteen
])
def test_parity_at_the_edges_of_the_lanes_of_a_wide_ring(pg, L, nc, mode, sel):
    # a second, short ring shares the batch: its clones leave all but the first lane empty
    pops = [dict(L=L, N=L // 3, n_clones=nc, seed=300 + L, weight_mode=mode, selection=sel),
            dict(L=11, N=5, n_clones=nc + 3, seed=301 + L, selection=sel)]
    run_parity(pg, pops, [10.0 / L ** 2, -0.1], 8.0 / L, 3)


@pytest.mark.parametrize("pops,s,dt,splits", [
    ([dict(L=20, N=10, n_clones=1, seed=1)], [0.3], 0.1, [2, 1]),
    ([dict(L=20, N=10, n_clones=31, seed=2), dict(L=50, N=25, n_clones=33, seed=3)], [0.3, -0.1], 0.1, [31, 1, 33]),
    ([dict(L=64, N=32, n_clones=1024, seed=4), dict(L=3, N=1, n_clones=32, seed=5, weight_mode=MOD)],
     [0.02, 0.4], 0.2, [34]),                    # every thread a clone; MODIFIED beside plain
    ([dict(L=65, N=30, n_clones=1023, seed=6, weight_mode=MOD), dict(L=12, N=0, n_clones=40, seed=7, weight_mode=MOD)],
     [-0.05, 0.3], 0.3, [40]),                   # two words; an empty ring
    ([dict(L=128, N=64, n_clones=700, seed=8), dict(L=40, N=20, n_clones=900, seed=9)], [0.5, 2.5], 0.2, [33]),
    ([dict(L=128, N=1, n_clones=1000, seed=10)], [1e-4], 3000.0, [2]),  # activities over more bins than shared memory counts
    ([dict(L=16, N=8, n_clones=40, seed=11)], [0.1], 0.1, [1030]),      # more intervals than one launch takes
])
def test_one_tile_populations_run_equals_steps(pg, pops, s, dt, splits):
    a = pg.PopulationBatch(pops)
    b = pg.PopulationBatch(pops)
    for n in splits:
        a.run(dt, s, n)
    assert a.launch_count()["gather_evolve"] == sum((n + 1023) // 1024 for n in splits)
    for _ in range(sum(splits)):
        b.evolve(dt, s)
        b.resample()
    for p in range(len(pops)):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), (p, key)
    pa, ka, ta = a.estimate_psi()
    pb, kb, tb = b.estimate_psi()
    np.testing.assert_allclose(pa * ta, pb * tb, rtol=1e-15)
    np.testing.assert_allclose(ka * ta, kb * tb, rtol=1e-14)
    np.testing.assert_array_equal(a.events(), b.events())
    a.evolve(dt, s)                             # and the per-step calls go on from there
    b.run(dt, s, 1)
    a.resample()
    assert np.array_equal(a.copy_state(0)["lattice"], b.copy_state(0)["lattice"])


def test_one_tile_populations_tune_and_time_without_changing_results(pg):
    pops = [dict(L=50, N=25, n_clones=500 + 100 * i, seed=80 + i) for i in range(4)]
    s = [0.01, 0.02, -0.01, 0.0]
    a, b, c = (pg.PopulationBatch(pops) for _ in range(3))
    assert a.autotune(0.1, s)["tuned_us_per_interval"] > 0.0
    for x in (a, b):
        x.run(0.1, s, 36)
    kt = c.kernel_times(0.1, s, 36)
    assert kt["gather_evolve"][1] == 1 and kt["gather_evolve"][2] == int(c.events().sum())
    for p in range(4):
        ga, gb, gc = (x.copy_state(p) for x in (a, b, c))
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]) and np.array_equal(gc[key], gb[key]), (p, key)


def test_many_one_tile_populations_keep_the_launch_sequence(pg):
    # four times as many populations as blocks of 1024 threads the device holds
    import torch
    P = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    pops = [dict(L=20, N=10, n_clones=1000 + i % 3, seed=i) for i in range(P)]
    a = pg.PopulationBatch(pops)
    a.run(0.1, [0.05] * P, 3)
    assert a.launch_count()["evolve"] == 1
    b = pg.PopulationBatch(pops[:5])
    b.run(0.1, [0.05] * 5, 3)
    for p in range(5):
        assert np.array_equal(a.copy_state(p)["lattice"], b.copy_state(p)["lattice"])


@pytest.mark.parametrize("mode,sel", [(0, IID), (MOD, IID), (0, 0)])
@pytest.mark.parametrize("L,nc,s,dt", [
    (40, 5000, 2.5, 0.3),    # long runs of tiny weights
    (10, 9000, 6.0, 2.0),    # a few clones own nearly every new slot, more than a tile's map holds
    (20, 2049, -1.5, 0.3),   # the largest activity is the reference; a tile of one clone
])
def test_parity_under_strong_bias(pg, L, nc, s, dt, mode, sel):
    run_parity(pg, [dict(L=L, N=L // 2, n_clones=nc, seed=600 + L, weight_mode=mode, selection=sel)], [s], dt, 3)


def test_positions_too_close_to_a_slot_are_settled_exactly(pg, tmp_path):
    # the cloning stage takes a clone's new slots from 64-bit positions and settles those
    # within POP_POS_MARGIN of a slot by 128-bit comparisons; by default that is one clone
    # in 2^28 at N_c = 2^20.  A library built with the margin 2^17 times as wide takes that
    # path for about a clone in two thousand (four tiles in ten): separate and fused stages against
    # the per-step calls of the ordinary library, which the oracle tests check
    import ctypes
    import subprocess
    from paper_1711_05095_gb300 import build as b
    so = str(tmp_path / "libpop_margin.so")
    subprocess.run([b.nvcc(), "-O3", "-std=c++17", *b.ARCH, "-Xcompiler", "-fPIC", "-shared", "-DPOP_POS_MARGIN=(1ull<<30)",
                    "-I", b.ROOT + "/include", *b.SOURCES, "-o", so], check=True)
    pops = [dict(L=50, N=25, n_clones=200 * 1024 + 7, seed=90), dict(L=128, N=64, n_clones=2 ** 20, seed=91),
            dict(L=30, N=15, n_clones=70 * 1024, seed=92, weight_mode=MOD)]
    few = [dict(L=40, N=20, n_clones=60 * 1024 + 3, seed=93), dict(L=20, N=10, n_clones=9 * 1024, seed=94)]
    cases = ((pops, [0.02, 0.001, -0.01]), (few, [0.3, -0.1]))
    want = []
    for q, s in cases:
        a = pg.PopulationBatch(q)
        for _ in range(4):
            a.evolve(0.1, s)
            a.resample()
        want.append([a.copy_state(p) for p in range(len(q))])
        a.close()
    saved, path = pg._lib, pg.LIB_PATH
    try:
        pg._lib, pg.LIB_PATH = None, so
        for (q, s), w in zip(cases, want):
            for fused in (True, False):
                a = pg.PopulationBatch(q)
                if fused:
                    a.run(0.1, s, 4)
                else:
                    for _ in range(4):
                        a.evolve(0.1, s)
                        a.resample()
                for p in range(len(q)):
                    g = a.copy_state(p)
                    for key in ("lattice", "K", "anc", "dK"):
                        assert np.array_equal(g[key], w[p][key]), (p, key, fused)
                a.close()
    finally:
        pg._lib, pg.LIB_PATH = saved, path


def test_one_tile_launches_are_bounded_and_stop_at_the_step_limit(pg):
    # 64 active bonds at rate 1 or so for dt = 100: some thousands of draws per clone and
    # interval, so a launch takes five intervals (32768 draws over 0.5 x 128 x 100 + 1)
    a = pg.PopulationBatch([dict(L=128, N=64, n_clones=40, seed=70)])
    a.run(100.0, [0.0], 11)
    assert a.launch_count()["gather_evolve"] == 3
    b = pg.PopulationBatch([dict(L=128, N=64, n_clones=40, seed=70)])
    for _ in range(11):
        b.evolve(100.0, [0.0])
        b.resample()
    for key in ("lattice", "K", "anc", "dK"):
        assert np.array_equal(a.copy_state(0)[key], b.copy_state(0)[key]), key
    # intervals that only the step limit ends: the first is reported and the others are not
    # run, so sixteen take the time of one (and not sixteen times that)
    import time

    def seconds(n):
        c = pg.PopulationBatch([dict(L=128, N=1, n_clones=1, seed=71)])
        t = time.perf_counter()
        c.run(1e7, [0.0], n)
        with pytest.raises(pg.PopError) as e:
            c.events()
        assert e.value.status == pg.POP_ERR_RANGE
        t = time.perf_counter() - t
        c.close()
        return t

    one = seconds(1)
    assert seconds(16) < 4.0 * one


@pytest.mark.parametrize("pops", [[dict(L=30, N=15, n_clones=300, seed=73), dict(L=20, N=10, n_clones=1024, seed=74)],
                                  [dict(L=30, N=15, n_clones=3000, seed=75)]])
def test_a_captured_run_goes_on_from_the_population_when_replayed(pg, pops):
    # the interval number is the device's, not one fixed when the call was captured: two
    # intervals replayed three times after a first are intervals 2 .. 7, and the next call is
    # the eighth (one-tile populations, and the fused launches)
    import torch
    s = [0.02] * len(pops)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        a = pg.PopulationBatch(pops)
        a.run(0.1, s, 1)
        g = torch.cuda.CUDAGraph()
        st.synchronize()
        with torch.cuda.graph(g, stream=st):
            a.run(0.1, s, 2)
        for _ in range(3):
            g.replay()
        a.run(0.1, s, 1)
        b = pg.PopulationBatch(pops)
        b.run(0.1, s, 8)
        st.synchronize()
    np.testing.assert_array_equal(a.events(), b.events())
    for p in range(len(pops)):
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(a.copy_state(p)[key], b.copy_state(p)[key]), (p, key)


def test_events_of_a_share_of_more_than_2_to_the_32_hops(pg):
    # one block: 32768 clones to a warp, some 139800 hops each (4300 x 32.5), 4.6e9 > 2^32
    b = pg.PopulationBatch([dict(L=64, N=32, n_clones=2 ** 17, seed=76)])
    b.set_tuning(evolve_grid=1)
    b.evolve(4300.0, [0.0])
    hops = int(b.copy_state(0)["dK"].astype(np.int64).sum())
    assert hops > 4 * 2 ** 32
    assert int(b.events()[0]) == hops


@pytest.mark.parametrize("L", [40, 64, 100, 200, 400, 1000, 2000, 3000])
@pytest.mark.parametrize("mode", [0, MOD])
def test_long_intervals_counted_in_64_bits_match_oracle(pg, L, mode):
    # from 2^20 hops per clone on the dynamical stage counts in 64 bits, in kernels of its own
    # (two active bonds for dt = 530000; e^-s nearly 1); a short ring beside the others
    pops = [dict(L=L, N=1, n_clones=5 if L <= 128 else 1, seed=400 + L, weight_mode=mode), dict(L=9, N=1, n_clones=2, seed=401 + L)]
    s = [-1e-6, 0.0]
    b = pg.PopulationBatch(pops)
    b.evolve(530000.0, s)
    events = b.events()
    for p, q in enumerate(pops):
        o = oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"], modified=q.get("weight_mode", 0) == MOD)
        o.evolve(530000.0, s[p])
        g = b.copy_state(p)
        assert np.array_equal(g["lattice"], oracle.sites_to_words(o.sites, b.W)), p
        assert np.array_equal(g["K"], o.K) and np.array_equal(g["dK"], o.dK), p
        assert int(events[p]) == int(o.dK.astype(np.int64).sum()), p


def test_setting_one_tuned_parameter_leaves_the_others(pg):
    # the fused kernel's form stays the rule's (fuse_threads 0: 256 threads in a batch within
    # one wave) until it is set itself, and can be given back to the rule
    pops = [dict(L=50, N=25, n_clones=5000, seed=31), dict(L=40, N=20, n_clones=3000, seed=32)]
    s = [0.01, 0.02]
    a = pg.PopulationBatch(pops)
    before = a.get_tuning()
    assert before["fuse_threads"] == 0
    a.set_tuning()
    assert a.get_tuning() == before
    b = pg.PopulationBatch(pops)
    b.run(0.1, s, 5)
    for cfg in (dict(chains=1), dict(hist_mode=0), dict(evolve_grid=5), dict(gather_threads=256), dict(fuse_clones=2),
                dict(fuse_threads=128), dict(fuse_threads=128, fuse_clones=2), dict(fuse_threads=256, fuse_clones=1)):
        c = pg.PopulationBatch(pops)
        c.set_tuning(**cfg)
        got = c.get_tuning()
        assert got == dict(before, **cfg), cfg
        c.run(0.1, s, 5)
        for p in range(2):
            for key in ("lattice", "K", "anc", "dK"):
                assert np.array_equal(b.copy_state(p)[key], c.copy_state(p)[key]), (cfg, p, key)
        c.set_tuning(**{k: before[k] for k in cfg})
        assert c.get_tuning() == before
    with pytest.raises(pg.PopError):
        a.set_tuning(fuse_threads=256, fuse_clones=2)


@pytest.mark.parametrize("rings", [[(50, 0), (64, 1), (64, 5), (64, 6), (20, 20)], [(128, 6), (128, 7), (65, 1), (40, 7)],
                                   [(256, 8), (256, 9), (30, 8)], [(1025, 8), (1025, 9), (4096, 2), (17, 1)],
                                   [(64, 5), (30, 0), (64, 1)], [(128, 6), (100, 3)], [(4096, 8), (200, 1)]])
def test_density_mode_of_few_particles_matches_oracle(pg, rings):
    # either side of the line between the sums by particles and by sites, rings shorter than
    # the batch's words among them; a tile and a ragged one.  Both sum a clone in FP32 in the
    # order of the sites, so only the FP64 sum over the clones may differ
    pops = [dict(L=L, N=N, n_clones=1025 + 3 * i, seed=500 + i) for i, (L, N) in enumerate(rings)]
    b = pg.PopulationBatch(pops)
    orcs = [oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"]) for q in pops]
    for n in (1, 2):
        got = b.density_mode(n)
        for p, o in enumerate(orcs):
            np.testing.assert_allclose(got[p], oracle.density_mode(o.sites, n), rtol=1e-12, err_msg=str(rings[p]))


# what the forms of the fused kernel differ in beside RUN_CASES: MODIFIED weights and rings
# that fill their words in populations of more than 64 tiles, which scan their tile sums
FORM_CASES = dict({k: v for k, v in RUN_CASES.items() if k != "iid_unfused"},
                  w1_modified_scan=([dict(L=30, N=15, n_clones=65 * 1024 + 5, seed=27, weight_mode=1),
                                     dict(L=64, N=32, n_clones=66 * 1024, seed=28)], [0.05, -0.01], [4]),
                  w1_full_modified=([dict(L=64, N=32, n_clones=3000, seed=29, weight_mode=1)], [0.02], [4]),
                  w1_full_scan=([dict(L=64, N=32, n_clones=66 * 1024, seed=30)], [0.02], [4]),
                  w2_full_scan=([dict(L=128, N=64, n_clones=65 * 1024 + 1, seed=31)], [0.01], [4]),
                  w2_modified_scan=([dict(L=100, N=50, n_clones=65 * 1024 + 1, seed=32, weight_mode=1)], [0.01], [4]),
                  w2_full_modified_scan=([dict(L=128, N=64, n_clones=65 * 1024 + 1, seed=33, weight_mode=1)], [0.01], [4]))


@pytest.mark.parametrize("form", [dict(fuse_threads=128, fuse_clones=1), dict(fuse_threads=128, fuse_clones=2),
                                  dict(fuse_threads=256, fuse_clones=1)], ids=["128", "128x2", "256"])
@pytest.mark.parametrize("case", sorted(FORM_CASES))
def test_every_form_of_the_fused_stage_equals_steps(pg, case, form):
    pops, s, splits = FORM_CASES[case]
    a = pg.PopulationBatch(pops)
    a.set_tuning(**form)
    b = pg.PopulationBatch(pops)
    for n in splits:
        a.run(0.1, s, n)
    for _ in range(sum(splits)):
        b.evolve(0.1, s)
        b.resample()
    for p in range(len(pops)):
        ga, gb = a.copy_state(p), b.copy_state(p)
        for key in ("lattice", "K", "anc", "dK"):
            assert np.array_equal(ga[key], gb[key]), (p, key)
    pa, _, ta = a.estimate_psi()
    pb, _, tb = b.estimate_psi()
    np.testing.assert_allclose(pa * ta, pb * tb, rtol=1e-15)
    np.testing.assert_array_equal(a.events(), b.events())


def test_step_limit_of_every_stage(pg, tmp_path):
    # a library whose step limit is 64 steps (32 draws) per interval: intervals within it give
    # what the ordinary library gives (a lane of the fused stage makes more draws than that, of
    # several clones), longer ones end and are reported, by every form of every stage
    import ctypes
    import subprocess
    from paper_1711_05095_gb300 import build as b
    so = str(tmp_path / "libpop_limit.so")
    subprocess.run([b.nvcc(), "-O3", "-std=c++17", *b.ARCH, "-Xcompiler", "-fPIC", "-shared", "-DPOP_STEP_LIMIT=64u",
                    "-I", b.ROOT + "/include", *b.SOURCES, "-o", so], check=True)
    forms = [dict(fuse_threads=128, fuse_clones=1), dict(fuse_threads=128, fuse_clones=2),
             dict(fuse_threads=256, fuse_clones=1)]
    batches = [[dict(L=20, N=10, n_clones=9000, seed=95)], [dict(L=20, N=10, n_clones=5000, seed=96, weight_mode=MOD)],
               [dict(L=20, N=10, n_clones=5000, seed=97), dict(L=100, N=2, n_clones=3000, seed=98)],
               [dict(L=100, N=2, n_clones=3000, seed=99, weight_mode=MOD)]]
    small = [[dict(L=20, N=10, n_clones=700, seed=85)], [dict(L=100, N=2, n_clones=1000, seed=86, weight_mode=MOD)]]
    s = [0.3, 0.1]

    def run(q, dt, n, form):
        a = pg.PopulationBatch(q)
        if form:
            a.set_tuning(**form)
        a.run(dt, s[:len(q)], n)
        return a

    # at rate 10.5 (L = 20) or 4 an interval of 1 takes 6 draws, hardly ever 32
    want = []
    for q in batches + small:
        x = run(q, 1.0, 6, None)
        want.append([x.copy_state(p) for p in range(len(q))])
        x.close()
    saved, path = pg._lib, pg.LIB_PATH
    try:
        pg._lib, pg.LIB_PATH = None, so
        for i, q in enumerate(batches + small):
            for form in forms if i < len(batches) else [None]:
                x = run(q, 1.0, 6, form)
                for p in range(len(q)):
                    g = x.copy_state(p)
                    for key in ("lattice", "K", "anc", "dK"):
                        assert np.array_equal(g[key], want[i][p][key]), (i, form, p, key)
                x.close()
        # the first interval, by the separate dynamical stage, stays within the limit (61, 62, 62
        # and 61 hops at most, by the oracle); of the other 39, by the fused stage or the
        # one-tile launch, several do not
        for q, dt in (([dict(L=20, N=10, n_clones=9000, seed=81)], 3.4),
                      ([dict(L=20, N=10, n_clones=9000, seed=82, weight_mode=MOD)], 3.4 / np.e),
                      ([dict(L=20, N=10, n_clones=9000, seed=83), dict(L=80, N=0, n_clones=3000, seed=84)], 3.2),
                      ([dict(L=20, N=10, n_clones=1024, seed=85)], 3.4)):
            sq = [-1.0] * len(q)
            x = pg.PopulationBatch(q)
            x.evolve(dt, sq)
            assert int(x.events()[0]) > 0          # no error
            x.close()
            for form in forms:
                x = pg.PopulationBatch(q)
                x.set_tuning(**form)
                x.run(dt, sq, 40)
                with pytest.raises(pg.PopError) as e:
                    x.events()
                assert e.value.status == pg.POP_ERR_RANGE
                x.close()
        # the dynamical stages
        for q in ([dict(L=20, N=10, n_clones=500, seed=87)], [dict(L=200, N=3, n_clones=50, seed=88)],
                  [dict(L=40, N=20, n_clones=50, seed=89, weight_mode=pg.POP_GUIDED)]):
            x = pg.PopulationBatch(q)
            x.evolve(50.0, [0.0])
            with pytest.raises(pg.PopError) as e:
                x.events()
            assert e.value.status == pg.POP_ERR_RANGE
            x.close()
    finally:
        pg._lib, pg.LIB_PATH = saved, path


@pytest.mark.parametrize("L,nc", [(20, 3), (20, 1500), (100, 2100), (300, 70)])
def test_a_population_without_weights_selects_in_range(pg, L, nc):
    # MODIFIED weights at e^-s beyond FP32: infinity times the clones' differences, so every
    # weight is 0 or not a number, which counts as 0.  [iid]: every point lies at the last
    # clone; [eq]: no point, so the clones stay as they are.  dt = 1e-38 at rates 4.5e38 makes
    # some 45 hops per clone, more than the smallest population has clones
    q = dict(L=L, N=L // 2, n_clones=nc, weight_mode=MOD)
    b = pg.PopulationBatch([dict(q, seed=610, selection=IID), dict(q, seed=611)])
    for _ in range(3):
        before = b.copy_state(1)
        b.evolve(1e-38 if L == 20 else 2e-39, [-89.0, -89.0])
        x = b.copy_state(0)
        assert x["dK"].max() > 3
        b.resample()
        g = b.copy_state(0)
        assert (g["anc"] == nc - 1).all()
        assert np.array_equal(g["lattice"], np.repeat(x["lattice"][-1:], nc, axis=0))
        assert np.array_equal(g["K"], np.repeat(x["K"][-1:], nc))
        after = b.copy_state(1)
        assert np.array_equal(after["lattice"], before["lattice"]) and np.array_equal(after["K"], before["K"])
    assert not np.isfinite(b.estimate_psi()[0]).any()


def test_kernel_times_of_one_tile_populations_are_per_interval(pg):
    # a launch of 30 intervals and launches of 3000: both some microseconds per interval
    us = []
    for n in (30, 3000):
        b = pg.PopulationBatch([dict(L=20, N=10, n_clones=1000, seed=77)])
        b.kernel_times(0.1, [0.05], 30)   # warm
        us.append(b.kernel_times(0.1, [0.05], n)["gather_evolve"][0])
    assert 0.2 < us[0] / us[1] < 5.0, us  # a sum over the launch would be a hundredth


@pytest.mark.parametrize("kind", ["plain", "modified", "wide", "guided"])
def test_even_shares_of_many_part_filled_populations(pg, kind):
    # 70 populations (the search for a warp's first one takes two rounds) of 1 to 2051 clones:
    # shares that begin and end anywhere in them, empty ones included, against the oracle
    g = np.random.default_rng(7)
    sizes = [1, 32, 33, 1024, 1025, 2051] + [int(v) for v in np.floor(2.0 ** g.uniform(0, 8, 64))]
    L = [20 if kind == "guided" else int(v) for v in g.integers(5, 60, 70)]
    if kind == "wide":
        L[3] = 300
    mode = {"modified": MOD, "guided": pg.POP_GUIDED}.get(kind, 0)
    pops = [dict(L=L[i], N=L[i] // 2, n_clones=sizes[i], seed=700 + i, weight_mode=mode) for i in range(70)]
    s = [float(v) for v in g.uniform(-0.1, 0.1, 70)]
    phi = g.normal(0.0, 0.3, 512).astype(np.float32)
    orcs = []
    for p, q in enumerate(pops):
        o = oracle.Population(q["L"], q["N"], q["n_clones"], q["seed"], modified=mode == MOD,
                              phi=phi if kind == "guided" else None)
        o.evolve(0.3, s[p])
        orcs.append(o)
    for grid in (None, 1, 3, 50):
        b = pg.PopulationBatch(pops)
        if kind == "guided":
            for p in range(70):
                b.set_potential(p, phi)
        if grid is not None:
            b.set_tuning(evolve_grid=grid)
        b.evolve(0.3, s)
        events = b.events()
        for p, o in enumerate(orcs):
            c = b.copy_state(p)
            assert np.array_equal(c["lattice"], oracle.sites_to_words(o.sites, b.W)), (grid, p)
            assert np.array_equal(c["dK"], o.dK) and np.array_equal(c["K"], o.K), (grid, p)
            assert int(events[p]) == int(o.dK.astype(np.int64).sum())
        b.close()
