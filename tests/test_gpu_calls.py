"""Calls of one generation and batches at the borders of their forms, bit for bit
against the CPU oracle: the ordered survivor list for slots of any length, and
members of every kind on one block or several."""
import numpy as np
import pytest

import oracle
import spegg_synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def gpu_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_09255_gb300 import build
    build.build()


def spegg():
    from paper_1603_09255_gb300 import spegg as m
    return m


def kinds(n, n_loci, seed):
    """A workload of every kind of member: plain, dominance, map, weights, both,
    and effects of two digits."""
    def base(i):
        return S.single_species(n=n, n_loci=n_loci, mu=1e-3, seed=seed, replicate=100 * n_loci + i)
    import dataclasses
    rng = np.random.default_rng(n_loci)
    wide = dataclasses.replace(base(5), effects=rng.integers(-32768, 32768, n_loci).astype(np.int16), bias=1 << 23,
                               shift=12)
    wide.surv_table = S.stabilizing_table(wide.bias, wide.shift, 1e-5)
    return [base(0), S.with_dominance(base(1)), S.with_linkage(base(2)), S.with_weights(base(3)),
            S.with_weights(S.with_linkage(base(4))), wide]


def assert_member(b, i, w, gens):
    orc = oracle.OraclePopulation.from_workload(w)
    so, sg = orc.step(gens), b.read_stats(i, 1, gens)
    for name in so.dtype.names:
        assert np.array_equal(so[name], sg[name]), (i, name)
    if w.allele_model == 0:
        assert np.array_equal(orc.genotypes(), b.genotypes(i)), i
    else:
        assert np.array_equal(orc.values(), b.values(i)), i
    assert np.array_equal(orc.survivors(), b.survivors(i)), i
    a, g = orc.state(), b.state(i)
    for k in ("gen", "S", "status", "f", "R"):
        assert a[k] == g[k], (i, k)


# slots of 1 word, of several (31 and 32 words: one pass; 33: two), the last one ragged
@pytest.mark.parametrize("n", [1000, 100_001, 2_412_480, 2_490_331, 2_490_400])
def test_list_of_slots_of_any_length(n):
    w = S.single_species(n=n, n_loci=32, mu=1e-3, seed=n)
    orc = oracle.OraclePopulation.from_workload(w)
    gpu = spegg().Population.from_workload(w, stats_capacity=4)
    orc.step(1)
    gpu.step(1)
    assert np.array_equal(orc.survivors(), gpu.survivors())
    assert np.array_equal(orc.genotypes(), gpu.genotypes())


def assert_population(gpu, orc, so, gens):
    sg = gpu.read_stats(1, gens)
    for name in so.dtype.names:
        assert np.array_equal(so[name], sg[name]), name
    assert np.array_equal(orc.genotypes(), gpu.genotypes())
    assert np.array_equal(orc.survivors(), gpu.survivors())
    a, g = orc.state(), gpu.state()
    for k in ("gen", "S", "status", "f", "R"):
        assert a[k] == g[k], k


@pytest.mark.parametrize("kind", range(6))
@pytest.mark.parametrize("n", [513, 15_361, 30_721, 77_825])
def test_one_generation_calls_of_every_kind(n, kind):
    """Calls of one generation, among longer ones, of every kind of population,
    with one, two and six runs of slots in the directory and slots of two words."""
    L = (32, 64, 128, 256)[(kind + n) % 4]
    w = kinds(n, L, 11)[kind]
    orc = oracle.OraclePopulation.from_workload(w)
    gpu = spegg().Population.from_workload(w, stats_capacity=8)
    for k in (1, 1, 2, 1):
        gpu.step(k)
    assert_population(gpu, orc, orc.step(5), 5)


@pytest.mark.parametrize("n", [700, 40_000])
def test_one_generation_calls_with_a_drawn_growth_rate(n):
    w = S.with_beverton_holt(S.consumer_resource(n=n, n_loci=64, K=50.0 * n, mu=1e-3, seed=n))
    orc = oracle.OraclePopulation.from_workload(w)
    gpu = spegg().Population.from_workload(w, stats_capacity=16)
    for _ in range(9):
        gpu.step(1)
    assert_population(gpu, orc, orc.step(9), 9)


@pytest.mark.parametrize("n", [400, 3000, 30_000])
def test_one_generation_call_under_stream_capture(n):
    w = S.single_species(n=n, n_loci=64, mu=1e-3, seed=8)
    stream = torch.cuda.Stream()
    gpu = spegg().Population.from_workload(w, stats_capacity=16, stream=stream)
    gpu.step(1)
    gpu.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        gpu.step(1)
        gpu.step(1)
    with torch.cuda.stream(stream):
        for _ in range(3):
            graph.replay()
    gpu.step(1)
    orc = oracle.OraclePopulation.from_workload(w)
    assert_population(gpu, orc, orc.step(8), 8)


def continuous(n, n_loci, seed):
    return S.continuous_trait(n=n, n_loci=n_loci, seed=seed, replicate=7)


@pytest.mark.parametrize("sizes", [(33, 700), (5000, 40_000)])
def test_batch_of_every_kind(sizes):
    """Records, survivors and state of members of every kind, sizes and locus
    counts mixed, after calls of one generation and of several."""
    ws = [w for n in sizes for L in (32, 128, 256) for w in kinds(n + L, L, 7)] + [continuous(sizes[0], 64, 3)]
    b = spegg().Batch(ws, stats_capacity=8)
    for k in (1, 1, 3):
        b.step(k)
    for i, w in enumerate(ws):
        assert_member(b, i, w, 5)


def test_batch_of_every_kind_longer_than_a_launch():
    """One member of each kind, over more generations than a launch holds."""
    ws = kinds(300, 32, 5) + [continuous(200, 32, 5)]
    b = spegg().Batch(ws, stats_capacity=600)
    b.step(530)
    b.step(7)
    for i, w in enumerate(ws):
        assert_member(b, i, w, 537)


def test_batch_of_every_kind_under_stream_capture():
    """The kinds' launches fork from the captured stream and join it."""
    ws = kinds(2000, 64, 6)
    stream = torch.cuda.Stream()
    b = spegg().Batch(ws, stats_capacity=16, stream=stream)
    b.step(1)
    b.step(3)
    b.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        b.step(3)
        b.step(1)
    with torch.cuda.stream(stream):
        graph.replay()
        graph.replay()
    b.step(1)
    for i, w in enumerate(ws):
        assert_member(b, i, w, 13)


def test_served_jobs_of_every_kind():
    ws = kinds(3000, 64, 8) + kinds(200, 256, 9) + [continuous(1000, 64, 8)]
    gens = [20 + 5 * (i % 4) for i in range(len(ws))]
    sv = spegg().Server(gens_per_tick=8, max_resident=9)
    jobs = [sv.submit(w, g, 0.0) for w, g in zip(ws, gens)]
    sv.drain()
    for w, g, j in zip(ws, gens, jobs):
        so, sg = oracle.OraclePopulation.from_workload(w).step(g), sv.job_stats(j, 1, g)
        for name in so.dtype.names:
            assert np.array_equal(so[name], sg[name]), (w.name, name)


def test_populations_on_streams_of_their_own():
    """Small and large populations stepped at the same time, with calls of one
    generation and of several, equal to the oracle's."""
    ws = [S.single_species(n=n, n_loci=32, mu=1e-3, seed=20 + i) for i, n in enumerate((10_000, 24_321, 300, 120_000, 10_000))]
    pops = [spegg().Population.from_workload(w, stats_capacity=32) for w in ws]
    for k in (5, 1, 1, 7):
        for p in pops:
            p.step(k)
    for w, p in zip(ws, pops):
        orc = oracle.OraclePopulation.from_workload(w)
        assert_population(p, orc, orc.step(14), 14)


@pytest.mark.parametrize("gens", [1, 3, 40])
def test_continuous_members_under_stream_capture_are_refused(gens):
    """Before anything is enqueued: the batch goes on afterwards."""
    m = spegg()
    ws = kinds(600, 32, 6)[:2] + [continuous(500, 32, 6)]
    stream = torch.cuda.Stream()
    b = m.Batch(ws, stats_capacity=64, stream=stream)
    b.step(gens)
    b.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        with pytest.raises(m.SpeggError):
            b.step(gens)
    b.step(2)
    for i, w in enumerate(ws):
        assert_member(b, i, w, gens + 2)
