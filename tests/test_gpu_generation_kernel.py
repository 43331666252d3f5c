"""The generation kernel (single biallelic populations, batch members), the
continuous-allele kernel and the spatial pool at the sizes and values where their own branches change, bit for
bit against the CPU oracle: one block or several, whole and ragged groups and
slots, one- and two-digit values, 64-bit bins, calls longer than a launch,
extinction inside a call, rare survivors, several blocks per member, stream
capture, and a spatial pool that has to move its records often."""
import dataclasses

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


def assert_same(orc, gpu, so, sg, continuous=False):
    assert len(so) == len(sg)
    for name in so.dtype.names:
        assert np.array_equal(so[name], sg[name]), name
    read = "values" if continuous else "genotypes"
    assert np.array_equal(getattr(orc, read)(), getattr(gpu, read)())
    assert np.array_equal(orc.survivors(), gpu.survivors())
    a, b = orc.state(), gpu.state()
    for k in ("gen", "S", "status", "f", "R"):
        assert a[k] == b[k], (k, a[k], b[k])


def check(w, n_gen):
    orc = oracle.OraclePopulation.from_workload(w)
    gpu = spegg().Population.from_workload(w, stats_capacity=n_gen + 2)
    so = orc.step(n_gen)
    gpu.step(n_gen)
    assert_same(orc, gpu, so, gpu.read_stats(1, gpu.state()["gen"]), w.allele_model == 1)


# groups of 32; 512 is one block's 16 groups; 77,824 = 2,432 slots of one group
@pytest.mark.parametrize("n_loci", [32, 64, 128, 256])
@pytest.mark.parametrize("n", [1, 31, 33, 511, 512, 513, 1025, 77_823, 77_824, 77_825])
def test_group_and_slot_edges(n, n_loci):
    check(S.single_species(n=n, n_loci=n_loci, mu=1e-3, seed=n + n_loci), 4)


@pytest.mark.parametrize("dominance", [False, True])
@pytest.mark.parametrize("n_loci", [32, 64, 128, 256])
def test_two_digit_values(n_loci, dominance):
    """Effects and deviations over the whole int16 range."""
    rng = np.random.default_rng(n_loci)
    w = S.single_species(n=3000, n_loci=n_loci, mu=1e-3, seed=5)
    e = rng.integers(-32768, 32768, n_loci).astype(np.int16)
    e[:2] = -32768, 32767
    d = rng.integers(-32768, 32768, n_loci).astype(np.int16) if dominance else None
    w = dataclasses.replace(w, effects=e, dominance=d, bias=1 << 23, shift=12)
    w.surv_table = S.stabilizing_table(w.bias, w.shift, 1e-5)
    check(w, 6)


@pytest.mark.parametrize("bias", [(1 << 31) - 1, -(1 << 31), 1 << 30, (1 << 30) - 1])
def test_bins_of_a_large_bias(bias):
    w = S.single_species(n=2000, n_loci=64, mu=1e-3, seed=9)
    w = dataclasses.replace(w, bias=bias, shift=19)
    w.surv_table = np.full(4096, 0x9000_0000, np.uint32)
    check(w, 4)


@pytest.mark.parametrize("n", [400, 3000])
def test_call_longer_than_a_launch(n):
    check(S.consumer_resource(n=n, n_loci=64, K=50.0 * n, mu=1e-3, seed=2), 1030)


@pytest.mark.parametrize("n", [300, 5000, 80_000])
def test_extinction_inside_a_call(n):
    """The last generation's records, survivors and state of a population that
    stops before the call's end."""
    w = S.consumer_resource(n=n, n_loci=64, K=50.0 * n, seed=3)
    w.attack = S.constant_table(2 ** 30)
    check(w, 12)


@pytest.mark.parametrize("n_loci", [32, 256])
@pytest.mark.parametrize("n", [300, 513, 5000, 16_384, 16_385])
def test_calls_of_one_generation(n, n_loci):
    """One-generation calls back to back, among longer ones, with a resource
    and per-locus counts."""
    w = S.consumer_resource(n=n, n_loci=n_loci, K=50.0 * n, mu=1e-3, seed=n)
    orc = oracle.OraclePopulation.from_workload(w)
    gpu = spegg().Population.from_workload(w, stats_capacity=16)
    gpu.set_locus_counts()
    counts, so = [], []
    for k in (1, 1, 1, 2, 1, 1):
        gpu.step(k)
    for _ in range(7):
        so.append(orc.step(1))
        counts.append(orc.locus_counts())
    assert_same(orc, gpu, np.concatenate(so), gpu.read_stats(1, 7))
    assert np.array_equal(gpu.locus_counts(1, 7), np.stack(counts))


def test_extinction_in_a_call_of_one_generation():
    w = S.consumer_resource(n=5000, n_loci=64, K=2.5e5, seed=3)
    w.attack = S.constant_table(2 ** 30)
    orc = oracle.OraclePopulation.from_workload(w)
    gpu = spegg().Population.from_workload(w, stats_capacity=16)
    so = orc.step(4)
    for _ in range(4):
        gpu.step(1)
    assert_same(orc, gpu, so, gpu.read_stats(1, gpu.state()["gen"]))


@pytest.mark.parametrize("p", [0x0100_0000, 0x0010_0000])
def test_rare_survivors(p):
    """1 in 256 and 1 in 4,096 survive: most slots are empty, so the directory
    is walked over several."""
    w = S.single_species(n=200_000, n_loci=32, mu=1e-3, seed=4)
    w.surv_table = S.constant_table(p)
    check(w, 4)


def test_members_on_several_blocks():
    """Members of very different sizes and locus counts, some on many blocks,
    against the oracle."""
    ws = [S.single_species(n=n, n_loci=L, mu=1e-3, seed=31 + i, replicate=i)
          for i, (n, L) in enumerate([(300_000, 128), (20_000, 32), (500, 256), (77_825, 64), (33, 32), (60_000, 256)])]
    b = spegg().Batch(ws, stats_capacity=8)
    b.step(3)
    b.step(2)
    for i, w in enumerate(ws):
        orc = oracle.OraclePopulation.from_workload(w)
        so, sg = orc.step(5), b.read_stats(i, 1, 5)
        for name in so.dtype.names:
            assert np.array_equal(so[name], sg[name]), (i, name)
        assert np.array_equal(orc.genotypes(), b.genotypes(i)), i


@pytest.mark.parametrize("n", [400, 30_000])
def test_step_under_stream_capture(n):
    """A captured call replayed twice advances by twice its generations."""
    w = S.single_species(n=n, n_loci=64, mu=1e-3, seed=8)
    stream = torch.cuda.Stream()
    gpu = spegg().Population.from_workload(w, stats_capacity=16, stream=stream)
    gpu.step(1)
    gpu.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        gpu.step(3)
    with torch.cuda.stream(stream):
        graph.replay()
        graph.replay()
    orc = oracle.OraclePopulation.from_workload(w)
    so = orc.step(7)
    assert_same(orc, gpu, so, gpu.read_stats(1, 7))


@pytest.mark.parametrize("per_offspring", [0.5, 4.0, 7.0])
@pytest.mark.parametrize("n_loci", [32, 64, 128, 256])
def test_continuous_mutations_and_extreme_values(n_loci, per_offspring):
    """Below, around and above the 128 mutations of 32 offspring that are
    listed ahead, with values over the whole int16 range."""
    n = 1003
    w = S.continuous_trait(n=n, n_loci=n_loci, mu=per_offspring / (2 * n_loci), seed=n_loci)
    rng = np.random.default_rng(n_loci)
    v = rng.integers(-32768, 32768, (n, 2 * n_loci)).astype(np.int16)
    v[:40] = -32768
    v[40:80] = 32767
    v[80:120, ::2] = 0
    check(dataclasses.replace(w, init_values=v, bias=1 << 23, shift=12,
                              surv_table=np.full(4096, 0xC000_0000, np.uint32)), 4)


def test_space_pool_moves_its_records():
    """A pool little larger than the population: the records move every step
    or two."""
    c = S.spatial_community(X=3, Y=3, n0=200, n_loci=64, mu=1e-3, disp=0.2, seed=21)
    orc = oracle.OracleSpace(c)
    so = orc.step(12)
    gpu = spegg().Space(c, capacity=int(orc.sizes().sum()) + 500, stats_capacity=32)
    gpu.step(12)
    sg = gpu.read_stats(1, 12)
    for name in so.dtype.names:
        assert np.array_equal(so[name], sg[name]), name
    for s in range(gpu.ns):
        for p in range(gpu.c.patches):
            rg, ag = gpu.deme(s, p)
            ro, ao = orc.deme(s, p)
            assert np.array_equal(ag, ao) and np.array_equal(rg, ro), (s, p)
