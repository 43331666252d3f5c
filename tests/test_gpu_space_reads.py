"""Reading a spatial community takes no device memory: a read works on a device
that is full."""
import numpy as np
import pytest

import oracle
import spegg_synth as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_loci", [32, 256])
def test_reading_a_deme_allocates_nothing(n_loci):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1603_09255_gb300 import build, spegg
    build.build()

    class Counting(spegg.TorchAllocator):
        calls = 0

        def _do_alloc(self, nbytes, ctx):
            self.calls += 1
            return super()._do_alloc(nbytes, ctx)

    c = S.spatial_community(X=2, Y=2, n0=200, n_loci=n_loci, mu=1e-3, disp=0.2, seed=5)
    alloc = Counting()
    gpu, orc = spegg.Space(c, stats_capacity=16, allocator=alloc), oracle.OracleSpace(c)
    for steps in (1, 6):  # the records' pool, and the other one once they have moved
        gpu.step(steps)
        orc.step(steps)
        before = alloc.calls
        for s in range(gpu.ns):
            for p in range(c.patches):
                rg, ag = gpu.deme(s, p)
                ro, ao = orc.deme(s, p)
                assert np.array_equal(ag, ao) and np.array_equal(rg, ro), (s, p)
        assert alloc.calls == before


def test_two_threads_read_their_demes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import threading

    from paper_1603_09255_gb300 import build, spegg
    build.build()
    c = S.spatial_community(X=2, Y=2, n0=400, n_loci=64, mu=1e-3, disp=0.2, seed=6)
    gpu = spegg.Space(c, stats_capacity=16)
    gpu.step(5)
    want = [gpu.deme(s, p) for s in range(gpu.ns) for p in range(c.patches)]
    wrong = []

    def reader(offset):
        for k in range(200):
            d = (k + offset) % len(want)
            rg, ag = gpu.deme(d // c.patches, d % c.patches)
            if not (np.array_equal(rg, want[d][0]) and np.array_equal(ag, want[d][1])):
                wrong.append(d)

    threads = [threading.Thread(target=reader, args=(5 * i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
