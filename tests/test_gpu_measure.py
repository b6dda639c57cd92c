"""The measuring kernels against the CPU oracle and against one another (tolerance
zero): energies, overlaps and hashes of single lattices, whose result the kernel's
last block writes to the host, and of all replicas of a batch in one launch.
Sizes: rows that fill no word, one and several words a row, one and several
blocks and chunks per lattice."""
import numpy as np
import pytest

from oracle import OracleSim

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def isg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1411_0127_gb300 import build
    build.build()
    import paper_1411_0127_gb300 as m
    return m


@pytest.mark.parametrize("L", [4, 6, 30, 64, 66, 128, 130, 150])
def test_single_lattice_measures(isg, L):
    a, b = isg.Sim(L, 3, 4, 1.0, "minstd"), isg.Sim(L, 3, 5, 1.0, "minstd")
    oa, ob = OracleSim(L, 3, 4, 1.0, 0), OracleSim(L, 3, 5, 1.0, 0)
    for n in (0, 1, 2):
        for x, o in ((a, oa), (b, ob)):
            x.sweep(n)
            o.sweep(n)
            for _ in range(2):                       # the words are left zero for the next call
                assert x.energy() == o.energy() == x.tracked_energy()
                assert x.hash() == o.hash()
        assert a.overlap(b) == b.overlap(a) == oa.overlap(ob)
        assert a.overlap(a) == L ** 3


@pytest.mark.parametrize("kind", ["minstd", "mt19937"])
def test_batch_measures(isg, kind):
    """Every replica against its lone handle, with the run on another stream than
    the reads, and with one output alone."""
    import torch
    L = [4, 10, 64, 66, 130, 192, 258]
    n = len(L)
    b = isg.Batch(L, range(n), range(10, 10 + 2 * n), [1.0 + 0.1 * s for s in range(n)], kind)
    lone = [isg.Sim(L[r // 2], r // 2, 10 + r, 1.0 + 0.1 * (r // 2), kind) for r in range(2 * n)]
    st = torch.cuda.Stream()
    for sweeps in (0, 3):
        b.run(sweeps, 2, st)
        Et, H = b.tracked(st)
        Et2, H2 = b.tracked()
        E, Q = b.measure()
        for r, x in enumerate(lone):
            x.sweep(sweeps)
            assert E[r] == Et[r] == Et2[r] == x.energy(), (r, sweeps)
            assert H[r] == H2[r] == x.hash(), (r, sweeps)
        for s in range(n):
            assert Q[s] == lone[2 * s].overlap(lone[2 * s + 1])
    Q2 = np.zeros(n, dtype=np.int64)
    assert isg.lib().isg_batch_measure(b._h, None, Q2.ctypes.data, None) == isg.ISG_OK
    assert np.array_equal(Q2, Q)
    assert isg.lib().isg_batch_measure(b._h, None, None, None) == isg.ISG_OK
    assert isg.lib().isg_batch_tracked(b._h, None, None, None) == isg.ISG_OK


@pytest.mark.parametrize("L", [4, 48, 66, 128])
def test_overlap_needs_planes_of_one_word_width(isg, L):
    """A batch's replica (64-bit words) against a lone lattice of the same sample:
    counted where that one has 64-bit words too, refused where it has not (at L = 4
    the padded planes are equally long all the same)."""
    b = isg.Batch([L], [1], [2, 3], [1.0], "minstd")
    m, x, o = b.member(0), isg.Sim(L, 1, 3, 1.0, "minstd"), b.member(1)
    if x.info()["word_bits"] == 64:
        assert m.overlap(x) == x.overlap(m) == m.overlap(o)
    else:
        for p, q in ((m, x), (x, m)):
            with pytest.raises(isg.IsgError) as ei:
                p.overlap(q)
            assert ei.value.code == isg.ISG_ERR_MISMATCH
    b.close()


@pytest.mark.parametrize("L", [[4], [256], [30, 66] * 3, [384, 30], [512]])
def test_batch_measures_in_chunks(isg, L):
    """Batches whose chunks are of one thread's word each, of some hundred words that
    end within a row group, and of the most that there are."""
    n = len(L)
    b = isg.Batch(L, range(n), range(10, 10 + 2 * n), [1.0] * n, "minstd")
    b.run(1)
    Et, H = b.tracked()
    E, Q = b.measure()
    for r in range(2 * n):
        x = isg.Sim(L[r // 2], r // 2, 10 + r, 1.0, "minstd")
        x.sweep_plain(1)
        assert E[r] == Et[r] == x.energy() and H[r] == x.hash(), r
        if r % 2 == 0:
            y = isg.Sim(L[r // 2], r // 2, 11 + r, 1.0, "minstd")
            y.sweep_plain(1)
            assert Q[r // 2] == x.overlap(y)
            y.close()
        x.close()
    b.close()
