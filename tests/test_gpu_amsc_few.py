"""Multispin ensembles with few RNG streams, whose levels are made ahead of the
passes (isg_levels.cuh): systems against lone lattices swept by the plain kernel,
bit for bit.  Sizes: rows of a multiple of four sites per colour and others,
short last streams, streams cut into parts, more passes than are made at once."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("kind", ["minstd", "mt19937", "parisi_rapuano"])
@pytest.mark.parametrize("L,calls", [(4, (1, 70)), (6, (3,)), (34, (1, 65, 2)), (66, (2, 1)), (100, (3, 2)),
                                     (130, (2,)), (264, (1, 1))])
def test_few_streams(isg, L, calls, kind):
    J = [100 + 7 * b for b in range(32)]
    S = [500 + 3 * b for b in range(32)]
    beta = 1 / 1.2
    m = isg.Amsc(L, J, S, 77, beta, kind)
    done = 0
    for n in calls:
        m.sweep(n)
        done += n
        E = m.energies()
        for b in (0, 13, 31):
            x = isg.Sim(L, J[b], S[b], beta, kind, seed_rng=77)
            x.sweep_plain(done)
            assert E[b] == x.energy(), (b, done)
            assert np.array_equal(m.spins(b), x.read_spins()), (b, done)
    m.close()
