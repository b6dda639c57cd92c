"""Resident sweep launches (lattices with few RNG streams, isg_resident.cu)
against the plain kernel and the CPU oracle, bit for bit (tolerance zero).

Sizes: one stream and several, streams cut into parts with empty and short ones,
several streams per block, short last streams, both word widths, rows that fill
no word; calls of 1 to 9 sweeps, so that draws left over from a pass, the
generator states that a call stores and the next one loads, and the calls of the
plain kernel in between all take part."""
import numpy as np
import pytest

from oracle import OracleSim

pytestmark = pytest.mark.gpu

KINDS = ["minstd", "mt19937", "parisi_rapuano"]


@pytest.fixture(scope="module")
def isg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1411_0127_gb300 import build
    build.build()
    import paper_1411_0127_gb300 as m
    return m


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L", [4, 6, 14, 32, 40, 42, 62, 66, 96, 102, 128, 150, 192, 256, 300, 320, 378, 384, 428])
def test_resident_equals_plain(isg, L, kind):
    a = isg.Sim(L, 11, 12, 1 / 0.9, kind)
    b = isg.Sim(L, 11, 12, 1 / 0.9, kind)
    S = a.info()["streams"]
    for n in (1, 2, 9, 1, 4):
        a.sweep(n)
        b.sweep_plain(n)
        assert a.hash() == b.hash(), n
        assert a.tracked_energy() == b.tracked_energy() == a.energy()
        for t in {0, S // 2, S - 1}:
            assert np.array_equal(a.peek_draws(t, 700), b.peek_draws(t, 700)), (n, t)
        a.sweep_plain(1)
        b.sweep_plain(1)
    a.close()
    b.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L", [6, 34, 46, 100])
def test_resident_against_oracle(isg, L, kind):
    g = isg.Sim(L, 3, 4, 1 / 1.1, kind)
    o = OracleSim(L, 3, 4, 1 / 1.1, isg.RNG_KINDS[kind])
    for n in (3, 1, 6):
        g.sweep(n)
        o.sweep(n)
        assert np.array_equal(g.read_spins(), o.spins())
        assert g.tracked_energy() == o.tracked_energy()


@pytest.mark.parametrize("kind", KINDS)
def test_members_and_streams(isg, kind):
    """Batch members swept by their handles (64-bit words, counts made on first
    use), and four lattices swept at once on streams of their own."""
    import torch
    b = isg.Batch([48, 100], [1, 2], [3, 4, 5, 6], [1.0, 1.2], kind)
    for i in range(4):
        m = b.member(i)
        m.sweep(3)
        ref = isg.Sim(m.L, 1 + i // 2, 3 + i, m.beta, kind)
        ref.sweep_plain(3)
        assert m.hash() == ref.hash() and m.tracked_energy() == ref.tracked_energy()
    b.run(4, 2)
    m.sweep(2)
    ref.sweep_plain(6)
    assert m.hash() == ref.hash()
    sims = [isg.Sim(L, 1, 2, 1 / 0.9, kind) for L in (256, 128, 200, 256)]
    streams = [torch.cuda.Stream() for _ in sims]
    for _ in range(5):
        for s, st in zip(sims, streams):
            s.sweep(4, stream=st)
    torch.cuda.synchronize()
    for s in sims:
        r = isg.Sim(s.L, 1, 2, 1 / 0.9, kind)
        r.sweep_plain(20)
        assert s.hash() == r.hash()


def test_resident_wait_gives_up_with_a_status(isg):
    """A resident launch whose second pass waits for a pass that never comes: its
    bounded waits run out, the next energy read reports ISG_ERR_TIMEOUT once, and
    other lattices sweep on."""
    g = isg.Sim(128, 1, 2, 1 / 0.9, "mt19937")
    assert isg.lib().isg_resident_test_stall(g.handle) == isg.ISG_OK
    g.sweep(2)
    with pytest.raises(isg.IsgError) as ei:
        g.tracked_energy()
    assert ei.value.code == isg.ISG_ERR_TIMEOUT
    g.tracked_energy()
    big = isg.Sim(512, 1, 2, 1.0, "minstd")
    assert isg.lib().isg_resident_test_stall(big.handle) == isg.ISG_ERR_STATE
    a, o = isg.Sim(66, 1, 2, 1 / 0.9, "mt19937"), OracleSim(66, 1, 2, 1 / 0.9, 1)
    a.sweep(3)
    o.sweep(3)
    assert a.tracked_energy() == o.tracked_energy() == a.energy()


@pytest.mark.parametrize("L", [10, 12, 64, 100, 256])
def test_exchange_outputs(isg, L):
    """isg_exchange_async's outputs in pageable memory, in pinned memory that the
    kernel writes (small lattices, whole words) and at a pinned address that is
    not aligned to words; nothing behind the last byte is touched."""
    import torch
    nb = (L ** 3 + 7) // 8
    g = isg.Sim(L, 5, 6, 1 / 0.9, "minstd")
    pin = torch.zeros(nb + 16, dtype=torch.uint8).pin_memory().numpy()
    for out in (np.zeros(nb + 8, dtype=np.uint8), pin[:nb + 8], pin[1:nb + 9]):
        out[nb:] = 0xA5
        for E in (np.zeros(1, dtype=np.int64), torch.zeros(1, dtype=torch.int64).pin_memory().numpy()):
            g.exchange_async(None, out, 1, E)
            torch.cuda.synchronize()
            assert np.array_equal(out[:nb], g.read_spins_packed())
            assert int(E[0]) == g.tracked_energy() == g.energy()
            assert (out[nb:] == 0xA5).all()
            E[0] = 0
            g.exchange_async(None, None, 1, E)
            torch.cuda.synchronize()
            assert int(E[0]) == g.tracked_energy()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("sizes", [[4, 6, 14, 16] * 40, [32, 48, 100, 192], [256, 300, 4, 64]])
def test_batch_in_resident_launches(isg, sizes, kind):
    """Batches with few streams: many tiny lattices, and large beside small ones,
    in runs of several lengths, against the plain kernel."""
    n = len(sizes)
    b = isg.Batch(sizes, range(n), range(2 * n), [1.0 + 0.01 * s for s in range(n)], kind)
    for sweeps in (1, 5):
        b.run(sweeps)
    E, H = b.tracked()
    Em, _ = b.measure()
    assert np.array_equal(E, Em)
    for r in list(range(8)) + list(range(2 * n - 4, 2 * n)):
        if r >= 2 * n:
            continue
        x = isg.Sim(sizes[r // 2], r // 2, r, 1.0 + 0.01 * (r // 2), kind)
        x.sweep_plain(6)
        assert H[r] == x.hash() and E[r] == x.tracked_energy(), r
    b.close()


@pytest.mark.parametrize("kind", ["mt19937", "parisi_rapuano"])
def test_batch_resident_wait_gives_up_with_a_status(isg, kind):
    L = [48, 64, 20]
    b = isg.Batch(L, [1, 2, 3], range(6), [1.0] * 3, kind)
    assert isg.lib().isg_batch_test_stall(b._h) == isg.ISG_OK
    b.run(2)
    with pytest.raises(isg.IsgError) as ei:
        b.tracked()
    assert ei.value.code == isg.ISG_ERR_TIMEOUT
    b.tracked()                               # reported once; the counts start again
    b.run(3)
    Em, _ = b.measure()
    Et, _ = b.tracked()
    assert np.array_equal(Em, Et)


@pytest.mark.parametrize("kind", KINDS)
def test_server_quanta_in_resident_launches(isg, kind):
    """Jobs of several sizes and lengths in one server, each ending in another
    quantum, against lone lattices."""
    srv = isg.Server(quantum_sweeps=4)
    jobs = [(32, 3), (64, 9), (100, 4), (34, 17), (128, 1)]
    ids = [srv.submit(L, 10 + j, 20 + j, 1.1, kind, n) for j, (L, n) in enumerate(jobs)]
    srv.run()
    for j, (L, n) in enumerate(jobs):
        x = isg.Sim(L, 10 + j, 20 + j, 1.1, kind)
        x.sweep_plain(n)
        r = srv.job(ids[j])
        assert r["status"] == 2 and r["E"] == x.energy() and r["H"] == x.hash(), j
    srv.close()


@pytest.mark.parametrize("kind", KINDS)
def test_server_quantum_changes_engine(isg, kind):
    """Too many streams for a resident launch until the short jobs have ended:
    the pass engine first, the resident launch for the rest of the quantum."""
    srv = isg.Server(quantum_sweeps=4)
    jobs = [1] * 11 + [6, 3, 9, 4]
    ids = [srv.submit(256, 10 + j, 20 + j, 1.1, kind, n) for j, n in enumerate(jobs)]
    srv.run()
    for j, n in enumerate(jobs):
        x = isg.Sim(256, 10 + j, 20 + j, 1.1, kind)
        x.sweep_plain(n)
        r = srv.job(ids[j])
        assert r["status"] == 2 and r["E"] == x.energy() and r["H"] == x.hash(), j
        x.close()
    srv.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L", [32, 64, 150, 256])
def test_sweeps_replayed_from_a_graph(isg, L, kind):
    """isg_sweep captured into a CUDA graph, replayed three times between direct
    calls; a batch member, which has made no resident launch before, as well."""
    import torch
    a = isg.Sim(L, 11, 12, 1 / 0.9, kind)
    r = isg.Sim(L, 11, 12, 1 / 0.9, kind)
    b = isg.Batch([32, L], [1, 11], [5, 6, 7, 12], [1 / 0.9] * 2, kind)
    m = b.member(3)
    a.sweep(1)
    m.sweep_plain(1)
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        a.sweep(3, s)
        m.sweep(3, s)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    a.sweep(2)
    m.sweep(2)
    r.sweep_plain(12)
    assert a.hash() == r.hash() == m.hash()
    assert a.energy() == r.energy() == a.tracked_energy()
    a.close()
    r.close()
    b.close()


@pytest.mark.parametrize("kind", KINDS)
def test_batch_replayed_from_a_graph(isg, kind):
    """isg_batch_run captured as the first run of a batch, replayed twice, then
    runs of its own."""
    import torch
    L = [32, 64, 48]
    b = isg.Batch(L, [1, 2, 3], range(6), [1.1] * 3, kind)
    c = isg.Batch(L, [1, 2, 3], range(6), [1.1] * 3, kind)
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        b.run(3, 64, s)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    b.run(4)
    c.run(10)
    assert all(np.array_equal(x, y) for x, y in zip(b.tracked(), c.tracked()))
    b.close()
    c.close()


@pytest.mark.parametrize("kind", KINDS)
def test_server_quantum_of_several_launches(isg, kind):
    """A quantum of more passes than a resident launch takes (1024), with jobs that
    end in its first launch, in a later one and in the next quantum."""
    srv = isg.Server(quantum_sweeps=1100)
    jobs = [(6, 1300), (34, 1030), (32, 513), (14, 512), (48, 3)]
    ids = [srv.submit(L, 10 + j, 20 + j, 1.1, kind, n) for j, (L, n) in enumerate(jobs)]
    srv.run()
    assert srv.stats()["iterations"] == 2
    for j, (L, n) in enumerate(jobs):
        x = isg.Sim(L, 10 + j, 20 + j, 1.1, kind)
        x.sweep_plain(n)
        r = srv.job(ids[j])
        assert r["status"] == 2 and r["E"] == x.energy() and r["H"] == x.hash(), j
        x.close()
    srv.close()


def test_server_quantum_of_more_draws_than_32_bits_count(isg):
    """L = 40 has one stream of 32 000 draws a pass, so that 68 000 passes use more
    than 2^31 of them: one quantum against calls of 500 sweeps."""
    n = 34000
    srv = isg.Server(quantum_sweeps=n)
    j = srv.submit(40, 1, 2, 1.1, "mt19937", n)
    srv.run()
    assert srv.stats()["iterations"] == 1
    x = isg.Sim(40, 1, 2, 1.1, "mt19937")
    for _ in range(n // 500):
        x.sweep(500)
    r = srv.job(j)
    assert r["status"] == 2 and r["E"] == x.energy() == x.tracked_energy() and r["H"] == x.hash()
    srv.close()


def test_info_calls_name_the_launches_that_run(isg):
    """isg_sweep_info and isg_amsc_info on both sides of the stream counts up to
    which lattices run in resident launches and ensembles make their levels ahead."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for kind, most in (("minstd", 16), ("mt19937", 16), ("parisi_rapuano", 8)):
        for L in (4, 64, 256, 300, 320, 352, 380, 400, 428, 440, 512):
            s = isg.Sim(L, 1, 2, 1.0, kind)
            assert s.passes_per_launch() == (1024 if s.info()["streams"] < most * sms else 1), (kind, L)
            s.close()
    b = isg.Batch([48], [1], [2, 3], [1.0], "minstd")
    assert b.member(1).passes_per_launch() == 1024
    for L, form in ((4, 1), (64, 1), (256, 1), (322, 1), (390, 8), (432, 4)):
        m = isg.Amsc(L, range(32), range(32), 1, 1.0, "minstd")
        assert m.info()["form"] == form, L
        m.close()


@pytest.mark.parametrize("L", [280, 300, 352, 364, 400, 412])
def test_blocks_of_one_pair(isg, L):
    """MT19937 lattices of 5, 6, 9, 10, 13 and 14 streams on the fullest SM, as many
    blocks of one pair of warps there, against the plain kernel; a call of more
    than one launch at the smallest of them."""
    a = isg.Sim(L, 11, 12, 1 / 0.9, "mt19937")
    b = isg.Sim(L, 11, 12, 1 / 0.9, "mt19937")
    assert a.passes_per_launch() == 1024
    for n in (1, 2, 9, 514 if L == 280 else 1):
        a.sweep(n)
        b.sweep_plain(n)
        assert a.hash() == b.hash(), n
        assert a.tracked_energy() == b.tracked_energy() == a.energy()
    a.close()
    b.close()


@pytest.mark.parametrize("sizes", [[64] * 40, [96] * 20, [48, 64, 96, 128] * 6, [128] * 16])
def test_batch_of_one_pair_blocks(isg, sizes):
    """MT19937 batches of 5 to 14 streams per SM, resident launches of blocks of one pair."""
    n = len(sizes)
    b = isg.Batch(sizes, range(n), range(2 * n), [1.0 + 0.01 * s for s in range(n)], "mt19937")
    for sweeps in (1, 6):
        b.run(sweeps)
    E, H = b.tracked()
    for r in list(range(8)) + list(range(2 * n - 4, 2 * n)):
        x = isg.Sim(sizes[r // 2], r // 2, r, 1.0 + 0.01 * (r // 2), "mt19937")
        x.sweep_plain(7)
        assert H[r] == x.hash() and E[r] == x.tracked_energy(), r
        x.close()
    b.close()


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("L", [6, 34, 48])
def test_calls_of_several_launches(isg, L, kind):
    """Calls of more sweeps than a resident launch takes (512): counts, draws left
    over, stored states, the exchange's bond count of the first pass and a batch's run
    go on from launch to launch."""
    import torch
    a = isg.Sim(L, 11, 12, 1 / 0.9, kind)
    b = isg.Sim(L, 11, 12, 1 / 0.9, kind)
    for n in (513, 1030):
        a.sweep(n)
        b.sweep_plain(n)
        assert a.hash() == b.hash(), n
        assert a.tracked_energy() == b.tracked_energy() == a.energy()
        S = a.info()["streams"]
        assert np.array_equal(a.peek_draws(S - 1, 700), b.peek_draws(S - 1, 700))
    nb = (L ** 3 + 7) // 8
    bits = np.random.default_rng(L).integers(0, 256, nb, dtype=np.uint8)
    out, E = np.zeros(nb, dtype=np.uint8), np.zeros(1, dtype=np.int64)
    a.exchange_async(bits, out, 600, E)
    torch.cuda.synchronize()
    b.write_spins_packed(bits)
    b.sweep_plain(600)
    assert a.hash() == b.hash() and np.array_equal(out, b.read_spins_packed())
    assert int(E[0]) == a.tracked_energy() == b.tracked_energy() == a.energy()
    c = isg.Batch([L, 32], [11, 1], [12, 13, 5, 6], [1 / 0.9] * 2, kind)
    c.run(513)
    r = isg.Sim(L, 11, 12, 1 / 0.9, kind)
    r.sweep_plain(513)
    Et, H = c.tracked()
    assert H[0] == r.hash() and Et[0] == r.tracked_energy()
    c.close()


def test_exchange_output_registered_in_part(isg):
    """Spins into host memory of which only the first page is registered: the kernel
    does not write it directly; the call answers as a copy there does (an error
    status, or all bytes), and the lattice goes on."""
    import torch
    L, page = 64, 65536
    nb = L ** 3 // 8                                  # 32 KiB
    raw = np.zeros(4 * page, dtype=np.uint8)
    base = -raw.ctypes.data % page
    out = raw[base + page - 4096:base + page - 4096 + nb]    # its first 4096 bytes are registered
    rt = torch.cuda.cudart()
    assert int(rt.cudaHostRegister(raw.ctypes.data + base, page, 0)) == 0
    try:
        g = isg.Sim(L, 5, 6, 1 / 0.9, "minstd")
        try:
            g.exchange_async(None, out, 1, None)
            torch.cuda.synchronize()
            assert np.array_equal(out, g.read_spins_packed())
        except isg.IsgError as e:
            assert e.code == isg.ISG_ERR_CUDA
        g.sweep(1)
        assert g.energy() == g.tracked_energy()
        g.close()
    finally:
        assert int(rt.cudaHostUnregister(raw.ctypes.data + base)) == 0


@pytest.mark.parametrize("L", [106, 112, 128, 146, 164, 190, 200, 230, 256, 288, 300])
def test_short_minstd_calls(isg, L):
    """Calls of one sweep as launches of one pass each: every layout of them (parts of
    streams, even shares of two and four blocks an SM), between longer
    calls, as a batch's replica, with spins in (the first pass counts the bonds),
    captured and replayed, and with equal checkpoints."""
    import torch
    a = isg.Sim(L, 11, 12, 1 / 0.9, "minstd")
    b = isg.Sim(L, 11, 12, 1 / 0.9, "minstd")
    c = isg.Batch([L], [11], [5, 12], [1 / 0.9], "minstd")
    m = c.member(1)
    for n in (1, 2, 1, 3, 1):
        a.sweep(n)
        m.sweep(n)
        b.sweep_plain(n)
        assert a.hash() == b.hash() == m.hash(), n
        assert a.tracked_energy() == b.tracked_energy() == a.energy() == m.tracked_energy()
    assert a.save() == b.save()
    nb = L ** 3 // 8
    bits = np.random.default_rng(L).integers(0, 256, nb, dtype=np.uint8)
    E = np.zeros(1, dtype=np.int64)
    for n in (1, 2):
        a.exchange_async(bits, None, n, E)
        torch.cuda.synchronize()
        b.write_spins_packed(bits)
        b.sweep_plain(n)
        assert a.hash() == b.hash() and int(E[0]) == a.tracked_energy() == b.tracked_energy() == a.energy()
    torch.cuda.synchronize()
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        a.sweep(1, s)
        a.sweep(1, s)
        a.sweep(2, s)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    a.sweep(1)
    b.sweep_plain(13)
    assert a.hash() == b.hash() and a.energy() == b.energy() == a.tracked_energy()
    for x in (a, b, c):
        x.close()


@pytest.mark.parametrize("kind", KINDS)
def test_loaded_replica(isg, kind):
    """A batch's replica of 64-bit words where a lone lattice has 32-bit ones, saved
    and loaded: the handle runs the launches of its size, on the same trajectory."""
    for L in (64, 640):
        b = isg.Batch([L], [1], [2, 3], [1.1], kind)
        m = b.member(1)
        m.sweep(2)
        x = isg.Sim.load(m.save())
        lone = isg.Sim(L, 1, 3, 1.1, kind)
        assert x.info()["word_bits"] == 64
        assert x.passes_per_launch() == lone.passes_per_launch()
        for n in (1, 9):
            x.sweep(n)
            m.sweep_plain(n)
            assert x.hash() == m.hash() and x.tracked_energy() == m.tracked_energy() == x.energy()
        for s in (x, lone, b):
            s.close()
