"""The column form of a run (rule R1 from equal rows: one row of angle indices stands for the
population), bit for bit against the CPU oracle.

The cases lie where its cuts change: shares short enough for one block, for blocks that meet
through posts, for the grid barrier, and long ones taken from a queue; lists that shrink from
whole vectors to single quads to nothing inside a run and across runs; ragged last vectors; the
three item-sum forms; and every way the population enters or leaves the form (checkpoints with
equal and with different rows, batches, autotuning, reset). All results are whole numbers: the
tolerance is zero."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2609_30862_gb300 import qieo as Q
from paper_2609_30862_gb300 import workload as W
from saturated import load_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    Q.load()


def _problem(ng, items):
    if items == "byte":
        return W.knapsack(ng, ng + 11)
    r = np.random.RandomState(ng)
    if items == "mid":           # items below 2^20, at the limit
        w = r.randint(0, 1 << 20, ng)
        w[::2] = (1 << 20) - 1
        v = np.full(ng, (1 << 20) - 1)
    else:
        w = r.randint(0, 2**31 - 1, ng)
        v = r.randint(-2**31 + 1, 2**31 - 1, ng)
    return W.custom_problem(w, v, int(w.astype(np.int64).sum()) // 2)


def check(I, st, gens):
    k, t = I.state()
    assert t == gens == int(st.t[0])
    e, f = I.history(0, gens)
    assert np.array_equal(e, st.hist_e), int(np.argmax(e != st.hist_e))
    assert np.array_equal(f, st.hist_f)
    assert np.array_equal(k, st.k), "angle indices differ"
    assert np.array_equal(I.fitness(), st.f)
    assert np.array_equal(I.alleles(), st.x), "alleles differ"
    assert np.array_equal(I.allele_row(len(st.f) - 1), st.x[-1])
    bits, bf, bg, bc = I.best()
    assert (bf, bg, bc) == tuple(int(v) for v in st.best)
    assert np.array_equal(bits, st.best_x)


@pytest.mark.parametrize("ng,np_,D,items,chunks", [
    (1, 1, 100, "byte", [5]), (4, 7, 4, "byte", [1, 1, 6]), (9, 2, 12, "wide", [40]),
    (33, 511, 100, "byte", [30, 1, 1]), (100, 64, 100, "byte", [500]), (257, 513, 40, "mid", [25, 30]),
    (1023, 40, 100, "byte", [150, 60]), (2048, 300, 100, "byte", [70]), (2049, 65, 8, "wide", [20, 5]),
    (4100, 130, 100, "mid", [60, 90]), (6000, 16, 4000, "byte", [40]), (20003, 3, 100, "byte", [120]),
    (300, 20000, 100, "byte", [25, 90]), (20000, 4000, 12, "byte", [30]), (300001, 40, 100, "byte", [12]),
    (70, 50000, 100, "wide", [60]),
])
def test_column_form(ng, np_, D, items, chunks):
    prob = _problem(ng, items)
    gens = sum(chunks)
    st = O.run(prob, np_, gens, seed=ng, inst=3, D=D, lam=2, kind="omp")
    with Q.Instance(prob, np_, seed=ng, inst=3, D=D, lam=2) as I:
        for g in chunks:
            I.run(g)
        check(I, st, gens)
        I.reset()                # a second solve on the same words
        for g in chunks:
            I.run(g)
        check(I, st, gens)


def test_state_moves_between_the_forms():
    """Batches and other row-by-row runs between column runs; the checkpoint of a column run
    loaded elsewhere; a checkpoint whose rows differ, which the column form cannot hold."""
    prob, np_, seed = W.knapsack(2603, 5), 90, 5
    st = O.run(prob, np_, 155, seed=seed)
    with Q.Instance(prob, np_, seed=seed) as I, Q.Instance(prob, np_, seed=seed) as J:
        I.autotune(2)
        I.run(40)
        with Q.Batch([I]) as b:
            b.run(30)
        I.run(25)
        J.run(3)
        J.load(I.save())
        J.run(60)
        check(J, st, 155)
        I.run(60)
        check(I, st, 155)
    rng = np.random.default_rng(9)
    for rows_equal in (True, False):
        k0 = rng.integers(-25, 26, size=(1 if rows_equal else np_, 2603)).astype(np.int16).repeat(np_ if rows_equal else 1, 0)
        st = O.State(np_, prob.ng)
        st.k[:] = k0
        O.run(prob, np_, 70, seed=seed, state=st)
        with Q.Instance(prob, np_, seed=seed) as I:
            load_state(I, k0)
            assert np.array_equal(I.state()[0], k0)
            I.run(30)
            I.run(40)
            check(I, st, 70)
            I.reset()
            I.run(20)
            check(I, O.run(prob, np_, 20, seed=seed), 20)


@pytest.mark.parametrize("ng,np_", [(40, 30), (600, 50), (3000, 700)])
def test_convergence_stop(ng, np_):
    """The stop inside a run, with the generation after it never run, and a stop while the list
    is already empty; the allele plane of the last generation."""
    prob = W.knapsack(ng, 21)
    ref = O.run(prob, np_, 600, seed=21, window=20)
    n = int(ref.t[0])
    assert ref.stopped
    for chunks in ([600], [n - 1, 40], [n, 7], [11] * 60):
        with Q.Instance(prob, np_, seed=21, flags=Q.QIEO_FLAG_CONVERGE) as I:
            for g in chunks:
                I.run(g)
            k, t = I.state()
            assert t == n and np.array_equal(k, ref.k)
            e, f = I.history(0, n)
            assert np.array_equal(e, ref.hist_e) and np.array_equal(f, ref.hist_f)
            bits, bf, bg, bc = I.best()
            assert (bf, bg, bc) == tuple(int(v) for v in ref.best) and np.array_equal(bits, ref.best_x)
            assert np.array_equal(I.fitness(), ref.f)
            assert I.convergence() == (True, 20)


def test_wait_that_runs_out_is_reported():
    """A 1 ns bound on the wait between generations ends the run with a timeout, no trap and no
    hang; after a reset the instance runs correctly again."""
    for ng, np_ in ((400, 300), (2000, 300), (5000, 100)):
        prob = W.knapsack(ng, 16)
        with Q.Instance(prob, np_, seed=16) as I:
            I.set_wait_timeout(1)
            I.run(30)
            try:
                I.synchronize()
            except Q.QieoError as e:
                assert e.status == Q.QIEO_ERR_TIMEOUT
            I.set_wait_timeout(10 * 10**9)
            I.reset()
            I.run(30)
            check(I, O.run(prob, np_, 30, seed=16), 30)


@pytest.mark.parametrize("sizes,copies,D,items,chunks", [
    ([(1, 1), (40, 30)], 1, 4, "byte", [3, 1, 9]),                    # a member per block, empty lists
    ([(20000, 60), (2048, 33), (700, 500), (31, 128)], 1, 12, "byte", [25, 8]),
    ([(4500, 3), (260, 5), (9, 2)], 110, 20, "byte", [20, 4]),        # several members a block; three tiles on one
    ([(4100, 90), (50, 20), (2500, 40)], 2, 100, "mid", [60, 20]),
    ([(3000, 64), (257, 40), (12, 300)], 2, 100, "wide", [60, 20]),
])
def test_batched_column_form(sizes, copies, D, items, chunks):
    """Members on several blocks, on one, and several on one, against the oracle; a second solve."""
    specs = [(ng, np_, 10 * c + i) for c in range(copies) for i, (ng, np_) in enumerate(sizes)]
    probs = {ng: _problem(ng, items) for ng, _ in sizes}
    insts = [Q.Instance(probs[ng], np_, seed=7, inst=k, D=D, lam=2) for ng, np_, k in specs]
    gens = sum(chunks)
    sample = [i for i in range(len(specs)) if i < len(sizes) or i % 29 == 0]
    refs = {i: O.run(probs[specs[i][0]], specs[i][1], gens, seed=7, inst=specs[i][2], D=D, lam=2) for i in sample}
    with Q.Batch(insts) as b:
        for solve in range(2):
            for g in chunks:
                b.run(g)
            for i in sample:
                check(insts[i], refs[i], gens)
            for I in insts:
                I.reset()
    for I in insts:
        I.close()


def test_batch_whose_members_change_form():
    """A member that loads a checkpoint with different rows leaves the column form for the
    row-by-row one, and comes back after a reset; the others, one of rule R2 and one that stops by
    convergence among them, go on."""
    prob, np_ = W.knapsack(1500, 8), 40
    k0 = np.random.default_rng(3).integers(-25, 26, size=(np_, 1500)).astype(np.int16)
    conv = W.knapsack(200, 3)
    ref = O.run(conv, 30, 400, seed=3, window=20)
    insts = [Q.Instance(prob, np_, seed=i + 1, rule=1 if i == 2 else 0) for i in range(3)]
    insts.append(Q.Instance(conv, 30, seed=3, flags=Q.QIEO_FLAG_CONVERGE))
    with Q.Batch(insts) as b:
        b.run(15)
        load_state(insts[0], k0)         # (a checkpoint of generation 15 with other angles)
        st = O.run(prob, np_, 15, seed=1)
        st.k[:] = k0
        st = O.run(prob, np_, 30, seed=1, state=st)
        b.run(15)
        b.run(15)
        check(insts[0], st, 45)
        check(insts[1], O.run(prob, np_, 45, seed=2), 45)
        check(insts[2], O.run(prob, np_, 45, seed=3, rule=1), 45)
        insts[0].reset()
        b.run(355)
        check(insts[0], O.run(prob, np_, 355, seed=1), 355)
    k, t = insts[3].state()
    assert ref.stopped and t == int(ref.t[0]) and np.array_equal(k, ref.k)
    bits, bf, bg, bc = insts[3].best()
    assert (bf, bg, bc) == tuple(int(v) for v in ref.best) and np.array_equal(bits, ref.best_x)
    for I in insts:
        I.close()


@pytest.mark.parametrize("items,D", [("byte", 100), ("mid", 12), ("wide", 40)])
def test_served_column_form(items, D):
    """A server's solves: populations too small to hold the form's words where their state would
    lie (these run row by row), larger ones, and one that stops by convergence."""
    specs = [(1, 1), (300, 4), (90, 250), (2500, 60), (4100, 128), (33, 400)]
    with Q.Server(gens_per_step=7) as srv:
        ids = [srv.submit(_problem(ng, items), np_, 40, seed=ng, inst=2, D=D, lam=2) for ng, np_ in specs]
        stops = srv.submit(W.knapsack(200, 3), 300, 400, seed=3, flags=Q.QIEO_FLAG_CONVERGE)
        for rid, (ng, np_) in zip(ids, specs):
            res, bits = srv.poll(rid, wait_ms=60000)
            st = O.run(_problem(ng, items), np_, 40, seed=ng, inst=2, D=D, lam=2)
            assert res.state == Q.QIEO_SOLVE_DONE and res.generations_run == 40
            assert (res.fitness, res.generation, res.chromosome) == tuple(int(v) for v in st.best)
            assert np.array_equal(bits, st.best_x)
        res, bits = srv.poll(stops, wait_ms=60000)
        ref = O.run(W.knapsack(200, 3), 300, 400, seed=3, window=20)
        assert res.converged == 1 and res.generations_run == int(ref.t[0])
        assert np.array_equal(bits, ref.best_x)


@pytest.mark.parametrize("ng,np_,D,items,start", [
    (1, 1, 4, "byte", None), (9, 35, 12, "byte", None), (257, 700, 100, "mid", None), (2100, 300, 40, "byte", None),
    (20003, 70, 100, "byte", None), (100, 90, 100, "wide", None), (4100, 700, 20, "mid", "equal"),
    (1500, 40, 100, "byte", "mixed"),
])
def test_row_blocks(ng, np_, D, items, start):
    """A population in two row blocks, the elite exchanged here, from the start, from a checkpoint with
    equal rows and from one whose rows differ (which runs row by row): the oracle's unsharded run."""
    prob, cut = _problem(ng, items), (np_ + 2) // 3
    k0 = np.zeros((np_, ng), dtype=np.int16)
    if start:
        k0[:] = np.random.default_rng(4).integers(-(D // 4), D // 4 + 1, size=(1 if start == "equal" else np_, ng))
    st = O.State(np_, ng)
    st.k[:] = k0
    O.run(prob, np_, 40, seed=ng, inst=3, D=D, lam=2, state=st)
    blocks = [Q.Instance(prob, b - a, seed=ng, inst=3, D=D, lam=2, row0=a) for a, b in ((0, cut), (cut, np_)) if b > a]
    rows0 = [0, cut]
    for solve in range(2):
        for I, r0 in zip(blocks, rows0):
            I.reset()
            if start:
                load_state(I, k0[r0:r0 + I.np_], D)
        he, hf = [], []
        for t in range(40):
            found = [I.rows_observe(t) for I in blocks]
            f, row = max(((f, -c) for f, c in found))
            owner = 1 if len(blocks) > 1 and -row >= cut else 0
            elite = blocks[owner].allele_row(-row - rows0[owner])
            for I in blocks:
                I.rows_rotate(elite)
            he.append(-row)
            hf.append(f)
        assert np.array_equal(he, st.hist_e) and np.array_equal(hf, st.hist_f)
        assert np.array_equal(np.concatenate([I.state()[0] for I in blocks]), st.k)
        assert np.array_equal(np.concatenate([I.fitness() for I in blocks]), st.f)
        assert np.array_equal(np.concatenate([I.alleles() for I in blocks]), st.x)
    for I in blocks:
        I.close()


@pytest.mark.parametrize("ng,np_,D,items,chunks", [
    (1, 1, 4, "byte", [1] * 6), (50, 33, 100, "byte", [1] * 90), (1023, 40, 100, "byte", [1] * 70 + [20] + [1] * 5),
    (700, 300, 12, "wide", [1] * 20 + [3, 1]), (4100, 130, 100, "mid", [30, 1, 1, 25, 1]),
    (40000, 400, 8, "byte", [1, 4, 1, 1]), (300, 20000, 16, "byte", [1, 7, 1]),
])
def test_runs_of_one_generation(ng, np_, D, items, chunks):
    """Runs of one generation (two plain launches) between longer ones, through the points where genes
    reach their bounds."""
    prob, gens = _problem(ng, items), sum(chunks)
    st = O.run(prob, np_, gens, seed=ng, inst=3, D=D, lam=2, kind="omp")
    with Q.Instance(prob, np_, seed=ng, inst=3, D=D, lam=2) as I:
        for solve in range(2):
            for g in chunks:
                I.run(g)
            check(I, st, gens)
            I.reset()
    conv = W.knapsack(60, 21)
    ref = O.run(conv, 17, 600, seed=21, window=20)
    n = int(ref.t[0])
    with Q.Instance(conv, 17, seed=21, flags=Q.QIEO_FLAG_CONVERGE) as I:
        for _ in range(n + 7):
            I.run(1)
        k, t = I.state()
        assert ref.stopped and t == n and np.array_equal(k, ref.k)
        assert np.array_equal(I.history(0, n)[0], ref.hist_e)
        assert np.array_equal(I.best()[0], ref.best_x) and I.convergence() == (True, 20)


def _few_bits(ng):
    """Items of three bits: with millions of genes a row's sums still fit the packed row word."""
    r = np.random.RandomState(ng)
    w, v = r.randint(0, 8, ng), r.randint(0, 8, ng)
    return W.custom_problem(w, v, int(w.sum()) // 2)


@pytest.mark.parametrize("ng,np_,items", [(640_001, 3, "byte"), (1_000_003, 2, "wide"), (8_190_001, 3, "bits")])
def test_more_tiles_than_blocks(ng, np_, items):
    """Lists that a grid covers in several turns, cut into more tiles than they fill; 8,190,001 genes
    fill 4,000 tiles, whose cut no longer fits the 12-bit count of a packed row word. Alone, and as a
    member of a batch (fewer blocks each)."""
    prob = _few_bits(ng) if items == "bits" else _problem(ng, items)
    st = O.run(prob, np_, 6, seed=ng, inst=3, lam=2, kind="omp")
    with Q.Instance(prob, np_, seed=ng, inst=3, lam=2) as I, Q.Instance(prob, np_, seed=9, inst=1, lam=2) as J:
        I.run(6)
        check(I, st, 6)
        I.reset()
        with Q.Batch([I, J]) as b:
            b.run(6)
        check(I, st, 6)


@pytest.mark.parametrize("ng,np_", [(400, 300), (2000, 300), (5000, 100), (20000, 1000)])
def test_timed_out_run_is_reported_until_the_reset(ng, np_):
    """Blocks that meet at the grid barrier, in column_small_kernel and (20,000 x 1,000, long shares
    from a queue, with column_small_kernel launched behind it) in column_run_kernel: a 1 ns bound
    runs out and is reported; later runs, of one generation or many, do nothing to the population
    until the reset, after which a run is right again."""
    prob = W.knapsack(ng, 16)
    with Q.Instance(prob, np_, seed=16) as I:
        I.set_wait_timeout(1)
        I.run(30)
        with pytest.raises(Q.QieoError) as e:
            I.synchronize()
        assert e.value.status == Q.QIEO_ERR_TIMEOUT
        I.set_wait_timeout(10 * 10**9)
        for g in (1, 30):
            I.run(g)
            with pytest.raises(Q.QieoError) as e:
                I.best()
            assert e.value.status == Q.QIEO_ERR_TIMEOUT
        I.reset()
        I.run(30)
        check(I, O.run(prob, np_, 30, seed=16, kind="omp"), 30)


def test_row_by_row_batch_wait_that_runs_out_is_reported():
    """Members of rule R2 run row by row: batch_run_kernel's bounded wait for a member's previous
    generation. The member whose bound is 1 ns reports the timeout, the other is unaffected."""
    probs = [W.knapsack(3000, 41), W.knapsack(2500, 42)]
    with Q.Instance(probs[0], 120, seed=41, rule=1) as a, Q.Instance(probs[1], 90, seed=42, rule=1) as b:
        a.set_wait_timeout(1)
        with Q.Batch([a, b]) as bt:
            bt.run(6)
        with pytest.raises(Q.QieoError) as e:
            a.synchronize()
        assert e.value.status == Q.QIEO_ERR_TIMEOUT
        check(b, O.run(probs[1], 90, 6, seed=42, rule=1), 6)
        a.set_wait_timeout(10 * 10**9)
        a.reset()
        with Q.Batch([a]) as bt:
            bt.run(6)
        check(a, O.run(probs[0], 120, 6, seed=41, rule=1), 6)


def test_served_solve_whose_wait_runs_out_fails_alone():
    """A served solve on several blocks whose waits are bounded by 1 ns is reported as failed with the
    timeout; solves beside it, and one that needs the arena memory it leaves, are right."""
    prob, small = W.knapsack(20000, 5), W.knapsack(300, 6)
    with Q.Server(memory_bytes=64 << 20, gens_per_step=7) as srv:
        before = srv.submit(small, 40, 60, seed=1)
        srv.set_wait_timeout(1)
        bad = [srv.submit(prob, 500, 60, seed=2), srv.submit(prob, 500, 60, seed=2, flags=Q.QIEO_FLAG_CONVERGE)]
        srv.set_wait_timeout(10 * 10**9)
        after = srv.submit(prob, 500, 60, seed=3)
        for rid in bad:
            res, _ = srv.poll(rid, wait_ms=60000)
            assert (res.state, res.status) == (Q.QIEO_SOLVE_FAILED, Q.QIEO_ERR_TIMEOUT)
        for rid, p, n, seed in ((before, small, 40, 1), (after, prob, 500, 3)):
            res, bits = srv.poll(rid, wait_ms=60000)
            ref = O.run(p, n, 60, seed=seed, kind="omp")
            assert res.state == Q.QIEO_SOLVE_DONE
            assert (res.fitness, res.generation, res.chromosome) == tuple(int(v) for v in ref.best)
            assert np.array_equal(bits, ref.best_x)
        assert srv.stats()["completed"] == 2


def test_drawn_vectors_of_short_and_long_runs():
    """A long run counts the vectors on its list; a run of one generation draws every vector, fixed or
    not, and says so."""
    prob, np_ = W.knapsack(8000, 5), 2000
    with Q.Instance(prob, np_, seed=5, D=12) as I:
        assert I.shape().fixed_words == 1
        I.run(60)
        I.run(1)
        I.run(20)
        got = I.drawn_vectors(0, 81)
        assert got[0] == got[60] == np_ * 1000
        assert got[59] < np_ * 100 and got[61:].max() < np_ * 100
        check(I, O.run(prob, np_, 81, seed=5, D=12, kind="omp"), 81)


@pytest.mark.parametrize("start", ["checkpoint", "batch"])
def test_captured_run_goes_on_with_every_replay(start):
    """A run captured right after the population came from elsewhere: a checkpoint with equal rows, or a
    batch that ran row by row (a member asks for one launch per generation). Each replay of the
    graph continues where the one before stopped."""
    torch = pytest.importorskip("torch")
    prob, np_ = W.knapsack(2603, 5), 90
    stream = torch.cuda.Stream()
    with Q.Instance(prob, np_, seed=5, stream=stream.cuda_stream) as I:
        if start == "checkpoint":
            with Q.Instance(prob, np_, seed=5) as J:
                J.run(12)
                I.load(J.save())
        else:
            with Q.Instance(prob, np_, seed=6, stream=stream.cuda_stream, flags=Q.QIEO_FLAG_PER_GENERATION) as J:
                with Q.Batch([I, J]) as b:
                    b.run(12)
                J.synchronize()
        I.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            I.run(6)
        for _ in range(4):
            graph.replay()
        torch.cuda.synchronize()
        st = O.run(prob, np_, 36, seed=5)
        k, t = I.state()
        assert t == 36 and np.array_equal(k, st.k)
        bits, bf, bg, bc = I.best()
        assert (bf, bg, bc) == tuple(int(v) for v in st.best) and np.array_equal(bits, st.best_x)
        assert np.array_equal(I.fitness(), st.f)


@pytest.mark.parametrize("ng,np_,row", [(4096, 64, None), (4096, 64, 63), (4104, 64, None), (4104, 64, 1), (33, 9000, 8999),
                                        (1, 1, None), (20001, 300, None), (20001, 300, 299)])
def test_checkpoint_rows_are_compared(ng, np_, row):
    """A loaded population, with equal rows or with one gene of one row changed, on both sides of the
    size (512 KB: 4,096 x 64) from which the device compares the rows."""
    prob = W.knapsack(ng, 4)
    k0 = np.random.default_rng(ng).integers(-25, 26, size=(1, ng)).astype(np.int16).repeat(np_, 0)
    if row is not None:
        k0[row, ng - 1] = 25 if k0[row, ng - 1] < 25 else -25
    st = O.State(np_, ng)
    st.k[:] = k0
    O.run(prob, np_, 9, seed=4, state=st)
    with Q.Instance(prob, np_, seed=4) as I:
        load_state(I, k0)
        I.run(9)
        check(I, st, 9)


@pytest.mark.parametrize("before", ["", "run", "batch"])
def test_captured_row_by_row_batch_goes_on_with_every_replay(before):
    """A member that could run in the column form, in a batch that runs row by row: reset, perhaps a run in
    the column form, alone or in another batch, then a captured run of the batch, replayed."""
    torch = pytest.importorskip("torch")
    prob, np_ = W.knapsack(2603, 5), 90
    stream = torch.cuda.Stream()
    with Q.Instance(prob, np_, seed=5, stream=stream.cuda_stream) as I, \
            Q.Instance(prob, np_, seed=6, stream=stream.cuda_stream, flags=Q.QIEO_FLAG_PER_GENERATION) as J:
        with Q.Batch([I, J]) as b:
            b.run(3)
            I.reset()
            J.reset()
            if before == "run":
                I.run(8)
            if before == "batch":
                with Q.Batch([I]) as alone:
                    alone.run(8)
            I.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                b.run(6)
            for _ in range(4):
                graph.replay()
            torch.cuda.synchronize()
            for X, seed, gens in ((I, 5, 32 if before else 24), (J, 6, 24)):
                st = O.run(prob, np_, gens, seed=seed)
                k, t = X.state()
                assert t == gens and np.array_equal(k, st.k)
                assert np.array_equal(X.best()[0], st.best_x) and np.array_equal(X.fitness(), st.f)
        I.run(30)                # a run of its own goes on from there
        I.reset()
        I.run(30)
        check(I, O.run(prob, np_, 30, seed=5), 30)


@pytest.mark.parametrize("ng,np_,D,items,chunks", [
    (1, 1, 4, "byte", [2, 3, 4, 2]), (50, 33, 100, "byte", [4] * 24), (300, 70, 40, "wide", [2, 3, 4, 1] * 8),
    (4100, 130, 100, "mid", [3, 2, 5, 5, 5, 4, 4, 4, 5]), (2049, 65, 100, "byte", [4, 30, 2, 3, 40, 2, 4, 1, 2]),
    (600_001, 2, 100, "byte", [12, 4, 9, 4, 2]), (9, 300_000, 12, "byte", [4, 3, 2, 30, 4]),
])
def test_short_runs(ng, np_, D, items, chunks):
    """Runs of two to five generations as plain launches, each taking the CIP of the one before: before any
    gene can be fixed, later, and between runs in the cooperative form; a few rows of many genes and
    many rows of a few, where longer runs go this way."""
    prob, gens = _problem(ng, items), sum(chunks)
    st = O.run(prob, np_, gens, seed=ng, inst=3, D=D, lam=2, kind="omp")
    with Q.Instance(prob, np_, seed=ng, inst=3, D=D, lam=2) as I:
        for solve in range(2):
            for g in chunks:
                I.run(g)
            check(I, st, gens)
            I.reset()


@pytest.mark.parametrize("items,D,chunks", [("byte", 100, [1] * 12 + [5] + [1] * 3), ("mid", 12, [1] * 14), ("wide", 8, [2, 1, 1, 3, 1])])
def test_batched_runs_of_one_generation(items, D, chunks):
    """Runs of one generation of a batch (two plain launches), through 3 K generations, from which on they are
    cooperative; a member of rule R2 and one that stops by convergence among them."""
    specs = [(1, 1), (40, 30), (2049, 33), (4100, 90), (300, 257)]
    insts = [Q.Instance(_problem(ng, items), np_, seed=ng, D=D) for ng, np_ in specs]
    insts.append(Q.Instance(_problem(700, items), 40, seed=7, D=D, rule=1))
    conv = W.knapsack(60, 21)
    insts.append(Q.Instance(conv, 17, seed=21, flags=Q.QIEO_FLAG_CONVERGE))
    gens = sum(chunks)
    with Q.Batch(insts) as b:
        for solve in range(2):
            for g in chunks:
                b.run(g)
            for I, (ng, np_) in zip(insts, specs):
                check(I, O.run(_problem(ng, items), np_, gens, seed=ng, D=D), gens)
            check(insts[5], O.run(_problem(700, items), 40, gens, seed=7, D=D, rule=1), gens)
            check(insts[6], O.run(conv, 17, gens, seed=21), gens)
            for I in insts:
                I.reset()
        ref = O.run(conv, 17, 600, seed=21, window=20)
        n = int(ref.t[0])
        for _ in range(n + 5):
            b.run(1)
        k, t = insts[6].state()
        assert ref.stopped and t == n and np.array_equal(k, ref.k) and insts[6].convergence() == (True, 20)
    for I in insts:
        I.close()


@pytest.mark.parametrize("ng,np_,flags,shape,lam,items", [
    (5000, 90, 0, None, 1, "byte"), (5000, 90, Q.QIEO_FLAG_FORCE_WIDE, None, 1, "byte"), (5000, 90, 0, (32, 2, 0), 1, "byte"),
    (5000, 90, 0, (4, 1, 7), 1, "byte"), (5000, 90, 0, (32, 8, 40), 1, "byte"), (5000, 90, 0, (1, 1, 64), 1, "byte"),
    (5000, 90, Q.QIEO_FLAG_TIME_GENERATIONS, None, 1, "byte"), (900, 70, 0, None, 7, "mid"), (700, 40, 0, None, 1, "wide"),
    (2100, 12, 0, (1, 1, 0), 1, "byte"), (32800, 12, 0, (1, 1, 0), 1, "byte"),     # 263 and 4,100 tiles of one lane
    (263000, 4, 0, None, 1, "255"), (263200, 4, 0, None, 1, "255"),                # packed row sums just below and above 2^26
    (2050, 6000, 0, (32, 8, 2), 1, "byte"),
])
def test_rule_r1_row_by_row(ng, np_, flags, shape, lam, items):
    """Rule R1 from rows that differ, which the column form cannot hold: the resident form, the streamed
    one and their shapes, as the older tests of these forms had them run before the column form."""
    prob = W.custom_problem(np.full(ng, 255), np.full(ng, 255), 255 * ng // 2) if items == "255" else _problem(ng, items)
    k0 = np.random.default_rng(ng).integers(-25, 26, size=(np_, ng)).astype(np.int16)
    st = O.State(np_, ng)
    st.k[:] = k0
    st = O.run(prob, np_, 16, seed=ng, lam=lam, state=st, kind="omp")
    with Q.Instance(prob, np_, seed=ng, lam=lam, flags=flags) as I:
        if shape:
            I.set_shape(*shape)
        load_state(I, k0)
        for g in (7, 7, 2):
            I.run(g)
        check(I, st, 16)


def test_rule_r1_row_by_row_in_a_batch():
    """The persistent row-by-row form of a batch under rule R1: members whose rows differ; a wait that runs
    out; then one launch per generation (a member asks for it)."""
    prob, sizes = W.knapsack(3000, 41), ((120, 3), (90, 4))
    k0 = [np.random.default_rng(s).integers(-25, 26, size=(n, 3000)).astype(np.int16) for n, s in sizes]
    refs = []
    for (n, s), k in zip(sizes, k0):
        st = O.State(n, 3000)
        st.k[:] = k
        refs.append(O.run(prob, n, 12, seed=s, state=st))
    insts = [Q.Instance(prob, n, seed=s) for n, s in sizes]
    other = Q.Instance(prob, 20, seed=5, flags=Q.QIEO_FLAG_PER_GENERATION)
    for members in (insts, insts + [other]):
        with Q.Batch(members) as b:
            for I, k in zip(insts, k0):
                load_state(I, k)
            if members is insts:
                insts[0].set_wait_timeout(1)
                b.run(6)
                with pytest.raises(Q.QieoError) as e:
                    insts[0].synchronize()
                assert e.value.status == Q.QIEO_ERR_TIMEOUT
                insts[0].set_wait_timeout(10 * 10**9)
                for I, k in zip(insts, k0):
                    I.reset()
                    load_state(I, k)
            b.run(7)
            b.run(5)
            for I, st in zip(insts, refs):
                check(I, st, 12)
                I.reset()
    for I in members:
        I.close()


@pytest.mark.parametrize("np_", [30, 3000])
def test_generation_times_of_a_run_that_stops(np_):
    """The generations that a converged run does not execute take no time; nor does a run after it."""
    prob = W.knapsack(200, 3)
    with Q.Instance(prob, np_, seed=3, flags=Q.QIEO_FLAG_CONVERGE | Q.QIEO_FLAG_TIME_GENERATIONS) as I:
        I.run(700)
        n = I.state()[1]
        assert n < 690 and I.convergence() == (True, 20)
        ms = np.asarray(I.generation_times(700))
        assert len(ms) == 700 and ms[:n].min() > 0 and ms[:n].max() < 10 and not ms[n:].any()
        I.run(700)
        assert not np.asarray(I.generation_times(700)).any()


@pytest.mark.parametrize("rule,ng,np_,D", [(0, 200, 30, 100), (1, 40, 60, 8)])
@pytest.mark.parametrize("extra", [0, 1, 2])
def test_alleles_after_a_stop(rule, ng, np_, D, extra):
    """The alleles of the last generation that ran, whatever parity the generations asked for have."""
    prob = W.knapsack(ng, 3)
    ref = O.run(prob, np_, 900, seed=3, rule=rule, D=D, window=20)
    n = int(ref.t[0])
    assert ref.stopped
    for chunks in ([n + 5 + extra], [n + extra], [n - 2, 9 + extra]):
        with Q.Instance(prob, np_, seed=3, D=D, rule=rule, flags=Q.QIEO_FLAG_CONVERGE) as I:
            for g in chunks:
                I.run(g)
            assert I.state()[1] == n
            assert np.array_equal(I.alleles(), ref.x) and np.array_equal(I.allele_row(7), ref.x[7])


def test_kernel_times_of_repeated_runs():
    """Runs of one length, one launch per generation and timed: the second would replay a graph."""
    prob = W.knapsack(2603, 5)
    with Q.Instance(prob, 60, seed=5, rule=1, flags=Q.QIEO_FLAG_PER_GENERATION | Q.QIEO_FLAG_TIME_KERNELS) as I:
        for k in range(1, 5):
            I.run(6)
            ms, launches = I.kernel_time()
            assert launches == 6 * k and ms > 0
        check(I, O.run(prob, 60, 24, seed=5, rule=1), 24)


def test_more_resident_solves_than_a_work_list_starts_with():
    """4,500 small solves at once: the work lists grow between steps."""
    probs = [W.knapsack(320, s) for s in range(3)]
    with Q.Server(memory_bytes=1 << 30, max_active=5000, gens_per_step=1) as srv:
        ids = [srv.submit(probs[i % 3], 40, 400, seed=i + 1) for i in range(4500)]
        for i, rid in enumerate(ids):
            res, bits = srv.poll(rid, wait_ms=60000)
            assert res.state == Q.QIEO_SOLVE_DONE and res.generations_run == 400
            if i % 300 == 0:
                st = O.run(probs[i % 3], 40, 400, seed=i + 1)
                assert (res.fitness, res.generation, res.chromosome) == tuple(int(v) for v in st.best)
                assert np.array_equal(bits, st.best_x)
        assert srv.stats()["max_active"] > 3450
