"""The forms that the dispatch chooses by size, each against the oracle or against
the plain kernel, at the sizes where they can go wrong: edges of tiles, chunks and
row blocks, remainders, the smallest and largest of their range.  Integers bit for
bit."""
import threading

import numpy as np
import pytest

import oracle
from oracle import learned as OL
from paper_2310_07486_gb300 import qsg as Q

pytestmark = pytest.mark.gpu


def _context(shape, seed, ladder=None, **options):
    ctx = Q.Context([shape])
    ctx.qsg_init_samples(seed, [np.linspace(0.25, 0.35, shape.n_k) if ladder is None else ladder])
    for name, value in options.items():
        ctx.qsg_set_option(getattr(Q, "OPT_" + name), value)
    return ctx


@pytest.fixture
def chunked_sweep():
    """The fused kernel instead of the resident one where both serve a shape (the
    kernel form is process-wide: put back afterwards)."""
    shape = Q.Shape(8, 16, 1, 1, 1)
    Q.Context([shape]).qsg_set_option(Q.OPT_WAVEFRONT_VARIANT, 1)
    yield
    Q.Context([shape]).qsg_set_option(Q.OPT_WAVEFRONT_VARIANT, 0)


SMALL = [(2, 2), (2, 6), (4, 34), (6, 32), (8, 48), (10, 200), (12, 100), (14, 146), (16, 110), (22, 58), (28, 18), (32, 26)]


@pytest.mark.parametrize("L,Ltau", SMALL)
@pytest.mark.parametrize("algo,boundary", [(Q.METROPOLIS, Q.APBC), (Q.HEATBATH, Q.PBC)])
@pytest.mark.parametrize("K", [2, 20])
def test_resident_sweeps_match_the_plain_kernel(L, Ltau, algo, boundary, K):
    """20 ladder values make 80 slots, which stay resident; few large slots are chunked."""
    shape = Q.Shape(L, Ltau, 70, 2, K, algo, boundary)
    plain, fused = _context(shape, 3, SWEEP_KERNEL=1), _context(shape, 3)
    for n in (1, 4, 2):
        plain.qsg_sweep(n)
        fused.qsg_sweep(n)
    assert np.array_equal(plain.qsg_get_spins(0), fused.qsg_get_spins(0))


def test_long_calls_of_resident_sweeps_are_cut():
    """2^36 site-word updates per launch: 16,644 sweeps of 4.1 M words here."""
    shape = Q.Shape(8, 48, 64, 42, 32, Q.HEATBATH, Q.PBC)
    whole, halves = _context(shape, 5), _context(shape, 5)
    before = Q.qsg_kernel_launches()
    whole.qsg_sweep(17000)
    assert Q.qsg_kernel_launches() == before + 2
    for n in (16000, 1000):
        halves.qsg_sweep(n)
    assert np.array_equal(whole.qsg_get_spins(0), halves.qsg_get_spins(0))


@pytest.mark.parametrize("L,Ltau", [(6, 2), (6, 4), (6, 18), (6, 820), (8, 30), (10, 310), (12, 6), (14, 34), (16, 130),
                                    (18, 1022), (20, 50), (22, 14), (24, 66), (26, 20), (30, 36), (32, 10)])
@pytest.mark.parametrize("algo,boundary", [(Q.METROPOLIS, Q.PBC), (Q.HEATBATH, Q.APBC)])
def test_chunked_sweeps_of_any_ltau_match_the_plain_kernel(chunked_sweep, L, Ltau, algo, boundary):
    shape = Q.Shape(L, Ltau, 70, 1, 2, algo, boundary)
    plain, fused = _context(shape, 4, SWEEP_KERNEL=1), _context(shape, 4)
    plain.qsg_sweep(3)
    fused.qsg_sweep(3)
    assert np.array_equal(plain.qsg_get_spins(0), fused.qsg_get_spins(0))


# short extents (up to 4 words of sites), one and several row blocks, a last offset that
# is mirrored (L_tau / 2 a whole number of blocks) or not, streamed column blocks (L > 24)
CORR = [(2, 2), (4, 64), (8, 238), (8, 254), (8, 256), (10, 240), (12, 192), (14, 144), (16, 146), (16, 384), (6, 258),
        (12, 512), (18, 128), (18, 126), (20, 640), (22, 300), (24, 256), (24, 1024), (26, 512), (32, 256), (30, 130)]


@pytest.mark.parametrize("L,Ltau", CORR)
@pytest.mark.parametrize("boundary", [Q.PBC, Q.APBC])
def test_correlator_forms_match_the_integer_kernel(L, Ltau, boundary):
    shape = Q.Shape(L, Ltau, 66, 2, 2, Q.HEATBATH, boundary)
    got = []
    for kernel in (Q.CORR_TENSOR, Q.CORR_INTEGER):
        ctx = _context(shape, 5, CORR_KERNEL=kernel)
        for _ in range(2):
            ctx.qsg_sweep(2)
            ctx.qsg_measure_correlators()
        got.append(ctx.qsg_read_correlators(0, raw=True))
    for key in ("C_raw", "Q2_raw", "q2_raw"):
        assert np.array_equal(got[0][key], got[1][key]), key


def test_frozen_spins_reach_the_largest_correlator_sums():
    """All spins equal: every Gram element is L^2, the largest of every running sum."""
    shape = Q.Shape(24, 2048, 1, 2, 1, Q.HEATBATH, Q.PBC)
    ctx = _context(shape, 6)
    ctx.qsg_set_spins(0, np.zeros((shape.slots, shape.Ltau, 24, 24), dtype=np.uint64))
    ctx.qsg_measure_correlators()
    got = ctx.qsg_read_correlators(0, raw=True)
    assert np.all(got["C_raw"] == 2048 * 576) and np.all(got["Q2_raw"] == 2048 * 576 ** 2)


@pytest.mark.parametrize("spacing", [2e-4, 3e-2])
def test_tempering_tables_beyond_their_shared_heads_match_oracle(spacing):
    """A fine ladder (table entries past those held in shared memory) and a coarse one."""
    shape = Q.Shape(12, 64, 70, 2, 5, Q.METROPOLIS, Q.PBC)
    ladder = 0.3 + spacing * np.arange(5)
    ctx = _context(shape, 7, ladder)
    orc = oracle.OracleGroup(12, 64, 70, 2, 5, algo="metropolis")
    orc.init(7, ladder)
    for _ in range(3):
        ctx.qsg_sweep(1)
        orc.sweep(1)
        ctx.qsg_tempering_swap()
        orc.swap()
    assert np.array_equal(Q.unpack_spins(ctx.qsg_get_spins(0), shape), orc.spins())
    assert np.array_equal(ctx.qsg_read_accepts(0), orc.accepts())


def test_overlapped_groups_equal_groups_in_turn():
    """Tempering and measurements of groups with and without a scratch of their own, on
    side streams and one after another."""
    shapes = [Q.Shape(8, 48, 70, 3, 4, Q.HEATBATH, Q.PBC), Q.Shape(24, 512, 64, 4, 12, Q.HEATBATH, Q.APBC),
              Q.Shape(12, 64, 64, 4, 6, Q.HEATBATH, Q.PBC), Q.Shape(16, 256, 64, 2, 3, Q.HEATBATH, Q.PBC)]
    ladders = [np.linspace(0.25, 0.3, s.n_k) for s in shapes]
    got = []
    for mode in (1, 3):
        ctx = Q.Context(shapes)
        ctx.qsg_init_samples(9, ladders)
        ctx.qsg_set_option(Q.OPT_PERSISTENT, mode)
        for _ in range(3):
            ctx.qsg_sweep(2)
            ctx.qsg_tempering_swap()
            ctx.qsg_measure_correlators()
        got.append([(ctx.qsg_get_spins(g), ctx.qsg_read_correlators(g, raw=True), ctx.qsg_read_onetime(g)["raw"],
                     ctx.qsg_read_accepts(g), ctx.qsg_read_energies(g)) for g in range(len(shapes))])
    for a, b in zip(*got):
        assert np.array_equal(a[0], b[0])
        assert all(np.array_equal(a[1][k], b[1][k]) for k in a[1])
        assert all(np.array_equal(x, y) for x, y in zip(a[2:], b[2:]))


@pytest.mark.parametrize("L,Ltau,n_meas", [(2, 4, 1), (6, 34, 3), (14, 70, 7), (22, 258, 5), (32, 26, 49)])
def test_finish_rounds_like_one_division(L, Ltau, n_meas):
    ctx = _context(Q.Shape(L, Ltau, 70, 3, 2, Q.HEATBATH, Q.APBC), 15)
    for _ in range(n_meas):
        ctx.qsg_sweep(1)
        ctx.qsg_measure_correlators()
    got = ctx.qsg_read_correlators(0, raw=True)
    n, L2 = float(n_meas), float(L * L)
    assert np.array_equal(got["C"], got["C_raw"].astype(float) / (n * L2 * Ltau))
    assert np.array_equal(got["Q2"], got["Q2_raw"].astype(float) / (n * L2 * L2 * Ltau))


@pytest.mark.parametrize("L,Ltau,R", [(2, 4, 3), (14, 34, 8), (24, 66, 6), (26, 40, 4), (32, 130, 8)])
def test_onetime_sums_of_many_replicas_match_oracle(L, Ltau, R):
    shape = Q.Shape(L, Ltau, 3, R, 1, Q.METROPOLIS, Q.PBC)
    lad = np.array([0.3])
    ctx = _context(shape, 8, lad)
    orc = oracle.OracleGroup(L, Ltau, 3, R, 1, algo="metropolis")
    orc.init(8, lad)
    ctx.qsg_measure_correlators()
    orc.measure()
    assert np.array_equal(ctx.qsg_read_onetime()["raw"], orc.read_onetime()["raw"])


@pytest.mark.parametrize("n", [1, 608, 609, 3000])
def test_prediction_tiles_match_oracle(n):
    X = np.random.default_rng(n).random((n, 64), dtype=np.float32)
    theta = OL.init_params(3)
    m = Q.MLP(n, 16)
    m.set_params(theta)
    ref, e, _ = OL.fp32_forward_bound(theta.astype(np.float64), X)
    assert np.all(np.abs(m.predict(X, bf16=False).astype(np.float64) - ref) <= e)


@pytest.mark.parametrize("batch", [15, 3000])
def test_training_steps_of_one_call_equal_single_calls(batch):
    """257 steps (two launches) for a small batch; more tiles than SMs for a large one."""
    rng = np.random.default_rng(batch)
    X = rng.random((3000, 64), dtype=np.float32)
    T = np.full((3000, 33), 1.0 / 32, dtype=np.float32)
    steps = 257 if batch < 100 else 3
    idx = rng.integers(0, 3000, size=(steps, batch)).astype(np.int32)
    params, losses = [], []
    for cuts in ([0, steps], [0, 1, 2, steps]):
        m = Q.MLP(3000, batch)
        m.set_params(OL.init_params(4))
        m.set_data(X, T)
        losses.append(np.concatenate([m.train(idx[a:b], 1e-3) for a, b in zip(cuts, cuts[1:])]))
        params.append(m.get_params())
    assert np.array_equal(losses[0], losses[1]) and np.array_equal(params[0], params[1])
    assert np.all(np.isfinite(params[0]))


@pytest.mark.parametrize("shapes", [[Q.Shape(8, 48, 64, 4, 4, Q.HEATBATH)], [Q.Shape(16, 256, 64, 2, 8)],
                                    [Q.Shape(12, 64, 64, 2, 8), Q.Shape(8, 32, 64, 1, 2)]])
def test_graph_follows_a_second_initialisation_with_another_seed(shapes):
    """Captured sweeps hold the seed: resident, chunked and few-slot forms, one and two
    groups, against direct launches; another seed, then the first one again."""
    lads = [np.linspace(0.25, 0.35, s.n_k) for s in shapes]
    graphed, direct = Q.Context(shapes), Q.Context(shapes)
    graphed.qsg_set_option(Q.OPT_GRAPH, 3)
    for seed in (3, 2 ** 40 + 3, 3):
        for ctx in (graphed, direct):
            ctx.qsg_init_samples(seed, lads)
            ctx.qsg_sweep(7)
            ctx.qsg_tempering_swap()
        for g in range(len(shapes)):
            assert np.array_equal(graphed.qsg_get_spins(g), direct.qsg_get_spins(g)), (seed, g)


def test_long_calls_on_few_slots_are_cut_by_time():
    """Two small slots: 600,000 sweeps are half a second on two SMs, whatever the words
    add up to; a launch takes a quarter of one at most."""
    shape = Q.Shape(6, 32, 1, 2, 1, Q.METROPOLIS, Q.PBC)
    whole, parts = _context(shape, 5), _context(shape, 5)
    before = Q.qsg_kernel_launches()
    whole.qsg_sweep(600000)
    assert 2 <= Q.qsg_kernel_launches() - before <= 4
    for _ in range(6):
        parts.qsg_sweep(100000)
    assert np.array_equal(whole.qsg_get_spins(0), parts.qsg_get_spins(0))


# pairs of shapes whose launches share a kernel instance and need different amounts of
# shared memory above 48 KB: resident slots, ladder decisions, one-time sums
SHARED = [("qsg_sweep", Q.Shape(16, 50, 1, 1, 1), Q.Shape(16, 64, 1, 1, 1)),
          ("qsg_tempering_swap", Q.Shape(2, 2, 1, 1, 40), Q.Shape(2, 2, 1, 1, 128)),
          ("qsg_measure_correlators", Q.Shape(24, 128, 1, 6, 1), Q.Shape(24, 128, 1, 7, 1))]


@pytest.mark.parametrize("call,small,large", SHARED)
def test_threads_with_contexts_of_different_sizes(call, small, large):
    """Two host threads, each with its own context and stream: a launch of one must not
    lower the shared-memory limit that the other has just set."""
    torch = pytest.importorskip("torch")
    errors, start = [], threading.Barrier(2)

    def work(shape):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                ctx = _context(shape, 3, np.linspace(0.25, 0.35, shape.n_k))
                start.wait()
                for _ in range(4000):
                    getattr(ctx, call)()
                ctx.qsg_get_spins(0)
        except Exception as e:
            errors.append(e)

    threads = [threading.Thread(target=work, args=(s,)) for s in (small, large)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_graph_of_resident_groups_of_different_sizes():
    shapes = [Q.Shape(12, 160, 64, 2, 30, Q.HEATBATH), Q.Shape(12, 144, 64, 2, 30, Q.HEATBATH)]
    lads = [np.linspace(0.25, 0.35, 30)] * 2
    graphed, direct = Q.Context(shapes), Q.Context(shapes)
    graphed.qsg_set_option(Q.OPT_GRAPH, 4)
    for ctx in (graphed, direct):
        ctx.qsg_init_samples(5, lads)
        ctx.qsg_sweep(9)
    for g in range(2):
        assert np.array_equal(graphed.qsg_get_spins(g), direct.qsg_get_spins(g))


def test_finish_of_sums_over_a_count_set_to_zero_is_that_of_a_division():
    """Infinities with the sums' signs, NaN for 0 / 0; chi_lin adds up the C of every lag
    and replica."""
    shape = Q.Shape(8, 10, 70, 2, 2, Q.HEATBATH, Q.APBC)
    ctx = _context(shape, 15)
    ctx.qsg_sweep(3)
    ctx.qsg_measure_correlators()
    ctx.qsg_set_counters(3, 0, 0)
    got = ctx.qsg_read_correlators(0, raw=True)
    with np.errstate(divide="ignore", invalid="ignore"):
        C = got["C_raw"] / 0.0
        assert np.array_equal(got["C"], C, equal_nan=True) and np.isinf(C).any()
        assert np.array_equal(got["Q2"], got["Q2_raw"] / 0.0, equal_nan=True)
        chi = ctx.qsg_read_onetime()["chi_lin"]
        assert np.array_equal(chi, C.sum(axis=(0, 3)), equal_nan=True) and np.isnan(chi).any()


@pytest.mark.parametrize("L,Ltau,slots", [(6, 16, 1), (8, 16, 3), (16, 32, 7), (20, 16, 2), (24, 16, 7), (4, 32, 2)])
@pytest.mark.parametrize("algo,boundary", [(Q.METROPOLIS, Q.APBC), (Q.HEATBATH, Q.PBC)])
def test_graphs_of_few_small_slots_match_the_plain_kernel(L, Ltau, slots, algo, boundary):
    """One kernel per sweep as the larger slots have; the largest resident one (8,192 words)
    and one beyond it."""
    shape = Q.Shape(L, Ltau, 64, 1, slots, algo, boundary)
    plain, graph = _context(shape, 3, SWEEP_KERNEL=1), _context(shape, 3, GRAPH=4)
    for n in (4, 9, 1):
        plain.qsg_sweep(n)
        graph.qsg_sweep(n)
    assert np.array_equal(plain.qsg_get_spins(0), graph.qsg_get_spins(0))
    before = Q.qsg_kernel_launches()
    graph.qsg_sweep(4)
    assert Q.qsg_kernel_launches() - before == 4 + 2  # the counter set after direct sweeps, and advanced


@pytest.mark.parametrize("L,Ltau,K,launches", [(18, 50, 1, 6), (12, 100, 8, 6), (20, 34, 8, 1), (18, 50, 16, 1)])
def test_direct_sweeps_of_few_words_take_the_cheaper_form(L, Ltau, K, launches):
    """Extents that are no multiple of 16: two plain launches per sweep for few words in
    large slots, else one resident launch for the call."""
    ctx = _context(Q.Shape(L, Ltau, 64, 1, K, Q.HEATBATH, Q.PBC), 3)
    before = Q.qsg_kernel_launches()
    ctx.qsg_sweep(3)
    assert Q.qsg_kernel_launches() - before == launches


@pytest.mark.parametrize("L,Ltau,R,K", [(8, 64, 2, 1), (8, 64, 2, 2), (16, 128, 2, 9), (16, 128, 2, 10), (4, 240, 2, 7),
                                        (12, 16, 2, 1), (12, 18, 2, 1)])
def test_short_extents_on_both_sides_of_the_sample_line(L, Ltau, R, K):
    """Tensor tiles for few sample bits, the integer form for many: the same sums."""
    shape = Q.Shape(L, Ltau, 64, R, K, Q.HEATBATH, Q.APBC)
    got = []
    for kernel in (Q.CORR_TENSOR, Q.CORR_INTEGER):
        ctx = _context(shape, 5, CORR_KERNEL=kernel)
        ctx.qsg_sweep(2)
        ctx.qsg_measure_correlators()
        got.append(ctx.qsg_read_correlators(0, raw=True))
    for key in ("C_raw", "Q2_raw", "q2_raw"):
        assert np.array_equal(got[0][key], got[1][key]), key


@pytest.mark.parametrize("L,Ltau", [(4, 86), (8, 100), (12, 128), (16, 88), (18, 84), (20, 90), (24, 128), (26, 86), (28, 126),
                                    (26, 128), (26, 130), (32, 160), (30, 254), (32, 256), (26, 84), (28, 258)])
@pytest.mark.parametrize("boundary", [Q.PBC, Q.APBC])
def test_tiles_of_one_and_two_row_blocks(L, Ltau, boundary):
    """The triangle of row pairs at the ends of its range and the offsets beyond them, in the
    lags, in the largest sums (all spins equal) and for few sample bits."""
    shape = Q.Shape(L, Ltau, 64, 2, 1, Q.HEATBATH, boundary)
    got = []
    for kernel in (Q.CORR_TENSOR, Q.CORR_INTEGER):
        ctx = _context(shape, 5, CORR_KERNEL=kernel)
        ctx.qsg_sweep(2)
        ctx.qsg_measure_correlators()
        ctx.qsg_set_spins(0, np.zeros((shape.slots, Ltau, L, L), dtype=np.uint64))
        ctx.qsg_measure_correlators()
        got.append(ctx.qsg_read_correlators(0, raw=True))
    for key in ("C_raw", "Q2_raw", "q2_raw"):
        assert np.array_equal(got[0][key], got[1][key]), key


def test_workspace_without_the_groups_own_scratch():
    """Two small groups in a workspace that holds one correlator scratch: the same results;
    a byte less is refused."""
    shapes = [Q.Shape(8, 48, 70, 3, 4, Q.HEATBATH), Q.Shape(12, 64, 64, 4, 6, Q.HEATBATH, Q.APBC)]
    lads = [np.linspace(0.25, 0.3, s.n_k) for s in shapes]
    own = [s.n_replicas * 64 * s.Ltau * ((s.L ** 2 + 63) // 64) * s.words * s.n_k * 8 for s in shapes]
    features = max(s.words for s in shapes) * 64 * 64 * 4
    full = Q.qsg_workspace_bytes(shapes)
    lean = full - sum(own) - features + max(own)
    assert all(v % 256 == 0 for v in own) and max(own) > features
    with pytest.raises(Q.QSGError) as e:
        Q.Context(shapes, workspace_bytes=lean - 1)
    assert e.value.status == -6
    got = []
    for size in (full, full - 1, lean):
        ctx = Q.Context(shapes, workspace_bytes=size)
        ctx.qsg_init_samples(9, lads)
        for _ in range(2):
            ctx.qsg_sweep(2)
            ctx.qsg_measure_correlators()
        got.append([(ctx.qsg_read_correlators(g, raw=True), ctx.qsg_read_onetime(g)["raw"], ctx.qsg_sample_features(g))
                    for g in range(2)])
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert all(np.array_equal(a[0][k], b[0][k]) for k in a[0])
            assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


def test_contexts_are_made_and_destroyed_beside_running_work():
    """Neither waits for the device; the words of the flag's copies are given back and more
    contexts than there are serve all the same."""
    torch = pytest.importorskip("torch")
    busy = _context(Q.Shape(24, 1024, 64, 4, 16, Q.HEATBATH), 1)
    small = Q.Shape(8, 16, 1, 1, 1)
    _context(small, 2).close()
    torch.cuda.synchronize()
    busy.qsg_sweep(3000)  # 0.2 s
    done = torch.cuda.Event()
    done.record()
    with torch.cuda.stream(torch.cuda.Stream()):
        for _ in range(3):
            Q.Context([small]).close()
    assert not done.query()
    many = [Q.Context([small]) for _ in range(520)]
    for ctx in (many[0], many[-1]):
        ctx.qsg_init_samples(2, [[0.3]])
        ctx.qsg_sweep(2)
    assert np.array_equal(many[0].qsg_get_spins(0), many[-1].qsg_get_spins(0))
