"""Batched 1D Riemann tubes (one persistent launch) against the FP64 oracle, tube by tube."""
import numpy as np
import pytest

from tests.parity import assert_fp32, assert_fp64, field_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def msh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1210_5246_gb300 import msh as m
    m.load()
    return m


def _random_tubes(lengths, seed):
    from paper_1210_5246_gb300 import inputs
    t = inputs.tubes(ntubes=len(lengths), seed=seed)
    t.length = np.asarray(lengths, dtype=np.int32)
    return t


def _oracle_tube(oracle, tubes, k, dtype=np.float64):
    n = int(tubes.length[k])
    W = tubes.initial_tube(k).astype(dtype).astype(np.float64)
    g = oracle.Grid((n,), (0.0,), (1.0,), ((1, 1),), tubes.cfl)
    U, steps, t, rc, _ = oracle.run(g, oracle.prim_to_cons(W), tubes.t_end)
    return U.reshape(10, n), steps, t, rc


LENGTHS = [4, 5, 17, 64, 127, 128, 129, 255, 256, 257, 300, 513, 1000, 1024]


def test_batch_fp64_matches_oracle(msh, oracle):
    tubes = _random_tubes(LENGTHS, seed=41)
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    b.run(threads=256)
    U = b.get_state()
    steps, t, cu = b.info()
    for k in range(len(LENGTHS)):
        Uo, so, to, rc = _oracle_tube(oracle, tubes, k)
        assert rc == 0 and steps[k] == so and t[k] == to == tubes.t_end
        assert_fp64(b.tube(U, k), Uo, what=f"tube {k} (len {LENGTHS[k]})")
    assert cu == int((steps * tubes.length).sum())
    b.close()


def test_batch_fp32_matches_oracle(msh, oracle):
    tubes = _random_tubes(LENGTHS[:-2] + [1500, 2048], seed=42)
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP32)
    b.run(threads=128)
    W = b.get_state(msh.PRIMITIVE).astype(np.float64)
    for k in range(len(tubes.length)):
        Uo, _, _, _ = _oracle_tube(oracle, tubes, k, np.float32)
        assert_fp32(b.tube(W, k), oracle.cons_to_prim(Uo), what=f"tube {k}")
    b.close()


def test_block_sizes_and_autotune_agree_bitwise(msh):
    tubes = _random_tubes([37, 400, 1000, 129, 2048, 6], seed=43)
    out = []
    for nt in (128, 256, 512, 0):
        b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP32)
        b.run(threads=nt)
        out.append(b.get_state())
        b.close()
    for o in out[1:]:
        np.testing.assert_array_equal(o, out[0])


def test_per_tube_launches_match_batch(msh):
    tubes = _random_tubes([64, 300, 129, 1000], seed=44)
    b1 = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    b1.run()
    b2 = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    b2.run_per_tube()
    s1, t1, _ = b1.info()
    s2, t2, _ = b2.info()
    np.testing.assert_array_equal(s1, s2)
    np.testing.assert_array_equal(t1, t2)
    assert_fp64(b2.get_state(), b1.get_state(), tol=1e-12, what="per-tube vs batch")
    b1.close()
    b2.close()


def test_reset_reproduces_run(msh):
    tubes = _random_tubes([100, 200], seed=45)
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP32)
    b.run(threads=256)
    a = b.get_state()
    b.reset()
    b.run(threads=256)
    np.testing.assert_array_equal(b.get_state(), a)
    b.close()


def test_step_cap_reports_timeout(msh):
    tubes = _random_tubes([200], seed=46)
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP32)
    with pytest.raises(msh.MshError) as ei:
        b.run(threads=128, max_steps=3)
    assert ei.value.status == msh.MSH_E_TIMEOUT
    b.close()


def test_rejects_bad_tubes(msh):
    from paper_1210_5246_gb300 import inputs
    t = inputs.tubes(ntubes=2, seed=47)
    with pytest.raises(msh.MshError):
        msh.Batch(np.array([3, 10]), t.WL, t.WR, t.t_end)
    bad = t.WL.copy()
    bad[1, 0] = -1.0
    with pytest.raises(msh.MshError) as ei:
        msh.Batch(t.length.clip(4, 100), bad, t.WR, t.t_end)
    assert ei.value.status == msh.MSH_E_REALIZABILITY


def _oracle_tubes(oracle, tubes, ks, dtype):
    """Oracle runs of tubes ks (from the initial states rounded to dtype), in parallel threads
    (the oracle's C code is re-entrant and runs without the GIL; one OpenMP thread each)."""
    import concurrent.futures as cf
    import os

    def one(k):
        oracle.set_num_threads(1)
        return k, _oracle_tube(oracle, tubes, k, dtype)
    with cf.ThreadPoolExecutor(max_workers=max(1, min(32, os.cpu_count() or 1))) as ex:
        return dict(ex.map(one, ks))


def test_full_workload_4096_tubes(msh, oracle):
    """The full batched workload (4096 tubes, 128..2048 cells, FP32, t = 0.1) in one persistent
    launch, against the oracle run of every tube from the FP32-rounded input:
    * the workload as one state (all tubes back to back, the norm of every other workload):
      relative L1 <= 2e-4 on rho and <= 5e-4 on each P_ij;
    * every tube realizable at t_end; per tube the same tolerances for all but at most 1 %
      of the tubes (a tube with near-vacuum states can take a different but valid path where
      a rounding-level difference flips a discontinuous decision: a face state's
      positivity check or an a-posteriori fallback tag), and every tube within 4x them.
    The tubes of up to 1024 cells (the FP64 batch limit) also run as one FP64 batch: every
    tube within the FP32 tolerances, 99 % of them element by element at 1e-10 with the
    oracle's step count, among them every one whose run took no fallback."""
    from paper_1210_5246_gb300 import inputs
    tubes = inputs.tubes()
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP32)
    b.run()
    steps, t, cu = b.info()
    fb = b.fallback_steps()
    assert np.all(t == tubes.t_end)
    W = b.get_state(msh.PRIMITIVE).astype(np.float64)
    b.close()
    assert np.all(W[0] > 0) and np.all(W[4] > 0)
    assert len(np.nonzero(fb)[0]) > 0  # the workload exercises the fallback
    ref = _oracle_tubes(oracle, tubes, range(4096), np.float32)
    Wo = np.concatenate([oracle.cons_to_prim(ref[k][0]) for k in range(4096)], axis=1)
    assert all(ref[k][3] == 0 for k in range(4096))
    assert_fp32(W, Wo, what="4096 tubes as one state")
    worst = np.zeros(4096)
    for k in range(4096):
        e = field_errors(b.tube(W, k), oracle.cons_to_prim(ref[k][0]), "l1")
        worst[k] = max(e[0] / 2e-4, max(e[4:]) / 5e-4)
    assert (worst > 1).sum() <= 41 and worst.max() <= 4, (int((worst > 1).sum()), float(worst.max()))
    # FP64: the tubes that fit an FP64 batch
    from paper_1210_5246_gb300 import inputs as I
    k64 = [k for k in range(4096) if tubes.length[k] <= 1024]
    sub = I.Tubes(tubes.length[k64], tubes.WL[k64], tubes.WR[k64], tubes.t_end, tubes.cfl)
    b64 = msh.Batch(sub.length, sub.WL, sub.WR, sub.t_end, sub.cfl, msh.FP64)
    b64.run()
    s64, t64, _ = b64.info()
    fb64 = b64.fallback_steps()
    U64 = b64.get_state()
    b64.close()
    ref64 = _oracle_tubes(oracle, sub, list(range(len(k64))), np.float64)
    exact = 0
    for i, k in enumerate(k64):
        Uo, so, to, rc = ref64[i]
        assert rc == 0 and t64[i] == to
        e = field_errors(b64.tube(U64, i), Uo, "linf").max()
        if e <= 1e-10 and s64[i] == so:
            exact += 1
        else:
            assert_fp32(oracle.cons_to_prim(b64.tube(U64, i)), oracle.cons_to_prim(Uo), what=f"fp64 tube {k}")
            assert fb64[i] > 0 or e <= 1e-8, (k, e)
    assert exact >= 0.99 * len(k64), (exact, len(k64))


def test_iterated_fallback_tube_fp64(msh, oracle):
    """Tube 3519 of the batched workload (density ratio 33, P_xx = 0.016 on the light side)
    needs more than one fallback pass: the batch kernel and the 1D grid kernel both match
    the oracle run to t_end."""
    from paper_1210_5246_gb300 import inputs
    full = inputs.tubes()
    k = 3519
    tubes = _random_tubes([int(full.length[k])], seed=48)
    tubes.WL[0], tubes.WR[0] = full.WL[k], full.WR[k]
    Uo, so, to, rc = _oracle_tube(oracle, tubes, 0)
    assert rc == 0 and to == tubes.t_end
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    b.run(threads=128)
    steps, t, _ = b.info()
    assert steps[0] == so and t[0] == to
    assert_fp64(b.tube(b.get_state(), 0), Uo, what="batch tube 3519")
    b.close()
    n = int(tubes.length[0])
    g = msh.Grid((n,), (0.0,), (1.0,), ((1, 1),), tubes.cfl, msh.FP64)
    g.set_state(tubes.initial_tube(0), msh.PRIMITIVE)
    ns, tg = g.run(tubes.t_end)
    assert ns == so and tg == to
    assert_fp64(g.get_state(), Uo.reshape(10, 1, 1, n), what="grid tube 3519")
    g.close()


@pytest.mark.parametrize("prec,lengths", [
    ("FP64", [29, 30, 31, 59, 60, 61, 91, 240, 241, 256, 257, 512, 513]),
    ("FP32", [29, 30, 31, 59, 60, 61, 91, 481, 512, 513, 961, 1024, 1025]),
])
def test_segment_and_class_edges(msh, oracle, prec, lengths):
    # lengths around the 30-cell segments of a warp and the limits of the length classes, all
    # classes in one batch: the same bits as with one block size for all, and the oracle's states
    tubes = _random_tubes(lengths, seed=47)
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, getattr(msh, prec))
    b.run()
    U = b.get_state().copy()
    W = b.get_state(msh.PRIMITIVE).astype(np.float64)
    b.reset()
    b.run(threads=128)
    assert np.array_equal(U, b.get_state())
    steps, _, _ = b.info()
    for k in range(len(lengths)):
        Uo, so, _, rc = _oracle_tube(oracle, tubes, k, np.float64 if prec == "FP64" else np.float32)
        assert rc == 0
        if prec == "FP64":
            assert steps[k] == so
            assert_fp64(b.tube(U, k), Uo, what=f"tube {k} (len {lengths[k]})")
        else:
            assert_fp32(b.tube(W, k), oracle.cons_to_prim(Uo), what=f"tube {k} (len {lengths[k]})")
    b.close()


def test_fp64_batch_larger_than_the_chip(msh, oracle):
    # more FP64 tubes than SMs sweep chunk by chunk through shared memory: lengths around the chunks
    # of each class's blocks (64, 128, 256 cells, and two ghost cells) against the oracle
    edges = [4, 61, 62, 63, 64, 126, 127, 190, 253, 254, 255, 256, 257, 382, 510, 511, 512, 513, 766, 1024]
    tubes = _random_tubes(edges + [5] * 1300, seed=48)
    tubes.t_end = 0.02
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    b.run()
    U = b.get_state()
    steps, _, _ = b.info()
    for k in range(len(edges) + 3):
        Uo, so, _, rc = _oracle_tube(oracle, tubes, k)
        assert rc == 0 and steps[k] == so
        assert_fp64(b.tube(U, k), Uo, what=f"tube {k} (len {tubes.length[k]})")
    b.close()


def test_fp64_sweep_form_edges(msh, oracle):
    # lengths at which an FP64 tube changes between segments and chunks, in a batch whose medium
    # tubes fill a class of their own: against the oracle, and the same bits at every block size
    edges = [119, 120, 121, 126, 127, 239, 240, 241, 254, 255, 361, 382, 383, 480, 481, 510, 511, 842, 894, 895]
    tubes = _random_tubes(edges + [100] * 310 + [20] * 310, seed=49)
    tubes.t_end = 0.02
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    b.run()
    U = b.get_state()
    steps, _, _ = b.info()
    for k in list(range(len(edges))) + [len(edges), len(tubes.length) - 1]:
        Uo, so, _, rc = _oracle_tube(oracle, tubes, k)
        assert rc == 0 and steps[k] == so
        assert_fp64(b.tube(U, k), Uo, what=f"tube {k} (len {tubes.length[k]})")
    for threads in (128, 256, 512):
        b.reset()
        b.run(threads=threads)
        assert np.array_equal(U, b.get_state())
    b.close()


def test_fp64_tubes_too_long_for_512_threads_are_refused(msh):
    tubes = _random_tubes([1000], seed=50)
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    with pytest.raises(msh.MshError) as ei:
        b.run(threads=512)
    assert ei.value.status == msh.MSH_E_INVALID_ARG and "512 threads" in str(ei.value)
    b.close()


def test_first_run_with_chosen_block_sizes_starts_over(msh):
    """The first run with threads = 0 starts from the initial state, also after runs with an
    explicit block size; later runs go on from where the tubes are."""
    tubes = _random_tubes([60, 200, 333], seed=51)
    b = msh.Batch(tubes.length, tubes.WL, tubes.WR, tubes.t_end, tubes.cfl, msh.FP64)
    b.run(threads=256)
    U = b.get_state()
    b.run()
    np.testing.assert_array_equal(b.get_state(), U)
    b.run()
    assert not np.array_equal(b.get_state(), U)
    b.close()
