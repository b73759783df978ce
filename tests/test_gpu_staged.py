"""The staged step (the default of FP64 grids and of small FP32 grids) against the streaming
step kernels (a grid whose tiling was set): the same arithmetic per cell and face, so the
states, times and fallback tags have to agree bit for bit, at sizes around a group of 32
items, with every kind of boundary, scheme, gravity and with fallback passes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BCS = {"per": (0, 0), "out": (1, 1), "ref": (2, 2), "mix": (2, 1)}


@pytest.fixture(scope="module")
def msh():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1210_5246_gb300 import msh as m
    m.load()
    return m


def _state(shape, seed, extreme=False):
    rng = np.random.default_rng(seed)
    W = np.zeros((10,) + shape)
    s = 2.0 if extreme else 0.5
    W[0] = np.exp(rng.uniform(-s, s, shape))
    W[1:4] = rng.uniform(-1.5, 1.5, (3,) + shape)
    d = [rng.uniform(0.2, 1.0, shape) for _ in range(3)]
    a, b, c = (rng.normal(0.0, 0.2, shape) for _ in range(3))
    W[4], W[5], W[6] = d[0] ** 2, a * d[0], b * d[0]
    W[7], W[8], W[9] = a * a + d[1] ** 2, a * b + c * d[1], b * b + c * c + d[2] ** 2
    return W


def _run(msh, n, bc, prec, scheme, W, steps, tiling, phi=None, G=0.0):
    nd = len(n)
    g = msh.Grid(n, (0.0,) * nd, (1.0, 1.5, 0.5)[:nd], (bc,) * nd, 0.3, prec)
    if tiling:
        g.set_tiling(8, 0 if nd == 3 else 4)
    g.set_scheme(scheme)
    if phi is not None:
        g.set_potential(phi)
    if G:
        g.set_self_gravity(G)
    g.set_state(W.astype(g.dtype), msh.PRIMITIVE)
    dt = g.step()
    n_, t = g.run(max_steps=steps)
    out = (dt, n_, t, g.get_state(), g.diagnostics())
    g.close()
    return out


def _same(a, b):
    assert a[:3] == b[:3]
    np.testing.assert_array_equal(a[3], b[3])
    # the totals are summed in another order (FP32 streaming sums start in FP32)
    scale = np.abs(b[4][0]).max()
    assert np.abs(a[4][0] - b[4][0]).max() <= (1e-12 if a[3].dtype == np.float64 else 1e-6) * scale
    assert a[4][1:] == b[4][1:]


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
@pytest.mark.parametrize("scheme", ["MUSCL_HANCOCK", "MUSCL_HANCOCK_ROE", "MUSCL_HANCOCK_HLLC", "KT"])
@pytest.mark.parametrize("n,bc", [((2,), "ref"), ((33,), "mix"), ((260,), "per"), ((31, 2), "out"), ((45, 33), "mix"),
                                  ((64, 32), "per"), ((2, 3, 2), "ref"), ((33, 7, 19), "mix"), ((17, 32, 9), "per")])
def test_staged_equals_streaming(msh, n, bc, scheme, prec):
    W = _state(n[::-1] if len(n) == 3 else (1,) * (3 - len(n)) + n[::-1], sum(n))
    p, s = getattr(msh, prec), getattr(msh, scheme)
    if scheme == "KT":
        W[1:4] *= 0.3
    _same(_run(msh, n, BCS[bc], p, s, W, 20, False), _run(msh, n, BCS[bc], p, s, W, 20, True))


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
@pytest.mark.parametrize("n", [(45, 33), (33, 7, 19)])
def test_staged_gravity_equals_streaming(msh, n, prec):
    W = _state((1,) * (3 - len(n)) + n[::-1], 3)
    rng = np.random.default_rng(5)
    pad = tuple(m + 2 for m in n[::-1])
    phi = 0.01 * rng.uniform(-1.0, 1.0, (1,) * (3 - len(n)) + pad)
    p = getattr(msh, prec)
    _same(_run(msh, n, BCS["out"], p, 0, W, 20, False, phi), _run(msh, n, BCS["out"], p, 0, W, 20, True, phi))
    _same(_run(msh, n, BCS["per"], p, 0, W, 40, False, phi, 0.2), _run(msh, n, BCS["per"], p, 0, W, 40, True, phi, 0.2))


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
@pytest.mark.parametrize("scheme", ["MUSCL_HANCOCK", "MUSCL_HANCOCK_ROE", "MUSCL_HANCOCK_HLLC"])
@pytest.mark.parametrize("n,bc", [((300,), "out"), ((60, 41), "mix"), ((25, 18, 12), "ref")])
def test_staged_fallback_equals_streaming(msh, n, bc, scheme, prec):
    """Extreme states over steps longer than the CFL rule allows: cells are tagged and fallback
    passes run; tags counted per step and the states agree."""
    W = _state((1,) * (3 - len(n)) + n[::-1], 7, extreme=True)
    nd, out = len(n), []
    for tiling in (False, True):
        g = msh.Grid(n, (0.0,) * nd, (1.0,) * nd, (BCS[bc],) * nd, 0.5, getattr(msh, prec))
        if tiling:
            g.set_tiling(4, 5)
        g.set_scheme(getattr(msh, scheme))
        g.set_state(W.astype(g.dtype), msh.PRIMITIVE)
        _, dt, _ = g.reduce_layers(0, n[-1])
        tags = []
        for f in (1.0, 1.2, 1.0):
            try:
                tags.append(g.step_dt(f * dt))
            except msh.MshError as e:  # a cell that stays non-realizable: the state is kept
                tags.append((e.status, str(e)))
                break
        out.append((tags, g.get_state()))
        g.close()
    assert out[0][0] == out[1][0] and out[0][0][0] != 0
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
@pytest.mark.parametrize("n,bc", [((40,), "mix"), ((2,), "ref"), ((33, 18), "mix"), ((32, 9), "per"), ((21, 30), "out"),
                                  ((3, 2), "ref"), ((12, 7, 9), "mix"), ((8, 6, 33), "per"), ((2, 3, 2), "out")])
def test_staged_reverse_equals_pencils(msh, n, bc, prec):
    """Three reverse steps (K = 2: a recomputed state in one segment) with gravity: the staged
    reverse steps and the pencil kernels apply the same adjoint to the same forward states and
    differ in the order of the sums that reach a cell, at most 4 ndim + 4 terms per step:
    well within 1e-12 (FP64) and 2e-5 (FP32) of the largest entry."""
    nd = len(n)
    W = _state((1,) * (3 - nd) + n[::-1], 11)
    W[1:4] *= 0.5
    rng = np.random.default_rng(3)
    phi = 0.01 * rng.uniform(-1.0, 1.0, (1,) * (3 - nd) + tuple(m + 2 for m in n[::-1]))
    lam = rng.normal(size=W.shape)
    out = []
    for tiling in (False, True):
        g = msh.Grid(n, (0.0,) * nd, (1.0, 1.5, 0.5)[:nd], (BCS[bc],) * nd, 0.3, getattr(msh, prec))
        if tiling:
            g.set_tiling(8, 0 if nd == 3 else 4)
        g.set_potential(phi)
        g.set_state(W.astype(g.dtype), msh.PRIMITIVE)
        _, dt, _ = g.reduce_layers(0, n[-1])
        out.append(g.adjoint_run(W.astype(g.dtype), [0.9 * dt, 0.8 * dt, 0.7 * dt], lam.astype(g.dtype), K=2,
                                 kind=msh.PRIMITIVE).astype(np.float64))
        g.close()
    tol = 1e-12 if prec == "FP64" else 2e-5
    assert np.abs(out[0] - out[1]).max() <= tol * np.abs(out[1]).max()


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
@pytest.mark.parametrize("n,tiling", [((60, 41), (4, 5)), ((90, 70), (16, 9)), ((25, 18, 12), (8, 0)), ((64, 33, 20), (8, 5))])
def test_run_that_tags_cells(msh, n, tiling, prec):
    """A streaming run launches its steps without fallback passes until one tags cells; profiled
    runs launch every pass.  Extreme states tag cells in the first steps and later: states,
    times and the error of a run that stays non-realizable agree, also over short runs."""
    nd = len(n)
    W = _state((1,) * (3 - nd) + n[::-1], 7, extreme=True)
    out = []
    for profiled in (False, True):
        g = msh.Grid(n, (0.0,) * nd, (1.0,) * nd, (BCS["mix"],) * nd, 0.5, getattr(msh, prec))
        g.set_tiling(*tiling)
        g.set_profiling(profiled)
        g.set_state(W.astype(g.dtype), msh.PRIMITIVE)
        seen = []
        for steps in (3, 40, 1):
            try:
                seen.append(g.run(max_steps=steps))
            except msh.MshError as e:
                seen.append((e.status, str(e)))
                break
        out.append((seen, g.get_state(), g.time(), g.diagnostics()[1:]))
        g.close()
    assert out[0][0] == out[1][0] and out[0][2:] == out[1][2:]
    np.testing.assert_array_equal(out[0][1], out[1][1])
    # the first step tags cells
    g = msh.Grid(n, (0.0,) * nd, (1.0,) * nd, (BCS["mix"],) * nd, 0.5, getattr(msh, prec))
    g.set_tiling(*tiling)
    g.set_state(W.astype(g.dtype), msh.PRIMITIVE)
    _, dt, _ = g.reduce_layers(0, n[-1])
    try:
        assert g.step_dt(dt) > 0
    except msh.MshError:
        pass
    g.close()


def test_noalloc_thin_box_fits_the_fixed_scratch(msh):
    # a box two cells wide and deep whose default shape for a grid would be 18695 blocks, more
    # partials than the allocation-free step's scratch holds: stepped all the same, to the same bits
    import torch
    n, bc = (2, 261730, 2), ((0, 0),) * 3
    W = _state((n[2], n[1], n[0]), seed=61)
    g = msh.Grid(n, (0.0,) * 3, (1.0, 1.5, 0.5), bc, 0.3, msh.FP32)
    g.set_tiling(8, 0)
    g.set_state(W.astype(np.float32), msh.PRIMITIVE)
    U0 = g.get_state()
    dt = g.step()
    U1 = g.get_state()
    g.close()
    u0 = torch.tensor(U0, device="cuda")
    u1 = torch.empty_like(u0)
    e = msh.msh_step_noalloc(n, (0.0,) * 3, (1.0, 1.5, 0.5), bc, msh.FP32, 0.3, u0, u1)
    assert abs(e - dt) <= 1e-12 * dt
    assert np.array_equal(u1.cpu().numpy().reshape(U1.shape), U1)


def _after_step_ms(g, reps=6):
    """Time that a profiled step takes after its step kernel: fallback passes and finalize of a
    streaming step (five launches), nothing but two events of a staged one."""
    ms = []
    for _ in range(reps):
        g.set_profiling(True)
        g.run(max_steps=1)
        ms.append(g.profile()[1])
        g.set_profiling(False)
    return min(ms)


@pytest.mark.parametrize("prec,n,staged", [("FP32", 3000, True), ("FP32", 600000, True), ("FP32", 1500000, False),
                                           ("FP64", 1500000, True)])
def test_large_1d_grids(msh, n, prec, staged):
    """1D grids around the size at which the staged step's buffers leave L2: the default takes the
    staged step below it only (FP32), and gives the bits of the streaming step."""
    rng = np.random.default_rng(6)
    W = np.zeros((10, 1, 1, n))
    W[0] = rng.uniform(0.8, 1.2, n)
    W[1:4] = rng.uniform(-0.2, 0.2, (3, 1, 1, n))
    W[4] = W[7] = W[9] = rng.uniform(0.9, 1.1, n)
    out, after = [], []
    for tiling in (False, True):
        g = msh.Grid((n,), (0.0,), (1.0,), ((1, 1),), 0.4, getattr(msh, prec))
        if tiling:
            g.set_tiling(8, 1)
        g.set_state(W.astype(g.dtype), msh.PRIMITIVE)
        g.run(max_steps=3)
        out.append((g.time(), g.get_state()))
        after.append(_after_step_ms(g))
        g.close()
    assert (after[0] < 0.5 * after[1]) == staged
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("prec,n", [("FP64", (200, 150)), ("FP64", (40, 30, 20)), ("FP32", (900, 700)), ("FP32", (64, 64, 64)),
                                    ("FP32", (48, 40, 32))])
def test_autotune_keeps_a_form_of_the_step(msh, prec, n):
    """Autotune leaves the state and time as they were and returns the streaming shape; whichever form
    it keeps, the run's bits are the default's, an explicit tiling streams, and an FP32 grid too
    large for the staged step streams in any case."""
    nd = len(n)
    W = _state((1,) * (3 - nd) + n[::-1], 21)
    W[1:4] *= 0.2
    out = []
    for tune in (False, True):
        g = msh.Grid(n, (0.0,) * nd, (1.0,) * nd, (BCS["per"],) * nd, 0.3, getattr(msh, prec))
        g.set_state(W.astype(g.dtype), msh.PRIMITIVE)
        if tune:
            U = g.get_state()
            shape = g.autotune()
            np.testing.assert_array_equal(g.get_state(), U)
            assert g.tiling() == shape and g.time() == (0.0, 0)
        g.run(max_steps=20)
        out.append((g.time(), g.get_state()))
        if tune:
            after = _after_step_ms(g)
            g.set_tiling(*shape)
            after_streaming = _after_step_ms(g)
            assert after_streaming > 0.012  # fallback passes and finalize: five launches
            if n == (900, 700):
                assert after > 0.012
        g.close()
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])
