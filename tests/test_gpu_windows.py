"""The windows of a launch run side by side (their replicas start from their own snapshots). One bd_step over many windows
equals the same steps taken a window (or less) at a time, bit for bit: the noise is keyed by the step, not by the launch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2206_05851_gb300 import bdra, inputs as I  # noqa: E402


def _fene(n, r, flow=I.FLOW_SHEAR):
    return I.Chain(n_beads=n, n_replicas=r, spring=I.SPRING_FENE, flow=flow, b=40.0, rate=0.5, f_c=0.5 * 40 ** 0.5, k0=1e-3, dx=0.2)


def _globule(n, r, hi):
    ch = I.collapsed_chain(r, n_beads=n)
    ch.hi_a = 1.0 if hi else 0.0
    return ch


# few units a launch (each window its own CTAs), one unit, uneven variants side by side, more units than warps, RPY (both kernels)
BATCHES = {
    "one": [_fene(20, 16)],
    "dumbbell": [_fene(2, 1)],
    "uneven": [_fene(n, r) for n, r in ((3, 5), (17, 8), (50, 33), (61, 2), (100, 7), (230, 3), (500, 2))],
    "many": [_fene(50, 24) for _ in range(160)],
    "collapsed": [_globule(n, r, False) for n, r in ((8, 3), (50, 7), (120, 2))],
    "rpy": [_globule(n, r, True) for n, r in ((7, 2), (50, 3), (60, 2))],
}


def _run(chains, calls, S, windows, prec, flags):
    wl = I.custom(chains, 4e-5 if chains[0].spring == I.SPRING_HARMONIC else 1e-3, S, S * windows)
    ctx = bdra.Context(chains, wl.dt, S, 11, I.initial_positions(wl, seed=5), precision=prec, max_windows=windows,
                       thr_mask=7, bell_mask=7, flags=flags, stream=torch.cuda.current_stream().cuda_stream)
    for n in calls:
        ctx.step(n)
    W = sum(calls) // S
    out = [ctx.replica_average(w) for w in range(W)] + [ctx.time_average(w) for w in range(W)]
    out.append(ctx.positions(True))
    if calls[0] % S == 0:      # a call that ends inside a window adds its part of the hazard to the total there: another order of sums
        out += ctx.kinetics()
    if flags & bdra.BD_FLAG_CONFORMATION:
        out += [a for w in range(W) for a in ctx.conformation(w)]
    assert ctx.info().windows_done == W
    ctx.close()
    return out


@pytest.mark.parametrize("conf", [False, True])
@pytest.mark.parametrize("prec", [bdra.BD_PREC_FP32, bdra.BD_PREC_FP64])
@pytest.mark.parametrize("batch", sorted(BATCHES))
def test_windows_side_by_side_equal_one_at_a_time(batch, prec, conf):
    chains = BATCHES[batch]
    if batch == "many" and prec == bdra.BD_PREC_FP64:
        chains = chains[:24]
    S, W = (7, 9) if batch != "many" else (5, 4)
    flags = bdra.BD_FLAG_CONFORMATION if conf else 0
    one = _run(chains, [S] * W + [3], S, W + 1, prec, flags)
    for calls in ([S * W + 3], [2, S * W + 1]):                # from a window start; from inside a window
        # RPY positions are rebuilt from the stored bonds at the start of every call, so only equal calls give equal bits there
        if batch == "rpy" and calls != [S * W + 3]:
            continue
        got = _run(chains, calls, S, W + 1, prec, flags)
        want = one if calls[0] % S == 0 else one[:2 * W + 1] + one[2 * W + 4:]
        for a, b in zip(want, got, strict=True):
            if batch == "rpy":
                tol = 1e-3 if prec == bdra.BD_PREC_FP32 else 1e-10
                assert np.abs(a - b).max() <= tol * max(1.0, np.abs(a).max())
            else:
                np.testing.assert_array_equal(a, b)


def test_float64_noise_tables_outlive_the_context_that_filled_them():
    """The float64 contexts of a device share their noise tables: one closed early leaves the others' results unchanged, and
    one opened after all were closed fills them again."""
    chains = BATCHES["uneven"][:4]
    want = _run(chains, [20], 10, 2, bdra.BD_PREC_FP64, 0)
    wl = I.custom(chains, 1e-3, 10, 20)

    def make():
        return bdra.Context(chains, wl.dt, 10, 11, I.initial_positions(wl, seed=5), precision=bdra.BD_PREC_FP64, max_windows=2,
                            stream=torch.cuda.current_stream().cuda_stream)

    a, b = make(), make()
    a.step(5)
    a.close()
    b.step(20)
    np.testing.assert_array_equal(b.replica_average(1), want[1])
    b.close()
    c = make()
    c.step(20)
    np.testing.assert_array_equal(c.positions(True), want[4])
    c.close()


@pytest.mark.parametrize("batch", ["one", "dumbbell", "uneven", "collapsed"])
def test_small_batches_take_the_shortest_step(batch):
    """A batch that leaves every warp an SM sub-partition of its own runs on the tiles with the shortest step that fit its
    chains; float32 results do not depend on the tile."""
    chains = BATCHES[batch]
    wl = I.custom(chains, 4e-5 if batch == "collapsed" else 1e-3, 6, 12)
    got = []
    for hints in ({}, {"lanes_hint": 16, "layout_hint": 1}):
        ctx = bdra.Context(chains, wl.dt, 6, 11, I.initial_positions(wl, seed=5), max_windows=2,
                           stream=torch.cuda.current_stream().cuda_stream, **hints)
        if not hints:
            for c, v in zip(chains, ctx.plan()[0]):
                tiles = (202, 204, 205, 207, 216) if batch == "collapsed" else (4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16)
                assert v == next(t for t in tiles if -(-c.n_beads // (t % 100)) <= 32)
        ctx.step(12)
        got.append((ctx.replica_average(1), ctx.positions(True)))
        ctx.close()
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("beads", [(2,), (200, 57), (200, 58), (200, 59), (500, 500, 500, 500, 53), (500, 500, 500, 500, 54)])
def test_event_list_and_survival_at_the_edges_of_the_one_cta_form(beads):
    """M = 1, 255, 256, 257 and 2048 springs (one CTA), 2049 (block counts): the list equals the first-event arrays in its
    documented order, the log-survival the hazards' sums."""
    chains = [_fene(n, 3) for n in beads]
    wl = I.custom(chains, 5e-3, 10, 60)
    ctx = bdra.Context(chains, wl.dt, 10, 3, I.initial_positions(wl, seed=9), max_windows=6, thr_mask=7, bell_mask=7,
                       stream=torch.cuda.current_stream().cuda_stream)
    ctx.step(60)
    ev, surv = ctx.events()
    dev_list = torch.zeros((6 * ctx.M, 24), dtype=torch.uint8, device="cuda")
    dev_surv = torch.zeros((len(chains), 3), dtype=torch.float64, device="cuda")
    n = bdra.bd_detect_events(ctx.ptr, dev_list, 6 * ctx.M, dev_surv)
    haz, thr, bell = ctx.kinetics()
    ctx.close()
    want, at = [], 0
    for c, ch in enumerate(chains):
        for i in range(ch.n_beads - 1):
            for q in range(3):
                want += [(c, i, q, k, int(a[q, at + i])) for k, a in ((0, thr), (1, bell)) if a[q, at + i] >= 0]
        at += ch.n_beads - 1
    assert [tuple(int(x) for x in e) for e in ev] == want and n == len(want)
    np.testing.assert_array_equal(dev_list.cpu().numpy()[:n].reshape(-1).view(bdra.EVENT_DTYPE), ev)
    assert len(beads) == 1 or want
    at = 0
    for c, ch in enumerate(chains):
        s = -haz[:, at:at + ch.n_beads - 1].sum(axis=1)
        np.testing.assert_allclose(surv[c], s, rtol=ch.n_beads * 2.0 ** -52)     # another order of the sum
        at += ch.n_beads - 1
    np.testing.assert_array_equal(dev_surv.cpu().numpy(), surv)


@pytest.mark.parametrize("prec", [bdra.BD_PREC_FP32, bdra.BD_PREC_FP64])
@pytest.mark.parametrize("batch", sorted(BATCHES))
def test_overlapped_schedule_equals_parents_first(batch, prec):
    """Parents beside replicas (small batches, chains with hydrodynamic interaction) and parents before replicas (while the two
    are timed) give the same bits on equal calls: over several windows, one window, a start and an end inside a window."""
    chains = BATCHES[batch]
    if batch == "many" and prec == bdra.BD_PREC_FP64:
        chains = chains[:24]
    S, W = 6, 8
    wl = I.custom(chains, 4e-5 if chains[0].spring == I.SPRING_HARMONIC else 1e-3, S, S * W)
    got = []
    for timing in (False, True):
        ctx = bdra.Context(chains, wl.dt, S, 11, I.initial_positions(wl, seed=5), precision=prec, max_windows=W,
                           thr_mask=7, bell_mask=7, stream=torch.cuda.current_stream().cuda_stream)
        bdra.bd_enable_timing(ctx.ptr, timing)
        for n in (3 * S, S, 2, S + 3, S + 1):
            ctx.step(n)
        got.append([ctx.replica_average(w) for w in range(7)] + [ctx.time_average(w) for w in range(7)] +
                   [ctx.positions(True), *ctx.kinetics(), np.array(ctx.info().overextensions)])
        ctx.close()
    for a, b in zip(*got, strict=True):
        np.testing.assert_array_equal(a, b)
