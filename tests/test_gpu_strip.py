"""The strip kernel (one strip of the signal per thread block, its incoming state from a warm-up) against
the float64 oracle at the sizes where it can go wrong, and against the lookback kernel.

Bounds: the suite's stated ones (1e-4 of the peak up to pole radius 0.99, 2e-3 beyond).
"""
import numpy as np
import pytest

import oracle
import workloads
from workloads import designs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROW, UNIT, SMS = 64, 8192, 152  # samples of a row and of a unit of 128 rows; strips of a long signal


@pytest.fixture(scope="module")
def dev():
    from paper_2607_23763_gb300 import build
    build.build()
    return torch.device("cuda:0")


def _filter(sos, **kw):
    from paper_2607_23763_gb300 import SosFilter
    return SosFilter(sos, **kw)


# the edges of rows, units, strips of half a unit, strips of one unit and of several, one strip per SM
SIZES = [1, ROW - 1, ROW, ROW + 1, UNIT - 1, UNIT, UNIT + 1, UNIT + UNIT // 2, 3 * UNIT + ROW, SMS * UNIT // 2 - 1,
         SMS * UNIT // 2 + 1, SMS * (UNIT - 10 * ROW) + 3, SMS * UNIT + 1, 3 * SMS * UNIT + 77]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("order,cutoff,solver", [(2, 0.2, 0), (4, 0.3, 0), (6, 0.1, 0), (6, 0.4, 0), (10, 0.1, 0),
                                                 (12, 0.4, 0), (16, 0.05, 0), (16, 0.4, 0), (16, 0.4, 4), (14, 0.1, 0)])
def test_sizes_alignment_and_state(dev, order, cutoff, solver, n):
    """Every size with an initial and a final state, aligned, at odd offsets of input and output, in place
    with the final state over the initial one; all match the oracle, and the in-place result is the
    out-of-place one bit for bit."""
    sos = designs.butter_lowpass(order, cutoff)
    K = order // 2
    x = workloads.normal_f32(7 + order, n)
    zi = (0.01 * np.random.default_rng(n).standard_normal((K, 2))).astype(np.float32)
    ref, zref = oracle.sosfilt(sos, x, zi=zi.astype(np.float64), return_state=True)
    f = _filter(sos, tuning={"solver": solver})
    first = None
    for ox, oy in [(0, 0), (1, 2), (3, 0), (0, 1)]:
        xd = torch.empty(n + ox, device=dev)[ox:]
        xd.copy_(torch.from_numpy(x))
        y = torch.full((n + oy + 8,), 7.0, device=dev)
        z, zf = torch.from_numpy(zi).to(dev), torch.empty(K, 2, device=dev)
        f.run(xd, y[oy:oy + n], zi=z, zf=zf)
        assert f.sync_status() == 0
        got = y.cpu().numpy()
        assert np.all(got[:oy] == 7.0) and np.all(got[oy + n:] == 7.0)  # nothing written outside
        got = got[oy:oy + n]
        assert oracle.rel_err(got, ref) < 1e-4
        assert np.abs(zf.cpu().numpy() - zref).max() < 1e-4 * np.abs(zref).max()
        if first is None:
            first = got
    xd, z = torch.from_numpy(x).to(dev), torch.from_numpy(zi).to(dev)
    f.run(xd, xd, zi=z, zf=z)
    assert f.sync_status() == 0
    assert np.array_equal(xd.cpu().numpy(), first)
    assert np.abs(z.cpu().numpy() - zref).max() < 1e-4 * np.abs(zref).max()
    f.close()


@pytest.mark.parametrize("order", [2, 8, 16])
@pytest.mark.parametrize("n", [40000, 1 << 21, (1 << 23) + 5])
def test_matches_the_lookback_kernel(dev, order, n):
    """The same signal through the lookback kernel (10 groups per tile, which never takes strips)."""
    sos = designs.butter_lowpass(order, 0.1)
    x = torch.randn(n, device=dev, generator=torch.Generator(device=dev).manual_seed(n))
    a, b = _filter(sos), _filter(sos, tuning={"solver": 2, "groups_per_cta": 10})
    za, zb = torch.empty(order // 2, 2, device=dev), torch.empty(order // 2, 2, device=dev)
    ya, yb = a.run(x, zf=za), b.run(x, zf=zb)
    assert a.sync_status() == 0 and b.sync_status() == 0
    assert float((ya - yb).abs().max()) < 2e-5 * float(yb.abs().max())
    assert float((za - zb).abs().max()) < 2e-5 * float(zb.abs().max())
    a.close()
    b.close()


@pytest.mark.parametrize("n", [2048 * ROW, (1 << 20) + 77, 3 * SMS * UNIT + ROW - 1])
@pytest.mark.parametrize("zero_b0", [False, True])
@pytest.mark.parametrize("order", [6, 8, 10, 12, 16])
def test_recurrences_of_a_quiet_cascade(dev, order, zero_b0, n):
    """Cascades of little float32 noise (below 5e-7 of the output) are done by the recurrences, even counts of
    sections two at a time, with every section's b0 factored out and with a b0 of zero (the general class).
    Bound: ten times that noise."""
    sos = designs.butter_lowpass(order, 0.5)
    if zero_b0:
        sos[1] = [0.0, 1.0, 0.5, sos[1, 3], sos[1, 4]]
    x = workloads.normal_f32(order, n)
    zi = (0.01 * np.random.default_rng(n).standard_normal((order // 2, 2))).astype(np.float32)
    ref, zref = oracle.sosfilt(sos, x, zi=zi.astype(np.float64), return_state=True)
    f = _filter(sos)
    zf = torch.empty(order // 2, 2, device=dev)
    y = f.run(torch.from_numpy(x).to(dev), zi=torch.from_numpy(zi).to(dev), zf=zf)
    assert f.sync_status() == 0
    assert oracle.rel_err(y.cpu().numpy(), ref) < 5e-6
    assert np.abs(zf.cpu().numpy() - zref).max() < 5e-6 * max(np.abs(zref).max(), np.abs(ref).max())
    f.close()


@pytest.mark.parametrize("radius", [0.9, 0.999, 0.99999])
def test_long_memory(dev, radius):
    """Cascades that remember for a part of a strip, for several units, and for longer than a strip (those
    run the lookback kernel), on a decaying impulse whose tail crosses every strip."""
    sos = designs.resonator_bank(4, radius=radius)
    n = 1 << 21
    x = np.zeros(n, np.float32)
    x[100] = 1.0
    x[n // 2:] = workloads.normal_f32(3, n - n // 2)
    f = _filter(sos)
    y = f.run(torch.from_numpy(x).to(dev))
    assert f.sync_status() == 0
    ref = oracle.sosfilt(sos, x)
    got = y.cpu().numpy()
    assert oracle.rel_err(got, ref) < 2e-3
    assert oracle.rel_err(got[:n // 2], ref[:n // 2]) < 2e-3
    f.close()


@pytest.mark.parametrize("order", [4, 16])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("n,at", [(5000, 4000), (1 << 20, 70001), (1 << 20, (1 << 20) - 2), (3 * SMS * UNIT, 9 * UNIT)])
def test_a_value_that_is_not_finite_spreads_to_the_end(dev, order, bad, n, at):
    """What follows a NaN or an infinity in a recurrence is not finite, to the signal's end and in the final
    state, also in the strips that never saw it; what comes before is untouched.  The next run is clean."""
    sos = designs.butter_lowpass(order, 0.2)
    x = workloads.normal_f32(5, n)
    ref, zref = oracle.sosfilt(sos, x, return_state=True)
    f = _filter(sos)
    xd = torch.from_numpy(x).to(dev)
    xb = xd.clone()
    xb[at] = bad
    zf = torch.empty(order // 2, 2, device=dev)
    y = f.run(xb, zf=zf).cpu().numpy()
    assert f.sync_status() == 0
    assert oracle.rel_err(y[:at], ref[:at]) < 1e-4
    assert not np.isfinite(y[at:]).any()
    assert not np.isfinite(zf.cpu().numpy()).any()
    y = f.run(xd, zf=zf).cpu().numpy()
    assert oracle.rel_err(y, ref) < 1e-4
    assert np.abs(zf.cpu().numpy() - zref).max() < 1e-4 * np.abs(zref).max()
    f.close()


def test_streams_and_filters_at_once(dev):
    """Eight filters on eight streams, in place, overlapping on the device: each as if alone."""
    sos = designs.butter_lowpass(8, 0.1)
    n = (1 << 20) + 3
    xs = [torch.randn(n, device=dev) for _ in range(8)]
    fs = [_filter(sos) for _ in xs]
    want = [f.run(x) for f, x in zip(fs, xs)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xs]
    for _ in range(3):
        ys = [x.clone() for x in xs]
        torch.cuda.synchronize()
        for f, y, s in zip(fs, ys, streams):
            f.run(y, y, stream=s)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(ys, want))
    assert all(f.sync_status() == 0 for f in fs)
    for f in fs:
        f.close()


def _long(dev, order):
    """Samples of a signal whose strips take TMA copies: 512 rows and more, and at one and two sections more than
    what is done without the tensor cores."""
    rows = {2: 3400, 4: 12300}.get(order, 640)
    return rows * torch.cuda.get_device_properties(dev).multi_processor_count * ROW


# what forms the outputs: recurrences of one and two sections, in pairs, one at a time; products (both solvers)
LONG = [(2, 0.2, 0), (4, 0.3, 0), (8, 0.5, 0), (12, 0.5, 0), (6, 0.5, 0), (16, 0.05, 0), (8, 0.1, 0), (16, 0.4, 4)]


@pytest.mark.parametrize("tail", [0, 77])
@pytest.mark.parametrize("order,cutoff,solver", LONG)
def test_strips_by_tma(dev, order, cutoff, solver, tail):
    """Strips long enough for TMA copies, with an initial and a final state: against the oracle, and the run in
    place, with the final state over the initial one, bit for bit the same."""
    sos = designs.butter_lowpass(order, cutoff)
    n = _long(dev, order) + tail
    x = workloads.normal_f32(11 + order, n)
    zi = (0.01 * np.random.default_rng(order).standard_normal((order // 2, 2))).astype(np.float32)
    ref, zref = oracle.sosfilt(sos, x, zi=zi.astype(np.float64), return_state=True)
    f = _filter(sos, tuning={"solver": solver})
    xd, z, zf = torch.from_numpy(x).to(dev), torch.from_numpy(zi).to(dev), torch.empty(order // 2, 2, device=dev)
    y = torch.full((n + 8,), 7.0, device=dev)
    f.run(xd, y[:n], zi=z, zf=zf)
    assert f.sync_status() == 0
    assert bool((y[n:] == 7.0).all())
    assert oracle.rel_err(y[:n].cpu().numpy(), ref) < 1e-4
    assert np.abs(zf.cpu().numpy() - zref).max() < 1e-4 * np.abs(zref).max()
    f.run(xd, xd, zi=z, zf=z)
    assert f.sync_status() == 0
    assert torch.equal(xd, y[:n]) and torch.equal(z, zf)
    f.close()


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("bad", [float("nan"), float("-inf")])
@pytest.mark.parametrize("order,cutoff", [(2, 0.2), (8, 0.5), (16, 0.05)])
@pytest.mark.parametrize("long", [False, True])
def test_values_that_are_not_finite_in_every_mode(dev, order, cutoff, bad, in_place, long):
    """The same for each way of forming the outputs (order 16 at 0.05: products, whose rows with such samples are
    done again), staged by TMA and by 16-byte copies, in place too."""
    sos = designs.butter_lowpass(order, cutoff)
    n = _long(dev, order) + 77 if long else (1 << 20) + 77
    at = n // 3 + 37
    x = workloads.normal_f32(6, n)
    ref = oracle.sosfilt(sos, x)
    f = _filter(sos)
    xb = torch.from_numpy(x).to(dev)
    xb[at] = bad
    zf = torch.empty(order // 2, 2, device=dev)
    y = f.run(xb, xb if in_place else None, zf=zf).cpu().numpy()
    assert f.sync_status() == 0
    assert oracle.rel_err(y[:at], ref[:at]) < 1e-4
    assert not np.isfinite(y[at:]).any()
    assert not np.isfinite(zf.cpu().numpy()).any()
    f.close()


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("budget", [1, 3000, 30000])
@pytest.mark.parametrize("order,cutoff", [(2, 0.2), (8, 0.5), (16, 0.05)])
def test_expired_waits_of_strips_by_tma(dev, order, cutoff, budget, in_place):
    """A wait that gives up while TMA copies and products are in flight (their own waits have a limit of their
    own): the run reports SOS_ETIMEOUT, its workspace is as it was, and the next run, on the same block of
    memory and the same SMs, is right.  With the longer budgets a run may also end in time."""
    sos = designs.butter_lowpass(order, cutoff)
    n = _long(dev, order) + 77
    x = torch.randn(n, device=dev, generator=torch.Generator(device=dev).manual_seed(order))
    good = _filter(sos)
    want = good.run(x)
    assert good.sync_status() == 0
    f = _filter(sos, tuning={"spin_budget_cycles": budget})
    for _ in range(3):
        b = x.clone()
        y = f.run(b, b if in_place else None)
        status = f.sync_status()
        assert status == -4 or (budget > 1 and status == 0)
        if status == 0:
            assert torch.equal(y, want)
        assert torch.equal(good.run(x), want) and good.sync_status() == 0
    f.close()
    good.close()


@pytest.mark.parametrize("ox,oy", [(1, 1), (0, 0), (3, 0), (0, 2)])
@pytest.mark.parametrize("rows", [300, 1300])
@pytest.mark.parametrize("order", [2, 4])
def test_strips_of_many_units_by_fmas(dev, order, rows, ox, oy):
    """One and two sections without the tensor cores, strips of several units: misaligned signals of any length and
    aligned ones of up to a few thousand rows a strip, with states, in place too."""
    sos = designs.butter_lowpass(order, 0.05)
    n = rows * torch.cuda.get_device_properties(dev).multi_processor_count * ROW + 77
    x = workloads.normal_f32(21 + order, n)
    zi = (0.01 * np.random.default_rng(order).standard_normal((order // 2, 2))).astype(np.float32)
    ref, zref = oracle.sosfilt(sos, x, zi=zi.astype(np.float64), return_state=True)
    f = _filter(sos)
    xd = torch.empty(n + ox, device=dev)[ox:]
    xd.copy_(torch.from_numpy(x))
    y = torch.full((n + oy + 8,), 7.0, device=dev)
    z, zf = torch.from_numpy(zi).to(dev), torch.empty(order // 2, 2, device=dev)
    f.run(xd, y[oy:oy + n], zi=z, zf=zf)
    assert f.sync_status() == 0
    assert bool((y[:oy] == 7.0).all()) and bool((y[oy + n:] == 7.0).all())
    assert oracle.rel_err(y[oy:oy + n].cpu().numpy(), ref) < 1e-4
    assert np.abs(zf.cpu().numpy() - zref).max() < 1e-4 * np.abs(zref).max()
    f.run(xd, xd, zi=z, zf=z)
    assert f.sync_status() == 0
    assert torch.equal(xd, y[oy:oy + n]) and torch.equal(z, zf)
    f.close()


@pytest.mark.parametrize("order,cutoff", [(2, 0.2), (4, 0.1), (6, 0.5), (6, 0.1), (8, 0.1), (10, 0.1), (12, 0.05), (16, 0.05)])
@pytest.mark.parametrize("n", [1 << 17, (1 << 18) + 5, 1 << 20, 3 << 20, 6 << 20])
def test_both_ways_agree_where_the_rule_changes(dev, order, cutoff, n):
    """Lengths around the lines between strips and lookback, aligned, misaligned and with the tensor-core solver: each
    against the lookback kernel of ten groups a tile, which never takes strips."""
    sos = designs.butter_lowpass(order, cutoff)
    x = torch.randn(n + 4, device=dev, generator=torch.Generator(device=dev).manual_seed(n + order))
    b = _filter(sos, tuning={"solver": 2, "groups_per_cta": 10})
    for solver in (0, 4):
        a = _filter(sos, tuning={"solver": solver})
        for o in (0, 1, 2):
            za, zb = torch.empty(order // 2, 2, device=dev), torch.empty(order // 2, 2, device=dev)
            ya, yb = a.run(x[o:o + n], zf=za), b.run(x[o:o + n], zf=zb)
            assert a.sync_status() == 0 and b.sync_status() == 0
            assert float((ya - yb).abs().max()) < 2e-5 * float(yb.abs().max())
            assert float((za - zb).abs().max()) < 2e-5 * float(zb.abs().max())
        a.close()
    b.close()


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("long", [False, True])
@pytest.mark.parametrize("order,cutoff,solver", [(2, 0.2, 0), (4, 0.3, 0), (8, 0.5, 0), (6, 0.5, 0), (16, 0.05, 0), (8, 0.1, 4)])
def test_samples_next_to_the_largest_float32(dev, order, cutoff, solver, long, in_place):
    """Finite outputs where the lookback kernel's are, though such samples round to an infinite TF32 value; in own
    rows and in the rows that warm the next strip up."""
    sos = designs.butter_lowpass(order, cutoff)
    n = _long(dev, order) + 77 if long else (1 << 20) + 77
    x = 1e36 * torch.randn(n, device=dev, generator=torch.Generator(device=dev).manual_seed(order))
    x[5] = -3.4028234e38
    x[20011::50021] = 3.4028234e38
    x[-3] = 3.4028e38
    f, g = _filter(sos, tuning={"solver": solver}), _filter(sos, tuning={"solver": 2, "groups_per_cta": 10})
    zf, zg = torch.empty(order // 2, 2, device=dev), torch.empty(order // 2, 2, device=dev)
    want = g.run(x, zf=zg)
    y = f.run(x, x if in_place else None, zf=zf)
    assert f.sync_status() == 0 and g.sync_status() == 0
    assert bool(torch.isfinite(want).all()) and bool(torch.isfinite(zg).all())
    assert float((y - want).abs().max()) < 2e-5 * float(want.abs().max())
    assert float((zf - zg).abs().max()) < 2e-5 * float(zg.abs().max())
    f.close()
    g.close()
