"""The host code that decides whether a cascade's runs may go by strips (sosfilt_api.cpp, on the CPU against the
stand-ins of tests/api_host/): the rows after which a state is forgotten, the cascade's float32 noise, and the rule
that cuts a signal into strips (sosfilt_strip_rule.h)."""
import ctypes
import shutil

import numpy as np
import pytest

from workloads import designs

from .test_api_host import _LIB, KIND_LANE, KIND_TC, _create, _launches, _tune_costs, lib  # noqa: F401  (a fixture)

ROW = 64
SMS = 152  # of the device on which the rule's lines were measured; the stand-in has four


def _fields(lib, sos, tuning=None, n=1 << 22, offset=0):
    """(strips, rows a strip, warm-up rows, by FMAs, products, any tables) of each pass of a run."""
    f = _create(lib, sos, tuning)
    x = np.zeros(n + 8, np.float32)
    at = x.ctypes.data + (-x.ctypes.data) % 16 + 4 * offset
    lib.host_reset()
    assert lib.sos_filter_run(f, at, at, n, None, None, None) == 0
    out, got = (ctypes.c_int * 6)(), []
    for i in range(lib.host_launches()):
        assert lib.host_strip_fields(i, out) == 0
        got.append(tuple(out))
    lib.sos_filter_destroy(f)
    return got


def _transition(sos):
    """One sample of the transposed-direct-form-II cascade under zero input, [2K][2K]."""
    S = 2 * len(sos)
    M = np.zeros((S, S))
    for j in range(S):
        z, v = np.zeros(S), 0.0
        z[j] = 1.0
        for k, (b0, b1, b2, a1, a2) in enumerate(sos):
            y = b0 * v + z[2 * k]
            z[2 * k], z[2 * k + 1] = b1 * v - a1 * y + z[2 * k + 1], b2 * v - a2 * y
            v = y
        M[:, j] = z
    return M


def _resonator(sections, radius):
    return designs.resonator_bank(sections, radius=radius)


def _dc_blocker(radius):
    """A zero at frequency zero and a real pole beside it: quiet however long it remembers."""
    return np.array([[1.0, -1.0, 0.0, -radius, 0.0]])


def _smoother(radius):
    """A one-pole smoother."""
    return np.array([[1.0 - radius, 0.0, 0.0, -radius, 0.0]])


FORGETFUL = [designs.butter_lowpass(2, 0.2), designs.butter_lowpass(16, 0.05), designs.butter_lowpass(8, 0.5),
             _resonator(1, 0.99), _resonator(4, 0.98), _smoother(0.9), np.array([[0.5, 0.2, 0.1, 0.0, 0.0]])]


@pytest.mark.parametrize("i", range(len(FORGETFUL)))
def test_a_state_is_forgotten_after_the_warm_up_and_not_long_before(lib, i):  # noqa: F811
    """After warm_rows rows every entry of the transition, and of every later one, is below 2^-150 (zero in
    float32); at half of them (the rule is careful by a factor in size, not in time) it is not."""
    sos = FORGETFUL[i]
    (strips, _, rows, _, _, tables), = _fields(lib, sos)
    assert tables and strips and 1 <= rows < 4096
    Q = np.linalg.matrix_power(_transition(sos), ROW)
    P = np.linalg.matrix_power(Q, rows)
    for _ in range(64):
        assert np.abs(P).max() < 2.0 ** -150
        P = P @ Q
    if rows > 2:
        assert np.abs(np.linalg.matrix_power(Q, rows // 2)).max() > 2.0 ** -150


@pytest.mark.parametrize("sections,radius", [(1, 0.999), (1, 0.9995), (2, 0.9993), (4, 0.999), (8, 0.999)])
def test_slow_noisy_cascades_keep_the_lookback(lib, sections, radius):  # noqa: F811
    """Narrow resonators amplify float32 rounding by more than 1e-5 once their errors have piled up, which takes
    longer than their first 2048 samples: no strip tables."""
    assert _settled_noise(_resonator(sections, radius)) > 1e-5
    assert _fields(lib, _resonator(sections, radius))[0][0] == 0
    assert _fields(lib, _resonator(sections, radius))[0][5] == 0


@pytest.mark.parametrize("sos", [_resonator(1, 0.9999), _resonator(4, 0.9998), _smoother(0.9999), _dc_blocker(0.99999)])
def test_cascades_that_remember_too_long_are_never_warmed_up(lib, sos):  # noqa: F811
    """Beyond 4096 rows of memory no signal is cut into strips, whatever the noise over a single one."""
    assert _fields(lib, sos)[0][0] == 0


@pytest.mark.parametrize("radius", [0.99, 0.999, 0.9995])
def test_slow_quiet_cascades_still_take_strips(lib, radius):  # noqa: F811
    (strips, _, rows, _, _, _), = _fields(lib, _dc_blocker(radius))
    assert strips == 4 and rows > 0


def test_one_slow_pass_keeps_all_passes_from_strips(lib):  # noqa: F811
    """Nine sections are two passes; a pole that remembers too long, in either, leaves neither a warm-up."""
    slow = _smoother(0.9999)
    for sos in (np.vstack([designs.butter_lowpass(16, 0.1), slow]), np.vstack([slow, designs.butter_lowpass(16, 0.1)])):
        got = _fields(lib, sos)
        assert len(got) == 2 and all(g[0] == 0 for g in got)


def _cut(lib, K, products, odd, tc, n, warm, sms=SMS):
    out = (ctypes.c_int * 4)()
    lib.host_strip_cut.argtypes = [ctypes.c_int] * 4 + [ctypes.c_longlong] + [ctypes.c_int] * 2 + [ctypes.c_void_p]
    return tuple(out) if lib.host_strip_cut(K, products, odd, tc, n, warm, sms, out) else None


@pytest.mark.parametrize("sms", [1, 4, 152, 300])
@pytest.mark.parametrize("K", range(1, 9))
def test_every_cut_covers_the_signal_and_warms_up_in_one_neighbour(lib, K, sms):  # noqa: F811
    """What the kernel relies on, for every section count, mode, alignment, length and warm-up."""
    rng = np.random.default_rng(K)
    taken = 0
    for _ in range(4000):
        products, odd, tc = (int(v) for v in rng.integers(0, 2, 3))
        products &= K > 2
        tc &= not odd
        n, warm = int(2 ** rng.uniform(0, 31)), int(2 ** rng.uniform(-1, 13))
        c = _cut(lib, K, products, odd, tc, n, warm, sms)
        if c is None:
            continue
        taken += 1
        strips, rows, w, fma = c
        n_rows = -(-n // ROW)
        assert 1 <= strips <= min(sms, 256)
        assert (strips - 1) * rows < n_rows <= strips * rows
        assert w == (0 if strips == 1 and n_rows <= 128 else warm) and w <= rows
        assert not (fma and K > 2)
        assert warm > 0 or n_rows <= 128
    assert taken > 400


# (sections, products, x misaligned, against the tensor-core kernel, log2 samples, warm-up rows) and which of the two
# was measured faster; the strips' mode for one and two sections
LINES = [
    ((3, 1, 1, 0, 22, 100), None), ((3, 1, 1, 0, 26, 100), 0),  # order 6 by products, misaligned: 26.6 us against 23.5
    ((5, 0, 1, 0, 21.5, 100), None), ((5, 0, 1, 0, 18, 16), 0),
    ((5, 1, 1, 0, 22, 300), None), ((8, 1, 1, 0, 22, 300), 0),
    ((3, 1, 0, 0, 18, 100), None), ((3, 0, 0, 0, 18, 100), 0), ((3, 1, 0, 0, 22, 100), 0), ((3, 1, 0, 1, 18, 100), 0),
    ((4, 1, 0, 0, 18, 200), None), ((4, 1, 0, 0, 18, 100), 0), ((5, 1, 0, 0, 17, 100), None), ((8, 1, 0, 0, 17, 100), 0),
    ((1, 0, 0, 1, 28, 16000), None), ((1, 0, 0, 1, 28, 11000), 0), ((2, 0, 0, 0, 28, 19000), 0), ((2, 0, 0, 1, 28, 19000), None),
    ((3, 0, 0, 1, 28, 27000), None), ((3, 0, 0, 0, 28, 27000), 0), ((8, 1, 0, 1, 28, 27000), 0),
    ((1, 0, 0, 0, 20, 4), 1), ((1, 0, 0, 0, 24, 1600), 1), ((1, 0, 0, 0, 26, 100), 0), ((1, 0, 1, 0, 28, 100), 1),
    ((2, 0, 0, 0, 26, 100), 1), ((2, 0, 0, 0, 28, 100), 0), ((2, 0, 1, 0, 24, 1600), 1), ((1, 0, 1, 0, 25, 3300), None),
    ((2, 0, 0, 0, 15, 256), None), ((2, 0, 0, 0, 20, 256), 1), ((1, 0, 0, 0, 12, 0), 1), ((3, 0, 0, 0, 12, 4), None),
]


@pytest.mark.parametrize("case,want", LINES)
def test_the_faster_way_is_taken(lib, case, want):  # noqa: F811
    K, products, odd, tc, log2n, warm = case
    c = _cut(lib, K, products, odd, tc, int(2 ** log2n), warm)
    assert (None if c is None else c[3]) == want


def test_runs_are_cut_by_the_rule_and_the_alignment(lib):  # noqa: F811
    """The cut that a launch receives: by products or not as the filter's noise says, by FMAs where x is misaligned
    (one or two sections), and none at N = 32, with ten groups or with cyclic reduction."""
    o2, o16 = designs.butter_lowpass(2, 0.2), designs.butter_lowpass(16, 0.05)
    assert _fields(lib, o2)[0][3] == 0 and _fields(lib, o2, offset=1)[0][3] == 1
    assert _fields(lib, o16)[0][4] == 1 and _fields(lib, designs.butter_lowpass(8, 0.5))[0][4] == 0
    assert _fields(lib, o16)[0][:2] == (4, 16384)
    for tuning in ({"N": 32}, {"groups_per_cta": 10}):
        assert _fields(lib, o16, tuning)[0][0] == 0


def _settled_noise(sos):
    """Float32 direct-form-I error over the output in 2-norms, long after the start (numpy, one rounding per
    operation)."""
    rng = np.random.default_rng(5)
    n, skip = 60000, 30000
    x = rng.standard_normal(n).astype(np.float32)
    b0 = float(np.prod(sos[:, 0]))
    v, w = x * np.float32(b0), x.astype(np.float64) * b0
    for s in sos:
        q64 = np.array([s[1] / s[0], s[2] / s[0], -s[3], -s[4]])
        q = q64.astype(np.float32)
        y, z = np.zeros(n, np.float32), np.zeros(n)
        x1 = x2 = y1 = y2 = np.float32(0)
        X1 = X2 = Y1 = Y2 = 0.0
        for i in range(n):
            y0 = v[i] + q[0] * x1 + q[1] * x2 + q[2] * y1 + q[3] * y2
            x2, x1, y2, y1 = x1, v[i], y1, y0
            y[i] = y0
            Z = w[i] + q64[0] * X1 + q64[1] * X2 + q64[2] * Y1 + q64[3] * Y2
            X2, X1, Y2, Y1 = X1, w[i], Y1, Z
            z[i] = Z
        v, w = y, z
    return float(np.linalg.norm(v[skip:] - w[skip:]) / np.linalg.norm(w[skip:]))


def test_the_autotuner_keeps_a_choice_for_runs_by_strips_and_one_for_the_others(lib, tmp_path):  # noqa: F811
    """Where strips make the PH solver as fast as the tensor-core one, the choice for runs that keep the lookback
    is still the tensor cores'.  On a copy of the library, whose tuning no other test sees."""
    shared, path = lib, tmp_path / "libapi_host.so"
    shutil.copy(_LIB, path)
    lib = ctypes.CDLL(str(path))
    for name in ("sos_filter_create", "sos_filter_destroy", "sos_filter_run", "host_launch"):
        getattr(lib, name).argtypes = getattr(shared, name).argtypes
        getattr(lib, name).restype = getattr(shared, name).restype
    lib.sos_autotune.argtypes = [ctypes.c_int, ctypes.c_void_p]
    lib.host_set_strip_cost.argtypes = [ctypes.c_int, ctypes.c_float]
    lib.host_set_cost.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_float]
    K, n = 8, 1 << 20

    def kinds(sos, n=n, offset=0):
        f = _create(lib, sos)
        x = np.zeros(n + 8, np.float32)
        at = x.ctypes.data + (-x.ctypes.data) % 16 + 4 * offset
        lib.host_reset()
        assert lib.sos_filter_run(f, at, at, n, None, None, None) == 0
        got = [(l["kind"], l["N"]) for l in _launches(lib)]
        lib.sos_filter_destroy(f)
        return got

    def tune():
        lib.host_set_light(1)
        try:
            assert lib.sos_autotune(20, None) == 0
        finally:
            lib.host_set_light(0)
            lib.host_reset()

    _tune_costs(lib, lambda K: (KIND_TC, 64))       # lookback: the tensor cores are the fastest
    for k in range(1, 9):
        lib.host_set_strip_cost(k, 0.5)             # strips: both solvers are equal, the first is kept
    tune()
    assert kinds(designs.butter_lowpass(2 * K, 0.2)) == [(KIND_LANE, 64)]
    assert kinds(_resonator(K, 0.999)) == [(KIND_TC, 64)]                   # too noisy
    assert kinds(_resonator(K, 0.99999)) == [(KIND_TC, 64)]                 # remembers too long
    assert kinds(designs.butter_lowpass(2 * K, 0.2), n=60000) == [(KIND_TC, 64)]  # too short
