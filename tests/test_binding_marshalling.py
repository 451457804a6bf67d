"""The binding's two ways of marshalling a call: the native module (csrc/py/native.cpp) and the Python one that stands in
where it was not built.  What they refuse, what they accept, and (on a GPU) that both filter alike."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2607_23763_gb300 import _binding  # noqa: E402
from workloads import designs  # noqa: E402


class _Recorder:
    """In the native module's place: keeps what it was called with."""

    def run_batch(self, *args):
        self.args = args
        return 0


class _Filter:
    _hv = 1


def test_any_iterable_may_hold_the_outputs_of_a_batch(monkeypatch):
    """Outputs, filters and states that come from a generator are taken as they were before the native path."""
    rec = _Recorder()
    monkeypatch.setattr(_binding, "_native", rec)
    monkeypatch.setitem(_binding._fn, "sos_filter_run_batch_ex", 0)
    monkeypatch.setattr(_binding, "load_library", lambda path=None: None)
    xs = [torch.zeros(4), torch.zeros(5)]
    ys = [torch.empty(4), torch.empty(5)]
    out = _binding.run_batch((_Filter() for _ in xs), xs, (y for y in ys), (None for _ in xs), iter([None, None]))
    assert all(a is b for a, b in zip(out, ys)) and len(out) == 2
    assert rec.args[2] is xs and len(rec.args[1]) == len(rec.args[3]) == len(rec.args[4]) == len(rec.args[5]) == 2


def _native():
    try:
        from paper_2607_23763_gb300 import _native as mod
    except ImportError:
        pytest.skip("the native module is not built here")
    return mod


BAD = [torch.zeros(4), torch.zeros(4, dtype=torch.float64), np.zeros(4, np.float32), None, 3]


@pytest.mark.parametrize("i", range(len(BAD)))
def test_both_ways_refuse_what_is_no_float32_cuda_tensor(i):
    nat = _native()
    with pytest.raises(TypeError, match="x must be a contiguous float32 CUDA tensor"):
        nat.run(0, 0, BAD[i], BAD[i], None, None, None)
    with pytest.raises(TypeError, match="x must be a contiguous float32 CUDA tensor"):
        nat.run_batch(0, [_Filter()], [BAD[i]], [BAD[i]], None, None, None)
    with pytest.raises(TypeError, match="x must be a contiguous float32 CUDA tensor"):
        _binding._dptr(BAD[i], "x")


def test_the_native_way_refuses_lists_of_other_lengths():
    nat = _native()
    with pytest.raises(ValueError):
        nat.run_batch(0, [], [torch.zeros(4)], [torch.zeros(4)], None, None, None)
    with pytest.raises(AttributeError):
        nat.run_batch(0, [1], [torch.zeros(4)], [torch.zeros(4)], None, None, None)
    with pytest.raises(TypeError):
        nat.run(0, 0)


@pytest.mark.gpu
def test_both_ways_filter_alike(monkeypatch):
    from paper_2607_23763_gb300 import SosFilter, build, run_batch
    build.build()
    assert _binding._native_module(), "the native module was not built on this machine"
    dev = torch.device("cuda:0")
    fs = [SosFilter(designs.butter_lowpass(o, 0.1)) for o in (2, 8, 16)]
    xs = [torch.randn(70001 + i, device=dev) for i in range(3)]
    zs = [0.01 * torch.randn(f.K, 2, device=dev) for f in fs]
    side = torch.cuda.Stream()

    def all_ways():
        out = []
        for stream in (None, side):
            torch.cuda.synchronize()
            zf = [torch.empty_like(z) for z in zs]
            ys = [torch.empty_like(x) for x in xs]
            for f, x, y, z, w in zip(fs, xs, ys, zs, zf):
                f.run(x, y, zi=z, zf=w, stream=stream)
            yn = [torch.empty_like(x) for x in xs]
            for f, x, y in zip(fs, xs, yn):
                f.run_noalloc(x, y, stream=stream)
                torch.cuda.synchronize()
            zb = [torch.empty_like(z) for z in zs]
            yb = [torch.empty_like(x) for x in xs]
            run_batch(fs, xs, yb, [zs[0], None, zs[2]], [zb[0], zb[1], None], stream=stream)
            torch.cuda.synchronize()
            out += ys + zf + yn + yb + zb[:2]
        return out

    native = all_ways()
    with pytest.raises(TypeError):
        fs[0].run(torch.zeros(8, device=dev)[::2], torch.zeros(4, device=dev))
    monkeypatch.setattr(_binding, "_native", False)
    python = all_ways()
    assert all(torch.equal(a, b) for a, b in zip(native, python))
    with pytest.raises(TypeError):
        fs[0].run(torch.zeros(8, device=dev)[::2], torch.zeros(4, device=dev))
    for f in fs:
        f.close()
