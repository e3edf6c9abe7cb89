"""The binding's C module against the ctypes functions it stands in for: the
same results and refusals for every form of argument, on calls that the library
rejects on the host (no GPU needed)."""

import ctypes

import numpy as np
import pytest

try:
    from paper_1601_04033_gb300 import fasgd as f
except ImportError:                      # pragma: no cover - the library is not built
    pytest.skip("libfasgd.so is not built", allow_module_level=True)
if f._binding is None:
    pytest.skip("built without Python's headers", allow_module_level=True)

NAMES = f._binding.install({n: getattr(f, n) for n in f._binding.install(dict(vars(f)))})
COUNTS = {n: len(f.SIGNATURES[n][1]) - (n == "fasgd_pull") for n in NAMES}


def through_ctypes(name, args):
    if name == "fasgd_pull":
        T = ctypes.c_int64()
        return f.LIB.fasgd_pull(*args, ctypes.byref(T)), T.value
    return getattr(f.LIB, name)(*args)


def outcome(call, *args):
    try:
        return call(*args)
    except (TypeError, ctypes.ArgumentError):
        return "refused"


@pytest.fixture(autouse=True)
def slow_functions():
    """The module's own fallbacks, restored after a test replaced them."""
    f._binding.install({n: (lambda *a, _n=n: through_ctypes(_n, a)) for n in NAMES})
    yield
    f._binding.install({n: (lambda *a, _n=n: through_ctypes(_n, a)) for n in NAMES})


@pytest.mark.parametrize("name", NAMES)
def test_arguments_as_ctypes_takes_them(name):
    n = COUNTS[name]
    fast = getattr(f._binding, name)
    null = [None] + [0] * (n - 1)        # a null handle, or P = None / 0: rejected on the host
    for base in ([0] * n, null, [None] * n, [0] * (n - 1), [0] * (n + 1), []):
        assert outcome(fast, *base) == outcome(through_ctypes, name, list(base)), base
    for k in range(n):
        for bad in (None, 1.5, "x", True, -1, 1 << 70, np.int64(3), ctypes.c_void_p(), b"abc"):
            if k == 0 and bad is not None and bad != 1.5:
                continue                 # would be taken for a handle or a size
            args = [0] * n
            args[k] = bad
            assert outcome(fast, *args) == outcome(through_ctypes, name, args), (k, bad)


def test_keywords_reach_the_python_function():
    assert f.fasgd_apply_pending is f._binding.fasgd_apply_pending
    seen = []
    f._binding.install({n: (lambda *a, _n=n, **k: seen.append((_n, a, k)) or 7) for n in NAMES})
    assert f.fasgd_apply_pending(None, K=3) == 7
    assert seen == [("fasgd_apply_pending", (None,), {"K": 3})]
