"""The binding's C module against the ctypes functions it stands in for: the
same results and refusals for every form of argument, on calls that the library
rejects on the host (no GPU needed)."""

import ctypes
import glob
import inspect
import os
import shutil
import subprocess
import sys
import sysconfig

import numpy as np
import pytest

try:
    from paper_1601_04033_gb300 import fasgd as f
except ImportError:                      # pragma: no cover - the library is not built
    pytest.skip("libfasgd.so is not built", allow_module_level=True)
if f._binding is None:
    pytest.skip("built without Python's headers", allow_module_level=True)

NAMES = sorted(f._CTYPES)
COUNTS = {n: len(f.SIGNATURES[n][1]) - (n == "fasgd_pull") for n in NAMES}


def outcome(call, *args, **kwargs):
    try:
        return call(*args, **kwargs)
    except (TypeError, ctypes.ArgumentError):
        return "refused"


@pytest.mark.parametrize("name", NAMES)
def test_arguments_as_ctypes_takes_them(name):
    n = COUNTS[name]
    fast, slow = getattr(f, name), f._CTYPES[name]
    assert fast is getattr(f._binding, name) and fast is not slow
    null = [None] + [0] * (n - 1)        # a null handle, or P = None / 0: rejected on the host
    for base in ([0] * n, null, [None] * n, [0] * (n - 1), [0] * (n + 1), []):
        assert outcome(fast, *base) == outcome(slow, *base), base
    for k in range(n):
        for bad in (None, 1.5, "x", True, -1, 1 << 70, np.int64(3), ctypes.c_void_p(), b"abc"):
            if k == 0 and bad is not None and bad != 1.5:
                continue                 # would be taken for a handle or a size
            args = [0] * n
            args[k] = bad
            assert outcome(fast, *args) == outcome(slow, *args), (k, bad)


@pytest.mark.parametrize("name", NAMES)
def test_keywords_and_odd_types_reach_the_functions_that_ship(name):
    """Through the fallbacks fasgd.py installed, not stand-ins."""
    params = list(inspect.signature(f._CTYPES[name]).parameters)
    null = dict.fromkeys(params, 0)
    assert outcome(getattr(f, name), **null) == f._CTYPES[name](**null)
    assert outcome(getattr(f, name), **null, nonsense=1) == "refused"
    assert outcome(getattr(f, name), None, *[ctypes.c_int64(0)] * (len(params) - 1)) == \
        outcome(f._CTYPES[name], None, *[ctypes.c_int64(0)] * (len(params) - 1))


def test_fallbacks_are_kept_whole():
    """The module takes no function of its own as a fallback (a call would go
    round without end), and a refused install changes nothing."""
    own = {n: getattr(f._binding, n) for n in NAMES}
    for space in (own, {**f._CTYPES, NAMES[-1]: own[NAMES[-1]]}, dict(vars(f))):
        with pytest.raises(ValueError):
            f._binding.install(space)
    with pytest.raises(KeyError):
        f._binding.install({})
    assert f.fasgd_apply_pending(None, K=3) == f.EINVAL
    seen = []
    try:
        f._binding.install({n: (lambda *a, _n=n, **k: seen.append((_n, a, k)) or 7) for n in NAMES})
        assert f.fasgd_apply_pending(None, K=3) == 7
    finally:
        f._binding.install(f._CTYPES)
    assert seen == [("fasgd_apply_pending", (None,), {"K": 3})]
    assert f.fasgd_apply_pending(None, K=3) == f.EINVAL


@pytest.mark.parametrize("name, warns", [("_binding.cpython-39-x86_64-linux-gnu.so", False),
                                         ("_binding.so", True), ("_binding" + sysconfig.get_config_var("EXT_SUFFIX"), True)])
def test_only_this_interpreters_module_is_loaded(tmp_path, name, warns):
    """A module built for another Python is not looked at, and one that does not
    load is reported; the calls go through ctypes either way."""
    pkg = tmp_path / "paper_1601_04033_gb300"
    pkg.mkdir()
    for p in glob.glob(os.path.join(f._build.PKG, "*.py")):
        shutil.copy(p, pkg)
    os.symlink(f._build.LIB, pkg / "libfasgd.so")
    (pkg / name).write_bytes(b"not a module")
    code = ("import warnings\nwith warnings.catch_warnings(record=True) as w:\n"
            "    warnings.simplefilter('always')\n    from paper_1601_04033_gb300 import fasgd as f\n"
            "assert f._binding is None and f.fasgd_apply_pending(None, K=3) == f.EINVAL\n"
            "print(sum('ctypes' in str(x.message) for x in w))")
    r = subprocess.run([sys.executable, "-c", code], cwd=tmp_path, capture_output=True, text=True)
    assert r.returncode == 0 and int(r.stdout) == warns, r.stdout + r.stderr


def test_the_module_carries_the_interpreters_tag():
    assert f._binding.__file__ == f._build.BINDING
    assert f._build.BINDING.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert not os.path.exists(os.path.join(f._build.PKG, "_binding.so"))
