"""The build on the CPU: the library does not depend on the binding's native calls, and those are not used with another torch or
Python than they were built for; what the binding hands to them."""
import ctypes
import os
import sys
import types

import pytest

from paper_2503_18339_b200 import binding, build


@pytest.fixture
def elsewhere(monkeypatch, tmp_path):
    """The library is up to date, the native calls would be built into a folder of their own."""
    build.build()
    monkeypatch.setattr(build, "HOST", str(tmp_path / "_host.so"))
    monkeypatch.setattr(build, "HOST_RECORD", str(tmp_path / "record"))
    return tmp_path


def library_after(capfd):
    assert build.build() == build.LIB
    assert ctypes.CDLL(build.LIB).granq_status_string is not None
    assert not os.path.exists(build.HOST)
    assert len([line for line in capfd.readouterr().err.splitlines() if line.startswith("_host.so has not been built")]) == 1


def test_library_without_a_compiler_for_the_native_calls(elsewhere, monkeypatch, capfd):
    monkeypatch.setenv("CXX", "false")
    library_after(capfd)


def test_library_without_torch(elsewhere, monkeypatch, capfd):
    monkeypatch.setitem(sys.modules, "torch", None)
    library_after(capfd)


def test_native_calls_of_an_older_source_do_not_stay(elsewhere, monkeypatch, capfd):
    with open(build.HOST, "w") as f:
        f.write("old")
    os.utime(build.HOST, (0, 0))
    monkeypatch.setenv("CXX", "false")
    library_after(capfd)


def module_for(record):
    calls = []
    m = types.SimpleNamespace(setup=lambda *a: calls.append(a), calls=calls)
    if record is not None:
        m.built_for = record
    return m


@pytest.mark.parametrize("record", [None, "torch 1.0, cxx11 abi 1, python 3.8"])
def test_native_calls_of_other_versions_are_refused(monkeypatch, record):
    build.build()
    native = module_for(record)
    for name, value in (("_host_calls", native), ("_lib", None), ("_native", None)):
        monkeypatch.setattr(binding, name, value)
    with pytest.warns(UserWarning, match="_host.so was built for"):
        binding.lib()
    assert binding._native is None and not native.calls


def test_native_calls_of_these_versions_are_used(monkeypatch):
    build.build()
    native = module_for(build.host_record())
    for name, value in (("_host_calls", native), ("_lib", None), ("_native", None)):
        monkeypatch.setattr(binding, name, value)
    binding.lib()
    assert binding._native is native and len(native.calls) == 1
    from paper_2503_18339_b200 import _host
    assert _host.built_for == build.host_record()


def test_native_calls_of_other_versions_are_built_again(elsewhere, monkeypatch):
    for path, text in ((build.HOST, "module"), (build.HOST_RECORD, "torch 1.0, cxx11 abi 1, python 3.8")):
        with open(path, "w") as f:
            f.write(text)
    assert build._host_stale()
    with open(build.HOST_RECORD, "w") as f:
        f.write(build.host_record())
    assert not build._host_stale()


@pytest.mark.parametrize("want", [None, False, True, 0, 1, "yes"])
def test_want_params_is_a_truth_value(monkeypatch, want):
    import torch
    asked = []
    spy = lambda name: lambda *a: asked.append((name, a)) or "answered"
    monkeypatch.setattr(binding, "_native", types.SimpleNamespace(fused_call=spy("fused"), fwd_packmask_call=spy("fwd_packmask")))
    x, g = torch.zeros(1, 1, 2, 2), torch.zeros(1)
    for call in (lambda: binding.granq_fakequant_fused(x, 4, want_params=want),
                 lambda: binding.granq_fakequant_fused_fwd_packmask(x, 4, want_params=want),
                 lambda: binding.granq_fakequant_fused_stats(x, 4, want_params=want),
                 lambda: binding.granq_fakequant_fwd_packmask(x, 4, g, g, want_params=want)):
        assert call() == "answered"
    at = {"fused": 7, "fwd_packmask": 8}
    assert [a[at[name]] for name, a in asked] == [int(bool(want))] * 4
