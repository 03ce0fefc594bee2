"""How the binding passes arguments: the native call helper, and the ctypes form that takes its place where the helper is not
built.  No GPU needed: the calls fail their argument checks before any CUDA work."""
import ctypes
import os
import sys
import sysconfig
import threading

import pytest
import torch

from paper_2412_07174_b200 import binding, build

P = 0x10000  # a fake, 16-byte aligned, never dereferenced address


@pytest.fixture(params=["native", "ctypes"])
def form(request, monkeypatch):
    build.build()
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_call", None)
    monkeypatch.setattr(binding, "_entry", {})
    if request.param == "native":
        if not os.path.exists(build.CALL):
            pytest.skip("no C compiler or Python headers")
        binding.lib()
    else:
        monkeypatch.setitem(sys.modules, "paper_2412_07174_b200._scap_call", None)  # as if it were not there
        monkeypatch.delattr(sys.modules["paper_2412_07174_b200"], "_scap_call", raising=False)
        with pytest.warns(UserWarning, match="ctypes"):
            binding.lib()
    return request.param


def status(fn, *args, **kw):
    try:
        fn(*args, **kw)
    except binding.ScapError as e:
        return e.code
    return 0


def test_every_call_form_returns_the_library_s_status(form):
    bf = torch.bfloat16
    ws = torch.zeros(1 << 16, dtype=torch.uint8)
    x, W, v, y = torch.zeros(2, 64, dtype=bf), torch.zeros(64, 60, dtype=bf), torch.zeros(64), torch.zeros(2, 64)
    tau = torch.zeros(4)[:1]
    assert status(binding.scap_sparse_fc, x, W, v, tau, None, y, ws, stream=P) == 4              # N = 60
    assert status(binding.scap_sparse_fc, x, W[:, :56], v, None, None, y, ws, stream=0) == 1             # no threshold
    assert status(binding.scap_sparse_fc, x.repeat(9, 1), W, v, tau, None, y, ws, stream=0) == 2  # 18 rows
    assert status(binding.scap_sparse_fc, x, W[:, :56], v, tau, None, y, ws[:16], stream=0) == 5
    assert status(binding.scap_dense_fc, x, W, None, y, ws, stream=0) == 4
    q = torch.zeros(64, 24, dtype=torch.int8)
    assert status(binding.scap_sparse_fc_q8, x, q, v, v, tau, None, y, ws, stream=0) == 4
    assert status(binding.scap_dense_fc_q8, x, q, v, None, y, ws, stream=0) == 4
    z = torch.zeros(64, dtype=torch.uint8)
    assert status(binding.scap_sparse_fc_q4, x, q, v, z, 48, v, tau, None, y, ws, stream=0) == 2
    assert status(binding.scap_dense_fc_q4, x, q, v, z, 48, None, y, ws, stream=0) == 2
    assert status(binding.scap_sparse_fc_grouped, x, W, v, tau, None, y, [0, 1], ws, stream=0) == 4
    assert status(binding.scap_sparse_fc_grouped, x, W[:, :56], v, tau, None, y, [0, 16], ws, stream=0) == 1
    assert status(binding.scap_sparse_fc_host, x, W, v, tau, None, y, ws, stream=0) == 4
    assert status(binding.scap_glu_ffn, x, W, W, None, tau, None, None, tau, None, y, ws, stream=0) != 0


def test_a_full_argument_list_arrives_in_order(form):
    """The last arguments of the longest call travel on the stack: a workspace that is one byte short is told from one that is not."""
    h, W = torch.zeros(1, 64, dtype=torch.bfloat16), torch.zeros(64, 128, dtype=torch.bfloat16)
    tau, y = torch.zeros(4)[:1], torch.zeros(1, 64)
    need = binding.scap_glu_workspace(1, 64, 64)
    short = torch.zeros(need, dtype=torch.uint8)[: need - 1]
    assert status(binding.scap_glu_ffn, h, W, W[:, :64].contiguous(), None, tau, None, None, tau, None, y, short, stream=0) == 5


def test_wrong_types_raise_and_leave_the_call_undone(form):
    x, W = torch.zeros(1, 64, dtype=torch.bfloat16), torch.zeros(64, 64, dtype=torch.bfloat16)
    ws, y = torch.zeros(1 << 16, dtype=torch.uint8), torch.zeros(1, 64)
    with pytest.raises((AttributeError, TypeError)):
        binding.scap_sparse_fc(x, W, "m", torch.zeros(1), None, y, ws, stream=0)
    with pytest.raises((AttributeError, TypeError)):
        binding.scap_sparse_fc(x, W, None, 0.5, None, y, ws, stream=0)
    with pytest.raises(TypeError):
        binding.scap_sparse_fc(x, W.double(), None, torch.zeros(1), None, y, ws, stream=0)


def test_four_threads(form):
    x, W = torch.zeros(1, 64, dtype=torch.bfloat16), torch.zeros(64, 60, dtype=torch.bfloat16)
    ws, y, tau = torch.zeros(1 << 16, dtype=torch.uint8), torch.zeros(1, 64), torch.zeros(4)[:1]
    seen = []

    def work(expected):
        w, t = (W, tau) if expected == 4 else (W[:, :56], None)
        seen.append({status(binding.scap_sparse_fc, x, w, None, t, None, y, ws, stream=0) for _ in range(2000)} == {expected})
    threads = [threading.Thread(target=work, args=(e,)) for e in (4, 1, 4, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert seen == [True] * 4


def test_native_helper_arguments():
    build.build()
    if not os.path.exists(build.CALL):
        pytest.skip("no C compiler or Python headers")
    from paper_2412_07174_b200._scap_call import call
    entry = ctypes.cast(binding.lib().scap_sparse_fc, ctypes.c_void_p).value
    args = [P, P, None, P, None, P, 1, 64, 64, 1, None, None, P, 0, None]
    assert call(entry, *args) == 5                          # integers are addresses; a workspace of no bytes
    assert call(entry, 2 ** 64 - 16, *args[1:]) == 5        # an address in the upper half
    with pytest.raises(OverflowError):
        call(entry, 2 ** 64, *args[1:])
    with pytest.raises(TypeError):
        call(entry, *([0] * 25))
    with pytest.raises(TypeError):
        call()
    with pytest.raises(ValueError):
        call(0, 1)
    with pytest.raises(AttributeError):
        call(entry, 0.5)


def test_the_helper_belongs_to_one_interpreter_and_may_be_missing(tmp_path, monkeypatch, capsys):
    assert build.CALL.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    for cc in ("false", str(tmp_path / "no_such_compiler")):
        monkeypatch.setenv("CC", cc)
        assert build.build_call_helper(target=str(tmp_path / "helper.so")) is False
        assert "ctypes" in capsys.readouterr().err
    assert not (tmp_path / "helper.so").exists()
