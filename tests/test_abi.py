"""CPU-only checks of the C ABI: the library loads without a GPU, exports every symbol the
header declares, and rejects bad arguments on the host before anything could be launched."""
import ctypes
import os
import re
import subprocess
import sys
import sysconfig

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2601_16515_b200 import build
    build.build()
    from paper_2601_16515_b200 import salad
    return salad


def declared_functions():
    text = open(os.path.join(ROOT, "include", "salad.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(salad_[a-z_0-9]+)\s*\(", text)))


def test_header_symbols_are_exported(lib):
    names = declared_functions()
    assert set(names) == set(lib.EXPORTS)
    raw = ctypes.CDLL(lib.LIB_PATH)
    for n in names:
        assert hasattr(raw, n), n


def test_status_strings(lib):
    assert lib.status_string(0) == "SALAD_OK"
    for code, name in [(-1, "INVALID_ARG"), (-2, "UNSUPPORTED"), (-3, "WORKSPACE"), (-4, "CAPACITY"),
                       (-5, "CUDA"), (-6, "TIMEOUT"), (-7, "BAD_MASK")]:
        assert lib.status_string(code) == "SALAD_ERR_" + name
    assert lib.status_string(-99) == "SALAD_ERR_UNKNOWN"


def test_workspace_bytes(lib):
    assert lib.salad_workspace_bytes(1, 12, 32760, 128, 128, 64) > 12 * 128 * 128 * 2
    assert lib.salad_workspace_bytes(1, 12, 32760, 128, 128, 64) % 256 == 0
    assert lib.salad_workspace_bytes(1, 2, 1024, 64, 64, 64) > 0
    assert lib.salad_workspace_bytes(1, 2, 1024, 96, 64, 64) == 0       # head dim
    assert lib.salad_workspace_bytes(1, 2, 1024, 64, 32, 64) == 0       # Bq
    assert lib.salad_workspace_bytes(1, 2, 1024, 64, 64, 128) == 0      # Bk
    assert lib.salad_workspace_bytes(0, 2, 1024, 64, 64, 64) == 0
    # independent of N and of the block size, grows with batch*heads
    assert lib.salad_workspace_bytes(2, 1000, 64, 64, 64, 64) > lib.salad_workspace_bytes(2, 12, 64, 64, 64, 64)


def test_host_side_argument_checks(lib):
    L = lib._lib
    P = ctypes.c_void_p
    fake = P(0x1000)            # never dereferenced: validation fails first
    ws_bytes = lib.salad_workspace_bytes(1, 2, 1024, 64, 64, 64)
    rc = L.salad_sparse_attn_fwd(None, fake, fake, fake, None, 1, 2, 1024, 64, 64, 64, fake, fake, 1, 0.0,
                                 fake, ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_INVALID_ARG
    rc = L.salad_sparse_attn_fwd(fake, fake, fake, fake, None, 1, 2, 1024, 96, 64, 64, fake, fake, 1, 0.0,
                                 fake, ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_UNSUPPORTED
    rc = L.salad_sparse_attn_fwd(fake, fake, fake, fake, None, 1, 2, 1024, 64, 64, 64, fake, fake, 3, 0.0,
                                 fake, ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_INVALID_ARG                                  # Hm not in {1, H}
    rc = L.salad_sparse_attn_fwd(fake, fake, fake, fake, None, 1, 2, 1024, 64, 64, 64, fake, fake, 1, -1.0,
                                 fake, ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_INVALID_ARG                                  # negative scale
    rc = L.salad_sparse_attn_fwd(fake, fake, fake, fake, None, 1, 2, 1024, 64, 64, 64, fake, fake, 1, 0.0,
                                 fake, ws_bytes - 1, None, None)
    assert rc == lib.SALAD_ERR_WORKSPACE
    rc = L.salad_sparse_attn_fwd(fake, fake, fake, fake, None, 1, 2, 1024, 64, 64, 64, fake, fake, 1, 0.0,
                                 P(0x1010), ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_WORKSPACE                                    # misaligned workspace
    rc = L.salad_sparse_attn_fwd(P(0x1004), fake, fake, fake, None, 1, 2, 1024, 64, 64, 64, fake, fake, 1, 0.0,
                                 fake, ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_INVALID_ARG                                  # misaligned tensor
    rc = L.salad_fused_fwd(fake, fake, fake, fake, 1, 2, 1024, 64, 64, 64, fake, fake, 1, None, fake, 0.0, 1e-6,
                           fake, ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_INVALID_ARG                                  # missing scale
    rc = L.salad_linear_attn_fwd(fake, fake, fake, fake, None, None, 1, 2, 1024, 64, -1.0, fake, ws_bytes,
                                 None, None)
    assert rc == lib.SALAD_ERR_INVALID_ARG                                  # negative eps
    win = (ctypes.c_int32 * 3)(1, 1, 1)
    assert L.salad_mask_build(0, 4, 4, 64, 64, 1, win, fake, None, 0, None, None) == lib.SALAD_ERR_INVALID_ARG
    assert L.salad_mask_build(4, 4, 4, 64, 64, 1, None, fake, None, 0, None, None) == lib.SALAD_ERR_INVALID_ARG
    assert L.salad_mask_build(4, 4, 4, 64, 64, 1, win, fake, None, 5, None, None) == lib.SALAD_ERR_INVALID_ARG
    assert L.salad_mask_build(4, 4, 4, 64, 64, 1000, win, fake, None, 0, None, None) == lib.SALAD_ERR_UNSUPPORTED
    neg = (ctypes.c_int32 * 3)(1, -1, 1)
    assert L.salad_mask_build(4, 4, 4, 64, 64, 1, neg, fake, None, 0, None, None) == lib.SALAD_ERR_INVALID_ARG


def test_mask_validator_argument_checks(lib):
    L = lib._lib
    P = ctypes.c_void_p
    fake = P(0x1000)
    assert L.salad_csr_validate(None, fake, 10, 4, 8, fake, None) == lib.SALAD_ERR_INVALID_ARG     # no row_ptr
    assert L.salad_csr_validate(fake, fake, 10, 4, 8, None, None) == lib.SALAD_ERR_INVALID_ARG     # no status word
    assert L.salad_csr_validate(fake, None, 10, 4, 8, fake, None) == lib.SALAD_ERR_INVALID_ARG     # capacity without a list
    assert L.salad_csr_validate(fake, fake, -1, 4, 8, fake, None) == lib.SALAD_ERR_INVALID_ARG
    assert L.salad_csr_validate(fake, fake, 10, 0, 8, fake, None) == lib.SALAD_ERR_INVALID_ARG
    assert L.salad_csr_validate(fake, fake, 10, 4, 0, fake, None) == lib.SALAD_ERR_INVALID_ARG
    assert L.salad_set_mask_validation(-5) == lib.SALAD_ERR_INVALID_ARG
    assert L.salad_set_mask_validation(100) == lib.SALAD_OK
    assert L.salad_set_mask_validation(0) == lib.SALAD_OK


def test_no_gpu_means_error_not_fallback(lib):
    import torch
    if torch.cuda.is_available():
        pytest.skip("GPU present")
    L = lib._lib
    fake = ctypes.c_void_p(0x1000)
    ws_bytes = lib.salad_workspace_bytes(1, 2, 1024, 64, 64, 64)
    rc = L.salad_sparse_attn_fwd(fake, fake, fake, fake, None, 1, 2, 1024, 64, 64, 64, fake, fake, 1, 0.0,
                                 fake, ws_bytes, None, None)
    assert rc == lib.SALAD_ERR_CUDA


def test_a_cpu_device_is_refused(lib):
    # the builders allocate their outputs on the device they are given: host memory must not reach a kernel
    for call in (lambda: lib.salad_mask_build(2, 4, 4, 64, 64, [(1, 1, 1)], device="cpu"),
                 lambda: lib.salad_stswa_mask_build((2, 4, 4), [0, 1], [3, 3], device="cpu")):
        with pytest.raises(ValueError, match="Expected a cuda device"):
            call()


def test_host_only_entry_points_need_no_cuda_torch(lib):
    code = ("import torch\n"
            "for name in ('_cuda_getDevice', '_cuda_getCurrentRawStream'): delattr(torch._C, name)\n"
            "from paper_2601_16515_b200 import salad\n"
            "assert salad.salad_workspace_bytes(1, 2, 1024, 64, 64, 64) > 0 and salad.status_string(0) == 'SALAD_OK'\n")
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)


def test_native_calls_answer_like_ctypes(lib):
    """The calls that bypass ctypes (csrc/fastcall.cpp): the same answers on the host-side checks, and whatever they do not
    convert is left to ctypes, with its errors."""
    assert set(lib._fast) <= set(lib.EXPORTS) and "salad_fused_fwd" in lib._fast
    p, ws_bytes = 1 << 20, lib.salad_workspace_bytes(1, 2, 1024, 64, 64, 64)      # never dereferenced
    good = [p, p, p, p, 1, 2, 1024, 64, 64, 64, p, p, 2, p, p, 0.0, 1e-6, p, ws_bytes, None, None]
    for change in ({0: None}, {3: p + 8}, {7: 96}, {9: 32}, {12: 5}, {15: -1.0}, {15: float("nan")}, {16: float("inf")}, {17: p + 1},
                   {18: ws_bytes - 1}, {4: -1}, {6: 0}, {4: 2**32}):
        args = [change.get(i, a) for i, a in enumerate(good)]
        rc = lib._fast["salad_fused_fwd"](*args)
        assert isinstance(rc, int) and rc == lib._lib.salad_fused_fwd(*args) and rc < 0, change
    for change in ({0: 1.0}, {6: 1024.0}, {15: "0"}, {4: None}):
        args = [change.get(i, a) for i, a in enumerate(good)]
        assert lib._fast["salad_fused_fwd"](*args) is None
        with pytest.raises(ctypes.ArgumentError):
            lib._enter("salad_fused_fwd", *args)
    assert lib._fast["salad_fused_fwd"](*good[:-1]) is None


def test_no_registers_change_hands():
    """No kernel hands registers over between its warps: ptxas 12.9 lost values that live across setmaxnreg in forms of the attention
    kernel (wrong outputs, no warning), and the same sources without it were right."""
    csrc = os.path.join(ROOT, "paper_2601_16515_b200", "csrc")
    for name in sorted(os.listdir(csrc)):
        assert "setmaxnreg" not in re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read()), name


def test_tensor_memory_loads_wait_where_they_load():
    """tcgen05.ld is asynchronous and its wait names no register: one statement issues a load and waits for it, or the compiler
    may use (or copy) the registers in between."""
    csrc, loads = os.path.join(ROOT, "paper_2601_16515_b200", "csrc"), 0
    for name in sorted(os.listdir(csrc)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        for statement in re.findall(r"\basm\b[^;]*?\((?:\"(?:[^\"\\]|\\.)*\"|[^\"])*?\)\s*;", text):
            code = "".join(re.findall(r"\"((?:[^\"\\]|\\.)*)\"", statement))
            if "tcgen05.ld." in code or "tcgen05.wait::ld" in code:
                loads += 1
                assert "tcgen05.ld." in code and "tcgen05.wait::ld" in code[code.rindex("tcgen05.ld."):], (name, statement[:120])
    assert loads >= 4


def test_without_the_native_module(lib, tmp_path, monkeypatch):
    """The module that bypasses ctypes is named for its interpreter, the build goes on without it where it cannot be compiled (and
    leaves none of other sources), and the binding answers the same through ctypes."""
    from paper_2601_16515_b200 import build
    assert os.path.basename(build.FASTCALL) == "_fastcall" + sysconfig.get_config_var("EXT_SUFFIX")
    stale = tmp_path / os.path.basename(build.FASTCALL)
    monkeypatch.setattr(build, "FASTCALL", str(stale))
    for command in (["no-such-compiler"], [sys.executable, "-c", "raise SystemExit(1)"]):
        stale.write_bytes(b"")
        os.utime(stale, (0, 0))
        monkeypatch.setattr(build, "fastcall_command", lambda out: command)
        with pytest.warns(RuntimeWarning, match="not built"):
            assert build.build() == build.LIB
        assert not os.listdir(tmp_path)
    code = ("from paper_2601_16515_b200 import build\n"
            "build.FASTCALL += '.absent'\n"
            "from paper_2601_16515_b200 import salad\n"
            "p, n = 1 << 20, salad.salad_workspace_bytes(1, 2, 1024, 64, 64, 64)\n"
            "good = [p, p, p, p, 1, 2, 1024, 64, 64, 64, p, p, 2, p, p, 0.0, 1e-6, p, n, None, None]\n"
            "assert salad._fast == {}\n"
            "assert salad._enter('salad_fused_fwd', None, *good[1:]) == salad.SALAD_ERR_INVALID_ARG\n"
            "assert salad._enter('salad_fused_fwd', *good[:18], n - 1, None, None) == salad.SALAD_ERR_WORKSPACE\n")
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)


def test_stswa_call_bypasses_ctypes(lib):
    """The ST-SWA call, whose head flags are host memory, takes the way of the other calls of every layer, with ctypes' answers."""
    flags = (ctypes.c_int32 * 2)(0, 1)
    p, n = 1 << 20, lib._lib.salad_stswa_workspace_bytes(1, 2, 4, 16, 16, 64)
    good = [p, p, p, p, 1, 2, 1024, 64, 4, 16, 16, ctypes.addressof(flags), p, p, p, p, 0.5, 0.0, 1e-6, p, n, None, None]
    for change in ({0: None}, {3: p + 8}, {6: 1023}, {7: 96}, {8: 65}, {11: None}, {17: -1.0}, {18: float("nan")}, {19: p + 1}, {20: n - 1}):
        args = [change.get(i, a) for i, a in enumerate(good)]
        rc = lib._fast["salad_fused_stswa_fwd"](*args)
        assert isinstance(rc, int) and rc == lib._lib.salad_fused_stswa_fwd(*args) and rc < 0, change
