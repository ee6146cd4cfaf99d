"""The C-ABI library loads and exports every symbol that include/det.h and include/det_test.h declare (no GPU needed)."""
import ctypes
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    names = set()
    for h in ("det.h", "det_test.h"):
        src = open(os.path.join(ROOT, "include", h)).read()
        src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
        names |= set(re.findall(r"\b(det_[a-z0-9_]+)\s*\(", src))
    return sorted(names)


def test_header_symbols_are_exported():
    from paper_2609_17380_b200 import build
    so = build.build()
    lib = ctypes.CDLL(so)
    names = _declared()
    assert len(names) >= 35
    missing = [n for n in names if not hasattr(lib, n)]
    assert not missing, missing


def test_host_side_argument_checks():
    # error paths that return before any launch work without a GPU
    from paper_2609_17380_b200 import build
    lib = ctypes.CDLL(build.build())
    lib.det_sum_ws_bytes.restype = ctypes.c_size_t
    assert lib.det_sum_ws_bytes(ctypes.c_size_t(1200000000)) >= 4 * (1200000000 // 16384)
    assert lib.det_grad_accum_nbufs(8) == 5 and lib.det_grad_accum_nbufs(1) == 2 and lib.det_grad_accum_nbufs(7) == 4
    assert lib.det_grad_accum_nbufs(0) == -1
    assert lib.det_rmsnorm_fwd(0, None, None, 4, 8, ctypes.c_float(0), None, None, None) == -1      # DET_ERR_ARG
    buf = ctypes.create_string_buffer(4096)
    addr = ctypes.addressof(buf)
    a16 = ctypes.c_void_p((addr + 255) // 256 * 256)
    a1 = ctypes.c_void_p(a16.value + 4)
    assert lib.det_rmsnorm_fwd(0, a16, None, 4, 12, ctypes.c_float(0), a16, a16, None) == -2        # D % 8
    assert lib.det_rmsnorm_fwd(0, a1, None, 4, 8, ctypes.c_float(0), a16, a16, None) == -3          # alignment
    assert lib.det_linear_fwd(a16, a16, a16, a16, 100, 128, 128, a16, a16, None, None) == -2        # M % 128
    assert lib.det_linear_fwd(a16, a16, a16, a16, 128, 128, 1 << 17, a16, a16, None, None) == -5    # int32 range
    assert lib.det_attn_fwd(a16, a16, a16, 128, 1, 1, 1, 100, 0, a16, 128, a16, None) == -2         # S % 64
    assert lib.det_attn_fwd(a16, a16, a16, 512, 1, 4, 3, 128, 0, a16, 512, a16, None) == -2         # H % Hkv
    assert lib.det_attn_fwd(a16, a16, a16, 128, 1, 1, 1, 128, 100, a16, 128, a16, None) == -2       # window % 128
    assert lib.det_xent_fwd(a16, a16, 4, 8, ctypes.c_float(0), a16, a16, a16, a16, a16, ctypes.c_size_t(8), None, None) == -4
    # the attention forward of arithmetic version 2: shape limits, alignment, workspace size
    lib.det_attn_fwd_v2_ws_bytes.restype = ctypes.c_size_t
    need = lib.det_attn_fwd_v2_ws_bytes(1, 2, 256)
    assert need >= 2 * 256 * 256 * 6 and lib.det_attn_fwd_v2_ws_bytes(0, 2, 256) == 0
    big = ctypes.c_size_t(1 << 40)
    assert lib.det_attn_fwd_v2(a16, a16, a16, 768, 1, 2, 100, a16, 256, a16, a16, big, None, None) == -2      # S % 128
    assert lib.det_attn_fwd_v2(a16, a16, a16, 768, 1, 2, 16384, a16, 256, a16, a16, big, None, None) == -2    # S > 8192
    assert lib.det_attn_fwd_v2(a16, a16, a16, 128, 1, 2, 256, a16, 256, a16, a16, big, None, None) == -2      # ld < H * 128
    assert lib.det_attn_fwd_v2(a1, a16, a16, 768, 1, 2, 256, a16, 256, a16, a16, big, None, None) == -3       # alignment
    assert lib.det_attn_fwd_v2(a16, a16, a16, 768, 1, 2, 256, a16, 256, a16, a16, ctypes.c_size_t(need - 1), None, None) == -4
    assert lib.det_attn_fwd_v2(None, a16, a16, 768, 1, 2, 256, a16, 256, a16, a16, big, None, None) == -1     # null operand


# every tensor of a table is checked as a single argument is: one on the host, one with gaps or one that is too short is refused
# before anything is launched (no GPU needed: the refusal comes first)
def test_tables_are_checked():
    import pytest
    import torch
    import paper_2609_17380_b200 as det
    t = lambda n, dt=torch.float32: torch.zeros(n, dtype=dt)
    desc = det.det_adamw_desc(1e-3, 0.9, 0.95, 1e-8, 0.0, 1)
    bf = t(8, torch.int16)
    for args in (([desc], [det.DET_BF16], [bf], [t(8)], [t(8)], [t(8)]),              # on the host
                 ([desc], [det.DET_BF16], [bf], [t(4)], [t(8)], [t(8)]),              # a short gradient
                 ([desc], [det.DET_BF16], [bf], [t(8)], [t(8)], [t(4)]),              # a short moment
                 ([desc], [det.DET_F32], [bf], [t(8)], [t(8)], [t(8)]),               # 16 bits passed as 32
                 ([desc], [], [bf], [t(8)], [t(8)], [t(8)])):                         # no type given
        with pytest.raises(AssertionError):
            det.det_adamw_batch(*args)
    with pytest.raises(AssertionError):
        det.det_tensor_hash_batch([t(64, torch.uint8)], t(32, torch.uint8), t(4096, torch.uint8))


# the native callables take what an argument with a declared C type takes (integers of any kind, ctypes objects of that type or of one
# derived from it, anything with _as_parameter_) and refuse the rest as ctypes does, naming the argument; a status that is not DET_OK
# raises.  Rows of no values are refused and no rows return at once, so nothing is launched
def test_native_calls_convert_and_refuse():
    import numpy as np
    import pytest
    import torch
    import paper_2609_17380_b200 as det
    from paper_2609_17380_b200 import _binding
    lib = det.load()
    patterns = {n: p.replace("s", "p") for n, p in det._PATTERNS.items()}            # the stream as an argument: no device is touched
    calls = _binding.bind(det._SO, patterns, det._check, lib)
    swiglu, hash_, norm = calls["det_swiglu_bwd"], calls["det_tensor_hash_async"], calls["det_rmsnorm_fwd_q"]

    class Rows(ctypes.c_int):
        pass

    class Width:
        def __init__(self, v):
            self._as_parameter_ = v

    for width in (0, np.int64(0), False, ctypes.c_int(0), 1 << 32, torch.tensor(0), Rows(0), Width(0), Width(Rows(0))):   # 2^32 is 0 in a C int
        assert swiglu(16, 16, width, 8, 16, None) is None                        # no rows
        with pytest.raises(det.DetError) as e:
            swiglu(16, 16, 0, width, 16, None)
        assert e.value.code == -1
    for eps in (1, 1e-6, 1e300, np.float32(1e-6), np.float64(1e-6), torch.tensor(1e-6), ctypes.c_float(1e-6), Width(1e-6)):
        with pytest.raises(det.DetError) as e:                                    # rows of no values
            norm(16, 16, 0, 0, eps, 16, 16, 16, 16, None)
        assert e.value.code == -1
    for bad in (0.0, "0", None, ctypes.c_long(0), Width("0")):
        for call in (swiglu, lib.det_swiglu_bwd):                                 # the same from either
            with pytest.raises(ctypes.ArgumentError, match="argument 3"):
                call(16, 16, bad, 8, 16, None)
    for bad in ("1", None, 10 ** 400, ctypes.c_double(1.0)):
        for call in (norm, lib.det_rmsnorm_fwd_q):
            with pytest.raises(ctypes.ArgumentError, match="argument 5"):
                call(16, 16, 0, 0, bad, 16, 16, 16, 16, None)
    for bad in ("x", 1.0):
        with pytest.raises(TypeError):
            swiglu(bad, 16, 0, 8, 16, None)
    with pytest.raises(AssertionError):
        swiglu(torch.zeros(4), 16, 0, 8, 16, None)                                # not a CUDA tensor
    with pytest.raises(AttributeError):
        hash_(16, 0, 16, 16, None)                                                # a workspace has to be a tensor
    for n in (5, 7):
        with pytest.raises(TypeError):
            swiglu(*([0] * n))
    with pytest.raises(ImportError):
        _binding.bind(det._SO, dict(patterns, det_swiglu_bwd="pppppp"), det._check, lib)


# a second bind, one that is refused half-way included, leaves the callables of the first as they are: here they take the
# stream as an argument, where the package's take the current one
def test_bound_calls_stay_as_they_were_bound():
    import pytest
    import paper_2609_17380_b200 as det
    from paper_2609_17380_b200 import _binding
    lib = det.load()
    patterns = {n: p.replace("s", "p") for n, p in det._PATTERNS.items()}
    swiglu = _binding.bind(det._SO, patterns, det._check, lib)["det_swiglu_bwd"]
    other = lambda name, status: 1 / 0
    _binding.bind(det._SO, det._PATTERNS, other, lib)
    assert swiglu(16, 16, 0, 8, 16, None) is None
    with pytest.raises(ImportError):
        _binding.bind(det._SO, dict(det._PATTERNS, det_tensor_hash_async="p"), other, lib)
    assert swiglu(16, 16, 0, 8, 16, None) is None
    with pytest.raises(det.DetError):
        swiglu(16, 16, 0, 0, 16, None)


# a pattern with the current stream or a workspace where the entry point takes another pointer, the status word say, is refused, and so is
# one that is too short or too long; the table of C types and the patterns describe the same arguments
def test_patterns_fit_the_declarations():
    import pytest
    import paper_2609_17380_b200 as det
    from paper_2609_17380_b200 import _binding
    lib = det.load()
    for name, bad in (("det_linear_fwd", "ppppiiippps"), ("det_linear_fwd", "sppppiiippp"), ("det_linear_fwd", "ppppiiipps"),
                      ("det_linear_fwd", "ppppiiippspp"), ("det_sum", "pzipw"), ("det_sum", "pziwws"), ("det_sum", "wipws"), ("det_sum", ""),
                      ("det_sum", "vzipws"), ("det_sum", "pzipvzs"), ("det_xent_bwd", "pppiifis")):
        with pytest.raises(ImportError):
            _binding.bind(det._SO, dict(det._PATTERNS, **{name: bad}), det._check, lib)
    for name, p in det._PATTERNS.items():
        assert det._SIGNATURES[name] == "i" + p.replace("w", "pz").replace("s", "p"), name


def test_unknown_entry_point_is_an_attribute_error():
    import paper_2609_17380_b200 as det
    assert callable(det._c.det_sum) and not hasattr(det._c, "det_no_such_thing")


# the binding is compiled against torch's headers: another torch version makes the object stale although its source is older
def test_binding_follows_the_torch_version(monkeypatch):
    import subprocess
    import torch
    from paper_2609_17380_b200 import build
    build.build_binding()
    runs = []
    monkeypatch.setattr(subprocess, "run", lambda cmd, **k: runs.append(cmd) or subprocess.CompletedProcess(cmd, 1, "", "not run"))
    build.build_binding()
    assert not runs                                            # up to date
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".1")
    try:
        build.build_binding()
    except RuntimeError:
        pass
    assert len(runs) == 1


# a filling grid skips the wait at its start, so its last block has to wait at its end on every way out, that after an expired wait
# included, or what comes next on the stream overlaps the launch before.  No wait can be made to expire from outside: the source is read
def test_filling_kernels_always_reach_their_end():
    csrc = os.path.join(ROOT, "paper_2609_17380_b200", "csrc")
    found = 0
    for name in sorted(os.listdir(csrc)):
        if not name.endswith((".cu", ".cuh")) or name == "common.cuh":
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, name)).read())
        for body in src.split("__global__")[1:]:
            if "grid_fill_end()" not in body:
                continue
            found += 1
            body = body[:body.index("grid_fill_end()")]
            if "setmaxnreg.inc" in body:                        # producer warps leave on their own; the consumers go to the end
                body = body[body.index("setmaxnreg.inc"):]
            body = re.sub(r"\[&\]\([^)]*\)(?: -> \w+)? \{.*?\n  \};", "", body, flags=re.S)      # a lambda returns to its caller
            assert not re.search(r"\breturn\b", body), name
    assert found >= 3
