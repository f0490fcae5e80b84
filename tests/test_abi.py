"""The C-ABI library loads, exports every symbol the public header declares, and rejects bad
arguments on the host before touching a device.  No GPU needed."""
import ctypes
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    from paper_2506_09316_b200 import build
    return ctypes.CDLL(build.build())


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "dsla.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(dsla_[a-z_0-9]+)\s*\(", text)))


def test_header_symbols_are_exported(lib):
    names = declared_symbols()
    assert {"dsla_prefill", "dsla_decode_step", "dsla_state_alloc", "dsla_state_free"} <= set(names)
    for n in names:
        assert hasattr(lib, n), f"{n} declared in dsla.h but not exported"


def test_binding_covers_every_symbol(lib):
    import paper_2506_09316_b200 as dsla
    for n in declared_symbols():
        assert callable(getattr(dsla, n)), n


def test_status_strings(lib):
    lib.dsla_status_string.restype = ctypes.c_char_p
    got = [lib.dsla_status_string(i).decode() for i in range(6)]
    assert got == ["DSLA_OK", "DSLA_ERR_INVALID_ARG", "DSLA_ERR_UNSUPPORTED", "DSLA_ERR_CUDA", "DSLA_ERR_OOM",
                   "DSLA_ERR_TIMEOUT"]


def test_sizes_and_host_side_rejections(lib):
    from paper_2506_09316_b200 import binding as b
    assert b.dsla_state_bytes(128, 32, 128, 128) == 128 * 2 * 32 * 128 * 128 * 4
    assert b.dsla_state_bytes(0, 32, 128, 128) == 0 and b.dsla_state_bytes(1, 1, -1, 128) == 0
    h = ctypes.c_void_p()
    f = lib.dsla_state_alloc
    f.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_int,
                  ctypes.c_void_p, ctypes.c_size_t]
    assert f(None, 1, 1, 64, 64, None, 0) == b.DSLA_ERR_INVALID_ARG
    assert f(ctypes.byref(h), 0, 1, 64, 64, None, 0) == b.DSLA_ERR_INVALID_ARG
    assert f(ctypes.byref(h), 1, 1, 48, 48, None, 0) == b.DSLA_ERR_UNSUPPORTED
    assert f(ctypes.byref(h), 1, 1, 64, 128, None, 0) == b.DSLA_ERR_UNSUPPORTED
    assert f(ctypes.byref(h), 1, 1, 64, 64, ctypes.c_void_p(256), 8) == b.DSLA_ERR_INVALID_ARG   # too small
    assert f(ctypes.byref(h), 1, 1, 64, 64, ctypes.c_void_p(260), 1 << 20) == b.DSLA_ERR_INVALID_ARG  # misaligned
    # prefill / decode with a NULL state or NULL args never reach a launch
    a = b.dsla_prefill_args()
    assert lib.dsla_prefill(None, None, None) == b.DSLA_ERR_INVALID_ARG
    a.N, a.T, a.T_total, a.max_seqlen, a.H, a.d_k, a.d_v, a.chunk = 1, 8, 8, 8, 2, 64, 64, 64
    assert b._lib.dsla_prefill(ctypes.byref(a), None, None) == b.DSLA_ERR_INVALID_ARG
    a.d_k = a.d_v = 96
    assert b._lib.dsla_prefill(ctypes.byref(a), None, None) == b.DSLA_ERR_UNSUPPORTED
    a.d_k = a.d_v = 64
    a.chunk = 48
    assert b._lib.dsla_prefill(ctypes.byref(a), None, None) == b.DSLA_ERR_UNSUPPORTED
    a.chunk, a.T_total = 64, 9
    assert b._lib.dsla_prefill(ctypes.byref(a), None, None) == b.DSLA_ERR_INVALID_ARG      # N*T != T_total
    a.T_total, a.dtype = 8, 7
    assert b._lib.dsla_prefill(ctypes.byref(a), None, None) == b.DSLA_ERR_INVALID_ARG
    assert b._lib.dsla_prefill_workspace_bytes(None) == 0
    d = b.dsla_decode_args()
    assert b._lib.dsla_decode_step(ctypes.byref(d), None, None) == b.DSLA_ERR_INVALID_ARG
    assert b._lib.dsla_decode_step(None, None, None) == b.DSLA_ERR_INVALID_ARG
    assert b._lib.dsla_state_free(None) == b.DSLA_OK
    assert b._lib.dsla_state_zero(None, None, 0, None) == b.DSLA_ERR_INVALID_ARG
    assert b.dsla_launch_count() == 0


def test_product_package_does_not_import_the_checker():
    """Nothing under the CUDA package may import, load or name the CPU checker."""
    pkg = os.path.join(ROOT, "paper_2506_09316_b200")
    for dirpath, _, files in os.walk(pkg):
        for fn in files:
            if fn.endswith((".py", ".cu", ".cuh", ".h")):
                text = open(os.path.join(dirpath, fn)).read()
                assert "oracle" not in text, f"{fn} mentions the checker"


def test_workspace_query_knows_the_gate_layout(lib):
    """What dsla_prefill_workspace_bytes reports is what the kernel of that layout can use: with vector gates the summaries of the
    segments (fp32 [2][128][128] and [2][128] each), also through the C structure; without a layout, enough for either."""
    import torch
    from paper_2506_09316_b200 import binding as b
    entry = (2 * 128 * 128 + 2 * 128) * 4
    sizes = dict(T_total=4096, N=1, max_seqlen=4096, H=32, d=128, dense_T=4096)
    vec = b.dsla_prefill_workspace_bytes(gate_layout=b.DSLA_GATE_PER_KEY_CHANNEL, **sizes)
    assert vec == 32 * 4 * entry <= b.DSLA_STATIC_SCRATCH_BYTES
    assert b.dsla_prefill_workspace_bytes(**sizes) >= vec
    for other in (dict(dtype=torch.float32), dict(impl="simt"), dict(impl="tensor"), dict(d=64)):      # forms that kernel does not serve
        assert b.dsla_prefill_workspace_bytes(gate_layout=b.DSLA_GATE_PER_KEY_CHANNEL, **{**sizes, **other}) == 0


def test_workspace_is_what_the_kernel_uses(lib):
    """The single-CTA tensor kernel keeps its segment summaries on chip: no room for them is asked for, whatever the length; only the
    cluster variant and the visiting order of large packed batches need any."""
    from paper_2506_09316_b200 import binding as b

    def query(T, H, N=1, impl="tensor", dense=True):
        return b.dsla_prefill_workspace_bytes(N * T, N, T, H, 128, impl=impl, dense_T=T if dense else None, gate_layout=b.DSLA_GATE_SCALAR)

    for T in (64, 257, 385, 512, 777, 1152, 4096, 65536):
        for H in (1, 4, 16, 24, 32, 40):
            assert query(T, H) <= 256 and query(T, H, impl="auto") <= 256
    assert query(64, 2, N=64, dense=False) == 0 and query(64, 2, N=65, dense=False) >= 65 * 4
    assert query(4096, 32, impl="pair") > 2 * 32 * 2 * 128 * 128 * 4


def test_sequence_count_of_any_cu_seqlens_shape(lib):
    import torch
    from paper_2506_09316_b200 import binding as b
    cu = torch.tensor([0, 3, 3, 10], dtype=torch.int32)
    for shape in ((4,), (1, 4), (4, 1), (2, 2)):
        assert b._sequences(10, cu.view(shape), 7) == (3, 0, 7)
    assert b._sequences(12, None, 4) == (3, 4, 4) and b._sequences(12, None, None) == (1, 12, 12) and b._sequences(0, None, None)[0] == 0


def test_extension_module_reads_only_the_sizes_it_needs(lib):
    """v may have dimensions behind the head size and w any behind its first; q and x have exactly three and two.  No store is passed, so
    the C entry points refuse every call before they touch a device."""
    import torch
    from paper_2506_09316_b200 import _native, binding as b
    q, g, gamma = torch.zeros(4, 2, 64), torch.zeros(4, 2), torch.zeros(2)
    v, w = q.view(4, 2, 64, 1), torch.zeros(2, 4)
    gates = torch.stack([g, g])
    dense, steps = (None, 1, 4, 4, 64, 1.0, 0, 0, 0), (None, 1.0, 0)
    assert _native.prefill(q, q, v, v, g, g, gamma, None, None, None, *dense) == b.DSLA_ERR_INVALID_ARG
    assert _native.decode_step(q, q, v, v, g, g, gamma, None, None, *steps) == b.DSLA_ERR_INVALID_ARG
    assert _native.nstate_decode_step(q, q, v, v, gates, w, None, None, *steps) == b.DSLA_ERR_INVALID_ARG
    assert _native.nstate_prefill(q, q, v, v, gates, w, None, None, None, None, 1, 4, 4, 1.0, 0, 0, 0) == b.DSLA_ERR_INVALID_ARG
    assert _native.prefill_workspace(q, v, g, None, 1, 4, 4, 64, 0) == 0 and _native.nstate_prefill_workspace(q, v, gates, None, 1, 4, 4, 0) == 0
    x = torch.zeros(4, 64, dtype=torch.bfloat16)
    assert _native.gate_project(x, torch.zeros(6, 64, 1, dtype=torch.bfloat16), None, g, g, 0) == b.DSLA_ERR_UNSUPPORTED      # H = 3
    for bad in (lambda: _native.decode_step(v, q, v, v, g, g, gamma, None, None, *steps), lambda: _native.gate_project(q, x, None, g, g, 0)):
        with pytest.raises(ValueError):
            bad()


def test_prefill_of_whole_sequences_spills_no_registers(tmp_path):
    """The chunk loop of the tensor-core prefill keeps two 32-register sets alive at 96 registers a thread; ptxas reports what does not fit."""
    import shutil
    import subprocess
    from paper_2506_09316_b200 import build
    nvcc = shutil.which(build._nvcc())
    if nvcc is None:
        pytest.skip("no nvcc")
    out = subprocess.run([nvcc, *build.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, "dsla_prefill_tc.cu"), "-o",
                          str(tmp_path / "x.o")], capture_output=True, text=True, check=True)
    entry = [s for s in re.split("Compiling entry function", out.stderr + out.stdout)[1:] if "prefill_tc_kernelILb0ELb0E" in s]
    assert len(entry) == 1
    assert re.search(r"(\d+) bytes spill stores, (\d+) bytes spill loads", entry[0]).groups() == ("0", "0")
