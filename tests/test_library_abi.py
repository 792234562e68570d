"""The C-ABI library builds for sm_100a, loads, and exports every symbol include/dsbd.h declares
(no compute calls: this runs without a GPU)."""
import ctypes
import os
import re

import paper_2409_16560_b200 as dsbd
from paper_2409_16560_b200 import binding

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _declared():
    text = open(os.path.join(ROOT, "include", "dsbd.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(dsbd_[a-z_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported():
    lib = dsbd.load()
    names = _declared()
    assert set(binding.EXPORTS) <= set(names)
    for n in names:
        assert hasattr(lib, n), n
        assert isinstance(getattr(lib, n), ctypes._CFuncPtr)


def test_status_strings_and_workspace_queries_without_a_device():
    assert dsbd.status_string(0) == "ok"
    assert "workspace" in dsbd.status_string(-3)
    lib = dsbd.load()
    f = binding.ForestT()
    p = binding.VerifyParamsT()
    assert lib.dsbd_verify_workspace(ctypes.addressof(f), ctypes.addressof(p)) == 0   # invalid -> 0


def test_no_cpu_fallback():
    import numpy as np
    import pytest
    import torch
    arrays = dict(R=1, B=1, N=1, max_depth=0, req_beam_off=[0, 1], beam_node_off=[0, 1], parent=[-1], token=[0])
    f = dsbd.Forest(arrays, "cpu")
    z = torch.zeros(1, 8)
    out = dsbd.alloc_verify_out(f, np.array([0, 1]), "cpu")
    with pytest.raises(RuntimeError):
        dsbd.verify_step(f, dict(V=8), z, z, torch.zeros(1), torch.zeros(1), out)


def test_header_is_plain_c(tmp_path):
    """include/dsbd.h is a C header: a C99 compiler accepts it with warnings as errors."""
    import shutil
    import subprocess
    import pytest
    if shutil.which("gcc") is None:
        pytest.skip("no C compiler")
    src = tmp_path / "use_header.c"
    src.write_text('#include "dsbd.h"\n'
                   "int main(void) { dsbd_forest_t f; dsbd_verify_params_t p; dsbd_commit_params_t c;\n"
                   "  (void)f; (void)p; (void)c; return dsbd_status_string(0) == 0; }\n")
    subprocess.run(["gcc", "-std=c99", "-Wall", "-Wextra", "-pedantic", "-Werror", "-fsyntax-only",
                    "-I", os.path.join(ROOT, "include"), str(src)], check=True)


def test_forest_depths_match_a_plain_walk():
    """The binding computes node depths (they size the verification's launches) with array
    operations; a plain walk over the parent array must agree on random trees."""
    import numpy as np
    from paper_2409_16560_b200.binding import _node_depths
    rng = np.random.default_rng(0)
    for _ in range(100):
        n = int(rng.integers(1, 400))
        parent = np.array([-1] + [int(rng.integers(-1, i)) for i in range(1, n)])
        ref = np.zeros(n, np.int64)
        for i, p in enumerate(parent):
            ref[i] = 0 if p < 0 else ref[p] + 1
        assert np.array_equal(_node_depths(parent), ref)


def test_the_current_stream_without_torch_s_raw_calls(monkeypatch):
    """A torch without the raw calls is asked for its Stream object."""
    import types
    import torch
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=11))
    assert binding._stream_reader(types.SimpleNamespace())(None) == 11
    raw = types.SimpleNamespace(_cuda_getCurrentRawStream=lambda device: 70 + device, _cuda_getDevice=lambda: 2)
    for reader in (binding._stream_reader(types.SimpleNamespace()), binding._stream_reader(raw)):
        assert reader(types.SimpleNamespace(cuda_stream=5)) == 5
    assert binding._stream_reader(raw)(None) == 72


def test_a_merge_record_that_nobody_wrote_names_no_unit():
    """Records of cut attention units: tail, head_ends, g, rb, n_lo, n_tree.  N = 1000 nodes, 8 heads."""
    from paper_2409_16560_b200 import build
    lib = ctypes.CDLL(build.build_wait_test())
    ok = lambda *rec: bool(lib.dsbd_test_names_unit((ctypes.c_int32 * 8)(*rec), 1000, 8))
    big = 2 ** 31 - 1
    for n_lo, n_tree in [(0, 1), (999, 1), (936, 64), (0, 64), (1000, 0)]:
        assert ok(1, 0, 7, 2, n_lo, n_tree)
    for n_lo, n_tree in [(big, 1), (big, 64), (big - 63, 64), (1000, 1), (937, 64), (-1, 1), (-big - 1, 64), (0, 65), (0, -1),
                         (0, -big - 1), (0x11111111, 0x11111111), (big, -1)]:
        assert not ok(1, 0, 7, 2, n_lo, n_tree), (n_lo, n_tree)
    assert not ok(1, 0, 8, 2, 0, 1) and not ok(1, 0, -1, 2, 0, 1) and not ok(1, 0, 7, 65, 0, 1) and not ok(1, 0, 7, -1, 0, 1)


def _verify_shape(R, rows, V, top_k):
    f = binding.ForestT(R, R, R, 1, 1, 1, 1, 1, 0, 1, rows, rows)          # (the pointers are not followed)
    return f, binding.VerifyParamsT(V=V, temperature=1.0, thresh=0.7, W_min=1, W_max=1, W_nom=1, top_k=top_k, top_p=1.0)


def test_cluster_sizes_without_a_device_s_answer():
    """148 SMs of two CTAs over the cluster's size, and no clusters of 16, which not every device takes."""
    import pytest
    import torch
    if torch.cuda.is_available():
        pytest.skip("the device answers")
    lib = dsbd.load()
    resident = ctypes.c_int32()
    for top_k in (0, 10):
        for R, ctas in [(1, 8), (37, 8), (38, 4), (74, 4), (75, 2), (148, 2), (149, 1), (5000, 1)]:
            f, p = _verify_shape(R, 6, 16384, top_k)
            assert lib.dsbd_verify_cluster_ctas(ctypes.addressof(f), ctypes.addressof(p), ctypes.addressof(resident)) == ctas
            assert resident.value == 296 // ctas
    f, p = _verify_shape(0, 6, 16384, 0)
    assert lib.dsbd_verify_cluster_ctas(ctypes.addressof(f), ctypes.addressof(p), None) == 0


def test_every_time_stamp_of_the_verification_has_a_name():
    import bench
    text = open(os.path.join(ROOT, "paper_2409_16560_b200", "csrc", "dsbd_verify.cu")).read()
    assert {int(x) for x in re.findall(r"\bTS\((\d+)\)", text)} == set(bench.PHASE_NAMES)
