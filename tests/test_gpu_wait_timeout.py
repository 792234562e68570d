"""A bounded wait of the tensor-core attention kernels that runs out.

Every mbarrier wait of these kernels gives up after a limit, records DSBD_DEV_TIMEOUT, lets the
copies in flight land, frees its tensor memory and returns.  The product library offers no way
to make a wait run out, so this test builds a second library from the same sources with
DSBD_TEST_WAIT_TIMEOUT: the limit drops to about a millisecond and the copy producer of one CTA
leaves out one tile, whose barrier is then never completed.  Nothing faults and nothing hangs:
the call returns with the status set, the other CTAs finish their work, and the next launch
of the product library on the same context matches the oracle."""
import ctypes as C

import numpy as np
import pytest
import torch

import paper_2409_16560_b200 as dsbd
from paper_2409_16560_b200 import binding as bd
from paper_2409_16560_b200 import build as cuda_build
from paper_2409_16560_b200 import inputs
from parity_util import attention_close, to_host_f32
from test_gpu_attention import _custom, _gpu, _oracle_beams

pytestmark = pytest.mark.gpu

DEV_TIMEOUT = 5


def _wait_library():
    lib = C.CDLL(cuda_build.build_wait_test())
    lib.dsbd_forest_attention_workspace.restype = C.c_size_t
    lib.dsbd_forest_attention_workspace.argtypes = [C.c_void_p, C.c_void_p]
    lib.dsbd_forest_attention.restype = C.c_int
    lib.dsbd_forest_attention.argtypes = [C.c_void_p] * 10 + [C.c_size_t, C.c_void_p, C.c_void_p]
    lib.dsbd_forest_attention_paged_workspace.restype = C.c_size_t
    lib.dsbd_forest_attention_paged_workspace.argtypes = [C.c_void_p] * 3
    lib.dsbd_forest_attention_paged.restype = C.c_int
    lib.dsbd_forest_attention_paged.argtypes = [C.c_void_p] * 11 + [C.c_size_t, C.c_void_p, C.c_void_p]
    return lib


@pytest.mark.parametrize("sizes", [[9, 5, 12, 3], [20, 17, 25, 18], [20, 2, 3, 2]])
def test_a_wait_that_runs_out_sets_the_status_and_leaves_the_context_usable(sizes):
    """Trees of at most 48 query rows: the transposed kernel; of 68 to 100 and of 8 to 80: the 128-row and the 64-row
    instance of the kernel with the rows on the M side (their units are cut: the combination follows)."""
    lib = _wait_library()
    rng = np.random.default_rng(31)
    rand_tree = lambda n: [-1] + [int(rng.integers(0, i)) for i in range(1, n)]
    trees = [rand_tree(n) for n in sizes]
    L = [700, 300, 1000, 200]                              # every unit has several tiles
    forest, spec, t, poff = _custom(rng, trees, L, 8, 2, 128, torch.bfloat16)
    f = dsbd.Forest(forest, "cuda")
    fs = f.struct()
    desc = bd._attn_desc(8, 2, 128, torch.bfloat16, inputs.default_scale(128), poff)
    poff_dev = torch.as_tensor(poff).cuda()
    out = torch.zeros_like(t["q"])
    need = int(lib.dsbd_forest_attention_workspace(C.addressof(fs), C.addressof(desc)))
    ws = torch.zeros(max(need, 256), dtype=torch.uint8, device="cuda")
    for _ in range(2):                                     # (the first launch loads the kernel)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        begin, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        begin.record()
        rc = lib.dsbd_forest_attention(C.addressof(fs), C.addressof(desc), t["q"].data_ptr(), t["k_new"].data_ptr(),
                                       t["v_new"].data_ptr(), t["k_prefix"].data_ptr(), t["v_prefix"].data_ptr(),
                                       poff_dev.data_ptr(), out.data_ptr(), ws.data_ptr(), ws.numel(), status.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        end.record()
        assert rc == 0
        torch.cuda.synchronize()                           # returns: the wait was bounded
        assert int(status.item()) == DEV_TIMEOUT
    # about a millisecond (250 tries of 4 us, or 2e6 cycles) for the tile, and again for the copies in flight.  The
    # product library's limits are 1000 and 2000 times these: a second or two
    assert begin.elapsed_time(end) < 8.0
    assert "wait" in dsbd.status_string(DEV_TIMEOUT)
    # the CTAs whose tiles all arrived did their work: the last tree's rows are right
    nodes, ref = _oracle_beams(forest, spec, t, poff, list(range(len(trees))))
    bno = forest["beam_node_off"]
    last = slice(int(bno[-2]), int(bno[-1]))
    attention_close(to_host_f32(out[last]), ref[last], bf16=True)
    # the context is intact (tensor memory freed, no copy left in flight): the product library's
    # next launch on the same device gives the full, correct result
    good = _gpu(forest, spec, t, poff)
    attention_close(to_host_f32(good), ref, bf16=True)


def test_a_wait_that_runs_out_in_a_call_of_several_layers_with_cut_units():
    """The run of CTA 0 stops in the first layer.  Its records of the layers it never reached are empty, so
    that the merge, which runs over all layers, takes no unit from them; rows of other runs are right in all layers."""
    lib = _wait_library()
    runs = torch.cuda.get_device_properties(0).multi_processor_count
    R, L, Hq, Hkv, n_layers = 8, 10000, 8, 2, 3
    # 16 units of 80 tiles a layer: a run for every SM, units cut into about 9
    sizes = [9] * R
    bno = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    parent = np.concatenate([[-1] + list(range(b, b + 8)) for b in bno[:-1]]).astype(np.int32)
    forest = dict(R=1, B=R, N=int(bno[-1]), max_depth=8, req_beam_off=np.array([0, R], np.int32), beam_node_off=bno,
                  parent=parent, token=np.zeros(int(bno[-1]), np.int32))
    f = dsbd.Forest(forest, "cuda")
    poff = (L * np.arange(R + 1)).astype(np.int64)
    per = -(-L // 64)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    mk = lambda *s: torch.randn(*s, generator=g, device="cuda").to(torch.bfloat16)
    q, kn, vn = mk(n_layers, f.N, Hq, 128), mk(n_layers, f.N, Hkv, 128), mk(n_layers, f.N, Hkv, 128)
    kp, vp = mk(n_layers, R * per, Hkv, 64, 128), mk(n_layers, R * per, Hkv, 64, 128)
    table = torch.arange(R * per, dtype=torch.int32, device="cuda")
    page_off, poff_dev = (torch.as_tensor(x).cuda() for x in (per * np.arange(R + 1), poff))
    scale = inputs.default_scale(128)
    ref, status = dsbd.forest_attention_paged(f, Hq, Hkv, 128, scale, q, kn, vn, kp, vp, table, page_off, poff_dev, poff)
    assert int(status.item()) == 0
    fs, desc, pages = f.struct(), bd._attn_desc(Hq, Hkv, 128, torch.bfloat16, scale, poff), bd.KvPagesT()
    pages.page_table, pages.page_off, pages.n_pages = table.data_ptr(), page_off.data_ptr(), R * per
    pages.n_layers = n_layers
    pages.pool_layer_stride, pages.new_layer_stride, pages.q_layer_stride = kp.stride(0), kn.stride(0), q.stride(0)
    need = int(lib.dsbd_forest_attention_paged_workspace(*(C.addressof(x) for x in (fs, desc, pages))))
    assert need > 32 * runs * n_layers                     # records and partial results: units are cut
    ws = torch.full((need,), 0x11, dtype=torch.uint8, device="cuda")
    out = torch.zeros_like(q)
    rc = lib.dsbd_forest_attention_paged(C.addressof(fs), C.addressof(desc), *(x.data_ptr() for x in (q, kn, vn, kp, vp)),
                                         C.addressof(pages), poff_dev.data_ptr(), out.data_ptr(), ws.data_ptr(), need,
                                         status.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    assert int(status.item()) == DEV_TIMEOUT
    recs = ws[:32 * runs * n_layers].view(torch.int32).view(n_layers, runs, 8).cpu().numpy()
    assert (recs[1:, 0] == 0).all()
    assert np.isin(recs[..., :2], (0, 1)).all() and (recs[..., 2] < R).all() and (recs[..., 3] < Hkv).all()
    assert torch.equal(out[:, int(bno[-2]):], ref[:, int(bno[-2]):])          # the last beam
    again, status = dsbd.forest_attention_paged(f, Hq, Hkv, 128, scale, q, kn, vn, kp, vp, table, page_off, poff_dev, poff)
    assert int(status.item()) == 0 and torch.equal(again, ref)
