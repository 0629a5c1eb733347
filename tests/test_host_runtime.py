"""Host code of the library on a CUDA runtime that runs nothing
(fake_cudart.cpp): what launches ask for and what they share, without a GPU."""
import ctypes
import glob
import os
import re
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_2606_15991_gb300 as tp
from paper_2606_15991_gb300 import _lib, build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host_path(built_lib, tmp_path_factory):
    """libtp linked with the fake runtime."""
    out = tmp_path_factory.mktemp("host")
    obj, so = str(out / "fake.o"), str(out / "libtp_host.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-I" + inc, "-c", os.path.join(HERE, "fake_cudart.cpp"),
                    "-o", obj], check=True)
    subprocess.run([build.nvcc(), "-shared", "--cudart", "none", "-Xlinker", "-Bsymbolic", "-o", so, obj] +
                   sorted(glob.glob(os.path.join(build.BUILD, "*.o"))), check=True)
    return so


@pytest.fixture
def host(host_path, monkeypatch):
    L = ctypes.CDLL(host_path)
    for name, args in _lib._PROTOS.items():
        f = getattr(L, name)
        f.argtypes, f.restype = args, _lib._RESTYPES.get(name, ctypes.c_int32)
    monkeypatch.setattr(_lib, "_lib", L)
    for which in range(3):
        L.fake_seen(which, None, ctypes.c_int64(0))
    yield L
    L.fake_finish()


S1, S2 = 0x100, 0x200  # streams


def _exec(mode=_lib.SYNC, stream=S1, event=None):
    return tp.make_exec(mode, stream, event)


def test_shared_memory_limits_are_never_lowered(host):
    """A kernel's dynamic shared-memory limit belongs to the process: a launch
    that set it to its own size would fail a larger launch of another thread
    made between that thread's set and its launch."""
    ctx = tp.tp_ctx_create(0)
    for m, n, split in ((512, 512, 2), (1024, 512, 4), (512, 512, 4), (2048, 2048, 2), (64, 64, 2)):
        a, b, c = torch.zeros(m, 64), torch.zeros(64, n), torch.zeros(m, n)
        p = tp.tp_partition_create(ctx, c, (64, 64))
        tp.tp_gemm(ctx, p, a, b, tp.gemm_config(split_k=split), _exec())
        tp.tp_partition_destroy(p)
    for hidden in (160, 96, 128):
        m = tp.tp_mlp_create(ctx, 5, hidden, 72, 4, np.zeros(5 * hidden + hidden * hidden + 74 * hidden + 72, np.float32))
        tp.tp_mlp_forward(m, torch.zeros(4, 5), torch.zeros(4, 72), _exec())
        tp.tp_mlp_destroy(m)
    for k in (40000, 16384, 24576, 512, 20480):
        buf = torch.zeros(k + 8)
        at = -buf.data_ptr() // 4 % 4
        for off in (at, at + 1):      # streamed, where it fits, and per lane
            w, x, y = torch.zeros(256, k, dtype=torch.bfloat16), buf[off:off + k], torch.zeros(256)
            p = tp.tp_partition_create(ctx, y, (256,))
            tp.tp_gemv(ctx, p, w, x, _exec())
            tp.tp_decode_down_residual(ctx, p, w, x, _exec())
            tp.tp_partition_destroy(p)
    tp.tp_ctx_destroy(ctx)
    assert host.fake_lowered() == 0


def _wait_op(ctx, ok, ex):
    """An operation without an output partition whose kernel gives up (or not)."""
    tp.tp_diag_bounded_wait(ctx, 1_000_000, ok, ex)


def _times_out(event):
    with pytest.raises(tp.TPError) as e:
        tp.tp_event_wait(event)
    return e.value.status == _lib.ERR_TIMEOUT


def test_event_destroyed_in_flight_keeps_its_word(host):
    ctx = tp.tp_ctx_create(0)
    ev = tp.tp_event_create(ctx)
    _wait_op(ctx, False, _exec(tp.ASYNC, S1, ev))
    tp.tp_event_destroy(ev)
    fresh = tp.tp_event_create(ctx)
    _wait_op(ctx, True, _exec(tp.ASYNC, S2, fresh))
    host.fake_finish()
    tp.tp_event_wait(fresh)      # not the first event's late timeout
    tp.tp_event_destroy(fresh)
    tp.tp_ctx_destroy(ctx)


def test_graph_destroyed_in_flight_keeps_its_word(host):
    ctx = tp.tp_ctx_create(0)
    replay, fresh = tp.tp_event_create(ctx), None
    g = tp.tp_graph_begin(ctx, S1)
    _wait_op(ctx, False, _exec(tp.CAPTURE, S1))
    tp.tp_graph_end(g)
    tp.tp_graph_replay(g, _exec(tp.ASYNC, S1, replay))
    tp.tp_graph_destroy(g)
    fresh = tp.tp_event_create(ctx)
    _wait_op(ctx, True, _exec(tp.ASYNC, S2, fresh))
    host.fake_finish()
    tp.tp_event_wait(fresh)
    assert _times_out(replay)
    for ev in (replay, fresh):
        tp.tp_event_destroy(ev)
    tp.tp_ctx_destroy(ctx)


def test_any_number_of_events_report_their_own_errors(host):
    ctx = tp.tp_ctx_create(0)
    events = [tp.tp_event_create(ctx) for _ in range(5000)]
    for i, ev in enumerate(events):
        _wait_op(ctx, i % 2 == 0, _exec(tp.ASYNC, S1, ev))
    host.fake_finish()
    for i, ev in enumerate(events):
        assert i % 2 == 0 or _times_out(ev)
        tp.tp_event_wait(ev)
    _wait_op(ctx, True, _exec())
    for ev in events:
        tp.tp_event_destroy(ev)
    tp.tp_ctx_destroy(ctx)
    assert host.fake_hosts() == 0


def test_events_and_graphs_outlive_their_context(host_path):
    """In a process whose allocator overwrites what is freed."""
    child = f"""
import ctypes
L = ctypes.CDLL({host_path!r})
V = ctypes.c_void_p
ctx, ev, used, g = V(), V(), V(), V()
class Exec(ctypes.Structure):
    _fields_ = [("mode", ctypes.c_int32), ("flags", ctypes.c_int32)] + [(n, V) for n in "seco"]
def ok(st): assert st == 0, st
ok(L.tp_ctx_create(0, ctypes.byref(ctx)))
ok(L.tp_event_create(ctx, ctypes.byref(ev)))
ok(L.tp_event_create(ctx, ctypes.byref(used)))
ok(L.tp_graph_begin(ctx, V(0x100), ctypes.byref(g)))
ok(L.tp_graph_end(g))
ok(L.tp_diag_bounded_wait(ctx, ctypes.c_int64(1000000), 0, ctypes.byref(Exec(1, 0, 0x100, used.value))))
ok(L.tp_ctx_destroy(ctx))
ok(L.tp_event_destroy(ev))
ok(L.tp_graph_destroy(g))
assert L.tp_event_wait(used) == {_lib.ERR_TIMEOUT}
ok(L.tp_event_destroy(used))
assert L.fake_hosts() == 0
"""
    subprocess.run([sys.executable, "-c", child], check=True, timeout=120,
                   env={**os.environ, "MALLOC_PERTURB_": "165"})


def _down(ctx, h, p, ex, ni=16384):
    """A down projection over K slices: partial sums, and a finish kernel."""
    tp.tp_decode_down_residual(ctx, p, torch.zeros(h.numel(), ni, dtype=torch.bfloat16), torch.zeros(ni), ex)


def _addresses(host, which):
    out = (ctypes.c_uint64 * 4096)()
    n = host.fake_seen(which, out, ctypes.c_int64(4096))
    return list(out[:n])


def test_partial_sums_of_work_in_flight_do_not_share_a_buffer(host):
    ctx = tp.tp_ctx_create(0)
    hs = [torch.zeros(64) for _ in range(4)]
    ps = [tp.tp_partition_create(ctx, h, (64,)) for h in hs]
    g = tp.tp_graph_begin(ctx, S1)
    for _ in range(2):
        _down(ctx, hs[0], ps[0], _exec(tp.CAPTURE, S1))
    tp.tp_graph_end(g)
    graph = set(_addresses(host, 0))
    assert len(graph) == 1
    evs = [tp.tp_event_create(ctx) for _ in range(3)]
    seen = set()
    for _ in range(50):
        tp.tp_graph_replay(g, _exec(tp.ASYNC, S1, evs[0]))
        for i in (1, 2):
            _down(ctx, hs[i], ps[i], _exec(tp.ASYNC, S2 + i, evs[i]))
        _down(ctx, hs[3], ps[3], _exec(tp.SYNC, S2))
        now = _addresses(host, 0)
        assert len(set(now)) == 3 and not graph & set(now)
        seen |= set(now)
        for ev in evs:
            tp.tp_event_wait(ev)
    assert len(seen) == 3   # reused, not one for each operation
    for ev in evs:
        tp.tp_event_destroy(ev)
    tp.tp_graph_destroy(g)
    for p in ps:
        tp.tp_partition_destroy(p)
    tp.tp_ctx_destroy(ctx)


def test_tile_queues_of_work_in_flight_do_not_share_a_counter(host):
    ctx = tp.tp_ctx_create(0)
    x, z = torch.zeros(4096), [torch.zeros(4096) for _ in range(3)]
    ps = [tp.tp_partition_create(ctx, t, (512,)) for t in z]
    for p in ps:
        tp.tp_partition_map(p, _lib.MAP_QUEUE, 3)

    def run(i, ex):
        tp.tp_map_scale(ctx, ps[i], x, x, ex)

    g = tp.tp_graph_begin(ctx, S1)
    run(0, _exec(tp.CAPTURE, S1))
    tp.tp_graph_end(g)
    graph = _addresses(host, 1)
    ev = tp.tp_event_create(ctx)
    for _ in range(600):
        run(1, _exec(tp.ASYNC, S2, ev))
        run(2, _exec(tp.SYNC, S1))
        now = _addresses(host, 1)
        assert len(now) == 2 and len(set(now + graph)) == 3
        tp.tp_event_wait(ev)
    tp.tp_event_destroy(ev)
    tp.tp_graph_destroy(g)
    for p in ps:
        tp.tp_partition_destroy(p)
    tp.tp_ctx_destroy(ctx)


def test_mlp_outputs_over_their_input_are_copied_out_last(host):
    """An output that overlaps X is written when nothing reads X any more."""
    f, h, c, b = 9, 8, 4, 6
    ctx = tp.tp_ctx_create(0)
    m = tp.tp_mlp_create(ctx, f, h, c, b, np.zeros(f * h + h * h + h * c + 2 * h + c, np.float32))
    buf, t, loss = torch.zeros(400), torch.zeros(b, c), torch.zeros(1)
    x = buf[:b * f].view(b, f)
    for at in (0, 10, b * f - 1, b * f):
        y = buf[at:]
        want = [y.data_ptr()] if at < b * f else []
        tp.tp_mlp_forward(m, x, y, _exec())
        assert _addresses(host, 2) == want
        tp.tp_mlp_loss_grad(m, x, t, t, loss, y, _exec())
        assert _addresses(host, 2) == want
    tp.tp_mlp_destroy(m)
    tp.tp_ctx_destroy(ctx)


def test_counted_fp32_products_run_the_kernel_of_the_uncounted(host):
    """Write counts are evidence for the kernel that the operands' layout picks."""
    host.fake_last_kernel.restype = ctypes.c_char_p

    def form():      # fetch of A, fetch of B, split
        return re.search(rb"gemm_f32_kernelILi(\d)ELi(\d)ELb(\d)E", host.fake_last_kernel()).groups()

    ctx = tp.tp_ctx_create(0)
    m, n, k = 70, 66, 40
    c = torch.zeros(m, n)
    p = tp.tp_partition_create(ctx, c, (64, 64))
    counts = torch.zeros(m * n, dtype=torch.int32)

    def layouts(r, cols):
        buf = torch.zeros(r * 80 + 8)
        at = -buf.data_ptr() // 4 % 4
        yield buf[at:].as_strided((r, cols), (80, 1))
        yield buf[at + 1:].as_strided((r, cols), (80, 1))
        yield torch.zeros(cols, r).t()

    seen = set()
    for split in (1, 2):
        for a in layouts(m, k):
            for b in layouts(k, n):
                tp.tp_gemm(ctx, p, a, b, tp.gemm_config(split_k=split), _exec())
                plain = form()
                tp.tp_gemm(ctx, p, a, b, tp.gemm_config(split_k=split),
                           tp.make_exec(stream=S1, write_counts=counts, write_owner=counts))
                assert form() == plain
                seen.add(plain)
    assert len(seen) == 18
    tp.tp_partition_destroy(p)
    tp.tp_ctx_destroy(ctx)


def test_gemv_of_overlapping_rows_takes_no_tensor_map(host):
    host.fake_last_kernel.restype = ctypes.c_char_p
    ctx = tp.tp_ctx_create(0)
    rows, k = 256, 1024
    buf = torch.zeros(rows * k + 8, dtype=torch.bfloat16)
    buf = buf[-(buf.data_ptr() // 2) % 8:]
    xb = torch.zeros(k + 4)
    x, y = xb[-(xb.data_ptr() // 4) % 4:][:k], torch.zeros(rows)
    p = tp.tp_partition_create(ctx, y, (rows,))
    for stride, kernel in ((k, b"gemv_stream_kernel"), (8, b"gemv_kernel"), (0, b"gemv_kernel")):
        tp.tp_gemv(ctx, p, buf.as_strided((rows, k), (stride, 1)), x, _exec())
        assert kernel in host.fake_last_kernel()
    tp.tp_partition_destroy(p)
    tp.tp_ctx_destroy(ctx)
