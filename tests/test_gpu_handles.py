"""Gauge handles made and destroyed next to other work: while a stream of
another thread captures, while another thread solves (the solver captures
graphs of its own), and in the caller's memory."""
import threading

import numpy as np
import pytest
import torch

import oracle as O
from paper_1311_4521_gb300 import fields as F

pytestmark = pytest.mark.gpu
DIMS = (8, 8, 8, 8)
VH = 8 ** 4 // 2


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def in_thread(work):
    failed = []

    def body():
        try:
            work()
        except Exception as e:
            failed.append(e)

    t = threading.Thread(target=body)
    t.start()
    return t, failed


def test_handles_come_and_go_while_another_stream_captures():
    from paper_1311_4521_gb300 import tmhop
    c, other = tmhop.Context(0), tmhop.Context(0)
    U, psi = F.gauge_field(DIMS, 970, "random"), F.gaussian_spinor(VH, 970, 1)
    g, Ud = c.gauge(DIMS, U, "f32", 12), tmhop._as_real_dev(U, c.device)
    a, out = c.pack(psi, "f32"), c.empty(VH, "f32").zero_()
    c.Qtm(g, out, a, 0.16, 0.01)
    mine = torch.cuda.Stream()
    torch.cuda.synchronize()

    def handles():
        for prec in (tmhop.TM_F64, tmhop.TM_F32, tmhop.TM_F64):
            for _ in range(3):
                h = tmhop.tm_gauge_create(other.handle, DIMS, Ud, prec, 18, (-1, 1, 1, 1), mine)
                tmhop.tm_gauge_destroy(h)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="thread_local"):
        t, failed = in_thread(handles)
        t.join()
        c.Qtm(g, out, a, 0.16, 0.01)
    assert not failed, failed
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert rel(c.unpack(out, VH, "f32").cpu().numpy(), O.Qtm(DIMS, U, psi, 0.16, 0.01)) < 1e-6
    g.close()
    c.close()
    other.close()


def test_handles_come_and_go_while_another_thread_solves():
    from paper_1311_4521_gb300 import tmhop
    c, other = tmhop.Context(0), tmhop.Context(0)
    U, psi = F.gauge_field(DIMS, 971, "near", 0.3), F.gaussian_spinor(VH, 971, 1)
    g, lo, Ud = c.gauge(DIMS, U, "f64", 18), c.gauge(DIMS, U, "f32", 12), tmhop._as_real_dev(U, c.device)
    b, mine = c.pack(psi, "f64"), torch.cuda.Stream()
    torch.cuda.synchronize()
    stop = threading.Event()

    def handles():
        while not stop.is_set():
            tmhop.tm_gauge_destroy(tmhop.tm_gauge_create(other.handle, DIMS, Ud, tmhop.TM_F32, 18, (-1, 1, 1, 1), mine))

    t, failed = in_thread(handles)
    try:
        for _ in range(30):
            x = c.empty(VH, "f64").zero_()
            st, info = c.cg(g, x, b, 0.12, 0.05, 1e-9, 1000, lo)
            assert st == tmhop.TM_OK and info["true_relres"] <= 1e-9
    finally:
        stop.set()
        t.join()
    assert not failed, failed
    for h in (g, lo):
        h.close()
    c.close()
    other.close()


@pytest.mark.parametrize("prec,recon,tol", [("f64", 18, 1e-13), ("f64", 12, 1e-13), ("f64x", 18, 1e-13), ("f32", 12, 1e-6),
                                            ("f16", 12, 5e-3)])
def test_links_in_the_callers_memory(prec, recon, tol):
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    U, psi = F.gauge_field(DIMS, 972, "random"), F.gaussian_spinor(VH, 972, 1)
    P, bc, Ud = tmhop.PREC[prec], (-1, 1, 1, 1), tmhop._as_real_dev(U, c.device)
    n = tmhop.tm_gauge_storage_bytes(DIMS, P, recon)
    own = c.gauge(DIMS, U, prec, recon)
    a, want = c.pack(psi, prec), O.Qtm(DIMS, U, psi, 0.16, 0.01)
    ref = c.Qtm(own, c.empty(VH, prec), a, 0.16, 0.01)
    links = 8 * VH * {"f64": 8, "f64x": 8, "f32": 4, "f16": 2}[prec] * recon
    for size in (n, links):   # with the FP64 handle's fixed-point copy, and with its links alone
        mem = torch.full((n + 256,), 0xA5, dtype=torch.uint8, device=c.device)
        h = tmhop.tm_gauge_create_in(c.handle, DIMS, Ud, P, recon, bc, mem, size)
        out = c.empty(VH, prec)
        tmhop.tm_Qtm(c.handle, h, out, a, 0.16, 0.01)
        if size == n:
            assert torch.equal(out, ref) and tmhop.tm_gauge_bytes(h) == own.nbytes
        assert rel(c.unpack(out, VH, prec).cpu().numpy(), want) < tol
        assert bool((mem[size:] == 0xA5).all())   # nothing written past what was given
        tmhop.tm_gauge_destroy(h)
    for args in ((mem, links - 1), (mem[8:], n), (None, n)):
        with pytest.raises(tmhop.TmError):
            tmhop.tm_gauge_create_in(c.handle, DIMS, Ud, P, recon, bc, *args)
    own.close()
    c.close()


def test_handles_in_torch_memory_on_two_streams():
    """Closed with launches under way, one stream's memory does not go to the other's next handle too early."""
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    U = [torch.from_numpy(F.gauge_field(DIMS, s, "random")).cuda() for s in (973, 974)]
    src = c.pack(F.gaussian_spinor(VH, 973, 1), "f32")
    ref = []
    for u in U:
        g = c.gauge(DIMS, u, "f32", 12)
        ref.append(c.hopping_eo(g, c.empty(VH, "f32"), src, 0).clone())
        g.close()
    torch.cuda.synchronize()
    streams, outs = [torch.cuda.Stream(), torch.cuda.Stream()], [[], []]
    for k in range(40):
        with torch.cuda.stream(streams[k & 1]):
            g = tmhop.Gauge(c, DIMS, U[k & 1], "f32", 12, torch_memory=True)
            outs[k & 1].append(c.hopping_eo(g, c.empty(VH, "f32"), src, 0))
            g.close()
    torch.cuda.synchronize()
    for r, os in zip(ref, outs):
        assert all(torch.equal(r, o) for o in os)
    c.close()


@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (16, 16, 16, 16)])
def test_device_bytes_count_the_fixed_point_scratch(dims):
    from paper_1311_4521_gb300 import tmhop
    c, vh = tmhop.Context(0), int(np.prod(dims)) // 2
    g = c.gauge(dims, F.gauge_field(dims, 975, "near", 0.3), "f64", 18)
    a, out = c.pack(F.gaussian_spinor(vh, 975, 1), "f64"), c.empty(vh, "f64")
    assert tmhop.tm_ctx_device_bytes(c.handle) == 0
    c.Qtm(g, out, a, 0.16, 0.01)
    # two fields of 12 components of 16 bytes and a word a site, by blocks of 32 sites, and nothing else
    assert tmhop.tm_ctx_device_bytes(c.handle) == 2 * vh * (12 * 16 + 4)
    g.close()
    c.close()


def test_fixed_point_copies_can_be_refused_and_leave_room():
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    U, psi = F.gauge_field(DIMS, 976, "random"), F.gaussian_spinor(VH, 976, 1)
    a, want, links = c.pack(psi, "f64"), O.Qtm(DIMS, U, psi, 0.16, 0.01), 8 * VH * 144

    def handle(copies):
        g = c.gauge(DIMS, U, "f64", 18)
        assert g.nbytes == links * (2 if copies else 1)
        assert rel(c.unpack(c.Qtm(g, c.empty(VH, "f64"), a, 0.16, 0.01), VH, "f64").cpu().numpy(), want) < 1e-13
        return g

    handle(True).close()
    tmhop.tm_ctx_set_fixed_point(c.handle, False)
    g = handle(False)
    U_dev, n = tmhop._as_real_dev(U, c.device), tmhop.tm_gauge_storage_bytes(DIMS, tmhop.TM_F64, 18)
    mem = torch.empty(n, dtype=torch.uint8, device=c.device)
    h = tmhop.tm_gauge_create_in(c.handle, DIMS, U_dev, tmhop.TM_F64, 18, (-1, 1, 1, 1), mem, n)
    assert tmhop.tm_gauge_bytes(h) == links
    tmhop.tm_gauge_destroy(h)
    tmhop.tm_ctx_set_fixed_point(c.handle, True)
    handle(True).close()
    free, total = torch.cuda.mem_get_info()
    hold = torch.empty(free - total // 2 + (32 << 20), dtype=torch.uint8, device=c.device)   # less than half is left
    handle(False).close()
    del hold
    torch.cuda.empty_cache()
    handle(True).close()
    g.close()
    c.close()
