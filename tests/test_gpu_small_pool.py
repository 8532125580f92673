"""A handle in a device pool that does not hold the whole face buffer: it takes
half of it and updates what it leaves out in one pass, with the same bits, and
what is allocated later still fits."""
import contextlib
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

USED_HIGH = 8                                    # CU_MEMPOOL_ATTR_USED_MEM_HIGH


class _Location(C.Structure):
    _fields_ = [("type", C.c_int), ("id", C.c_int)]


class _Props(C.Structure):
    _fields_ = [("allocType", C.c_int), ("handleTypes", C.c_int), ("location", _Location),
                ("win32", C.c_void_p), ("maxSize", C.c_size_t), ("usage", C.c_ushort),
                ("reserved", C.c_ubyte * 54)]


def _ok(r):
    assert r == 0, r


@contextlib.contextmanager
def pool(limit):
    """The device's pool replaced by one of at most `limit` bytes (0: no limit)."""
    import torch
    torch.zeros(1, device="cuda")
    cu = C.CDLL("libcuda.so.1")
    old, new = C.c_void_p(), C.c_void_p()
    _ok(cu.cuDeviceGetMemPool(C.byref(old), 0))
    pr = _Props(allocType=1, handleTypes=0, location=_Location(1, 0), maxSize=limit)
    _ok(cu.cuMemPoolCreate(C.byref(new), C.byref(pr)))
    _ok(cu.cuDeviceSetMemPool(0, new))

    def used():
        v = C.c_uint64()
        _ok(cu.cuMemPoolGetAttribute(new, USED_HIGH, C.byref(v)))
        return v.value

    try:
        yield used
    finally:
        _ok(cu.cuDeviceSetMemPool(0, old))
        torch.cuda.synchronize()
        _ok(cu.cuMemPoolDestroy(new))


def _case(L, matched=False):
    p, f = synth.bumpy_dam_break(L=L, eps=0.0, seed=5)        # every finest cell a leaf, most of them wet
    return dict(p, flux_match=matched), f


def _run(p, f, uniform):
    from paper_2206_05761_gb300.sim import Simulation
    sim = Simulation(p, f)
    sim.advance(max_steps=2)
    if uniform:
        sim.advance_uniform(max_steps=2)
        sim.advance(max_steps=18)
    out = sim.fields(), sim.time(), sim.counters()[:4]
    sim.close()
    return out


def _same(a, b):
    for q in ("h", "qx", "qy"):
        assert np.array_equal(a[0][q], b[0][q]), q
    assert a[1:] == b[1:]


FULL = 192                                       # bytes of face buffer per finest cell


@pytest.mark.parametrize("matched", [False, True])
def test_a_handle_with_half_the_face_buffer(matched):
    L = 11
    p, f = _case(L, matched)
    with pool(0) as used:
        ref = _run(p, f, uniform=True)
        need = used()
    n = 1 << (2 * L)
    assert need > FULL * n
    # all but a third of the buffer: the whole of it does not fit, half of it does
    with pool(need - FULL * n // 3) as used:
        _same(_run(p, f, uniform=True), ref)
        assert used() <= need - FULL * n // 3


def test_a_later_allocation_takes_half_of_the_buffer():
    L = 11
    p, f = _case(L)
    with pool(0) as used:
        ref = _run(p, f, uniform=True)
        need = used()
    # the handle fits whole, the uniform steps' list of leaves (4 bytes a cell) does not
    with pool(need - 2 * (1 << (2 * L))):
        _same(_run(p, f, uniform=True), ref)


def test_a_batch_with_half_the_face_buffers():
    from paper_2206_05761_gb300.sim import Ensemble
    L, D = 10, 4
    cases = [_case(L) for _ in range(D)]

    def run():
        e = Ensemble(cases)
        e.advance(max_steps=3)
        out = [(e.member_fields(d), e.member_time(d)) for d in range(D)]
        e.close()
        return out

    with pool(0) as used:
        ref = run()
        need = used()
    with pool(need - D * FULL * (1 << (2 * L)) // 3):
        for a, b in zip(run(), ref):
            _same(a, b)


def test_a_member_takes_half_of_its_buffer_after_the_batch_was_planned():
    import paper_2206_05761_gb300.hwfv1 as H
    from paper_2206_05761_gb300.sim import Ensemble
    L, D = 10, 3
    cases = [_case(L) for _ in range(D)]

    def run():
        e = Ensemble(cases)
        e.advance(max_steps=2)
        # the uniform steps' list (4 bytes a cell each) is allocated on first use
        for d in range(D):
            H.hwfv1_advance_uniform(H.hwfv1_batch_member(e.bt, d), float("inf"), 1)
        e.advance(max_steps=2)
        out = [(e.member_fields(d), e.member_time(d)) for d in range(D)]
        e.close()
        return out

    with pool(0) as used:
        ref = run()
        need = used()
    with pool(need - 2 * (1 << (2 * L))):
        for a, b in zip(run(), ref):
            _same(a, b)


def test_too_small_a_pool_is_refused():
    import paper_2206_05761_gb300.hwfv1 as H
    from paper_2206_05761_gb300.sim import Simulation
    L = 11
    p, f = _case(L)
    with pool(64 << 20):
        with pytest.raises(H.Hwfv1Error) as e:
            Simulation(p, f)
        assert e.value.status == 2                # HWFV1_ERR_OOM
