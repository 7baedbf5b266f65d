"""The native marshalling of the per-request calls hands the library the same records ctypes would."""
import ctypes as C

import numpy as np
import pytest

from paper_2409_13761_b200 import kdn

pytestmark = pytest.mark.skipif(kdn._native is None, reason="no C compiler or no Python headers")


def records(n):
    return [kdn.XferOp(4096 + i, 7 + i, (1 << 33) + i, kdn.Chunk((1 << 63) + 16 * i, (1 << 40) + i, 5 + i, i % 7, i & 1, -3 - i)) for i in range(n)]


def same_bytes(p, n, record, want):
    assert C.string_at(p, n * C.sizeof(record)) == bytes(want)[:n * C.sizeof(record)]


@pytest.mark.parametrize("n", [0, 1, 16, 17, 300])
def test_transfers(n):
    ops, seen = records(n), []

    @C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p)
    def entry(ctx, pool, p, count, stream, side):
        seen.append((ctx, pool, count, stream, side))
        same_bytes(p, count, kdn.kdn_xfer_op, kdn.xfer_array(ops))
        return 4

    for ctx in (C.c_void_p(0x1230), 0x1230):
        assert kdn._native.call_xfer(C.cast(entry, C.c_void_p).value, ctx, 3, ops, 0x77, None) == 4
    assert seen == [(0x1230, 3, n, 0x77, None)] * 2

    keeps = [0x9000 + i for i in range(n)]

    @C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p)
    def sparse(ctx, pool, p, count, stream, side):
        same_bytes(p, count, kdn.kdn_sparse_op, kdn.sparse_array(ops, keeps))
        return count % 5

    assert kdn._native.call_sparse(C.cast(sparse, C.c_void_p).value, None, 0, tuple(ops), keeps, 0, 0) == n % 5


@pytest.mark.parametrize("n,parts", [(0, 0), (1, 0), (1, 10), (3, 6), (20, 2)])
def test_requests(n, parts):
    reqs = [kdn.ComposeReq(64 * i, 9, [o.chunk for o in records(parts)], list(np.arange(parts) * 100 + i), 5e5 + i, i & 1) for i in range(n)]

    @C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p)
    def entry(ctx, pool, p, count, stream, side):
        got, want = C.cast(p, C.POINTER(kdn.kdn_compose_req)), kdn.compose_array(reqs)
        assert count == n
        for i in range(n):
            a, b = got[i], want[i]
            for f in ("block_table", "n_table_blocks", "n_parts", "rope_theta", "rope_style", "reserved"):
                assert getattr(a, f) == getattr(b, f)
            same_bytes(a.parts, parts, kdn.kdn_chunk, C.string_at(b.parts, parts * C.sizeof(kdn.kdn_chunk)))
            assert [a.part_dst_pos[j] for j in range(parts)] == [b.part_dst_pos[j] for j in range(parts)]
        return 0

    assert kdn._native.call_compose(C.cast(entry, C.c_void_p).value, 8, 0, reqs, 0, 0) == 0


def test_selects():
    reqs = [kdn.ComposeReq(64, 9, [o.chunk for o in records(k)], list(range(k)), 1e4) for k in (3, 0, 20)]
    selects = [[None, (0x5000, 7), None], [], [(0x6000 + j, j) if j % 2 else None for j in range(20)]]

    @C.CFUNCTYPE(C.c_int, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p)
    def entry(ctx, pool, p, sel, count, stream, side):
        got = C.cast(sel, C.POINTER(kdn.kdn_select))
        assert count == 3 and (ctx, pool, stream, side) == (8, 1, 2, 3)
        for r, want in enumerate(selects):
            for j, w in enumerate(want):
                assert (got[r].part_select[j], got[r].part_n_select[j]) == (w if w else (None, 0))
        return 0

    assert kdn._native.call_compose_select(C.cast(entry, C.c_void_p).value, 8, 1, reqs, selects, 2, 3) == 0
    with pytest.raises(ValueError):
        kdn._native.call_compose_select(0, 8, 1, reqs, selects[:2], 2, 3)


def test_bad_arguments_raise_and_do_not_call():
    with pytest.raises(AttributeError):
        kdn._native.call_xfer(0, 0, 0, [object()], 0, 0)
    with pytest.raises(TypeError):
        kdn._native.call_xfer(0, 0, 0, 5, 0, 0)
    with pytest.raises(ValueError):
        kdn._native.call_compose(0, 0, 0, [kdn.ComposeReq(0, 0, [records(1)[0].chunk], [], 1.0)], 0, 0)


class Stream:
    """As torch.cuda.Stream has it."""
    _as_parameter_ = C.c_void_p(0x5150)


class Sub(kdn.Chunk):
    """A chunk that says itself where it is."""

    def c(self):
        return kdn.kdn_chunk(0xABC0, 64, 2, 0, 0, 0, 0)


def _sparse_less():
    return (records(3), [0x9000])


FORMS = {
    "stream": ("kdn_store", lambda: (records(2),), Stream()),
    "stream of compose": ("kdn_compose", lambda: ([kdn.ComposeReq(64, 9, [records(1)[0].chunk], [5], 5e5)],), Stream()),
    "sizes modulo 2^64": ("kdn_retrieve", lambda: ([kdn.XferOp(64, 3 + (1 << 32), -1, kdn.Chunk(16, (1 << 64) - 16, 4, 0, 0, (1 << 63) + 5))],), 7),
    "a chunk of a class of its own": ("kdn_store", lambda: ([kdn.XferOp(64, 3, 0, Sub(16, 16, 4))],), 7),
    "fewer keep-lists than ops": ("kdn_store_sparse", _sparse_less, 7),
    "fewer positions than parts": ("kdn_compose", lambda: ([kdn.ComposeReq(64, 9, [o.chunk for o in records(3)], [5], "5e5")],), 7),
    "positions of an array": ("kdn_compose", lambda: ([kdn.ComposeReq(64, 9, [o.chunk for o in records(3)], np.arange(3) * 64, 5e5)],), 7),
    "selects for the first request": ("kdn_compose_select", lambda: ([kdn.ComposeReq(64, 9, [records(1)[0].chunk], [5], 5e5)] * 2, [[(0x5000, 7)]]), 7),
    "more selects than parts": ("kdn_compose_select", lambda: ([kdn.ComposeReq(64, 9, [records(1)[0].chunk], [5], 5e5)], [[None, (0x5000, 7)]]), 7),
}
BAD = {
    "records of a generator": ("kdn_store", lambda: (iter(records(2)),), 7),
    "no record": ("kdn_store", lambda: ([object()],), 7),
    "a size that is no int": ("kdn_store", lambda: ([kdn.XferOp(64, 3.0, 0, records(1)[0].chunk)],), 7),
    "a stream that is none": ("kdn_store", lambda: (records(1),), 1.5),
    "a stream of another type": ("kdn_store", lambda: (records(1),), C.c_int(5)),
    "too many positions": ("kdn_compose", lambda: ([kdn.ComposeReq(64, 9, [records(1)[0].chunk], [5, 6], 5e5)],), 7),
    "fewer selects than parts": ("kdn_compose_select", lambda: ([kdn.ComposeReq(64, 9, [o.chunk for o in records(2)], [5, 6], 5e5)], [[None]]), 7),
}


def called(monkeypatch, native, name, args, stream):
    """What the library's entry point gets (or the exception) with and without the extension module."""
    seen = []
    record = {"kdn_store_sparse": kdn.kdn_sparse_op}.get(name, kdn.kdn_xfer_op)

    def entry(ctx, pool, p, *rest):
        sel, (count, stream, side) = (rest[0], rest[1:]) if len(rest) == 4 else (None, rest)
        if name in ("kdn_compose", "kdn_compose_select"):
            reqs, got = C.cast(p, C.POINTER(kdn.kdn_compose_req)), []
            for i in range(count):
                q = reqs[i]
                got.append((q.block_table, q.n_table_blocks, q.rope_theta, q.rope_style, C.string_at(q.parts, q.n_parts * C.sizeof(kdn.kdn_chunk)),
                            q.part_dst_pos[:q.n_parts]))
                if sel:
                    s = C.cast(sel, C.POINTER(kdn.kdn_select))[i]
                    got.append([(s.part_select[j], s.part_n_select[j]) if s.part_select else None for j in range(q.n_parts)])
        else:
            got = C.string_at(p, count * C.sizeof(record))
        seen.append((ctx, pool, count, stream, side, got))
        return 0

    vp = C.c_void_p
    middle = [vp, vp] if name == "kdn_compose_select" else [vp]
    fn = C.CFUNCTYPE(C.c_int, vp, C.c_int, *middle, C.c_int, vp, vp)(entry)
    monkeypatch.setattr(kdn, "lib", type("Lib", (), {name: staticmethod(fn)}))
    constant = {"kdn_store": "_STORE", "kdn_retrieve": "_RETRIEVE", "kdn_compose": "_COMPOSE", "kdn_store_sparse": "_STORE_SPARSE",
                "kdn_compose_select": "_COMPOSE_SELECT"}[name]
    monkeypatch.setattr(kdn, constant, C.cast(fn, vp).value)
    monkeypatch.setattr(kdn, "_native", native)
    try:
        getattr(kdn, name)(0x1230, 3, *args, stream)
    except Exception as exc:
        return type(exc)
    return seen


@pytest.mark.parametrize("form", list(FORMS) + list(BAD))
def test_what_ctypes_takes_and_refuses_is_taken_and_refused(monkeypatch, form):
    """A call is the same with the extension module as without it, also in the forms the module does not know."""
    name, args, stream = {**FORMS, **BAD}[form]
    with monkeypatch.context() as m:
        want = called(m, None, name, args(), stream)
    with monkeypatch.context() as m:
        got = called(m, kdn._native, name, args(), stream)
    assert got == want
    assert (isinstance(want, list) and len(want) == 1) if form in FORMS else issubclass(want, Exception)


def test_a_list_that_shrinks_while_it_is_read():
    ops = records(40)

    class Op:
        n_table_blocks, token_offset, chunk = 1, 0, ops[0].chunk

        @property
        def block_table(self):
            ops.clear()
            return 64

    ops[0] = Op()
    with pytest.raises(IndexError):
        kdn._native.call_xfer(0, 0, 0, ops, 0, 0)
