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
