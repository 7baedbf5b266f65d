"""What users of libkdn have it do, as cases that can be timed and compared.

A case is one call an engine makes: store, retrieve, compose (whole chunks, or only the listed tokens of each), or the
layer-wise retrieve, on a pool of Llama-3-8B or -70B shape as one rank of a tensor-parallel engine of 1, 2, 4 or 8
GPUs sees it (8, 4, 2 or 1 KV heads), with device tables, chunks and streams as bench.py and the tests have them.

    call     store | retrieve | compose | layerwise (retrieve in steps of `step` layers, an event per layer)
    codec    0 raw bf16, 1 / 2 int8 / int4 group-64, 3 / 4 the same with per-channel keys, 5 / 6 token-delta Rice
    layers, heads, block           the pool's shape (head_dim is 128 in both models)
    n, parts, tokens               n requests x parts chunks x tokens each (parts is 1 except in compose)
    offset   request position of a chunk's first token (compose: the parts follow one another from there)
    keep     share of the tokens that are listed: a keep-list for store and retrieve, a select-list for compose; 1 = all
    rho      correlation of neighbouring tokens in the input (the token-delta codecs are made for 0.9 and more)
    host     the chunks lie in page-locked host memory
"""
import numpy as np
import torch

from paper_2409_13761_b200 import kdn, synth

HEAD_DIM = 128
THETA = 500000.0
DEVICE = "cuda:0"
SEGMENT = 256          # the input's token correlation runs over stretches of this many tokens

# Bits per element the token-delta codecs come to on this input (scales, lengths and parameters included).
RICE_BITS = {(5, 0.0): 8.57, (5, 0.9): 7.70, (5, 0.99): 6.79, (6, 0.0): 4.44, (6, 0.9): 3.62, (6, 0.99): 2.86}
FIXED_BYTES = {0: 2.0, 1: 1.0625, 2: 0.5625, 3: 1.0625, 4: 0.5625}

ORDINARY = dict(call="retrieve", codec=0, layers=32, heads=8, block=16, n=1, parts=1, tokens=512, offset=0, keep=1.0, rho=0.0,
                host=False, step=0)


def listed():
    return [dict(ORDINARY, **c) for c in (
        # the smallest call: one of eight ranks takes a 128-token chunk into its blocks
        dict(name="one_head_retrieve", heads=1, tokens=128),
        # one turn of a conversation is put away as its request ends: an odd length at an odd position
        dict(name="turn_store_int8", call="store", codec=1, tokens=77, offset=1003),
        # the call made for each request that reuses a document: one chunk of ordinary length
        dict(name="doc_retrieve_raw"),
        # a library is filled: many chunks in one call
        dict(name="batch_store_int8", call="store", codec=1, n=32),
        # a batch of requests starts on documents of ragged length, in the most compact fixed-rate codec
        dict(name="batch_retrieve_int4", codec=2, n=32, tokens=509, offset=5),
        # retrieval-augmented request: ten documents side by side, keys re-rotated to where they now stand
        dict(name="rag_compose_raw", call="compose", parts=10, tokens=1024),
        # the same from compressed documents of a ragged length, two of eight heads of the larger model, several requests
        dict(name="rag_compose_td8_two_heads", call="compose", codec=5, layers=80, heads=2, n=4, parts=4, tokens=331, rho=0.9),
        # library of documents whose keys keep a scale per channel
        dict(name="batch_store_kc8", call="store", codec=3, n=16),
        # compression of a library for delivery, and decompression as requests arrive
        dict(name="batch_store_td8", call="store", codec=5, n=16, rho=0.9),
        dict(name="batch_retrieve_td4", codec=6, n=32, rho=0.9),
        # only the tokens a scorer kept, two of eight heads
        dict(name="half_kept_retrieve_int8", codec=1, heads=2, n=16, tokens=1024, keep=0.5),
        # one chunk comes from host memory, eight layers at a time
        dict(name="host_layerwise_int8", call="layerwise", codec=1, tokens=512, host=True, step=8),
    )]


# Elements a drawn call moves at most, so that none costs more than the largest listed one of its kind.
MOST = 3 << 28
MOST_RICE_STORE = 7 << 26
MOST_HOST = 1 << 24


def draw(rng):
    call = rng.choice(["store", "store", "store", "retrieve", "retrieve", "retrieve", "compose", "compose", "compose", "layerwise"])
    codec = rng.choice([0, 0, 1, 1, 2, 3, 4, 5, 6])
    c = dict(ORDINARY, call=call, codec=codec, layers=rng.choice([32, 32, 80]), heads=rng.choice([8, 8, 4, 2, 1]),
             block=rng.choice([16, 16, 32, 64]))
    c["rho"] = rng.choice([0.0, 0.9, 0.99]) if codec >= 5 else 0.0
    if call != "layerwise" and rng.random() < 0.2:
        c["keep"] = rng.choice([0.25, 0.5, 0.75])
    c["host"] = codec < 5 and c["keep"] == 1.0 and rng.random() < (0.5 if call == "layerwise" else 0.05)
    most = MOST_HOST if c["host"] else MOST_RICE_STORE if codec >= 5 and call == "store" else MOST
    rows = most // (c["layers"] * 2 * c["heads"] * HEAD_DIM)                     # tokens the call may have
    c["tokens"] = min(rows, int(round(2.0 ** rng.uniform(4.0, 12.0))))
    lots = int(min(64, rows // c["tokens"], max(1.0, 2.0 ** rng.uniform(-2.0, 6.0))))
    if call == "compose":
        c["parts"] = max(1, min(lots, rng.choice([2, 4, 10])))
    c["n"] = max(1, lots // c["parts"])
    offset = rng.choice([0, rng.randrange(2048)])
    # the codecs that group along tokens take whole chunks only at the start of a block
    c["offset"] = offset // c["block"] * c["block"] if codec >= 3 else offset
    c["step"] = rng.choice([4, 8, 16]) if call == "layerwise" else 0
    return c


class State:
    """A registered pool, its chunks and the records of the call; the context goes with it."""

    def __init__(self):
        self.ctx = kdn.kdn_create(0)

    def __del__(self):
        kdn.kdn_destroy(self.ctx)


def _kept(case):
    return max(1, int(case["tokens"] * case["keep"]))


def _place(case, part, tokens):
    """Position of a request's part: the parts follow one another, for the codecs that need it on block boundaries."""
    stride = -(-tokens // case["block"]) * case["block"] if case["codec"] >= 3 else tokens
    return case["offset"] + part * stride


def _fill(case, gen, planes, rows):
    """The input: N(0, 1) values with four loud channels a head, correlated along tokens, at the given pool rows."""
    L, H = case["layers"], case["heads"]
    gain = synth.outlier_gain(synth.KVShape("", L, H, HEAD_DIM, 1, 1, THETA)).view(2 * L, H * HEAD_DIM).to(DEVICE)
    m, rho = None, case["rho"]
    if rho:
        t = torch.arange(SEGMENT, device=DEVICE, dtype=torch.float64)
        m = torch.tril(rho ** (t[:, None] - t[None, :]).clamp(min=0))
        m[:, 1:] *= (1.0 - rho * rho) ** 0.5
        m = m.float()
    n = rows.numel()
    for p in range(2 * L):
        x = torch.randn((-(-n // SEGMENT) * SEGMENT, H * HEAD_DIM), generator=gen, device=DEVICE)
        if m is not None:
            x = torch.matmul(m, x.view(-1, SEGMENT, H * HEAD_DIM)).view(x.shape)
        planes[p].view(-1, H * HEAD_DIM).index_copy_(0, rows, (x[:n] * gain[p]).to(torch.bfloat16))


def prepare(case, seed):
    L, H, bs, codec, T = case["layers"], case["heads"], case["block"], case["codec"], case["tokens"]
    n, parts = case["n"], case["parts"]
    total, chunk_tokens = n * parts, T
    sparse = case["keep"] < 1.0
    storing, composing = case["call"] == "store", case["call"] == "compose"
    keep_list = sparse and not composing
    if keep_list:
        chunk_tokens = _kept(case)
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    rng = np.random.default_rng(seed)

    # block tables: every block somewhere else, as after an engine has run for a while
    req_tokens = _place(case, parts - 1, T) + T
    req_blocks, src_blocks = -(-req_tokens // bs), -(-T // bs)
    used = n * req_blocks if storing else max(n * req_blocks, total * src_blocks)
    n_blocks = used + used // 4 + 8
    s = State()
    s.case, s.stream = case, torch.cuda.current_stream().cuda_stream
    s.pool = torch.zeros((2 * L, n_blocks, bs, H, HEAD_DIM), dtype=torch.bfloat16, device=DEVICE)
    s.desc = kdn.pool_desc(L, H, HEAD_DIM, bs, n_blocks, [s.pool[2 * l].data_ptr() for l in range(L)],
                           [s.pool[2 * l + 1].data_ptr() for l in range(L)])
    s.pool_id = kdn.kdn_pool_register(s.ctx, s.desc)

    def tables(count, blocks):
        t = torch.from_numpy(rng.permutation(n_blocks)[:count * blocks].astype(np.int32).reshape(count, blocks)).to(DEVICE)
        return t

    def records(table, offset, bufs):
        return [kdn.XferOp(table[i].data_ptr(), table.shape[1], offset, bufs[i]) for i in range(len(bufs))]

    nbytes = kdn.kdn_chunk_bytes(s.desc, chunk_tokens, codec)
    stride = -(-nbytes // 256) * 256
    # (the bytes a token-delta chunk does not use are never written: zeros, so that outputs can be compared whole)
    on_gpu = torch.zeros((total, stride), dtype=torch.uint8, device=DEVICE)
    s.chunks = on_gpu if not case["host"] else torch.zeros((total, stride), dtype=torch.uint8, pin_memory=True)
    mem = kdn.KDN_MEM_PINNED_HOST if case["host"] else kdn.KDN_MEM_DEVICE
    at_device = [kdn.Chunk(on_gpu[i].data_ptr(), nbytes, chunk_tokens, codec) for i in range(total)]
    bufs = [kdn.Chunk(s.chunks[i].data_ptr(), nbytes, chunk_tokens, codec, mem) for i in range(total)]

    s.lists = None
    if sparse:
        s.lists = torch.stack([torch.randperm(T, generator=gen, device=DEVICE)[:_kept(case)].sort().values for _ in range(total)]).int().contiguous()
        s.keeps = [s.lists[i].data_ptr() for i in range(total)]

    s.table = tables(n, req_blocks)
    if storing:
        s.src, src_off = s.table, case["offset"]
    else:
        s.src, src_off = tables(total, src_blocks), 0
    pos = src_off + torch.arange(T, device=DEVICE)
    rows = (s.src[:, pos // bs].long() * bs + pos % bs).view(-1)
    _fill(case, gen, s.pool, rows)
    if not storing:
        # the chunks were stored by an earlier request, whose blocks have been given back since
        ops = records(s.src, 0, at_device)
        if keep_list:
            kdn.kdn_store_sparse(s.ctx, s.pool_id, ops, s.keeps, s.stream)
        else:
            kdn.kdn_store(s.ctx, s.pool_id, ops, s.stream)
        if kdn.kdn_status_sync(s.ctx, s.stream) != kdn.KDN_OK:
            raise RuntimeError("storing the input failed")
        if case["host"]:
            s.chunks.copy_(on_gpu)
        s.pool.zero_()
    if composing:
        where = [_place(case, j, T) for j in range(parts)]
        s.reqs = [kdn.ComposeReq(s.table[r].data_ptr(), req_blocks, bufs[r * parts:(r + 1) * parts], where, THETA) for r in range(n)]
        if sparse:
            s.selects = [[(s.keeps[r * parts + j], s.lists.shape[1]) for j in range(parts)] for r in range(n)]
    else:
        s.ops = records(s.table, case["offset"], bufs)
    if case["call"] == "layerwise":
        s.events = [torch.cuda.Event() for _ in range(L)]
        for e in s.events:
            e.record()
        s.handles = [e.cuda_event for e in s.events]
    return s


def run(s):
    call, sparse = s.case["call"], s.lists is not None
    if call == "store":
        if sparse:
            kdn.kdn_store_sparse(s.ctx, s.pool_id, s.ops, s.keeps, s.stream)
        else:
            kdn.kdn_store(s.ctx, s.pool_id, s.ops, s.stream)
        return s.chunks
    if call == "retrieve":
        if sparse:
            kdn.kdn_retrieve_sparse(s.ctx, s.pool_id, s.ops, s.keeps, s.stream)
        else:
            kdn.kdn_retrieve(s.ctx, s.pool_id, s.ops, s.stream)
    elif call == "layerwise":
        kdn.kdn_retrieve_layerwise(s.ctx, s.pool_id, s.ops, s.case["step"], s.stream, 0, s.handles)
    elif sparse:
        kdn.kdn_compose_select(s.ctx, s.pool_id, s.reqs, s.selects, s.stream)
    else:
        kdn.kdn_compose(s.ctx, s.pool_id, s.reqs, s.stream)
    return s.pool


def work(case):
    """bf16 on the pool side, the codec's bytes on the chunk side, each once; a product per coded element, three
    operations per re-rotated key element."""
    tokens = case["n"] * case["parts"] * (_kept(case) if case["keep"] < 1.0 else case["tokens"])
    elems = case["layers"] * 2 * tokens * case["heads"] * HEAD_DIM
    chunk = FIXED_BYTES[case["codec"]] if case["codec"] < 5 else RICE_BITS[case["codec"], case["rho"]] / 8.0
    flops = elems if case["codec"] else 0
    if case["call"] == "compose":
        flops += 3 * (elems // 2)
    return {"bytes": elems * (2.0 + chunk), "flops": float(flops)}


def tolerance(case):
    """Chunks and retrieved values are defined bit for bit.  A re-rotated key is an fp32 result rounded to bf16: against
    the same rotation in fp64, 1.4e-5 of the keys come out one step off, 9e-6 in the 2-norm and 7e-3 (a step) at most."""
    if case["call"] == "compose":
        return {"rel": 4e-5, "max": 0.016}
    return "exact"
