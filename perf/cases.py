"""What a user of this framework has it do, as timed cases.

Each case is one pass of a weight-sync call sequence through the public entry
points, on buffers that a user's program keeps: the plan, the trainer's shards,
the buckets, the checksums, the rollout's tensors and the pointer tables, all
made once by ``prepare``.

Kinds of pass (``op``):
  sync      trainer and rollout of one step: ``rr_pack``, then the receiver's
            stream-ordered ``rr_unpack_verify_async``
  receive   the receiver alone, blocking (``rr_unpack_verify``): a rollout that
            needs the answer before it goes on
  verify    a rollout that reconnects asks which of the buckets it holds are
            intact (``rr_verify_range`` with per-bucket flags, blocking)
  resume    one rank pulls its buckets again: ``rr_pack_range``, then the
            ranged ``rr_unpack_verify_async``
  relay     a rollout serves another of a different tensor-parallel degree from
            its loaded tensors (``rr_pack`` on a ``qwen3_relay`` layout)
  snapshot  a checkpoint in pinned host memory: ``rr_pack`` into host buckets,
            then a restore from them (``rr_unpack_verify``)
  host      the trainer's shards are in pinned host memory: ``rr_pack`` reads
            them there
"""
import math
from types import SimpleNamespace

import torch

import paper_2512_22492_gb300 as rr
from paper_2512_22492_gb300 import layouts

KIB, MIB = 1 << 10, 1 << 20


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------

def _case(op, layers, hidden, n_q, n_kv, head_dim, inter, vocab, *, tied=False, experts=0,
          src="f32", dst="bf16", shards=8, sharding="flat", tp=1, ep=False, src_tp=1,
          bucket=32 * MIB, align=16, tensor_align=256, name=None):
    c = dict(op=op, layers=layers, hidden=hidden, n_q=n_q, n_kv=n_kv, head_dim=head_dim,
             inter=inter, vocab=vocab, tied=tied, experts=experts, src=src, dst=dst,
             shards=shards, sharding=sharding, tp=tp, ep=ep, src_tp=src_tp, bucket=bucket,
             align=align, tensor_align=tensor_align)
    return dict(c, name=name) if name else c


def listed():
    return [
        # The smallest sync: the two-layer test model, where launches and latency count.
        _case("sync", 2, 256, 4, 2, 64, 688, 1024, shards=1, bucket=256 * KIB,
              name="sync_tiny"),
        # A small receiver that waits for its answer: four ranks' tensors, 64 KiB buckets.
        _case("receive", 2, 256, 4, 2, 64, 688, 1024, tp=4, bucket=64 * KIB,
              name="receive_tiny_tp4"),
        # An ordinary small model, whole.
        _case("sync", 28, 1024, 16, 8, 128, 3072, 151936, tied=True, name="sync_0.6b"),
        # The largest: FSDP2 trainer to a TP=8 rollout, half of Qwen3-8B's layers.
        _case("sync", 18, 4096, 32, 8, 128, 12288, 151936, sharding="rows", tp=8,
              bucket=128 * MIB, name="sync_8b_18layers_fsdp2_tp8"),
        # Mixture of experts, bf16 trainer, narrow expert slices per rank.
        _case("sync", 4, 2048, 32, 4, 128, 768, 151936, experts=128, src="bf16",
              sharding="rows", tp=8, bucket=64 * MIB, name="sync_30b_4layers_fsdp2_tp8"),
        # A rollout rank of the same model lost its relay and pulls its buckets again.
        _case("resume", 4, 2048, 32, 4, 128, 768, 151936, experts=128, src="bf16",
              sharding="rows", tp=8, bucket=64 * MIB, name="resume_30b_4layers_fsdp2_tp8"),
        # A float16 rollout from per-layer FSDP1 units.
        _case("sync", 6, 4096, 32, 8, 128, 12288, 151936, dst="f16", sharding="units", tp=4,
              bucket=128 * MIB, name="sync_8b_6layers_units_tp4_f16"),
        # A TP=8 rollout relays to a TP=4 one: row-parallel weights are put together from pieces.
        _case("relay", 2, 4096, 32, 8, 128, 12288, 8192, src="bf16", src_tp=8, tp=4,
              name="relay_8b_2layers_tp8_tp4"),
        # Odd widths (the odd test model, eight times as wide): rows that share no alignment.
        _case("sync", 4, 2057, 16, 8, 36, 5514, 30102, tp=2, bucket=8 * MIB,
              name="sync_odd_tp2"),
        # An unpadded bf16 FlatParameter of odd sizes, tensors back to back, buckets that
        # end in the middle of a 16-byte vector.
        _case("sync", 4, 2057, 16, 8, 36, 5513, 30101, src="bf16", shards=6, align=2,
              tensor_align=2, bucket=8 * MIB + 8, name="sync_odd_unpadded_bf16"),
        # A checkpoint to pinned host memory and back.
        _case("snapshot", 28, 1024, 16, 8, 128, 3072, 151936, tied=True, name="snapshot_0.6b"),
        # A reconnecting rollout checks what it holds.
        _case("verify", 28, 1024, 16, 8, 128, 3072, 151936, tied=True, name="verify_0.6b"),
    ]


def draw(rng):
    """One more case: any kind of pass, sizes over the listed range (spread by
    their logarithm), odd widths and every layout option among them."""
    ops = ["sync"] * 6 + ["receive", "verify", "resume", "relay", "snapshot", "host"]
    top = math.log(_params(listed()[3]))
    while True:
        op = rng.choice(ops)
        family = "dense" if op == "relay" else rng.choice(["dense", "dense", "moe", "odd"])
        tp = rng.choice([1, 1, 2, 4, 8])
        ep = family == "moe" and rng.random() < 0.3
        experts = rng.choice([8, 16, 32]) * (1 if family == "moe" else 0)
        n_kv = rng.choice([2, 4, 8])
        n_q = n_kv * rng.choice([1, 2, 4])
        if n_q % tp:
            continue
        target = math.exp(rng.uniform(math.log(1.5e6), top if op in ("sync", "verify", "resume")
                                      else math.log(6e8)))
        width = math.exp(rng.uniform(math.log(200), math.log(4200)))
        if family == "odd":
            head_dim, hidden = rng.choice([36, 60, 100]), int(width) | 1
            inter = tp * int(width * rng.uniform(1, 3) / tp + 1)
            vocab = tp * int(math.exp(rng.uniform(math.log(500), math.log(60000))) / tp + 1)
        else:
            head_dim, hidden = rng.choice([32, 64, 128]), max(64, int(width) // 64 * 64)
            inter = 8 * tp * max(1, int(width * (0.4 if experts else rng.uniform(2, 3.5)) / (8 * tp)))
            vocab = 64 * tp * int(math.exp(rng.uniform(math.log(500), math.log(152000))) / (64 * tp) + 1)
        src = rng.choice(["f32", "f32", "bf16"]) if op != "relay" else "bf16"
        dst = rng.choice(["bf16", "bf16", "bf16", "f16"]) if op != "relay" else "bf16"
        src_tp = rng.choice([1, 2, 4, 8]) if op == "relay" else 1
        if op == "relay" and (n_q % src_tp or inter % (8 * src_tp) or vocab % src_tp):
            continue
        bucket = 1 << rng.randint(16, 27)
        c = _case(op, 1, hidden, n_q, n_kv, head_dim, inter, vocab, tied=rng.random() < 0.3,
                  experts=experts, src=src, dst=dst, shards=rng.choice([1, 2, 4, 6, 8]),
                  sharding=rng.choice(["flat", "flat", "rows", "units"]), tp=tp, ep=ep,
                  src_tp=src_tp, bucket=bucket)
        if family == "odd" and rng.random() < 0.5:
            c.update(align=2 if src == "bf16" else 4, tensor_align=rng.choice([2, 16]),
                     bucket=bucket + 8 * rng.randint(0, 3))
        one, none = _params(dict(c, layers=1)), _params(dict(c, layers=0))
        c["layers"] = max(1, min(36 if not experts else 8, round((target - none) / (one - none))))
        pieces = c["layers"] * hidden * max(src_tp, tp) if op == "relay" else 0
        streams = _params(c) * 2 / tp
        if not 1.2e6 < _params(c) <= math.exp(top) or pieces > 80000:
            continue
        if not streams / 4000 < bucket < 2 * streams:   # neither a swarm of buckets nor mostly tail
            continue
        return c


# ---------------------------------------------------------------------------
# Shapes and sources, from the definitions
# ---------------------------------------------------------------------------

def _shape(c):
    return SimpleNamespace(layers=c["layers"], hidden=c["hidden"], n_q=c["n_q"], n_kv=c["n_kv"],
                           head_dim=c["head_dim"], intermediate=0 if c["experts"] else c["inter"],
                           vocab=c["vocab"], tied=c["tied"], n_experts=c["experts"],
                           moe_intermediate=c["inter"] if c["experts"] else 0)


def _shapes(c):
    """The trainer's parameters in registration order: (name, layer or -1, shape)."""
    h, d, m = c["hidden"], c["head_dim"], c["inter"]
    out = [("embed", -1, (c["vocab"], h))]
    for i in range(c["layers"]):
        out += [(f"{i}.q", i, (c["n_q"] * d, h)), (f"{i}.k", i, (c["n_kv"] * d, h)),
                (f"{i}.v", i, (c["n_kv"] * d, h)), (f"{i}.o", i, (h, c["n_q"] * d)),
                (f"{i}.q_norm", i, (d,)), (f"{i}.k_norm", i, (d,))]
        if c["experts"]:
            out.append((f"{i}.router", i, (c["experts"], h)))
        for e in range(c["experts"] or 1):
            out += [(f"{i}.{e}.gate", i, (m, h)), (f"{i}.{e}.up", i, (m, h)),
                    (f"{i}.{e}.down", i, (h, m))]
        out += [(f"{i}.input_ln", i, (h,)), (f"{i}.post_ln", i, (h,))]
    out.append(("norm", -1, (h,)))
    return out if c["tied"] else out + [("lm_head", -1, (c["vocab"], h))]


def _params(c):
    return sum(math.prod(s) for _, _, s in _shapes(c))


def _up(x, a):
    return -(-x // a) * a


def _source(c):
    """(bytes of every source buffer, pieces of every parameter): a piece is
    (buffer offset in the concatenation of all buffers, elements)."""
    es, n = 4 if c["src"] == "f32" else 2, c["shards"]
    align = max(c["align"], es)
    params = _shapes(c)
    if c["sharding"] == "rows":
        end, at = 0, []
        for _, _, s in params:
            rows, cols = s[0], math.prod(s[1:])
            chunk = -(-rows // n)
            end = _up(end, align)
            at.append([(k, end, (min((k + 1) * chunk, rows) - k * chunk) * cols)
                       for k in range(n) if k * chunk < rows])
            end += chunk * cols * es
        size = _up(end, 16)
        return [size] * n, [[(k * size + o, m) for k, o, m in p] for p in at]
    units = [layer + 1 if c["sharding"] == "units" else 0 for _, layer, _ in params]
    end, at = [0] * (max(units) + 1), []
    for (_, _, s), u in zip(params, units):
        end[u] = _up(end[u], align)
        at.append((u, end[u], math.prod(s)))
        end[u] += math.prod(s) * es
    size = [_up(e, 16 * n) for e in end]
    start = [sum(size[:u]) for u in range(len(size))]
    return [b // n for b in size for _ in range(n)], [[(start[u] + o, m)] for u, o, m in at]


def _values(nbytes, dtype, seed, pinned=False):
    """A block of weights, about N(0, 0.02), made from the seed on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.empty(nbytes // dtype.itemsize, dtype=dtype, device="cuda")
    x.normal_(0, 0.02, generator=g)
    if not pinned:
        return x
    return torch.empty(x.shape, dtype=dtype, pin_memory=True).copy_(x)


def _tensors(c, p):
    """The rollout's tensors from the trainer's parameters (by name), rank by
    rank, the way an inference engine's loader cuts and fuses them."""
    t, E, out = c["tp"], c["experts"], []

    def rows(x, r):
        return x.chunk(t, 0)[r]

    def cols(x, r):
        return x.chunk(t, 1)[r]

    def kv(x, r):
        return rows(x, r) if t <= c["n_kv"] else x.chunk(c["n_kv"], 0)[r * c["n_kv"] // t]

    for r in range(t):
        out.append(rows(p["embed"], r))
        for i in range(c["layers"]):
            out += [torch.cat([rows(p[f"{i}.q"], r), kv(p[f"{i}.k"], r), kv(p[f"{i}.v"], r)]),
                    cols(p[f"{i}.o"], r), p[f"{i}.q_norm"], p[f"{i}.k_norm"],
                    p[f"{i}.input_ln"], p[f"{i}.post_ln"]]
            if E:
                out.append(p[f"{i}.router"])
            mine = range(r * E // t, (r + 1) * E // t) if c["ep"] else range(E or 1)
            whole = c["ep"] and E
            gate_up = [x if whole else rows(x, r) for e in mine
                       for x in (p[f"{i}.{e}.gate"], p[f"{i}.{e}.up"])]
            down = [p[f"{i}.{e}.down"] if whole else cols(p[f"{i}.{e}.down"], r) for e in mine]
            out += [torch.cat(gate_up), torch.cat([x.reshape(-1) for x in down])]
        out.append(p["norm"])
        if not c["tied"]:
            out.append(rows(p["lm_head"], r))
    return out


def _layout(c):
    """(manifest, source layout, rollout layout) as a user describes them."""
    if c["op"] == "relay":
        return layouts.qwen3_relay(_shape(c), c["src_tp"], c["tp"])
    m, s, d = rr.qwen3_sync(_shape(c), c["src"], c["shards"], c["tp"], c["sharding"], ep=c["ep"],
                            dst_dtype=c["dst"])
    s.align_bytes, d.tensor_align_bytes = c["align"], c["tensor_align"]
    return m, s, d


# ---------------------------------------------------------------------------
# A pass
# ---------------------------------------------------------------------------

def _block(numel, dtype):
    """One zeroed block for the rollout's tensors, and the tensors in it (16-byte starts)."""
    starts, at = [], 0
    for n in numel:
        starts.append(at)
        at += _up(n, 8)
    block = torch.zeros(max(8, at), dtype=dtype, device="cuda")
    return block, [block[o:o + n] for o, n in zip(starts, numel)]


def _words(x):
    """The same memory as 64-bit words, the unit of the checksums."""
    return x.view(torch.int64)


def prepare(case, seed):
    op = case["op"]
    dtype = torch.float32 if case["src"] == "f32" else torch.bfloat16
    m, s, d = _layout(case)
    plan = rr.rr_plan_create(m, s, d, case["bucket"])
    st = SimpleNamespace(op=op, plan=plan)
    sizes = plan.source_buffer_bytes
    if op == "relay":
        st.source = _values(sum(_up(b, 256) for b in sizes), dtype, seed)
        st.base, at = [], st.source.data_ptr()
        for b in sizes:
            st.base.append(at)
            at += _up(b, 256)
    else:
        assert list(sizes) == _source(case)[0]
        st.source = _values(sum(sizes), dtype, seed, pinned=op == "host")
        ends = [sum(sizes[:i]) for i in range(len(sizes))]
        st.base = [st.source.data_ptr() + e for e in ends]
    n = plan.n_buckets
    stride = _up(plan.bucket_bytes, 16)
    host = dict(pin_memory=True) if op == "snapshot" else dict(device="cuda")
    st.store = torch.zeros((n, stride), dtype=torch.uint8, **host)
    st.checksums = torch.zeros(n, dtype=torch.int64, device="cuda")
    out = torch.float16 if case["dst"] == "f16" else torch.bfloat16
    st.t_src = rr.Pointers(plan, "src_shards", st.base)
    st.t_bkt = rr.Pointers(plan, "buckets", st.store[:, :plan.bucket_bytes])
    if op not in ("relay", "host", "verify"):
        st.block, st.tensors = _block(plan.tensor_numel, out)
        st.t_dst = rr.Pointers(plan, "dst", st.tensors)
        st.scratch = torch.zeros(n + 4, dtype=torch.int64, device="cuda")
        st.result = torch.zeros(2, dtype=torch.int64, device="cuda")
    if op == "resume":
        r = plan.tp // 2
        st.first = plan.first_bucket_of_rank[r]
        st.count = plan.first_bucket_of_rank[r + 1] - st.first
    if op in ("receive", "verify"):
        # A pulled image; a verifying rollout's has some buckets damaged on the way.
        rr.rr_pack(plan, st.t_src, st.t_bkt, st.checksums)
        st.source = st.base = None
        if op == "verify":
            st.bad = torch.zeros(n, dtype=torch.uint8, device="cuda")
            g = torch.Generator().manual_seed(seed)
            hit = torch.randperm(n, generator=g)[:max(1, n // 8)].cuda()
            st.store[hit, 8 * (seed % 97)] ^= 1
    torch.cuda.synchronize()
    return st


def run(st):
    op, plan = st.op, st.plan
    if op == "sync":
        rr.rr_pack(plan, st.t_src, st.t_bkt, st.checksums)
        rr.rr_unpack_verify_async(plan, st.t_bkt, st.checksums, st.t_dst, st.scratch, st.result)
        return {"buckets": _words(st.store), "checksums": st.checksums, "tensors": st.block,
                "result": st.result}
    if op == "receive":
        n_bad, first = rr.rr_unpack_verify(plan, st.t_bkt, st.checksums, st.t_dst)
        return {"tensors": st.block, "n_bad": n_bad, "first_bad": first}
    if op == "verify":
        n_bad, first = rr.rr_verify_range(plan, 0, plan.n_buckets, st.t_bkt, st.checksums, st.bad)
        return {"bad": st.bad, "n_bad": n_bad, "first_bad": first}
    if op == "resume":
        rr.rr_pack_range(plan, st.first, st.count, st.t_src, st.t_bkt, st.checksums)
        rr.rr_unpack_verify_async(plan, st.t_bkt, st.checksums, st.t_dst, st.scratch, st.result,
                                  first_bucket=st.first, n_buckets=st.count)
        mine = slice(st.first, st.first + st.count)
        return {"buckets": _words(st.store[mine]), "checksums": st.checksums[mine],
                "tensors": st.block, "result": st.result}
    if op == "snapshot":
        rr.rr_pack(plan, st.t_src, st.t_bkt, st.checksums)
        n_bad, first = rr.rr_unpack_verify(plan, st.t_bkt, st.checksums, st.t_dst)
        return {"buckets": _words(st.store), "checksums": st.checksums, "tensors": st.block,
                "n_bad": n_bad, "first_bad": first}
    rr.rr_pack(plan, st.t_src, st.t_bkt, st.checksums)   # relay, host
    return {"buckets": _words(st.store), "checksums": st.checksums}


# ---------------------------------------------------------------------------
# What a pass cannot do without, and what it should give
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: every source element that is needed read once, every bucket byte
    written once, every bucket byte read once by the receiver, every tensor
    element written once.  No arithmetic to speak of."""
    op, B, t = case["op"], case["bucket"], case["tp"]
    rank = [_sizes(case, r) for r in range(t)]
    stream, numel, need = [], [], []
    for sizes in rank:
        at = 0
        for n in sizes:
            at = _up(at, case["tensor_align"] if op != "relay" else 256) + 2 * n
        stream.append(_up(at, B))
        numel.append(sum(sizes))
    es = 4 if case["src"] == "f32" else 2
    if op == "resume":
        r = t // 2
        return {"bytes": es * numel[r] + 2 * stream[r] + 2 * numel[r], "flops": 0}
    source = es * _params(case)
    if op in ("sync", "snapshot"):
        total = source + 2 * sum(stream) + 2 * sum(numel)
    elif op == "receive":
        total = sum(stream) + 2 * sum(numel)
    elif op == "verify":
        total = sum(stream)
    else:
        total = source + sum(stream)
    return {"bytes": total, "flops": 0}


def _sizes(c, r):
    """Elements of every tensor of rank r, in stream order."""
    t, h, d, E, m = c["tp"], c["hidden"], c["head_dim"], c["experts"], c["inter"]
    kv = c["n_kv"] // t if t <= c["n_kv"] else 1
    layer = [(c["n_q"] // t + 2 * kv) * d * h, h * c["n_q"] * d // t, d, d, h, h]
    if E:
        layer += [E * h, 2 * E * m * h // t, E * m * h // t]
    else:
        layer += [2 * m * h // t, m * h // t]
    return ([c["vocab"] // t * h] + layer * c["layers"] + [h]
            + ([] if c["tied"] else [c["vocab"] // t * h]))


def tolerance(case):
    """Bits are fixed: the cast is round-to-nearest-even, the rest is movement and whole sums."""
    return "exact"


def exact(case, seed):
    """The rollout's tensors in 64 bits, straight from the trainer's values;
    buckets, checksums and counts are bytes and whole numbers."""
    if case["op"] in ("relay", "host", "verify"):
        return None
    es = 4 if case["src"] == "f32" else 2
    sizes, pieces = _source(case)
    src = _values(sum(sizes), torch.float32 if es == 4 else torch.bfloat16, seed)
    params = {}
    for (name, _, shape), at in zip(_shapes(case), pieces):
        parts = [src[o // es:o // es + n] for o, n in at]
        params[name] = (parts[0] if len(parts) == 1 else torch.cat(parts)).view(shape)
    tensors = _tensors(case, params)
    block, views = _block([x.numel() for x in tensors], torch.float64)
    if case["op"] == "resume":
        # Only the buckets of one rank were pulled: the other ranks' tensors stay zero.
        n, r = len(tensors) // case["tp"], case["tp"] // 2
        views, tensors = views[r * n:(r + 1) * n], tensors[r * n:(r + 1) * n]
    for v, x in zip(views, tensors):
        v.copy_(x.reshape(-1))
    return {"tensors": block}
