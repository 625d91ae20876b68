"""The performance cases of the library: what its users run, over the sizes and options they run it at.

A case names a kind of work and its sizes.  Kinds:

  prefill   one layer's whole looped prefill of one prompt through pipeline.LayerState: dense source loop, column
            selection, then per sparse loop token selection, residual quantization and loop attention.
  step      the sparse loops 2..R of one or more layers on stores that a serving engine keeps: the loop-r prefill step
            that the library exists for.  `rows` = False: no materialized rows are lent, attention dequantizes and adds
            in the kernel.  `packed` = True: the loop-1 base stays packed and is rebuilt before each loop.
  schedule  decaying token and column budgets: the old term is recomputed and the column sets pruned in every loop.
  dense     the source loop alone (all rows, with or without the column statistics).
  decode    single-token queries after the prompt, over the store that a prefill left.
  project   the projections of the active rows: Q/K/V (optionally with the residual codec as the epilogue) and the
            output projection added back into the hidden store.
  base      packing of a layer's loop-1 K and V and the rebuild of every row.

Inputs come from the library's own generator (workloads.DeviceStack: nested shrinking sets of changed rows, persistent
heavy key columns, small cross-loop residuals).  The projections that produce the sparse loops' Q, K and V rows belong
to the model around the library, so prepare() makes those rows.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2609_29812_b200 import binding as B
from paper_2609_29812_b200 import pipeline as P
from paper_2609_29812_b200 import workloads

_DEV = "cuda:0"


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def _loopcase(kind, name=None, *, L, heads=16, head_dim=128, dtype="bf16", loops=4, tokens=0.10, cols=1024,
              q_block=1024, bits=4, group=128, layers=1, rows=True, packed=False):
    c = dict(kind=kind, L=L, heads=heads, head_dim=head_dim, dtype=dtype, loops=loops, tokens=tokens, cols=cols,
             q_block=q_block, bits=bits, group=group, layers=layers, rows=rows, packed=packed)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the tiny single-layer check in f32: every call is short, latency and launches count
        _loopcase("prefill", "prefill_f32_tiny", L=512, heads=4, head_dim=64, dtype="f32", loops=2, tokens=0.25, cols=64,
                  q_block=64, group=64),
        # a short prompt of odd length with 8-bit residuals in small groups: two blocks, the second a short one
        _loopcase("prefill", "prefill_1k_ragged", L=1237, loops=3, tokens=0.20, cols=160, bits=8, group=64),
        # one layer of the 2.6B-shaped block at 8K, end to end
        _loopcase("prefill", "prefill_8k", L=8192, tokens=0.15, cols=512),
        # the headline configuration: loops 2..4 at 32K, four layers sharing each loop's token selection
        _loopcase("step", "step_32k", L=32768, layers=4),
        # the same step with the packed loop-1 base rebuilt in front of every loop
        _loopcase("step", "step_32k_packed", L=32768, packed=True),
        # the long-context configuration, one layer
        _loopcase("step", "step_128k", L=131072, cols=2048),
        # the deep model's decaying schedule: 90% -> 20% of the tokens, 2048 -> 256 columns, pruned in every loop
        _loopcase("schedule", "schedule_8k", L=8192, loops=8, tokens=0.90, cols=2048),
        # loop 1 at 32K with the statistics that loop 2 starts from: the longest launch of a prefill
        dict(kind="dense", name="dense_32k", L=32768, heads=16, q_block=1024, stats=True),
        # the decode phase of the long-context configuration: a batch of 32 queries
        dict(kind="decode", name="decode_128k_32", L=131072, heads=16, loops=4, queries=32, cols=2048, bits=4, group=128),
        # one user at a moderate context: the smallest decode call
        dict(kind="decode", name="decode_8k_1", L=8192, heads=16, loops=4, queries=1, cols=512, bits=4, group=128),
        # projections of the 10% active rows of a 32K prompt
        dict(kind="project", name="project_32k", L=32768, n=3277, d=2048, fused=False),
        # packing the loop-1 base of a prompt of odd length, and rebuilding all of it
        dict(kind="base", name="base_20k_ragged", L=20011, heads=16, bits=4, group=64, tail=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "step", "step", "step", "schedule", "dense", "decode", "decode", "project",
                       "base"])
    bits = rng.choice([2, 4, 4, 4, 8, 16])
    group = rng.choice([32, 64, 128, 128])
    if kind == "prefill":
        if rng.random() < 0.3:      # f32 storage or heads of 64: the binary32 path, used for checks and small models
            head_dim = 64
            return _loopcase(kind, L=_log(rng, 200, 1500), heads=rng.choice([4, 8, 16]), head_dim=head_dim,
                             dtype=rng.choice(["f32", "f32", "bf16"]), loops=rng.choice([2, 3, 4]),
                             tokens=rng.choice([0.1, 0.25, 0.5]), cols=_log(rng, 32, 160), q_block=rng.choice([64, 128, 256]),
                             bits=bits, group=min(group, head_dim))
        return _loopcase(kind, L=_log(rng, 400, 12000), heads=rng.choice([4, 8, 16, 16]), loops=rng.choice([2, 3, 4, 4, 6]),
                         tokens=round(rng.uniform(0.05, 0.30), 3), cols=_log(rng, 128, 1024),
                         q_block=rng.choice([512, 1024, 1024]), bits=bits, group=group)
    if kind == "step":
        L = _log(rng, 4096, 131072)
        packed = bits != 16 and rng.random() < 0.25
        return _loopcase(kind, L=L, loops=rng.choice([2, 3, 4, 4, 8]), tokens=round(rng.uniform(0.05, 0.20), 3),
                         cols=_log(rng, 128, 2048), q_block=rng.choice([512, 1024, 1024, 2048]), bits=bits, group=group,
                         rows=rng.random() < 0.8, packed=packed)
    if kind == "schedule":
        return _loopcase(kind, L=_log(rng, 1024, 8000), loops=rng.choice([3, 4, 6, 8]), tokens=round(rng.uniform(0.3, 0.9), 3),
                         cols=_log(rng, 256, 2048), bits=bits, group=group)
    if kind == "dense":
        return dict(kind=kind, L=_log(rng, 700, 30000), heads=rng.choice([4, 8, 16, 16]), q_block=rng.choice([512, 1024, 1024]),
                    stats=rng.random() < 0.8)
    if kind == "decode":
        return dict(kind=kind, L=_log(rng, 2048, 131072), heads=16, loops=rng.choice([2, 3, 4, 4]), queries=_log(rng, 1, 64),
                    cols=_log(rng, 64, 2048), bits=bits, group=group)
    if kind == "project":
        n = _log(rng, 60, 12000)
        return dict(kind=kind, L=n * rng.randint(2, 10), n=n, d=rng.choice([1024, 2048, 2048]), fused=rng.random() < 0.3)
    return dict(kind=kind, L=_log(rng, 700, 60000), heads=rng.choice([8, 16]), bits=rng.choice([2, 4, 4, 8]),
                group=rng.choice([32, 64, 64, 128]), tail=64)


# ------------------------------------------------------------------------------------------------
# sizes derived from a case
# ------------------------------------------------------------------------------------------------
def _budgets(case):
    """(tokens, columns) of loops 2..R."""
    R, L = case["loops"], case["L"]
    if case["kind"] == "schedule":      # linear decay to 20% of the rows and an eighth of the columns
        at = lambda a, b: [a + (b - a) * i / max(R - 2, 1) for i in range(R - 1)]
        fr = at(case["tokens"], min(case["tokens"], 0.20))
        cc = [max(32, int(round(x / 32.0)) * 32) for x in at(case["cols"], max(64, case["cols"] // 8))]
        return [max(1, int(f * L + 0.5)) for f in fr], cc
    return [max(1, int(case["tokens"] * L + 0.5))] * (R - 1), [case["cols"]] * (R - 1)


def _workload(case):
    R = case["loops"]
    if case["kind"] == "schedule":
        toks, _ = _budgets(case)
        changed = tuple(t / case["L"] for t in toks)
    else:
        changed = tuple(0.30 * 0.52 ** (r - 2) for r in range(2, R + 1))
    d = case["heads"] * case["head_dim"]
    big = case["dtype"] == "bf16"
    return workloads.Workload(case["kind"], L=case["L"], n_heads=case["heads"], head_dim=case["head_dim"], n_loops=R,
                              dtype=case["dtype"], changed_fracs=changed, delta_hi=0.3, delta_lo=1e-3, w_std=d ** -0.5,
                              heavy_frac=0.02 if big else 0.0, heavy_scale=8.0 if big else 1.0, token_frac=case["tokens"],
                              col_budget=case["cols"], q_block=case["q_block"], bits=case["bits"], group=case["group"],
                              n_layers=case.get("layers", 1))


def _tensor_path(case):
    return case["dtype"] == "bf16" and case["head_dim"] == 128


_CTX = {}


def _ctx():
    if "ctx" not in _CTX:       # one context per process, as a program keeps it
        _CTX["ctx"] = B.Context(0)
    return _CTX["ctx"]


# ------------------------------------------------------------------------------------------------
# prepare
# ------------------------------------------------------------------------------------------------
def prepare(case, seed):
    torch.cuda.set_device(0)
    with torch.no_grad():
        return {"prefill": _prepare_prefill, "step": _prepare_step, "schedule": _prepare_schedule, "dense": _prepare_dense,
                "decode": _prepare_decode, "project": _prepare_project, "base": _prepare_base}[case["kind"]](case, seed)


def _generator(seed):
    g = torch.Generator(device=_DEV)
    g.manual_seed(int(seed) % (1 << 31))
    return g


def _select_all(ctx, shape, G, toks):
    sels, cand = [], None
    for r, k in enumerate(toks, start=2):
        sel = P.select_tokens(ctx, shape, r, G[r - 2], G[r - 1], cand, k)
        sels.append(sel)
        cand = sel.active_idx
    return sels


def _prepare_prefill(case, seed):
    w, ctx = _workload(case), _ctx()
    stack = workloads.DeviceStack(w, seed=int(seed) % (1 << 30), device=_DEV)
    G = stack.stack_hidden()
    toks, _ = _budgets(case)
    shape = P.shape_of(w)
    sels = _select_all(ctx, shape, G, toks)
    gen = stack.layer(0)
    qkv1 = gen.qkv1()
    rows = {r: gen.rows(r, sels[r - 2].active_idx) for r in range(2, w.n_loops + 1)}
    gen.release()
    return SimpleNamespace(kind="prefill", w=w, ctx=ctx, shape=shape, G=G, toks=toks, qkv1=qkv1, rows=rows,
                           tensor=_tensor_path(case))


def _block_scores(q, k, shape, gen):
    """Column statistics of the dense loop, estimated from 64 queries of each block (the library accepts any scores)."""
    L, H, dh = q.shape
    nb = (L + shape.q_block - 1) // shape.q_block
    out = torch.zeros(H, nb, L, device=q.device)
    kt = k.permute(1, 2, 0)
    for b in range(nb):
        lo, hi = b * shape.q_block, min(L, (b + 1) * shape.q_block)
        m = min(64, hi - lo)
        pos = lo + torch.sort(torch.randperm(hi - lo, generator=gen, device=q.device)[:m])[0]
        s = torch.matmul(q[pos].permute(1, 0, 2).float(), kt[:, :, :hi].float()) * shape.sm_scale
        s.masked_fill_(torch.arange(hi, device=q.device)[None, None, :] > pos[None, :, None], float("-inf"))
        out[:, b, :hi] = torch.softmax(s, dim=-1).sum(dim=1) * ((hi - lo) / m)
    return out


def _stacked_streams(case, w, sels, layers):
    """Residual payloads of all layers, loop by loop: codes, scale, zero of K and V as [layers, n, ...] tensors."""
    out = []
    for sel in sels:
        one = []
        for _side in range(2):
            if w.bits == 16:
                one.append((torch.zeros(layers, sel.n, w.d, dtype=torch.bfloat16, device=_DEV), None, None))
            else:
                one.append((torch.zeros(layers, sel.n, w.d * w.bits // 8, dtype=torch.uint8, device=_DEV),
                            torch.zeros(layers, sel.n, w.d // w.group, dtype=torch.float16, device=_DEV),
                            torch.zeros(layers, sel.n, w.d // w.group, dtype=torch.float16, device=_DEV)))
        out.append(one)
    return out


def _streams_of_layer(payload, sels, l, side, ws=None, cur_only=()):
    out = []
    for i, sel in enumerate(sels):
        codes, scale, zero = payload[i][side]
        st = {"slot_of_pos": sel.slot_of_pos, "n_rows": sel.n, "codes": codes[l],
              "scale": None if scale is None else scale[l], "zero": None if zero is None else zero[l]}
        if ws is not None:
            st["rows_cur"] = ws[side][1][:sel.n]
            if i + 2 not in cur_only:      # a loop that reuses the carried old term reads nothing else
                st["rows_prev"] = ws[side][0][:sel.n]
        out.append(st)
    return out


def _prepare_sparse(case, seed, economy):
    """What the step and the schedule share: token sets, and per layer the dense loop's results and the rows."""
    w, ctx = _workload(case), _ctx()
    shape = P.shape_of(w)
    toks, cols = _budgets(case)
    stack = workloads.DeviceStack(w, seed=int(seed) % (1 << 30), device=_DEV)
    G = stack.stack_hidden()
    sels = _select_all(ctx, shape, G, toks)
    n_layers, R, n0 = case["layers"], w.n_loops, sels[0].n
    payload = _stacked_streams(case, w, sels, n_layers)
    ws = None
    if case["rows"]:
        ws = [[torch.empty(n0, w.d, dtype=torch.bfloat16, device=_DEV) for _ in range(2)] for _ in range(2)]
    s = SimpleNamespace(kind=case["kind"], w=w, ctx=ctx, shape=shape, G=G, toks=toks, cols=cols, sels=sels, payload=payload,
                        ws=ws, layers=[], g_out=G[0].clone(), packed=case["packed"],
                        status=torch.zeros(1, dtype=torch.int32, device=_DEV),
                        x=torch.empty(n0, w.d, dtype=torch.bfloat16, device=_DEV))
    P.lend_workspace(ctx, shape, _DEV)
    stores = [torch.empty(n_layers, w.L, w.n_heads, w.head_dim, dtype=torch.bfloat16, device=_DEV) for _ in range(2)]
    s.q_out, s.o_out = stores
    s.lse_out = torch.empty(n_layers, w.n_heads, w.L, device=_DEV)
    if economy:
        s.bg = torch.zeros_like(s.o_out)
        s.mass = torch.zeros_like(s.lse_out)
    if s.packed:                    # one rebuilt copy for the whole stack: the packed form is what stays
        s.k_buf = torch.zeros(w.L, w.n_heads, w.head_dim, dtype=torch.bfloat16, device=_DEV)
        s.v_buf = torch.zeros_like(s.k_buf)
    nb = (w.L + w.q_block - 1) // w.q_block
    s.col_idx = [torch.empty(n_layers, w.n_heads, nb, c, dtype=torch.int32, device=_DEV) for c in cols]
    s.col_cnt = [torch.empty(n_layers, w.n_heads, nb, dtype=torch.int32, device=_DEV) for c in cols]
    cur_only = range(3, R + 1) if economy else ()
    for l in range(n_layers):
        gen = stack.layer(l)
        q1, k1, v1 = gen.qkv1()
        y = SimpleNamespace()
        if s.packed:
            y.state = P.LayerState(ctx, w, _DEV)
            y.state.pack_base(k1, v1)
            y.state.rebuild_base(s.k_buf, s.v_buf)
            k1, v1 = s.k_buf, s.v_buf
        else:
            y.k, y.v = k1, v1
        y.q1, y.o1, y.lse1 = q1, torch.empty_like(q1), torch.empty(w.n_heads, w.L, device=_DEV)
        B.fl_dense_loop_attention(ctx, shape, q1, k1, v1, y.o1, y.lse1, None)
        y.scores = _block_scores(q1, k1, shape, _generator(seed * 64 + l))
        s.q_out[l], s.o_out[l], s.lse_out[l] = q1, y.o1, y.lse1
        y.hidden = gen.hidden(R)
        y.rows = {r: gen.rows(r, sels[r - 2].active_idx) for r in range(2, R + 1)}
        gen.release()
        y.store = B.make_store(k1, v1, _streams_of_layer(payload, sels, l, 0, ws, cur_only),
                               _streams_of_layer(payload, sels, l, 1, ws, cur_only))
        if economy:
            y.write, y.reuse = (B.make_carry(s.bg[l], s.mass[l], flag) for flag in (False, True))
        y.next_scores = [torch.zeros(w.n_heads, nb, c, device=_DEV) for c in cols] if not economy else None
        if s.packed:
            y.mask = torch.zeros(w.n_heads, (w.L + 31) // 32, dtype=torch.int32, device=_DEV)
        s.layers.append(y)
    return s


def _prepare_step(case, seed):
    return _prepare_sparse(case, seed, economy=True)


def _prepare_schedule(case, seed):
    return _prepare_sparse(case, seed, economy=False)


def _prepare_dense(case, seed):
    L, H = case["L"], case["heads"]
    g = _generator(seed)
    q, k, v = (torch.randn(L, H, 128, generator=g, device=_DEV).to(torch.bfloat16) for _ in range(3))
    heavy = torch.randperm(L, generator=g, device=_DEV)[:int(0.02 * L + 0.5)]
    k[heavy] *= 8.0
    nb = (L + case["q_block"] - 1) // case["q_block"]
    shape = B.make_shape(L, H, 128, B.FL_BF16, case["q_block"], 4, 128, 1e-6, 128 ** -0.5)
    return SimpleNamespace(kind="dense", ctx=_ctx(), shape=shape, q=q, k=k, v=v, o=torch.empty_like(q),
                           lse=torch.empty(H, L, device=_DEV),
                           scores=torch.zeros(H, nb, L, device=_DEV) if case["stats"] else None)


def _prepare_decode(case, seed):
    L, H, R, n, c = case["L"], case["heads"], case["loops"], case["queries"], min(case["cols"], case["L"])
    w = _workload(dict(case, kind="step", head_dim=128, dtype="bf16", tokens=0.10, q_block=1024))
    ctx, shape = _ctx(), P.shape_of(w)
    g = _generator(seed)
    bf = torch.bfloat16
    st = P.LayerState(ctx, w, _DEV)
    st.k_base, st.v_base = (torch.randn(L, H, 128, generator=g, device=_DEV).to(bf) for _ in range(2))
    order = torch.randperm(L, generator=g, device=_DEV)
    k_now, v_now = st.k_base, st.v_base
    for _r in range(2, R + 1):       # nested active sets of a tenth of the prompt
        m = w.k_tokens
        act = torch.sort(order[:m])[0]
        slot = torch.full((L,), -1, dtype=torch.int32, device=_DEV)
        slot[act] = torch.arange(m, dtype=torch.int32, device=_DEV)
        sel = P.TokenSelection(act.to(torch.int32), slot, None, m)
        st.alloc_stream(sel, rows=False)
        step = lambda x: (x[act].float() + 0.3 * torch.randn(m, H, 128, generator=g, device=_DEV)).to(bf)
        st.quantize(_r, step(k_now), step(v_now), sel)
    # subsets: ascending positions, every (query, head) its own
    idx = torch.empty(n * H, c, dtype=torch.int32, device=_DEV)
    for i in range(0, n * H, 64):
        keys = torch.rand(min(64, n * H - i), L, generator=g, device=_DEV)
        idx[i:i + 64] = torch.sort(torch.topk(keys, c, dim=1)[1], dim=1)[0].to(torch.int32)
    mk = lambda scale: (torch.randn(n, H, 128, generator=g, device=_DEV) * scale)
    q = [mk(1.0)]
    for _r in range(2, R + 1):
        q.append(q[-1] + mk(0.2))
    lse1 = torch.full((n, H), math.log(L) + 0.5, device=_DEV)
    new = lambda: torch.empty(n, H, 128, dtype=bf, device=_DEV)
    return SimpleNamespace(kind="decode", ctx=ctx, shape=shape, st=st, n=n, c=c, R=R, q=[x.to(bf) for x in q], o1=mk(0.3).to(bf),
                           lse1=lse1, idx=idx.view(n, H, c), cnt=torch.full((n, H), c, dtype=torch.int32, device=_DEV),
                           o=[new() for _ in range(R - 1)], lse=[torch.empty(n, H, device=_DEV) for _ in range(R - 1)],
                           p_new=torch.zeros(n, H, c, device=_DEV))


def _prepare_project(case, seed):
    L, n, d = case["L"], case["n"], case["d"]
    g = _generator(seed)
    bf = torch.bfloat16
    mk = lambda *shape: torch.randn(*shape, generator=g, device=_DEV)
    idx = torch.sort(torch.randperm(L, generator=g, device=_DEV)[:n])[0]
    s = SimpleNamespace(kind="project", ctx=_ctx(), L=L, n=n, d=d, fused=case["fused"], idx=idx.to(torch.int32),
                        hidden=mk(L, d).to(bf), w_qkv=(mk(3 * d, d) / d ** 0.5).to(bf), w_o=(mk(d, d) / d ** 0.5).to(bf),
                        attn=mk(n, d).to(bf), stream_rows=mk(n, d).to(bf), out=torch.zeros(L, d, dtype=bf, device=_DEV),
                        status=torch.zeros(1, dtype=torch.int32, device=_DEV))
    if s.fused:                     # loop 2 of a layer whose base is the previous loop's K and V
        w = _workload(dict(case, kind="step", heads=d // 128, head_dim=128, dtype="bf16", loops=2, tokens=n / L, cols=128,
                           q_block=1024, bits=4, group=128))
        s.shape = P.shape_of(w)
        slot = torch.full((L,), -1, dtype=torch.int32, device=_DEV)
        slot[idx] = torch.arange(n, dtype=torch.int32, device=_DEV)
        sel = P.TokenSelection(s.idx, slot, None, n)
        s.payload = _stacked_streams(case, w, [sel], 1)
        base = [mk(L, d).to(bf) for _ in range(2)]
        s.ws = [[torch.empty(n, d, dtype=bf, device=_DEV) for _ in range(2)] for _ in range(2)]
        s.keep = (base, slot)
        s.store = B.make_store(base[0], base[1], _streams_of_layer(s.payload, [sel], 0, 0, s.ws),
                               _streams_of_layer(s.payload, [sel], 0, 1, s.ws))
        s.q_rows = torch.empty(n, d, dtype=bf, device=_DEV)
    else:
        s.qkv = torch.empty(n, 3 * d, dtype=bf, device=_DEV)
    return s


def _prepare_base(case, seed):
    L, H = case["L"], case["heads"]
    w = _workload(dict(case, kind="step", head_dim=128, dtype="bf16", loops=2, tokens=0.1, cols=128, q_block=1024, group=128))
    g = _generator(seed)
    k, v = (torch.randn(L, H, 128, generator=g, device=_DEV).to(torch.bfloat16) for _ in range(2))
    k[torch.randperm(L, generator=g, device=_DEV)[:int(0.02 * L + 0.5)]] *= 8.0
    st = P.LayerState(_ctx(), w, _DEV)
    return SimpleNamespace(kind="base", st=st, k=k, v=v, group=case["group"], tail=case["tail"], k_out=torch.empty_like(k),
                           v_out=torch.empty_like(v))


# ------------------------------------------------------------------------------------------------
# run
# ------------------------------------------------------------------------------------------------
def run(s):
    return {"prefill": _run_prefill, "step": _run_step, "schedule": _run_schedule, "dense": _run_dense, "decode": _run_decode,
            "project": _run_project, "base": _run_base}[s.kind](s)


def _run_prefill(s):
    st = P.LayerState(s.ctx, s.w, _DEV)
    st.dense_loop(*s.qkv1)
    st.select_columns_dense()
    cand, out = None, {}
    for r, k in enumerate(s.toks, start=2):
        sel = P.select_tokens(s.ctx, st.shape, r, s.G[r - 2], s.G[r - 1], cand, k)
        cand = sel.active_idx
        q, kk, v = s.rows[r]
        if s.tensor:
            out["rows", r], _ = st.sparse_loop(r, q, kk, v, sel, indexed=True, carry="write" if r == 2 else "reuse",
                                               rows=True if r == 2 else "cur")
        else:
            out["rows", r], _ = st.sparse_loop(r, q, kk, v, sel)
        out["active", r] = sel.active_idx
    # the column lists themselves are not compared: near-ties move with the last bits of the scores
    for side, streams in (("k", st.k_streams), ("v", st.v_streams)):
        for r, x in enumerate(streams, start=2):
            out[side, "codes", r], out[side, "scale", r], out[side, "zero", r] = x["codes"], x["scale"], x["zero"]
    out["o"], out["q"], out["lse"], out["col_cnt"] = st.o_store, st.q_store, st.lse, st.col_cnt
    return out


def _select_and_gather(s, r, i):
    sel = s.sels[i]
    prev = s.sels[i - 1] if i else None
    B.fl_select_tokens(s.ctx, s.shape, r, s.G[r - 2], s.G[r - 1], prev.active_idx if i else None, prev.n if i else s.w.L,
                       s.toks[i], sel.scores, sel.active_idx, sel.slot_of_pos)
    return sel


def _run_step(s):
    ctx, shape, w, c = s.ctx, s.shape, s.w, s.cols[0]
    row_bytes = 2 * w.d
    for i, r in enumerate(range(2, w.n_loops + 1)):
        sel = _select_and_gather(s, r, i)
        for l, y in enumerate(s.layers):
            B.fl_gather_rows(ctx, y.hidden, sel.active_idx, sel.n, row_bytes, s.x)
            if r == 2:
                B.fl_select_columns(ctx, shape, y.scores, None, None, w.L, c, s.col_idx[0][l], s.col_cnt[0][l])
            if s.packed:
                if r == 2:
                    B.fl_mark_base_rows(ctx, shape, s.col_idx[0][l], s.col_cnt[0][l], c, sel.active_idx, sel.n, y.mask)
                B.fl_dequant_kv_base(ctx, shape, y.state.base_q, s.k_buf, s.v_buf, row_mask=y.mask)
            q, k, v = y.rows[r]
            B.fl_quant_kv_residual(ctx, shape, r, k, v, sel.active_idx, sel.n, y.store)
            # loop 2 reads the source loop's stores, later loops what the loop before left
            first = r == 2
            B.fl_loop_attention_indexed_carry(
                ctx, shape, r, q, y.q1 if first else s.q_out[l], s.q_out[l], sel.active_idx, sel.n, y.store,
                s.col_idx[0][l], s.col_cnt[0][l], c, y.lse1 if first else s.lse_out[l], s.lse_out[l],
                y.o1 if first else s.o_out[l], s.o_out[l], y.write if first else y.reuse, None, status=s.status)
        B.fl_scatter_update(ctx, s.x, sel.active_idx, sel.n, row_bytes, s.g_out)
    return _sparse_outputs(s, {"bg": s.bg, "mass": s.mass, "col_idx": s.col_idx[0], "col_cnt": s.col_cnt[0]})


def _run_schedule(s):
    ctx, shape, w = s.ctx, s.shape, s.w
    row_bytes = 2 * w.d
    last = w.n_loops
    for i, r in enumerate(range(2, last + 1)):
        sel = _select_and_gather(s, r, i)
        for l, y in enumerate(s.layers):
            B.fl_gather_rows(ctx, y.hidden, sel.active_idx, sel.n, row_bytes, s.x)
            idx, cnt, c = s.col_idx[i][l], s.col_cnt[i][l], s.cols[i]
            if r == 2:
                B.fl_select_columns(ctx, shape, y.scores, None, None, w.L, c, idx, cnt)
            q, k, v = y.rows[r]
            B.fl_quant_kv_residual(ctx, shape, r, k, v, sel.active_idx, sel.n, y.store)
            first = r == 2
            scores = y.next_scores[i] if r < last else None
            B.fl_loop_attention_indexed(
                ctx, shape, r, q, y.q1 if first else s.q_out[l], s.q_out[l], sel.active_idx, sel.n, y.store, idx, cnt, c,
                y.lse1 if first else s.lse_out[l], s.lse_out[l], y.o1 if first else s.o_out[l], s.o_out[l], scores,
                status=s.status)
            if r < last:
                B.fl_select_columns(ctx, shape, scores, idx, cnt, c, s.cols[i + 1], s.col_idx[i + 1][l], s.col_cnt[i + 1][l])
        B.fl_scatter_update(ctx, s.x, sel.active_idx, sel.n, row_bytes, s.g_out)
    # the first column lists come from scores made in prepare(); the pruned ones have near-ties (see _run_prefill)
    return _sparse_outputs(s, {"col_idx": s.col_idx[0], "col_cnt": s.col_cnt[-1]})


def _sparse_outputs(s, more):
    out = {"q": s.q_out, "o": s.o_out, "lse": s.lse_out, "g": s.g_out, **more}
    for i, sel in enumerate(s.sels):
        out["active", i] = sel.active_idx
        for side, (codes, scale, zero) in zip("kv", s.payload[i]):
            out[side, "codes", i], out[side, "scale", i], out[side, "zero", i] = codes, scale, zero
    return out


def _run_dense(s):
    B.fl_dense_loop_attention(s.ctx, s.shape, s.q, s.k, s.v, s.o, s.lse, s.scores)
    return {"o": s.o, "lse": s.lse, "scores": s.scores}


def _run_decode(s):
    o_prev, lse_prev = s.o1, s.lse1
    for i, r in enumerate(range(2, s.R + 1)):
        B.fl_decode_attention(s.ctx, s.shape, r, s.q[r - 1], s.q[r - 2], s.n, s.st.store, s.idx, s.cnt, s.c, lse_prev, s.lse[i],
                              o_prev, s.o[i], s.p_new if r == s.R else None)
        o_prev, lse_prev = s.o[i], s.lse[i]
    return {"o": s.o, "lse": s.lse, "p_new": s.p_new}


def _run_project(s):
    n, d, L = s.n, s.d, s.L
    if s.fused:
        B.fl_project_qkv_quant(s.ctx, s.shape, 2, s.hidden, L, s.idx, n, s.w_qkv, s.q_rows, None, s.store, status=s.status)
    else:
        B.fl_project_rows(s.ctx, s.hidden, L, s.idx, n, d, s.w_qkv, 3 * d, s.qkv, n, None, 0, status=s.status)
    # the rows of the residual stream go back to their positions, then the output projection is added into them
    B.fl_scatter_update(s.ctx, s.stream_rows, s.idx, n, 2 * d, s.out)
    B.fl_project_rows(s.ctx, s.attn, n, None, n, d, s.w_o, d, s.out, L, s.idx, 1, status=s.status)
    if s.fused:
        return {"q": s.q_rows, "payload": s.payload, "rows": s.ws, "out": s.out}
    return {"qkv": s.qkv, "out": s.out}


def _run_base(s):
    s.st.pack_base(s.k, s.v, s.group, s.tail)
    s.st.rebuild_base(s.k_out, s.v_out)
    return {"packed": s.st.base_tensors, "k": s.k_out, "v": s.v_out}


# ------------------------------------------------------------------------------------------------
# work and tolerance
# ------------------------------------------------------------------------------------------------
def _pairs(case, n, c):
    """(row, column) pairs of one head: the columns are drawn from the positions up to the end of the row's block."""
    L, qb = case["L"], case["q_block"]
    nb = (L + qb - 1) // qb
    return n / L * sum((min(L, (b + 1) * qb) - b * qb) * min(c, (b + 0.5) * qb) for b in range(nb))


def _touched(case, c):
    """Distinct columns of one head that are in some block's set, if the sets are independent."""
    L, qb = case["L"], case["q_block"]
    nb = (L + qb - 1) // qb
    left = 0.0
    for seg in range(nb):            # positions of this segment can be in the sets of its own and of later blocks
        miss = 1.0
        for b in range(seg, nb):
            miss *= 1.0 - min(1.0, c / min(L, (b + 1) * qb))
        left += (min(L, (seg + 1) * qb) - seg * qb) * (1.0 - miss)
    return left


def _dense_work(L, H, dh, e, stats, nb):
    pairs = 0.5 * L * (L + 1) * H
    return (4.0 * L * H * dh * e + 4.0 * H * L + (2.0 * H * nb * L if stats else 0.0),
            (4.0 if not stats else 6.0) * dh * pairs)


def work(case):
    kind = case["kind"]
    if kind == "dense":
        L, H = case["L"], case["heads"]
        by, fl = _dense_work(L, H, 128, 2, case["stats"], (L + case["q_block"] - 1) // case["q_block"])
        return {"bytes": by, "flops": fl}
    if kind == "decode":
        rows = float(case["queries"]) * case["heads"] * min(case["cols"], case["L"])
        return {"bytes": (case["loops"] - 1) * (rows * (2 * 128 * 2 + 4)), "flops": (case["loops"] - 1) * rows * 8.0 * 128}
    if kind == "project":
        n, d = case["n"], case["d"]
        return {"bytes": 2.0 * n * d * (1 + 3 + 1 + 1 + 2) + 8.0 * d * d, "flops": 8.0 * n * d * d}
    if kind == "base":
        full = case["L"] * case["heads"] * 128.0
        return {"bytes": 2 * full * (2 + 2 + 2 * case["bits"] / 8.0), "flops": 0.0}
    L, H, dh = case["L"], case["heads"], case["head_dim"]
    d, e = H * dh, 2 if case["dtype"] == "bf16" else 4
    nb = (L + case["q_block"] - 1) // case["q_block"]
    toks, cols = _budgets(case)
    bits, layers = case["bits"], case["layers"]
    payload = 2.0 * d * (e if bits == 16 else bits / 8.0 + 4.0 / case["group"])
    by = fl = 0.0
    cand = L
    for i, (n, c) in enumerate(zip(toks, cols)):
        n = min(n, cand)
        by += 2.0 * cand * d * e + 4.0 * L + 2.0 * n * d * e
        both = i == 0 or kind == "schedule"
        one = 2.0 * n * d * e                                              # hidden rows
        if i == 0:
            one += 4.0 * H * sum(min(L, (b + 1) * case["q_block"]) for b in range(nb))
        one += 4.0 * n * d * e + payload * n * (i + 1)                      # residual codec
        one += 2.0 * _touched(case, c) * d * e + (6.0 if both else 4.0) * n * d * e + 4.0 * H * nb * c
        if case.get("packed"):
            one += 2.0 * _touched(case, c) * d * (bits / 8.0 + e)
        by += layers * one
        fl += layers * H * _pairs(case, n, c) * 4.0 * dh * ((2.5 if kind == "schedule" else 2.0) if both else 1.0)
        cand = n
    if kind == "prefill":
        dby, dfl = _dense_work(L, H, dh, e, True, nb)
        by, fl = by + dby, fl + dfl
    return {"bytes": by, "flops": fl}


def tolerance(case):
    kind = case["kind"]
    if kind == "base":
        return "exact"
    if kind == "dense" or kind == "decode":
        return {"rel": 1e-2, "max": 5e-2}
    if case.get("dtype") == "f32":
        return {"rel": 1e-4, "max": 2e-2}
    return {"rel": 1e-2, "max": 1e-1, "differ": 2e-4}      # bf16 rows; a code at a rounding boundary may move
