"""The work a serving engine has this library do, as measurable cases.

A decode round of batched speculative verification is spec_allocate (D-cut),
the target forward (the caller's), spec_verify and spec_commit; the drafter's
side is spec_draft or, with the Markov head, spec_markov_draft; a target that
is split over tensor-parallel ranks runs the spec_shard_* calls through
ShardedRound.  The sizes are the library's workloads (workloads/synth.py:
concurrency 4-64, blocks of 4-16 drafts, vocabularies of 4K-201K) and, for the
allocator, its largest batch.  Every buffer is allocated in prepare(), as an
engine does once per batch slot; run() is one pass through the public entry
points on the current stream.
"""
import math
import weakref

import numpy as np
import torch

import paper_2607_25852_gb300 as spec
from paper_2607_25852_gb300.sharded import ShardedRound, even_bounds

DEV = "cuda"
V_MIN, V_MAX = 4096, 201088
MAX_BYTES = 64 * 17 * V_MAX * 2  # the stress round's logits: no drawn case streams more
RATIOS = ([1, 1, 3, 1], [4, 2, 4, 1])  # the budgets 1/4, 1/2, 3/4, 1 of the full block


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest whole round, driven call by call: launches and latency
        dict(name="round_tiny", kind="round", B=4, K=4, V=4096, t=1.0, dtype="f32", dense=False, H=64),
        # greedy decoding at concurrency 16
        dict(name="verify_greedy", kind="verify", B=16, K=16, V=128256, t=0.0, dtype="bf16", dense=False, packed=False),
        # sampled decoding at concurrency 32 against the drafter's distributions
        dict(name="verify_sampled", kind="verify", B=32, K=8, V=151936, t=0.8, dtype="bf16", dense=True, packed=False),
        # fp32 logits and q over an odd vocabulary (rows off the 16-byte grid), ragged depths
        dict(name="verify_ragged", kind="verify", B=12, K=7, V=100003, t=0.7, dtype="f32", dense=True, packed=True),
        # a budgeted round whose shape the device chooses, replayed as graphs
        dict(name="round_graph", kind="graph", B=64, K=16, V=128256, t=1.0, dtype="bf16", dense=False, H=4096),
        # the flagship: the whole round at concurrency 64 over the largest vocabulary
        dict(name="round_stress", kind="round", B=64, K=16, V=201088, t=1.0, dtype="bf16", dense=True, H=7168),
        # the drafter's step for that batch
        dict(name="draft_stress", kind="draft", B=64, K=16, V=201088, tau=1.0, dtype="bf16"),
        # greedy drafting at concurrency 16
        dict(name="draft_greedy", kind="draft", B=16, K=16, V=128256, tau=0.0, dtype="bf16"),
        # the Markov head over a block of 8 (7 drafts) at concurrency 64
        dict(name="markov_block", kind="markov", B=64, K=7, V=201088, r=256, tau=1.0),
        # greedy Markov drafting, a wide batch with a low-rank head
        dict(name="markov_greedy", kind="markov", B=96, K=4, V=128256, r=128, tau=0.0),
        # one rank's part of the flagship round under tensor parallelism 8, replayed as a graph
        dict(name="shard_rank", kind="shard", B=64, K=16, V=201088, S=8, rank=3, t=1.0, dtype="bf16", dense=True),
        # D-cut over the largest batch the allocator takes
        dict(name="allocate_large", kind="allocate", B=256, K=31, M=16),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_vocab(rng):
    """A vocabulary of the range: mostly whole groups of 64, sometimes any size."""
    V = _log_uniform(rng, V_MIN, V_MAX)
    return V if rng.random() < 0.3 else max(V_MIN, V // 64 * 64)


def _fit(B, rows_per_request, V, esize):
    """B lowered until the batch's rows stay within the largest listed case."""
    return max(1, min(B, MAX_BYTES // (rows_per_request * V * esize)))


def draw(rng):
    kind = rng.choice(["verify", "verify", "round", "graph", "draft", "draft", "markov", "shard", "allocate"])
    if kind == "allocate":
        K = _log_uniform(rng, 1, 31)
        return dict(kind=kind, B=_log_uniform(rng, 4, min(512, 8192 // (K + 1))), K=K, M=_log_uniform(rng, 1, 32))
    V, K = _draw_vocab(rng), rng.randint(1, 16)
    dtype = "bf16" if rng.random() < 0.75 else "f32"
    esize = 2 if dtype == "bf16" else 4
    if kind == "markov":
        K, r = rng.randint(1, 7), rng.choice([64, 128, 192, 256])
        B = _log_uniform(rng, 1, 128)
        while K > 1 and K * V * (r + B) > 7 * V_MAX * (256 + 64):
            K -= 1
        while V * (r + B) * K > 7 * V_MAX * (256 + 64):
            V //= 2
        return dict(kind=kind, B=B, K=K, V=V, r=r, tau=rng.choice([0.0, 0.6, 1.0]))
    if kind == "draft":
        return dict(kind=kind, B=_fit(_log_uniform(rng, 1, 64), K, V, esize), K=K, V=V,
                    tau=rng.choice([0.0, 0.7, 1.0]), dtype=dtype)
    B = _fit(_log_uniform(rng, 1, 64), K + 1, V, esize)
    t = rng.choice([0.0, 0.6, 0.8, 1.0, 1.0])
    dense = t > 0 and rng.random() < 0.6
    if kind == "verify":
        return dict(kind=kind, B=B, K=K, V=V, t=t, dtype=dtype, dense=dense, packed=rng.random() < 0.4)
    if kind == "shard":
        S = rng.choice([2, 4, 8])
        return dict(kind=kind, B=B, K=K, V=V, S=S, rank=rng.randrange(S), t=t, dtype=dtype, dense=dense)
    H = rng.choice([1024, 2048, 4096, 7168])
    return dict(kind=kind, B=B, K=K, V=V, t=t, dtype=dtype, dense=dense and kind == "round", H=H)


def work(case):
    kind, B, K = case["kind"], case["B"], case["K"]
    if kind == "allocate":
        n = B * (K + 1)
        return {"bytes": 4 * B * K * 2 + 12 * B + 12 * n + 8 * B + 8 * case["M"], "flops": n * math.log2(n)}
    V = case["V"]
    if kind == "markov":
        return {"bytes": K * V * (2 * case["r"] + 2 * B), "flops": K * B * V * (2 * case["r"] + 4)}
    e = 2 if case["dtype"] == "bf16" else 4
    if kind == "draft":
        return {"bytes": B * K * V * e + 12 * B * K, "flops": 4 * B * K * V}
    if kind == "graph":
        rows = spec.spec_budget_from_ratios(B, K, *RATIOS)[0]
    elif kind == "verify" and case["packed"]:
        rows = B * (K / 2 + 1)
    else:
        rows = B * (K + 1)
    if kind == "shard":
        V /= case["S"]
    moved = rows * V * e + (B * V * e if case["dense"] else 0)
    if kind in ("round", "graph"):
        moved += 2 * 2 * case["H"] * B * 2  # about two committed hidden rows per request, read and written
    return {"bytes": moved, "flops": 4 * rows * V}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _requests(B, rng):
    """Philox seeds, request ids and positions of a running batch."""
    i64 = lambda hi: torch.as_tensor(rng.integers(0, hi, B), dtype=torch.int64, device=DEV)
    return dict(seeds=i64(2**62), ids=i64(2**40), pos=i64(32768))


def _confidences(B, K, rng):
    """Half the requests chat-like, half code-like (confident drafters)."""
    half = B // 2
    c = np.concatenate([rng.beta(2.0, 2.0, (half, K)), rng.beta(8.0, 1.0, (B - half, K))])
    return np.maximum(c, 0.02).astype(np.float32)


def _dcut(conf, Ts, costs):
    """Section 4.2 in numpy: the chosen budget, the keep depths and U(T_m)."""
    B, K = conf.shape
    s = np.ones((B, K + 1), np.float32)
    for k in range(K):
        s[:, k + 1] = s[:, k] * conf[:, k]
    k_of, i_of = np.tile(np.arange(K + 1), B), np.repeat(np.arange(B), K + 1)
    order = np.lexsort((i_of, k_of, -s.reshape(-1)))
    prefix = np.cumsum(np.floor(s.reshape(-1)[order].astype(np.float64) * 2.0**40)) * 2.0**-40
    U = np.asarray([prefix[T - 1] for T in Ts])
    T = int(Ts[int(np.argmax(U / np.asarray(costs)))])
    return T, np.bincount(i_of[order[:T]], minlength=B) - 1, U


def _cost(T):
    return 1.0 + 0.004 * max(0, T - 256)  # flat until the target forward turns compute-bound


def _depths(case, rng):
    """Kept drafts per request, and what the allocator is given."""
    B, K, kind = case["B"], case["K"], case["kind"]
    if kind in ("round", "graph"):
        conf = _confidences(B, K, rng)
        Ts = spec.spec_budget_from_ratios(B, K, *RATIOS)
        # call by call at light load (a flat cost keeps every draft); graphs under the profiled cost
        costs = [1.0 if kind == "round" else _cost(T) for T in Ts]
        return _dcut(conf, Ts, costs)[1], dict(conf=conf, Ts=Ts, costs=costs)
    if case.get("packed"):
        return rng.integers(0, K + 1, B), None
    return np.full(B, K), None


def _verify_inputs(case, seed):
    """Target logits of the packed rows, the drafts and the drafter's q.

    With dense q the drafter is the target plus noise and the drafts are drawn
    from its softmax; otherwise a peak (row max + 8) sits at the draft with
    probability 0.8, else at another token."""
    B, K, V, t = case["B"], case["K"], case["V"], case["t"]
    rng = np.random.default_rng(seed)
    g = torch.Generator(device=DEV).manual_seed(seed)
    depth, alloc = _depths(case, rng)
    offs = np.concatenate([[0], np.cumsum(depth + 1)])
    R = int(offs[-1])
    dt = _dtype(case)
    drafts = torch.as_tensor(rng.integers(0, V, (B, K)), dtype=torch.int32, device=DEV)
    # graphs read one logits buffer of the full block's rows, whatever the budget
    logits = torch.zeros((B * (K + 1) if case["kind"] == "graph" else R, V), dtype=dt, device=DEV)
    q = torch.empty((B, K, V), dtype=dt, device=DEV) if case["dense"] else None
    for i in range(B):
        n, r0 = int(depth[i]), int(offs[i])
        rows = torch.randn((n + 1, V), generator=g, device=DEV) * 3.0
        if q is not None:
            noisy = torch.randn((K, V), generator=g, device=DEV)
            noisy[:n] += rows[:n]
            q[i] = torch.softmax(noisy / t, dim=-1).to(dt)
            race = torch.empty((K, V), device=DEV).exponential_(generator=g)
            drafts[i] = (q[i].float() / race).argmax(dim=-1).to(torch.int32)
        else:
            hit = torch.as_tensor(rng.random(n + 1) < 0.8, device=DEV)
            other = torch.as_tensor(rng.integers(0, V, n + 1), device=DEV)
            other[:n] = torch.where(hit[:n], drafts[i, :n].long(), other[:n])
            rows.scatter_(1, other[:, None], rows.amax(dim=1, keepdim=True) + 8.0)
        logits[r0:r0 + n + 1] = rows.to(dt)
    x = dict(logits=logits, drafts=drafts, q=q, depth=depth, offs=offs, alloc=alloc, **_requests(B, rng))
    if case["kind"] in ("round", "graph"):
        x["hidden"] = torch.randn((logits.shape[0], case["H"]), generator=g, device=DEV).to(torch.bfloat16)
        x["last"] = torch.as_tensor(rng.integers(0, V, B), dtype=torch.int32, device=DEV)
    return x


def _draft_inputs(case, seed):
    B, K, V = case["B"], case["K"], case["V"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    x = dict(logits=torch.empty((B, K, V), dtype=_dtype(case), device=DEV), **_requests(B, np.random.default_rng(seed)))
    for i in range(B):
        x["logits"][i] = (torch.randn((K, V), generator=g, device=DEV) * 3.1).to(_dtype(case))
    return x


def _markov_inputs(case, seed):
    B, K, V, r = case["B"], case["K"], case["V"], case["r"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    rng = np.random.default_rng(seed)
    normal = lambda *shape, std: (torch.randn(shape, generator=g, device=DEV) * std).to(torch.bfloat16)
    return dict(U=normal(B, K, V, std=2.5), W1=normal(V, r, std=0.3), W2T=normal(V, r, std=0.3),
                x0=torch.as_tensor(rng.integers(0, V, B), dtype=torch.int32, device=DEV), **_requests(B, rng))


def _allocate_inputs(case, seed):
    B, K, M = case["B"], case["K"], case["M"]
    rng = np.random.default_rng(seed)
    full = B * (K + 1)
    Ts = [max(B, full * (m + 1) // M) for m in range(M)]
    i32 = lambda *shape: torch.as_tensor(rng.integers(0, V_MAX, shape), dtype=torch.int32, device=DEV)
    return dict(conf=_confidences(B, K, rng), Ts=Ts, costs=[_cost(T) for T in Ts], last=i32(B), drafts=i32(B, K),
                pos=_requests(B, rng)["pos"])


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def _zeros(*shape, dtype=torch.int32):
    return torch.zeros(shape, dtype=dtype, device=DEV)


def _verify_outputs(B, K):
    return dict(accepted=_zeros(B), tokens=_zeros(B, K + 1), p_draft=_zeros(B, K, dtype=torch.float32),
                row_stats=_zeros(B * (K + 1), 2, dtype=torch.float32))


def _allocate_outputs(B, K, M):
    n = B * (K + 1)
    return dict(depth=_zeros(B), row_offsets=_zeros(B + 1), packed_tokens=_zeros(n),
                packed_pos=_zeros(n, dtype=torch.int64), chosen=_zeros(1), utility=_zeros(M, dtype=torch.float64))


class _Graphs:
    """Captured graphs, destroyed with the state that holds them."""

    def __init__(self):
        self.handles = []
        weakref.finalize(self, _Graphs._destroy, self.handles)

    @staticmethod
    def _destroy(handles):
        while handles:
            spec.spec_graph_destroy(handles.pop())

    def capture(self, stream, enqueue, device_launch=False):
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            spec.spec_graph_begin_capture(stream)
            enqueue()
            self.handles.append(spec.spec_graph_end_capture(stream, device_launch))
        return self.handles[-1]


def _run_allocate(s):
    x, o = s["x"], s["alloc"]
    a = x["alloc"] if "alloc" in x else x
    spec.spec_allocate(s["conf"], a["Ts"], a["costs"], x["last"], x["drafts"], x["pos"], o["depth"], o["row_offsets"],
                       o["packed_tokens"], o["packed_pos"], o["chosen"], o["utility"], s["status"])


def _run_verify(s, depth, offsets):
    x, o, c = s["x"], s["ver"], s["case"]
    spec.spec_verify(x["logits"], x["drafts"], x["q"], c["B"], c["K"], c["V"], c["t"], x["seeds"], x["ids"], x["pos"],
                     o["accepted"], o["tokens"], s["ws"], row_offsets=offsets, depth=depth, p_draft_out=o["p_draft"],
                     row_stats_out=o["row_stats"], status=s["status"])


def _run_commit(s):
    x, o, c = s["x"], s["com"], s["case"]
    spec.spec_commit(s["ver"]["accepted"], s["ver"]["tokens"], x["hidden"], c["B"], c["K"], o["tokens"], o["offsets"],
                     o["hidden"], row_offsets=s["alloc"]["row_offsets"], status=s["status"])


def _after_allocate(s):
    _run_verify(s, s["alloc"]["depth"], s["alloc"]["row_offsets"])
    _run_commit(s)


def _prepare_shard(case, s):
    """One rank's buffers, with the other ranks' records of this batch already
    gathered: the exchange is then the copy of the rank's own records."""
    B, K, V, S, rank, t = (case[k] for k in ("B", "K", "V", "S", "rank", "t"))
    x, o, bounds = s["x"], s["ver"], even_bounds(case["V"], case["S"])
    part = lambda a, k: None if a is None else a[..., bounds[k]:bounds[k + 1]].contiguous()
    every = ShardedRound(B, K, V, bounds, device=DEV, local=True)
    every.run([part(x["logits"], k) for k in range(S)], x["drafts"],
              None if x["q"] is None else [part(x["q"], k) for k in range(S)], t, x["seeds"], x["ids"], x["pos"],
              o["accepted"], o["tokens"], p_draft_out=o["p_draft"], row_stats_out=o["row_stats"], status=s["status"])

    def gather(local, out):
        out[rank * local.numel():(rank + 1) * local.numel()].copy_(local)

    mine = ShardedRound(B, K, V, bounds, rank=rank, device=DEV, gather=gather)
    mine.stats.copy_(every.stats)
    mine.races.copy_(every.races)
    lg, q = part(x.pop("logits"), rank), part(x.pop("q"), rank)
    s["stream"], s["graphs"] = torch.cuda.Stream(), _Graphs()
    s["keep"] = (mine, lg, q)
    s["graph"] = s["graphs"].capture(s["stream"], lambda: mine.run(
        lg, x["drafts"], q, t, x["seeds"], x["ids"], x["pos"], o["accepted"], o["tokens"], p_draft_out=o["p_draft"],
        row_stats_out=o["row_stats"], status=s["status"], stream=s["stream"]))


def prepare(case, seed):
    kind, B, K = case["kind"], case["B"], case["K"]
    s = dict(case=case, status=_zeros(1))
    if kind == "allocate":
        s["x"] = _allocate_inputs(case, seed)
        s["conf"] = torch.as_tensor(s["x"]["conf"], device=DEV)
        s["alloc"] = _allocate_outputs(B, K, case["M"])
        return s
    V = case["V"]
    if kind in ("draft", "markov"):
        s["x"] = _draft_inputs(case, seed) if kind == "draft" else _markov_inputs(case, seed)
        s["ws"] = spec.draft_workspace(B, K, V) if kind == "draft" else spec.markov_workspace(B, K, V, case["r"])
        s["out"] = dict(drafts=_zeros(B, K), conf=_zeros(B, K, dtype=torch.float32),
                        scores=_zeros(B, K + 1, dtype=torch.float32), row_stats=_zeros(B * K, 2, dtype=torch.float32))
        return s
    x = s["x"] = _verify_inputs(case, seed)
    s["ver"] = _verify_outputs(B, K)
    if kind == "shard":
        _prepare_shard(case, s)
        return s
    s["ws"] = spec.verify_workspace(B, K, V)
    if kind == "verify":
        packed = case["packed"]
        s["depth"] = torch.as_tensor(x["depth"], dtype=torch.int32, device=DEV) if packed else None
        s["offsets"] = torch.as_tensor(x["offs"], dtype=torch.int32, device=DEV) if packed else None
        return s
    s["conf"] = torch.as_tensor(x["alloc"]["conf"], device=DEV)
    s["alloc"] = _allocate_outputs(B, K, len(x["alloc"]["Ts"]))
    s["com"] = dict(tokens=_zeros(B * (K + 1)), offsets=_zeros(B + 1),
                    hidden=_zeros(B * (K + 1), case["H"], dtype=torch.bfloat16))
    if kind == "graph":
        s["stream"], s["graphs"], s["launched"] = torch.cuda.Stream(), _Graphs(), _zeros(1)
        Ts = x["alloc"]["Ts"]
        rounds = [s["graphs"].capture(s["stream"], lambda: _after_allocate(s), True) for _ in Ts]

        def choose():
            _run_allocate(s)
            spec.spec_select_round(s["alloc"]["chosen"], Ts, rounds, s["launched"], s["status"])

        s["graph"] = s["graphs"].capture(s["stream"], choose)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "allocate":
        _run_allocate(s)
        return [s["alloc"], s["status"]]
    if kind in ("draft", "markov"):
        x, o = s["x"], s["out"]
        if kind == "draft":
            spec.spec_draft(x["logits"], case["tau"], x["seeds"], x["ids"], x["pos"], o["drafts"], o["conf"], s["ws"],
                            scores_out=o["scores"], row_stats_out=o["row_stats"], status=s["status"])
        else:
            spec.spec_markov_draft(x["U"], x["W1"], x["W2T"], x["x0"], case["tau"], x["seeds"], x["ids"], x["pos"],
                                   o["drafts"], o["conf"], s["ws"], scores_out=o["scores"],
                                   row_stats_out=o["row_stats"], status=s["status"])
        return [o, s["status"]]
    if kind == "verify":
        _run_verify(s, s["depth"], s["offsets"])
        return [s["ver"], s["status"]]
    if kind == "shard":
        spec.spec_graph_launch(s["graph"])
        return [s["ver"], s["status"]]
    if kind == "graph":
        spec.spec_graph_launch(s["graph"])
    else:
        _run_allocate(s)
        _after_allocate(s)
    return [s["alloc"], s["ver"], s["com"], s["status"]]


# ---------------------------------------------------------------------------
# The same outputs in 64 bits
# ---------------------------------------------------------------------------
def _exact_temperature(t):
    return float(np.float32(t))  # the entry points take a float


def _exact_rows(logits, t, tokens):
    """(row statistics [R, 2], softmax probability at `tokens` [R]) of the rows."""
    st, p = [], []
    for r in range(logits.shape[0]):
        row = logits[r].double() / t
        m = row.max()
        S = torch.exp(row - m).sum()
        st.append(torch.stack([m, S.log()]))
        p.append(torch.exp(row[tokens[r]] - m) / S)
    return torch.stack(st), torch.stack(p)


def _exact_verify(case, x):
    B, K, t = case["B"], case["K"], case["t"]
    stats = torch.zeros((B * (K + 1), 2), dtype=torch.float64, device=DEV)
    p_draft = torch.zeros((B, K), dtype=torch.float64, device=DEV)
    for i in range(B):
        n, r0 = int(x["depth"][i]), int(x["offs"][i])
        rows = x["logits"][r0:r0 + n + 1]
        if t == 0:
            best, at = rows.double().max(dim=1)
            stats[r0:r0 + n + 1, 0] = best
            p_draft[i, :n] = (at[:n] == x["drafts"][i, :n]).double()
        else:
            z = torch.cat([x["drafts"][i, :n].long(), torch.zeros(1, dtype=torch.int64, device=DEV)])
            stats[r0:r0 + n + 1], p = _exact_rows(rows, _exact_temperature(t), z)
            p_draft[i, :n] = p[:n]
    return dict(accepted=None, tokens=None, p_draft=p_draft, row_stats=stats)


def _philox_words(position, request, seed, purpose, subs):
    """Philox4x32-10 words [len(subs) * 4] at the draw counters of spec.h."""
    u = lambda v: np.uint64(int(v) & 0xFFFFFFFF)
    n, low = len(subs), np.uint64(0xFFFFFFFF)
    c = [np.full(n, u(position)), np.full(n, u(request)), np.full(n, u(int(request) >> 32)),
         np.asarray(subs, np.uint64) | np.uint64(purpose << 28)]
    k = [int(seed) & 0xFFFFFFFF, (int(seed) >> 32) & 0xFFFFFFFF]
    for _ in range(10):
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ u(k[0]), b & low, (a >> np.uint64(32)) ^ c[3] ^ u(k[1]), a & low]
        k = [k[0] + 0x9E3779B9, k[1] + 0xBB67AE85]
    return np.stack(c, axis=1).reshape(-1)


def _race_variates(words):
    w = words.astype(np.uint32) >> np.uint32(9)
    return torch.as_tensor(-np.log((2.0 * w + 1.0) * 2.0**-24), device=DEV)


def _exact_draw(row, tau, position, request, seed):
    """One draft of the two-level race over a float64 row: (token, q(token), statistics)."""
    V = row.numel()
    row = row / (_exact_temperature(tau) if tau > 0 else 1.0)
    m = row.max()
    w = torch.exp(row - m)
    S = w.sum()
    if tau == 0:
        z = int(row.argmax())
    else:
        nb = -(-V // 256)
        pad = torch.zeros(nb * 256, dtype=torch.float64, device=DEV)
        pad[:V] = w
        E = _race_variates(_philox_words(position, request, seed, 4, np.arange(-(-nb // 4))))[:nb]
        b = int((E / pad.view(nb, 256).sum(dim=1)).argmin())
        E = _race_variates(_philox_words(position, request, seed, 5, np.arange(64) + 64 * b))
        z = 256 * b + int((E / pad.view(nb, 256)[b]).argmin())
    return z, w[z] / S, torch.stack([m, S.log()])


def _exact_block(case, x):
    """Drafts of a block in order (the Markov head's logits depend on the draft before)."""
    B, K, markov = case["B"], case["K"], case["kind"] == "markov"
    conf = torch.zeros((B, K), dtype=torch.float64, device=DEV)
    stats = torch.zeros((B * K, 2), dtype=torch.float64, device=DEV)
    ids, seeds, pos = (x[k].tolist() for k in ("ids", "seeds", "pos"))
    prev = x["x0"].long() if markov else None
    for k in range(K):
        bias = x["W1"][prev].double() @ x["W2T"].double().T if markov else None
        drawn = []
        for i in range(B):
            row = x["U"][i, k].double() + bias[i] if markov else x["logits"][i, k].double()
            z, conf[i, k], stats[i * K + k] = _exact_draw(row, case["tau"], pos[i] + k + 1, ids[i], seeds[i])
            drawn.append(z)
        prev = torch.as_tensor(drawn, device=DEV)
    scores = torch.cat([torch.ones((B, 1), dtype=torch.float64, device=DEV), conf.cumprod(dim=1)], dim=1)
    return dict(drafts=None, conf=conf, scores=scores, row_stats=stats)


def _exact_allocate(x):
    none = dict.fromkeys(("depth", "row_offsets", "packed_tokens", "packed_pos", "chosen"))
    return dict(none, utility=torch.as_tensor(_dcut(x["conf"], x["Ts"], x["costs"])[2]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "allocate":
        return [_exact_allocate(_allocate_inputs(case, seed)), None]
    if kind in ("draft", "markov"):
        return [_exact_block(case, (_draft_inputs if kind == "draft" else _markov_inputs)(case, seed)), None]
    x = _verify_inputs(case, seed)
    ver = _exact_verify(case, x)
    if kind in ("verify", "shard"):
        return [ver, None]
    return [_exact_allocate(x["alloc"]), ver, dict(tokens=None, offsets=None, hidden=None), None]
