"""What the library's speed is measured on: calls that a user of the trace finder makes.

A task runtime hashes its tasks to tokens, hands windows of its history to the
repeat finder (one at a time, as one batch, or through the server), matches the
traces found against the stream and replays them; a study of trace quality
solves short windows exactly.  Every case goes through the C ABI with
caller-owned buffers, as a runtime does (the served one through the Server
object).  The inputs are made on the GPU from the seed, in the shapes that the
repository's own workloads have: loop bodies with noise, nested loops of hashed
task descriptors, runs, uniform noise, phases of changing loops.

All outputs are whole numbers or bytes, so two correct runs agree exactly.  The
output arrays are zeroed once, when they are made: how many entries a call
writes is in its counts.  The doubling-round and selection-round counts are
diagnostics of one run and are not among the outputs.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2406_18111_gb300 as gb

_CTX = None


def _ctx():
    # a program keeps one context (its workspace grows to its largest call)
    global _CTX
    if _CTX is None:
        h = ctypes.c_void_p()
        _call(gb.lib().apo_create(ctypes.byref(h), 0))
        _CTX = h
    return _CTX


def _call(code):
    if code != gb.APO_OK:
        raise gb.ApoError(code, gb.lib().apo_last_error().decode(errors="replace"))


def _p(t):
    return None if t is None else t.data_ptr()


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _zeros(n, dtype=torch.int32):
    return torch.zeros(max(1, n), dtype=dtype, device="cuda")


# ------------------------------------------------------------------ inputs
def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(seed * 1000 + salt)


def _noise(s, share, alphabet, g):
    """Replaces about `share` of s by tokens uniform on [0, alphabet)."""
    hit = torch.rand(s.shape[0], device="cuda", generator=g) < share
    new = torch.randint(0, alphabet, (s.shape[0],), device="cuda", generator=g, dtype=s.dtype)
    return torch.where(hit, new, s)


def _spread(count, lo, hi):
    """`count` lengths spread over [lo, hi] by their logarithm, the same for every seed, in a mixed order."""
    q = (torch.arange(count, device="cuda", dtype=torch.float64) * 0.6180339887498949 + 0.37) % 1.0
    return torch.clamp((lo * torch.exp(q * math.log(hi / lo))).long(), lo, hi)


def _log_uniform(count, lo, hi, g):
    u = torch.rand(count, device="cuda", generator=g, dtype=torch.float64)
    return torch.clamp(torch.exp(math.log(lo) + u * (math.log(hi) - math.log(lo))).long(), lo, hi)


def _segments(lens, lo_period, hi_period, share, alphabet, g):
    """Back-to-back loops (period uniform on [lo_period, hi_period]) of the given lengths, with noise; int32."""
    n, k = int(lens.sum()), lens.shape[0]
    off = torch.cumsum(lens, 0) - lens
    period = torch.randint(lo_period, hi_period + 1, (k,), device="cuda", generator=g)
    pos = torch.arange(n, device="cuda") - torch.repeat_interleave(off, lens, output_size=n)
    s = (pos % torch.repeat_interleave(period, lens, output_size=n)).int()
    return _noise(s, share, alphabet, g)


def _phases(n, lo, hi, lo_period, hi_period, share, alphabet, g):
    """A stream of n tokens whose loop changes every lo .. hi tokens."""
    lens = _log_uniform(2 * n // lo + 2, lo, hi, g)
    end = torch.cumsum(lens, 0)
    k = int((end < n).sum()) + 1
    lens = lens[:k].clone()
    lens[-1] -= int(end[k - 1]) - n
    return _segments(lens, lo_period, hi_period, share, alphabet, g)


def _tasks(n, share, g):
    """Task descriptors of a nested loop (7 inner tasks in a body of 120, 25 bodies to the outer iteration), `share`
    of them replaced by one of 2^16 others; 1 to 8 region arguments each."""
    pool = 7 + 25 + (1 << 16)
    nargs = torch.randint(1, 9, (pool,), device="cuda", generator=g)
    first = torch.cumsum(nargs, 0) - nargs
    m = int(nargs.sum())
    tid = torch.randint(-2**31, 2**31, (pool,), device="cuda", generator=g).int()
    region = torch.randint(-2**31, 2**31, (m,), device="cuda", generator=g).int()
    mask = torch.randint(-2**63, 2**63 - 1, (m,), device="cuda", generator=g)
    priv = torch.randint(0, 4, (m,), device="cuda", generator=g).to(torch.uint8)
    tid[7:32] = tid[7].clone()
    region[first[7:32]] = 0x40000000 + torch.arange(25, device="cuda", dtype=torch.int32)
    j = torch.arange(n, device="cuda")
    o = j % 3000
    d = torch.where(o % 120 < 119, (o % 120) % 7, 7 + o // 120)
    hit = torch.rand(n, device="cuda", generator=g) < share
    d = torch.where(hit, torch.randint(32, pool, (n,), device="cuda", generator=g), d)
    na = nargs[d]
    arg_off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    arg_off[1:] = torch.cumsum(na, 0)
    total = int(arg_off[-1])
    src = torch.repeat_interleave(first[d] - arg_off[:-1], na, output_size=total) + torch.arange(total, device="cuda")
    return {"task_id": tid[d].contiguous(), "arg_off": arg_off.int(), "region": region[src].contiguous(),
            "field_mask": mask[src].contiguous(), "priv": priv[src].contiguous()}


def _window(case, seed):
    """One window's tokens: int32 (u32) or int64 (u64)."""
    n, g = case["n"], _gen(seed, 1)
    what = case["content"]
    if what == "loop":  # a loop body with 5% of irregular tasks
        s = (torch.arange(n, device="cuda") % case["period"]).int()
        s = _noise(s, 0.05, 1000, g)
    elif what == "tasks":  # hashed descriptors of a nested loop, 1% irregular
        return _hash_call(_tasks(n, 0.01, g))()
    elif what == "runs":  # a constant run, a period-2 run and a period-3 run, about a third each
        j = torch.arange(n, device="cuda")
        cut = torch.randint(0, n // 16 + 1, (2,), device="cuda", generator=g)
        t, u = n // 3 + cut[0], 2 * n // 3 + cut[1]
        s = torch.where(j < t, 0 * j, torch.where(j < u, 1 + (j - t) % 2, 3 + (j - u) % 3)).int()
    else:  # uniform u32
        s = torch.randint(-2**31, 2**31, (n,), device="cuda", generator=g).int()
    if case["bytes"] == 8:  # the same equalities over 64-bit tokens
        s = s.long() * 0x9E3779B97F4A7C1 + 12345
    return s


def _offsets(lens):
    off = np.zeros(len(lens) + 1, dtype=np.uint64)
    off[1:] = np.cumsum(lens)
    return off


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # Alg. 1's Hash over a history of 2^20 task descriptors
        {"name": "hash_1m", "kind": "hash", "n": 1 << 20},
        # one small history slice, every output asked for: launches and host waits count
        {"name": "repeats_4k", "kind": "repeats", "n": 4096, "content": "loop", "period": 50, "bytes": 4, "min_len": 5,
         "stages": True, "sa_lcp": False},
        # one large window of hashed tasks; SA and LCP are kept for the matcher
        {"name": "repeats_tasks_1m", "kind": "repeats", "n": 1 << 20, "content": "tasks", "period": 0, "bytes": 8,
         "min_len": 5, "stages": False, "sa_lcp": True},
        # the deepest repeats: a program that issues one, two or three tasks over and over
        {"name": "repeats_runs_16m", "kind": "repeats", "n": 1 << 24, "content": "runs", "period": 0, "bytes": 4,
         "min_len": 5, "stages": False, "sa_lcp": True},
        # nothing repeats: what a large irregular history costs
        {"name": "repeats_random_16m", "kind": "repeats", "n": 1 << 24, "content": "random", "period": 0, "bytes": 4,
         "min_len": 5, "stages": False, "sa_lcp": True},
        # the online finder's slices (unit 250, buffer 5000) of hashed tokens that one batch picks up
        {"name": "batched_slices", "kind": "batched", "windows": 40, "lo": 250, "hi": 5000, "bytes": 8, "min_len": 5,
         "stages": False},
        # many histories at once, of uneven length, every output asked for
        {"name": "batched_512", "kind": "batched", "windows": 512, "lo": 1024, "hi": 262144, "bytes": 4, "min_len": 5,
         "stages": True},
        # the traces of a window matched against that window, its suffix array at hand
        {"name": "match_traces_1m", "kind": "match_traces", "n": 1 << 20, "content": "tasks", "period": 0, "bytes": 8,
         "min_len": 5},
        # a large trace catalogue against a long recorded stream
        {"name": "match_stream_64m", "kind": "match_stream", "n": 1 << 26, "patterns": 10000, "lo": 5, "hi": 2000,
         "bytes": 4},
        # the replayer over a program whose loops change, with the traces the online finder reported
        {"name": "replay_1m", "kind": "replay", "n": 1 << 20, "max_trace_len": 0},
        # a burst of analysis requests from the host
        {"name": "served_burst", "kind": "served", "requests": 32, "lo": 4096, "hi": 1 << 20, "min_len": 5},
        # the quality study's short windows, solved exactly
        {"name": "optimum_64k", "kind": "optimum", "windows": 1 << 16, "n": 20, "min_len": 2},
    ]


def draw(rng):
    def log(lo, hi):
        return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))

    kind = rng.choice(["hash", "repeats", "repeats", "repeats", "batched", "batched", "match_traces", "match_stream",
                       "replay", "served", "optimum"])
    if kind == "hash":
        return {"kind": kind, "n": log(1 << 12, 1 << 20)}
    if kind in ("repeats", "match_traces"):
        content = rng.choice(["loop", "loop", "tasks", "runs", "random"] if kind == "repeats" else ["loop", "tasks"])
        case = {"kind": kind, "content": content, "period": rng.randint(3, 5000),
                "n": log(500, 1 << (20 if content in ("loop", "tasks") else 23)),
                "bytes": 8 if content == "tasks" else rng.choice([4, 8]), "min_len": rng.choice([5, 5, 25, 100])}
        if kind == "repeats":
            case |= {"stages": rng.random() < 0.5, "sa_lcp": content == "random" or rng.random() < 0.5}
        else:  # short enough a loop that there are traces to match
            case |= {"min_len": 5, "period": rng.randint(20, max(20, min(1000, case["n"] // 8)))}
        return case
    if kind == "batched":
        hi = log(1000, 1 << 17)
        return {"kind": kind, "windows": log(2, 300), "lo": max(100, hi // rng.randint(2, 100)), "hi": hi,
                "bytes": rng.choice([4, 8]), "min_len": rng.choice([5, 25]), "stages": rng.random() < 0.5}
    if kind == "match_stream":
        hi = log(20, 2000)
        return {"kind": kind, "n": log(1 << 13, 1 << 24), "patterns": log(10, 10000), "lo": 5, "hi": hi,
                "bytes": rng.choice([4, 8])}
    if kind == "replay":
        return {"kind": kind, "n": log(1 << 13, 1 << 20), "max_trace_len": rng.choice([0, 0, 200])}
    if kind == "served":
        return {"kind": kind, "requests": log(2, 40), "lo": 1000, "hi": log(4096, 1 << 19), "min_len": 5}
    return {"kind": kind, "windows": log(1 << 9, 1 << 15), "n": rng.randint(8, 20), "min_len": rng.choice([2, 3])}


# ------------------------------------------------------------------ the calls
def _hash_call(t):
    n = t["task_id"].shape[0]
    out = _zeros(n, torch.int64)
    tasks = gb.apo_tasks(n, _p(t["task_id"]), _p(t["arg_off"]), _p(t["region"]), _p(t["field_mask"]), _p(t["priv"]))
    keep = (t, out)

    def call(keep=keep):
        _call(gb.lib().apo_hash_tasks(_ctx(), ctypes.byref(tasks), _p(out), _stream()))
        return out
    return call


def _repeats_call(tokens, width, min_len, stages, sa_lcp, win_off=None):
    n = tokens.shape[0]
    m, k = 2 * n, n // min_len
    u8 = torch.uint8
    b = {"sa": _zeros(n) if stages or sa_lcp else None, "lcp": _zeros(n) if stages or sa_lcp else None,
         "cand_len": _zeros(m) if stages else None, "cand_id": _zeros(m) if stages else None,
         "cand_start": _zeros(m) if stages else None, "cand_accepted": _zeros(m, u8) if stages else None,
         "sel_start": _zeros(k), "sel_len": _zeros(k), "sel_trace": _zeros(k), "trace_len": _zeros(k),
         "trace_start": _zeros(k)}
    counts = np.zeros(4, dtype=np.uint64)
    offs = [] if win_off is None else [np.zeros(len(win_off), dtype=np.uint64) for _ in range(3)]
    names = ("cand_off", "sel_off", "trace_off")
    o = gb.apo_repeats_out(*[_p(b[x]) for x in ("sa", "lcp", "cand_len", "cand_id", "cand_start", "cand_accepted")],
                           m if stages else 0, *[_p(b[x]) for x in ("sel_start", "sel_len", "sel_trace")], max(1, k),
                           _p(b["trace_len"]), _p(b["trace_start"]), max(1, k), counts.ctypes.data,
                           *([x.ctypes.data for x in offs] or [None] * 3))
    par = gb.apo_repeats_params(min_len, 0)
    out = {x: v for x, v in b.items() if v is not None} | dict(zip(names, offs))
    if win_off is None:
        w = gb.apo_window(n, _p(tokens), width)
        f = gb.lib().apo_find_repeats
    else:
        w = gb.apo_windows(len(win_off) - 1, _p(tokens), width, win_off.ctypes.data)
        f = gb.lib().apo_find_repeats_batched
    keep = (tokens, win_off)

    def call(keep=keep):
        _call(f(_ctx(), ctypes.byref(w), ctypes.byref(par), ctypes.byref(o), _stream()))
        return out | {"counts": counts[:3]}
    return call


def _match_call(pat, stream, width, cap, pat_off=None, slices=None):
    n = stream.shape[0]
    end, pid = _zeros(cap), _zeros(cap)
    count = ctypes.c_uint64()
    if pat_off is not None:
        ps = gb.apo_patterns(len(pat_off) - 1, _p(pat), width, pat_off.ctypes.data, None, None)
    else:
        start, length, sa, lcp = slices
        ps = gb.apo_patterns(start.shape[0], _p(pat), width, None, _p(start), _p(length), _p(sa), _p(lcp), pat.shape[0])
    keep = (pat, stream, pat_off, slices)

    def call(keep=keep):
        _call(gb.lib().apo_match_candidates(_ctx(), ctypes.byref(ps), _p(stream), n, _p(end), _p(pid), cap,
                                            ctypes.byref(count), _stream()))
        return {"end": end, "id": pid, "count": int(count.value)}
    return call


def _replay_call(s, start, length, ingest, max_trace_len):
    n = s.shape[0]
    b = {"end": _zeros(n), "len": _zeros(n), "trace": _zeros(n), "traced": _zeros(n, torch.uint8), "curve": _zeros(n)}
    counts = np.zeros(8, dtype=np.uint64)
    t = gb.apo_replay_traces(start.shape[0], _p(start), _p(length), _p(ingest))
    par = gb.apo_replay_params(max_trace_len, 8, 1000, 17, 16, 5000)
    o = gb.apo_replay_out(_p(b["end"]), _p(b["len"]), _p(b["trace"]), n, _p(b["traced"]), _p(b["curve"]),
                          counts.ctypes.data)
    keep = (s, start, length, ingest)

    def call(keep=keep):
        _call(gb.lib().apo_replay(_ctx(), _p(s), n, 4, ctypes.byref(t), ctypes.byref(par), ctypes.byref(o), _stream()))
        return b | {"counts": counts[:3]}
    return call


def _served_call(requests, min_len):
    server = gb.Server(0, min_len=min_len, token_bytes=4, lanes=2)
    names = ("sel_start", "sel_len", "sel_trace", "trace_len", "trace_start")
    most = [len(q) // min_len for q in requests]
    b = {x: np.zeros(sum(most), dtype=np.uint32) for x in names}
    counts = np.zeros((len(requests), 2), dtype=np.int64)

    def call():
        ids = [server.submit(q) for q in requests]
        at = 0
        for k, i in enumerate(ids):
            r = server.wait(i)
            for x in names:
                v = getattr(r, x)
                b[x][at:at + len(v)] = v
            counts[k] = len(r.sel_start), len(r.trace_len)
            at += most[k]
        return b | {"counts": counts}
    return call


def _optimum_call(tokens, win_off, min_len):
    w, n = len(win_off) - 1, tokens.shape[0]
    b = {"best": _zeros(3 * w), "start": _zeros(n), "len": _zeros(n), "count": _zeros(w)}
    ws = gb.apo_windows(w, _p(tokens), 4, win_off.ctypes.data)
    keep = (tokens, win_off)

    def call(keep=keep):
        _call(gb.lib().apo_optimum_batched(_ctx(), ctypes.byref(ws), min_len, _p(b["best"]), _p(b["start"]),
                                           _p(b["len"]), _p(b["count"]), _stream()))
        return b
    return call


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed, 2)
    wide = 0x9E3779B97F4A7C1
    if kind == "hash":
        return _hash_call(_tasks(case["n"], 0.01, g))
    if kind == "repeats":
        return _repeats_call(_window(case, seed), case["bytes"], case["min_len"], case["stages"], case["sa_lcp"])
    if kind == "batched":
        lens = _spread(case["windows"], case["lo"], case["hi"])
        s = _segments(lens, 3, min(5000, case["hi"]), 0.05, 1000, g)
        s = s if case["bytes"] == 4 else s.long() * wide + 12345
        return _repeats_call(s, case["bytes"], case["min_len"], case["stages"], False, _offsets(lens.cpu().numpy()))
    if kind == "match_traces":
        s = _window(case, seed)
        r = _repeats_call(s, case["bytes"], case["min_len"], False, True)()
        t = int(r["counts"][2])
        return _match_call(s, s, case["bytes"], (100 if case["content"] == "tasks" else 256) * case["n"],
                           slices=(r["trace_start"][:t].clone(), r["trace_len"][:t].clone(), r["sa"], r["lcp"]))
    if kind == "match_stream":
        n, p = case["n"], case["patterns"]
        s = _phases(n, 4096, 1 << 20, 3, 5000, 0.05, 1000, g)
        lens = torch.clamp(_spread(p, case["lo"], case["hi"]), max=n)
        m = int(lens.sum())
        at = (torch.rand(p, device="cuda", generator=g, dtype=torch.float64) * (n - lens + 1)).long()
        off = torch.cumsum(lens, 0) - lens
        k = torch.repeat_interleave(torch.arange(p, device="cuda"), lens, output_size=m)
        copy = s[at[k] + torch.arange(m, device="cuda") - off[k]]  # even patterns occur, odd ones are noise
        other = torch.randint(0, 1000, (m,), device="cuda", generator=g, dtype=torch.int32)
        t = torch.where(k % 2 == 0, copy, other)
        if case["bytes"] == 8:
            s, t = s.long() * wide + 12345, t.long() * wide + 12345
        return _match_call(t, s, case["bytes"], min(32 * n, 1 << 29), pat_off=_offsets(lens.cpu().numpy()))
    if kind == "replay":
        n, unit, buffer = case["n"], 250, 5000
        s = _phases(n, 1 << 14, 1 << 17, 20, 600, 0.01, 1 << 16, g)
        i = np.arange(1, n // unit + 1)  # the finder's slices: unit * 2^ruler(i) tokens, at most the buffer
        size = np.minimum(np.minimum(unit * (i & -i), buffer), i * unit)
        off = _offsets(size)
        m = int(off[-1])
        begin = torch.from_numpy(i * unit - size).cuda()
        w = torch.repeat_interleave(torch.arange(len(i), device="cuda"), torch.from_numpy(size).cuda(), output_size=m)
        at = begin[w] + torch.arange(m, device="cuda") - torch.from_numpy(off[:-1].astype(np.int64)).cuda()[w]
        r = _repeats_call(s[at], 4, 5, False, False, off)()
        t = int(r["counts"][2])
        k = torch.repeat_interleave(torch.arange(len(i), device="cuda"),
                                    torch.from_numpy(np.diff(r["trace_off"].astype(np.int64))).cuda(), output_size=t)
        return _replay_call(s, (r["trace_start"][:t] + begin[k]).int(), r["trace_len"][:t].clone(),
                            ((k + 2) * unit).int(),  # ingested one analysis period after its analysis point
                            case["max_trace_len"])
    if kind == "served":
        lens = _spread(case["requests"], case["lo"], case["hi"])
        s = _segments(lens, 3, 5000, 0.05, 1000, g).cpu().numpy().view(np.uint32)
        off = _offsets(lens.cpu().numpy()).astype(np.int64)
        return _served_call([s[off[q]:off[q + 1]].copy() for q in range(case["requests"])], case["min_len"])
    # half uniform over four tokens, half short loops with noise
    w, n = case["windows"], case["n"]
    period = torch.randint(2, 7, (w, 1), device="cuda", generator=g)
    body = torch.randint(0, 4, (w, 6), device="cuda", generator=g, dtype=torch.int32)
    s = torch.gather(body, 1, torch.arange(n, device="cuda")[None, :] % period)
    any_ = torch.randint(0, 4, (w, n), device="cuda", generator=g, dtype=torch.int32)
    hit = torch.rand(w, n, device="cuda", generator=g) < 0.1
    hit[::2] = True
    return _optimum_call(torch.where(hit, any_, s).reshape(-1).contiguous(),
                         np.arange(0, w * n + 1, n, dtype=np.uint64), case["min_len"])


def run(state):
    return state()


def work(case):
    """Inputs read once and outputs written once; outputs whose number depends on the contents are taken at a round
    figure.  The operations are comparisons and integer arithmetic: per token, one pass over a radix-sorted suffix."""
    kind = case["kind"]
    if kind == "hash":  # 4.5 arguments a task: 13 bytes each, two operations a byte
        n = case["n"]
        return {"bytes": n * (16 + 4.5 * 13), "flops": n * 2 * (8 + 4.5 * 13)}
    if kind == "repeats":
        n = case["n"]
        out = (8 if case["stages"] or case["sa_lcp"] else 0) + (13 if case["stages"] and case["content"] != "random" else 0)
        return {"bytes": n * (case["bytes"] + out + 1), "flops": n * math.log2(max(2, n))}
    if kind == "batched":
        lo, hi = case["lo"], case["hi"]
        n = case["windows"] * (lo if hi <= lo else (hi - lo) / math.log(hi / lo))
        out = 21 if case["stages"] else 0
        return {"bytes": n * (case["bytes"] + out + 1), "flops": n * math.log2(max(2, hi))}
    if kind == "match_traces":  # the stream, its SA and LCP, about 8 matches a token
        n = case["n"]
        return {"bytes": n * (case["bytes"] + 8 + 64), "flops": n * 16}
    if kind == "match_stream":
        n = case["n"]
        m = case["patterns"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": (n + m) * case["bytes"] + n, "flops": (n + m) * 8}
    if kind == "replay":  # the stream, the traces (about one to 36 tasks), flags, curve and records
        n = case["n"]
        return {"bytes": n * (4 + 1 + 4 + 2), "flops": n * 32}
    if kind == "served":
        n = case["requests"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": n * 5, "flops": n * math.log2(case["hi"])}
    w, n = case["windows"], case["n"]
    return {"bytes": w * (4 * n + 16 + 8 * 6), "flops": w * n * n * n}


def exact(case, seed):
    """Whole numbers all through; the hashes are given from their definition (FNV-1a over the descriptor's bytes)."""
    if case["kind"] != "hash":
        return None
    t = {k: v.cpu().numpy() for k, v in _tasks(case["n"], 0.01, _gen(seed, 2)).items()}
    off = t["arg_off"].view(np.uint32).astype(np.int64)
    nargs = off[1:] - off[:-1]
    h = np.full(case["n"], 0xCBF29CE484222325, dtype=np.uint64)

    def feed(h, v, size):
        for b in range(size):
            h = (h ^ ((v >> np.uint64(8 * b)) & np.uint64(255))) * np.uint64(0x100000001B3)
        return h

    with np.errstate(over="ignore"):
        h = feed(feed(h, t["task_id"].view(np.uint32).astype(np.uint64), 4), nargs.astype(np.uint64), 4)
        for a in range(int(nargs.max())):
            at = np.nonzero(nargs > a)[0]
            k = off[at] + a
            x = feed(h[at], t["region"][k].view(np.uint32).astype(np.uint64), 4)
            x = feed(x, t["field_mask"][k].view(np.uint64), 8)
            h[at] = feed(x, t["priv"][k].astype(np.uint64), 1)
    return h.view(np.int64)
