"""What the framework is timed on: the calls that make up one expert-parallel AlltoAllv, as a serving or training program
issues them, and the host-buffer planner call.

Every case is one public call on buffers that such a program allocates once and keeps (plan, workspace, status, output):

* ``demand``   -- routing indices to demand rows (the scheduler's input)
* ``plan``     -- demand matrices to plans, on device tensors (one matrix per layer and step, or a batch of them)
* ``host``     -- the same through host buffers, only the plan rows in use coming back
* ``pack``     -- one rank's token rows into its staged send buffer (dispatch, sender)
* ``put``      -- the staged buffer into the receivers' buffers, with arrival counters (dispatch, transfer)
* ``unpack``   -- the receive buffer into expert-major rows (dispatch, receiver)
* ``return``   -- the experts' rows back into the token layout (combine, receiver)

Inputs are synthetic MoE routing with Zipf expert popularity (a permutation of the experts per matrix, as layers differ),
or sequence-parallel head/sequence redistribution.  All results are integers or copied bytes, so they compare exactly.
"""
from __future__ import annotations

import math
import struct
from functools import lru_cache

import torch

import paper_2609_34340_b200 as vp

DEVICE = "cuda:0"
LAMBDA_NS = 8000          # the default per-activation overhead


# ---- catalogs: a PCIe tree, two switches per node, four GPUs and one NIC per switch, every link 64 B/ns -----------------

def _topology_blob(nodes: int) -> bytes:
    g, bw, groups = 4, 64, 2 * nodes
    up, down, tx, rx = range(4)
    inst = []
    for a in range(groups):
        for d in range(groups):
            if a == d:
                inst.append((a, d, 0, g, ()))                                  # same switch: no shared link
                continue
            if a // 2 == d // 2:
                inst.append((a, d, 1, 1, (4 * a + up, 4 * d + down)))          # the other switch of the node
            inst.append((a, d, 2, 1, (4 * a + tx, 4 * d + rx)))                # over the two switches' NICs
    blob = struct.pack("<8I", 0x50545056, 1, groups * g, groups, g, 2, 4 * groups, len(inst))
    for a, d, kind, mult, res in inst:
        blob += struct.pack("<HHBBHI4H", a, d, kind, len(res), mult, bw, *(list(res) + [0] * (4 - len(res))))
    return blob


@lru_cache(maxsize=None)
def _catalog(nodes: int):
    topo = _topology_blob(nodes)
    channels = vp.build_catalog(topo)[0] if nodes <= 2 else vp.build_template_catalog(topo)[0]
    return vp.load_catalog(topo, channels, device=0)


# ---- inputs -------------------------------------------------------------------------------------------------------------

def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _popularity(B: int, E: int, skew: float, gen) -> torch.Tensor:
    """``[B, E]`` expert popularities, (1 + rank)^-s over a random order of the experts.  skew < 0: s drawn per matrix."""
    s = torch.rand(B, 1, device=DEVICE, generator=gen) * 1.5 if skew < 0 else torch.full((B, 1), skew, device=DEVICE)
    order = torch.rand(B, E, device=DEVICE, generator=gen).argsort(dim=1).to(torch.float32)
    p = torch.exp(-s * torch.log1p(order))
    return p / p.sum(dim=1, keepdim=True)


def _routing(T: int, topk: int, p: torch.Tensor, gen) -> torch.Tensor:
    """``[T, topk]`` distinct experts per token, in proportion to ``p`` (Gumbel top-k)."""
    u = torch.rand(T, p.numel(), device=DEVICE, generator=gen).clamp_(1e-20, 1 - 1e-7)
    return torch.topk(torch.log(p) - torch.log(-torch.log(u)), topk, dim=1).indices.to(torch.int32).contiguous()


def _moe_demand(N: int, tokens: torch.Tensor, topk: int, p: torch.Tensor, row_bytes: int, gen) -> torch.Tensor:
    """``[B, N, N]`` bytes that ``tokens[b, i]`` routed tokens per rank send: per expert a binomial number of a rank's tokens
    with the inclusion probability that top-k sampling without replacement gives it."""
    B, E = p.shape
    lo, hi = torch.zeros(B, 1, device=DEVICE), torch.full((B, 1), 1e9, device=DEVICE)
    for _ in range(60):
        c = (lo + hi) / 2
        over = (-torch.expm1(-c * p)).sum(dim=1, keepdim=True) > topk
        lo, hi = torch.where(over, lo, c), torch.where(over, c, hi)
    incl = -torch.expm1(-(lo + hi) / 2 * p)
    D = torch.empty(B, N, N, dtype=torch.int64, device=DEVICE)
    step = max(1, (1 << 25) // (N * E))
    for b in range(0, B, step):
        n = tokens[b:b + step].to(torch.float32).unsqueeze(2).expand(-1, -1, E).contiguous()
        got = torch.binomial(n, incl[b:b + step].unsqueeze(1).expand_as(n).contiguous(), generator=gen)
        D[b:b + step] = got.view(got.shape[0], N, N, E // N).sum(dim=3).to(torch.int64) * row_bytes
    D.diagonal(dim1=1, dim2=2).zero_()
    return D


def _sp_demand(B: int, N: int, gen) -> torch.Tensor:
    """Sequence-parallel redistribution in groups of eight ranks: 1,024 to 32,768 tokens per shard, five heads of 128 bf16
    values per peer."""
    shard = torch.randint(1024, 32769, (B, N, 1), device=DEVICE, generator=gen)
    same = torch.arange(N, device=DEVICE) // 8
    D = shard * (5 * 128 * 2) * (same.unsqueeze(0) == same.unsqueeze(1))
    D.diagonal(dim1=1, dim2=2).zero_()
    return D.contiguous()


def _experts(N: int) -> int:
    return 128 if N in (8, 64) else (192 if N == 96 else 256)


def _params(case: dict):
    N, granule = 8 * case["nodes"], 256 if case.get("load") in ("sp", "mixed") else case["row_bytes"]
    return vp.SchedParams(lambda_ns=LAMBDA_NS, granule_bytes=granule, k_target=2 * N, n_start=4, i_aa=3, k_max=_k_max(N))


def _k_max(N: int) -> int:
    return 8 * N if N < 96 else 16 * N


def _matrices(case: dict, gen) -> torch.Tensor:
    B, N, load = case["batch"], 8 * case["nodes"], case["load"]
    n_sp = {"moe": 0, "sp": B, "mixed": B // 2}[load]
    parts = [_sp_demand(n_sp, N, gen)] if n_sp else []
    if B > n_sp:
        shape = (B - n_sp, N)
        if load == "mixed":                                # the same number of tokens on every rank, 1 to 16,384 of them
            e = torch.randint(0, 15, (shape[0], 1), device=DEVICE, generator=gen)
            tokens = (2 ** e).expand(shape)
        else:
            tokens = torch.randint(max(1, case["tokens"] // 64), case["tokens"] + 1, shape, device=DEVICE, generator=gen)
        parts.append(_moe_demand(N, tokens, 8, _popularity(shape[0], _experts(N), -1.0, gen), case["row_bytes"], gen))
    D = torch.cat(parts)
    return D[torch.rand(B, device=DEVICE, generator=gen).argsort()].contiguous()


def _plan_outputs(plan) -> dict:
    return {"n_steps": plan.n_steps, "chan_id": plan.chan_id, "lane_dst": plan.lane_dst,
            "lane_inst": plan.lane_inst.view(torch.int16), "lane_bytes": plan.lane_bytes, "send_off": plan.send_off,
            "recv_off": plan.recv_off, "tau_ns": plan.tau_ns, "status": plan.status}


def _random_rows(n: int, row_bytes: int, gen) -> torch.Tensor:
    """``[n, row_bytes]`` rows of random bits; bf16 rows as a program holds them when the size allows."""
    if row_bytes % 8:
        return torch.randint(0, 256, (n, row_bytes), dtype=torch.uint8, device=DEVICE, generator=gen)
    bits = torch.randint(-2 ** 63, 2 ** 63 - 1, (n, row_bytes // 8), device=DEVICE, generator=gen)
    return bits.view(torch.int16)


def _one_call(case: dict, gen):
    """One AlltoAllv of ``tokens`` tokens per rank: (plan, demand, rank, that rank's routing, experts per rank).  The rank is
    one that receives at most twice the mean (a program that overflows its receive buffer is of no interest here)."""
    N, T, topk = 8 * case["nodes"], case["tokens"], case["topk"]
    E = _experts(N)
    p = _popularity(1, E, case["skew"], gen)
    D = _moe_demand(N, torch.full((1, N), T, device=DEVICE), topk, p, case["row_bytes"], gen)
    fits = D[0].sum(dim=0) <= 2 * T * topk * case["row_bytes"] * 0.95
    rank = int(torch.multinomial(fits.to(torch.float32), 1, generator=gen))
    idx = _routing(T, topk, p[0], gen)
    row = torch.bincount(idx.flatten().to(torch.int64) // (E // N), minlength=N) * case["row_bytes"]
    row[rank] = 0
    D[0, rank] = row
    if case["kind"] == "return":                           # the return call is an AlltoAllv of its own, with the demand transposed
        D = D.transpose(1, 2).contiguous()
    return vp.schedule_batch(_catalog(case["nodes"]), _params(case), D), D[0], rank, idx, E // N


def _i32(n: int) -> torch.Tensor:
    return torch.zeros(n, dtype=torch.int32, device=DEVICE)


def _bytes(n: int) -> torch.Tensor:
    return torch.empty(max(int(n), 1), dtype=torch.uint8, device=DEVICE)


# ---- the interface ------------------------------------------------------------------------------------------------------

def listed():
    return [
        # a decode step: the rank's own demand row from its routing, on the critical path of every layer
        dict(name="demand_decode", kind="demand", nodes=2, sources=1, tokens=128, topk=8, row_bytes=14336),
        # online planning of a single layer on one node: pure latency
        dict(name="plan_8_online", kind="plan", nodes=1, batch=1, load="moe", tokens=4096, row_bytes=14336),
        # planning a batch of layers on two nodes
        dict(name="plan_16_batch", kind="plan", nodes=2, batch=256, load="moe", tokens=8192, row_bytes=8192),
        # the 16 layers of one step at 64 GPUs, and 64 such steps
        dict(name="plan_64_step", kind="plan", nodes=8, batch=16, load="moe", tokens=16384, row_bytes=14336),
        dict(name="plan_64_batch", kind="plan", nodes=8, batch=1024, load="moe", tokens=16384, row_bytes=14336),
        # 256 GPUs, half MoE with few to many tokens, half sequence parallelism
        dict(name="plan_256_batch", kind="plan", nodes=32, batch=512, load="mixed", tokens=16384, row_bytes=14336),
        # a planner service: demand arrives in and plans leave through host memory
        dict(name="host_64", kind="host", nodes=8, batch=128, load="moe", tokens=16384, row_bytes=14336),
        # dispatch of a decode step and of a long prefill (bf16 rows of 7,168)
        dict(name="pack_decode", kind="pack", nodes=2, tokens=128, topk=8, row_bytes=14336, skew=0.8),
        dict(name="pack_prefill", kind="pack", nodes=2, tokens=16384, topk=8, row_bytes=14336, skew=1.2),
        # the staged buffer of an ordinary prefill chunk to its receivers
        dict(name="put_chunk", kind="put", nodes=2, tokens=2048, topk=8, row_bytes=14336, skew=0.8),
        # receive side of a prefill chunk: fp8 rows with their 56 float scales behind them (not a multiple of 128 bytes)
        dict(name="unpack_fp8", kind="unpack", nodes=2, tokens=4096, topk=8, row_bytes=7392, skew=0.8),
        # combine side of a ragged batch, top-6
        dict(name="return_ragged", kind="return", nodes=2, tokens=1531, topk=6, row_bytes=14336, skew=0.8),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["demand", "plan", "plan", "host", "pack", "put", "unpack", "return"])
    if kind == "demand":
        nodes = rng.choice([1, 2, 4, 8, 32])
        return dict(kind=kind, nodes=nodes, sources=rng.choice([1, 8 * nodes]), tokens=_log_int(rng, 16, 16384),
                    topk=rng.choice([1, 2, 4, 6, 8]), row_bytes=rng.choice([4096, 7392, 8192, 14336]))
    if kind in ("plan", "host"):
        nodes = rng.choice([1, 2, 4, 8, 12, 16, 32] if kind == "plan" else [1, 2, 8])
        most = {1: 4096, 2: 2048, 4: 512, 8: 1024, 12: 256, 16: 256, 32: 256}[nodes] if kind == "plan" else 256
        load = rng.choice(["moe", "moe", "sp", "mixed"])
        return dict(kind=kind, nodes=nodes, batch=_log_int(rng, 1, most), load=load, tokens=_log_int(rng, 128, 16384),
                    row_bytes=14336 if load != "moe" else rng.choice([4096, 7392, 8192, 14336]))
    # rows: bf16 hidden sizes, fp8 with scales, and one that is a multiple of four bytes only
    nodes, topk = rng.choice([1, 2, 2, 8]), rng.choice([1, 2, 4, 6, 8])
    row_bytes = rng.choice([1536, 4096, 4100, 7392, 8192, 14336])
    most = 8192 if kind != "put" else max(32, min(8192, (1 << 32) // (8 * nodes * topk * row_bytes)))   # all receivers: 4 GB
    return dict(kind=kind, nodes=nodes, tokens=_log_int(rng, 16, most), topk=topk, row_bytes=row_bytes,
                skew=rng.choice([0.0, 0.4, 0.8, 1.2]))


def prepare(case, seed):
    gen = _gen(seed)
    kind, N = case["kind"], 8 * case["nodes"]
    s = {"kind": kind}
    if kind == "demand":
        T, topk, n = case["tokens"], case["topk"], case["sources"]
        E = _experts(N)
        p = _popularity(1, E, -1.0, gen)[0]
        idx = torch.stack([_routing(T, topk, p, gen) for _ in range(min(n, 8))])
        if n > 8:                                          # more sources: the same draws in another order per rank
            pick = torch.randint(0, 8 * T, (n - 8, T), device=DEVICE, generator=gen)
            idx = torch.cat([idx, idx.view(8 * T, topk)[pick]])
        s.update(idx=idx.contiguous(), epr=E // N, N=N, row_bytes=case["row_bytes"],
                 out=torch.zeros(n, N, dtype=torch.int64, device=DEVICE), status=_i32(1))
        return s
    if kind in ("plan", "host"):
        cat, par, B = _catalog(case["nodes"]), _params(case), case["batch"]
        D = _matrices(case, gen)
        s.update(cat=cat, par=par)
        if kind == "plan":
            s.update(demand=D, plan=vp.Plan.empty(B, N, par.k_max, DEVICE), ws=_bytes(vp.schedule_workspace_bytes(cat, B, par)))
        else:
            plan = vp.Plan.empty(B, N, par.k_max, "cpu", pin=True)
            for t in _plan_outputs(plan).values():         # rows that are not in use stay as they are
                t.zero_()
            scratch = _bytes(vp.binding._load().vp_schedule_host_scratch_bytes(cat._h, B, par._c(N)))
            s.update(demand=D.cpu().pin_memory(), plan=plan, ws=scratch)
        s["out"] = _plan_outputs(s["plan"])
        return s
    plan, D, rank, idx, epr = _one_call(case, gen)
    rb, T, topk = case["row_bytes"], case["tokens"], case["topk"]
    s.update(plan=plan, rank=rank, idx=idx, epr=epr, status=_i32(1))
    # buffers have a fixed capacity, as in a program that does not wait for the routing: every copy leaves the rank and comes
    # back, and up to twice the mean arrives; what a call does not write stays zero
    most = T * topk
    if kind == "pack":
        rows = _random_rows(T, rb, gen)
        s.update(rows=rows, staged=torch.zeros(most, rows.shape[1], dtype=rows.dtype, device=DEVICE), src_map=_i32(most),
                 ws=_bytes(vp.pack_workspace_bytes(N, T, topk, plan.k_max)))
    elif kind == "put":
        caps = (D.sum(dim=0) + 255) // 256 * 256
        recv = torch.zeros(N * most * rb + 256 * N, dtype=torch.uint8, device=DEVICE)
        arrived = torch.zeros(N, dtype=torch.int64, device=DEVICE)
        s.update(staged=_random_rows(most, rb, gen), recv=recv, caps=caps, arrived=arrived,
                 recv_ptrs=recv.data_ptr() + torch.cumsum(caps, 0) - caps,
                 arrived_ptrs=arrived.data_ptr() + 8 * torch.arange(N, device=DEVICE))
    elif kind == "unpack":
        recv = _random_rows(2 * most, rb, gen)
        prob = torch.rand(epr, device=DEVICE, generator=gen) ** 2 + 1e-3
        s.update(recv=recv, expert=torch.multinomial(prob, 2 * most, replacement=True, generator=gen).to(torch.int32),
                 out=torch.zeros_like(recv), off=_i32(epr + 1), src=_i32(2 * most), map=_i32(2 * most),
                 ws=_bytes(vp.unpack_workspace_bytes(N, 2 * most, epr, plan.k_max)))
    else:
        recv = _random_rows(most, rb, gen)
        need = vp.binding._load().vp_unpack_tokens_workspace_bytes(N, T, topk, epr, most, plan.k_max)
        s.update(recv=recv, out=torch.zeros(most, recv.shape[1], dtype=recv.dtype, device=DEVICE), map=_i32(most),
                 ws=_bytes(need))
    return s


def run(s):
    kind = s["kind"]
    if kind == "demand":
        vp.demand_from_routing(s["idx"], s["epr"], s["N"], s["row_bytes"], out=s["out"], status=s["status"])
        return s["out"], s["status"]
    if kind == "plan":
        vp.schedule_batch(s["cat"], s["par"], s["demand"], plan=s["plan"], workspace=s["ws"])
        return s["out"]
    if kind == "host":
        vp.schedule_batch_host(s["cat"], s["par"], s["demand"], plan=s["plan"], scratch=s["ws"], used_only=True)
        return s["out"]
    if kind == "pack":
        vp.pack(s["plan"], 0, s["rank"], s["idx"], s["epr"], s["rows"], s["staged"], s["src_map"], s["status"], s["ws"])
        return s["staged"], s["src_map"], s["status"]
    if kind == "put":
        vp.exchange_put(s["plan"], 0, s["rank"], s["staged"], s["recv_ptrs"], s["caps"], s["arrived_ptrs"], s["status"])
        return s["recv"], s["arrived"], s["status"]
    if kind == "unpack":
        vp.unpack(s["plan"], 0, s["rank"], s["recv"], s["expert"], s["epr"], s["out"], s["off"], s["src"], s["map"], s["status"],
                  s["ws"])
        return s["out"], s["off"], s["src"], s["map"], s["status"]
    vp.unpack_tokens(s["plan"], 0, s["rank"], s["idx"], s["epr"], s["recv"], s["out"], s["map"], s["status"], s["ws"])
    return s["out"], s["map"], s["status"]


def work(case):
    kind, N = case["kind"], 8 * case["nodes"]
    if kind == "demand":
        copies = case["sources"] * case["tokens"] * case["topk"]
        return {"bytes": 4 * copies + 8 * case["sources"] * N + 4, "flops": copies}
    if kind in ("plan", "host"):
        # A plan has at least k_target activations (no lane of one moves more than the quantum allows); each has to bind its
        # channel, four starts of one sweep at least: two exact 4 x 4 assignments per group, 28 additions and maxima each.
        B, K = case["batch"], _k_max(N)
        flops = B * 2 * N * (4 * 2 * (N // 4) * 28 + N)
        rows = K if kind == "plan" else 2 * N              # every plan element is written; the host call returns rows in use
        return {"bytes": B * (N * N * 8 + rows * (28 * N + 4) + 16 * N + 16), "flops": flops}
    copies = case["tokens"] * case["topk"]
    rows = copies * (N - 1) / N                            # on average; copies to the rank itself do not travel
    rb = case["row_bytes"]
    if kind == "pack":                                     # source rows and routing in, staged rows and their sources out
        return {"bytes": case["tokens"] * rb + 4 * copies + rows * (rb + 4), "flops": 0}
    if kind == "put":
        return {"bytes": rows * 2 * rb, "flops": 0}
    if kind == "unpack":                                   # row, its expert in; row, its source and origin out
        return {"bytes": rows * (2 * rb + 12), "flops": 0}
    return {"bytes": rows * 2 * rb + 8 * copies, "flops": 0}


def tolerance(case):
    return "exact"
