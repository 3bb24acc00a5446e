"""GPU parity of the pack and both unpack directions where their index work changes form: one self-contained launch up to
16,384 items (return: 12,288) and 1,024 plan rows, chunked histograms beyond; the plan's senders read in place or resolved by a kernel of
their own; fewer rows than SMs (a row split over CTAs) and more; every copy width."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import tests.test_gpu_pack as tp
import tests.test_gpu_unpack as tu
from tests.test_gpu_pack import vp  # noqa: F401  (fixture)
from workloads import SchedParams as WParams
from workloads.configs import catalog_for
from workloads.demand import demand_from_routing, moe_routing

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _case(nodes, tokens, topk, row_bytes, k_max=0, seed=0):
    """One call on ``nodes`` nodes; row_bytes a multiple of two: int16 rows, otherwise bytes."""
    cat = catalog_for(nodes, "complete" if nodes <= 2 else "template")
    N = cat.topology.N
    E = 4 * N if N <= 128 else N
    rank = (seed * 5 + 3) % N
    idx = moe_routing(N * tokens, E, topk, 0.8, seed=seed, device="cuda")
    D = demand_from_routing(idx, torch.arange(N, device="cuda").repeat_interleave(tokens), N, E, row_bytes).cpu()
    gen = torch.Generator().manual_seed(seed)
    if row_bytes % 2:
        rows = torch.randint(0, 256, (tokens, row_bytes), dtype=torch.uint8, generator=gen)
    else:
        rows = torch.randint(-32768, 32768, (tokens, row_bytes // 2), dtype=torch.int16, generator=gen)
    w = WParams(granule_bytes=row_bytes, k_max=k_max).resolved(N)
    return dict(catalog=cat, demand=D.unsqueeze(0), params=w, rank=rank, rows=rows, row_bytes=row_bytes, topk=topk,
                expert_idx=idx.view(N, tokens, topk)[rank].cpu().contiguous(), experts_per_rank=E // N)


# (nodes, tokens, topk, row bytes, k_max): one CTA per token; a token over several CTAs; exactly the limit of the one-launch
# form and one token more; long plans (k_max above 1,024, above what a count CTA reads itself); 64, 128 and 256 ranks; rows that
# are multiples of 16, 4 and 1 bytes on both sides of 2 KB, rows of more than one 16 KB piece, and (return) both sides of 7 KB
CASES = [(2, 1, 1, 4096, 0), (2, 5, 8, 14336, 0), (1, 149, 3, 4100, 0), (2, 700, 6, 333, 0), (2, 1024, 8, 96, 0), (2, 1025, 8, 96, 0),
         (2, 2400, 8, 2064, 0), (2, 2100, 8, 4100, 0), (2, 300, 8, 2048, 1025), (2, 300, 8, 2048, 40000), (8, 40, 6, 7392, 0),
         (2, 1536, 8, 2064, 0), (2, 1537, 8, 2064, 0), (2, 2048, 8, 96, 0), (2, 2049, 8, 96, 0), (2, 600, 8, 33008, 0), (2, 297, 8, 2048, 0),
         (2, 74, 1, 2064, 0), (2, 75, 1, 16400, 0), (8, 1200, 8, 4096, 0), (8, 2300, 8, 1536, 0), (16, 30, 4, 4096, 2048), (32, 12, 8, 512, 4096), (2, 2100, 8, 16400, 0),
         (2, 1000, 8, 7152, 0), (2, 1000, 8, 7168, 0)]


@pytest.mark.parametrize("nodes,tokens,topk,row_bytes,k_max", CASES)
def test_pack_forms(vp, oracle_lib, nodes, tokens, topk, row_bytes, k_max):  # noqa: F811
    res = tp._run_case(vp, oracle_lib, _case(nodes, tokens, topk, row_bytes, k_max, seed=tokens))
    assert res[2] == 0
    tp._assert_pack(res)


@pytest.mark.parametrize("nodes,tokens,topk,row_bytes,k_max", CASES)
def test_unpack_forms(vp, oracle_lib, nodes, tokens, topk, row_bytes, k_max):  # noqa: F811
    case = _case(nodes, tokens, topk, row_bytes, k_max, seed=tokens + 1)
    oc, plan, one = tu._plans(vp, oracle_lib, case["catalog"], case["demand"], case["params"])
    R, recv, expert = tu._receive_case(case, case["rank"], case["experts_per_rank"], seed=1,
                                       dtype=torch.uint8 if row_bytes % 2 else torch.int16, extra_rows=5)
    got, want, cap = tu._run(vp, oc, plan, one, case["rank"], recv, expert, case["experts_per_rank"])
    assert got[4] == 0 and int(got[1][-1]) == R
    tu._assert_unpack(got, want, cap)


@pytest.mark.parametrize("nodes,tokens,topk,row_bytes,k_max", [c for c in CASES if c[3] % 2 == 0])
def test_unpack_tokens_forms(vp, oracle_lib, nodes, tokens, topk, row_bytes, k_max):  # noqa: F811
    case = _case(nodes, tokens, topk, row_bytes, k_max, seed=tokens + 2)
    oc, plan, one, R, recv = tu._return_case(vp, oracle_lib, case, case["rank"], seed=2, extra_rows=3)
    st, w_map = tu._run_tokens(vp, oc, plan, one, case["rank"], case["expert_idx"], case["experts_per_rank"], recv)
    assert st == 0 and int((w_map >= 0).sum()) == R


@pytest.mark.parametrize("tokens", [300, 2300])
def test_pack_mismatch_and_capacity_in_both_forms(vp, oracle_lib, tokens):  # noqa: F811
    case = _case(2, tokens, 8, 1024, seed=7)
    R = int(case["demand"][0, case["rank"]].sum().item() // 1024)
    res = tp._run_case(vp, oracle_lib, case, capacity_rows=R - 1)
    assert res[2] == vp.ST_PACK_CAPACITY == res[5] and not res[0][:R - 1].any()
    case["expert_idx"][0, 0] = 1 << 20                         # an expert on no rank
    res = tp._run_case(vp, oracle_lib, case)
    assert res[2] == vp.ST_PACK_MISMATCH and res[5] & vp.ST_PACK_MISMATCH


@pytest.mark.parametrize("sources,tokens,topk,N", [(1, 1, 1, 8), (1, 2049, 1, 16), (1, 4097, 4, 256), (8, 1024, 8, 8), (8, 1025, 8, 8),
                                                   (16, 3, 7, 256), (17, 3, 7, 256), (64, 5, 2, 64), (3, 30000, 8, 5)])
def test_demand_forms(vp, oracle_lib, sources, tokens, topk, N):  # noqa: F811
    """One cluster for all sources (up to 65,536 copies and 4,096 cells) or one per source, of one to eight CTAs."""
    epr = 3
    idx = torch.randint(-1, N * epr, (sources, tokens, topk), dtype=torch.int32, generator=torch.Generator().manual_seed(tokens))
    src0 = max(0, N - sources) if N >= sources else 0
    for last in (0, N * epr):                                  # the second time with an expert on no rank
        idx[-1, -1, -1] = last
        got, st = vp.demand_from_routing(idx.cuda(), epr, N, 768, src0=src0)
        want, bad = oracle_lib.demand_from_routing(idx.numpy(), epr, N, 768, src0=src0)
        assert int(st.item()) == bad == (1 if last else 0)
        assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("sources,tokens,topk,N", [(1, 1, 1, 8), (1, 4099, 3, 16), (200, 331, 7, 256), (256, 1100, 3, 256), (5, 9999, 3, 256)])
def test_demand_alignments(vp, oracle_lib, sources, tokens, topk, N):  # noqa: F811
    """Indices that start at any word: copies before, in and after the 16-byte loads; up to and beyond one wave of CTAs."""
    n = sources * tokens * topk
    for off in range(4):
        flat = torch.randint(-1, N * 2, (n + 3,), dtype=torch.int32, generator=torch.Generator().manual_seed(n + off))
        idx = flat[off:off + n].view(sources, tokens, topk)
        got, st = vp.demand_from_routing(flat.cuda()[off:off + n].view(sources, tokens, topk), 2, N, 4096)
        want, bad = oracle_lib.demand_from_routing(idx.numpy(), 2, N, 4096)
        assert int(st.item()) == bad == 0 and np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("nodes,T,topk,row_bytes", [(2, 3, 1, 16), (2, 700, 8, 14336), (2, 700, 8, 4100), (1, 500, 8, 333), (1, 90, 4, 1),
                                                    (2, 33, 6, 16400), (8, 40, 8, 7392), (8, 40, 8, 4102)])
def test_put_alignments(vp, oracle_lib, nodes, T, topk, row_bytes):  # noqa: F811
    """Chunk parts that go as bulk copies (addresses and sizes multiples of 16, more and less than one piece) and parts at every
    other alignment, into receive buffers at odd addresses, on plans of up to several hundred activations."""
    case = _case(nodes, T, topk, row_bytes, seed=T)
    cat, D, w, rank = case["catalog"], case["demand"][0], case["params"], case["rank"]
    N = cat.topology.N
    oc = oracle_lib.OracleCatalog(cat.topology.blob(), cat.blob())
    dc = vp.load_catalog(cat.topology.blob(), cat.blob())
    plan = vp.schedule_batch(dc, tp._params(vp, w), D.unsqueeze(0).cuda().contiguous())
    one = {k: (v[0] if isinstance(v, np.ndarray) else v) for k, v in oc.schedule_batch(D.unsqueeze(0).numpy(), w).items()}
    sent, cap = int(D[rank].sum()), D.sum(0).tolist()
    staged = torch.randint(0, 256, (sent + 1,), dtype=torch.uint8, generator=torch.Generator().manual_seed(T)).cuda()[:sent]
    step = 256 if row_bytes % 16 == 0 else 261
    bufs = torch.full((sum(cap) + N * 600,), 0xAB, dtype=torch.uint8, device="cuda")
    at = np.concatenate([[0], np.cumsum([(c + 511) // 256 * 256 + step - 256 for c in cap])[:-1]])
    counters = torch.zeros(N, dtype=torch.int64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    vp.exchange_put(plan, 0, rank, staged, bufs.data_ptr() + torch.from_numpy(at).cuda(), torch.tensor(cap, device="cuda"),
                    counters.data_ptr() + 8 * torch.arange(N, device="cuda"), status)
    torch.cuda.synchronize()
    want, want_arrived, st = oc.exchange(one, {i: (staged.cpu().numpy() if i == rank else np.zeros(int(D[i].sum()), np.uint8)) for i in range(N)})
    got = bufs.cpu().numpy()
    assert int(status.item()) == st == 0 and counters.cpu().tolist() == D[rank].tolist()
    mask = np.zeros(got.shape, bool)
    host = plan.cpu()
    for k in range(int(host["n_steps"][0])):
        j, n = int(host["lane_dst"][0, k, rank]), int(host["lane_bytes"][0, k, rank])
        if j >= 0 and n:
            r = int(host["recv_off"][0, k, j])
            assert np.array_equal(got[at[j] + r:at[j] + r + n], np.asarray(want[j]).reshape(-1)[r:r + n]), (k, j)
            mask[at[j] + r:at[j] + r + n] = True
    assert (got[~mask] == 0xAB).all()                          # nothing else is touched


@pytest.fixture
def large():
    """Gives the memory of a large test back to the device."""
    yield
    torch.cuda.empty_cache()


@pytest.mark.parametrize("tokens", [False, True])
def test_unpack_at_the_accepted_limit(vp, large, tokens):  # noqa: F811
    """2^31 - 1 rows of one byte, all of them in use: the last chunk ends where 32-bit indices do."""
    R, dev = 2 ** 31 - 1, "cuda"
    plan = vp.Plan.empty(1, 2, 1, dev)                         # one step: rank 0 sends to rank 1, or rank 1 returns to rank 0
    plan.n_steps.fill_(1)
    plan.lane_dst.copy_(torch.tensor([[[-1, 0] if tokens else [1, -1]]]))
    plan.lane_bytes.copy_(torch.tensor([[[0, R] if tokens else [R, 0]]]))
    plan.recv_off.copy_(torch.tensor([[[0, 0], [R, 0] if tokens else [0, R]]]))
    recv = torch.randint(-2 ** 63, 2 ** 63 - 1, (2 ** 28,), device=dev).view(torch.uint8)[:R].view(R, 1)
    expert = torch.randint(-2 ** 63, 2 ** 63 - 1, (2 ** 28,), device=dev).view(torch.uint8)[:R].to(torch.int32) & 1
    out = torch.zeros_like(recv)
    if tokens:                                                 # experts 2 and 3 live on rank 1
        st = vp.unpack_tokens(plan, 0, 0, (expert + 2).view(R, 1), 2, recv, out)
    else:
        off, st = vp.unpack(plan, 0, 1, recv, expert, 2, out)
    first = expert == 0
    n = int(first.sum())
    if not tokens:
        assert off.tolist() == [0, n, R]
    assert int(st.item()) == 0
    a, b = (out, recv) if tokens else (recv, out)              # a in the order of the routing, b sorted by expert
    assert torch.equal(a[first], b[:n]) and torch.equal(a[~first], b[n:])


@pytest.mark.parametrize("row_bytes,topk", [(2 ** 31 + 3, 1), (2 ** 31 + 3, 8193), (2 ** 33 + 4, 1)])
def test_rows_of_more_than_2_gb(vp, large, row_bytes, topk):  # noqa: F811
    """A row of more vectors (of one and four bytes) than 32 bits number: packed, unpacked and returned whole, by calls of few
    copies and of many (most of them dropped)."""
    plan = vp.Plan.empty(1, 2, 1, "cuda")
    row = torch.randint(-2 ** 63, 2 ** 63 - 1, (row_bytes // 8 + 1,), device="cuda").view(torch.uint8)[:row_bytes].view(1, row_bytes)
    idx = torch.full((1, topk), -1, dtype=torch.int32, device="cuda")
    idx[0, -1] = 1                                             # one copy, to rank 1

    def set_plan(src, dst):
        plan.n_steps.fill_(1)
        plan.lane_dst.fill_(-1)[0, 0, src] = dst
        plan.lane_bytes.zero_()[0, 0, src] = row_bytes
        plan.send_off.zero_()[0, 1, src] = row_bytes
        plan.recv_off.zero_()[0, 1, dst] = row_bytes

    set_plan(0, 1)
    out = torch.zeros_like(row)
    assert int(vp.pack(plan, 0, 0, idx, 1, row, out).item()) == 0 and torch.equal(out, row)
    out.zero_()
    off, st = vp.unpack(plan, 0, 1, row, torch.zeros(1, dtype=torch.int32, device="cuda"), 1, out)
    assert int(st.item()) == 0 and off.tolist() == [0, 1] and torch.equal(out, row)
    if topk == 1:
        set_plan(1, 0)
        out.zero_()
        assert int(vp.unpack_tokens(plan, 0, 0, idx, 1, row, out).item()) == 0 and torch.equal(out, row)


def test_demand_of_more_copies_than_32_bits_count(vp, large):  # noqa: F811
    """More than 2^32 copies from one source to one rank."""
    idx = torch.zeros((1, 2 ** 29 + 1, 8), dtype=torch.int32, device="cuda")
    idx[0, 7, :3], idx[0, -1, 0] = 1, -1                       # three copies to the source itself, one dropped
    got, st = vp.demand_from_routing(idx, 1, 2, 3, src0=1)
    assert int(st.item()) == 0 and got.tolist() == [[3 * (2 ** 32 + 8 - 4), 0]]


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("ring") / "libring.so")
    subprocess.check_call(["/usr/local/cuda/bin/nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O1", "-std=c++17", "-Xcompiler", "-fPIC",
                           "-shared", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2609_34340_b200", "csrc"),
                           os.path.join(ROOT, "tests", "own_ring_wait.cu"), "-o", out], timeout=300)
    fn = ctypes.CDLL(out).run_ring
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p,
                   ctypes.c_int, ctypes.c_void_p]
    return fn


@pytest.mark.parametrize("own,fanout,row_bytes", [(1, 1, 2048), (2, 8, 14336), (9, 3, 7392), (13, 1, 33008), (31, 2, 4096)])
@pytest.mark.parametrize("at", [0, 1, 4, 6])
def test_rows_are_complete_when_a_wait_gives_up(vp, ring, own, fanout, row_bytes, at):  # noqa: F811
    """The status bit of a wait that gave up may be overwritten by the CTA that writes the status, so no output may depend on it: what
    is left is moved by plain loads.  The wait runs out at the first, the second or the fifth stage of the rings, or (six) not at all."""
    gen = torch.Generator().manual_seed(own * 100 + at)
    rows = torch.randint(0, 256, (own + 3, row_bytes), dtype=torch.uint8, generator=gen)
    src = torch.randperm(own + 3, generator=gen)[:own].to(torch.int32)
    dst = torch.randperm(own * fanout + 5, generator=gen)[:own * fanout].to(torch.int32)
    dst[torch.rand(own * fanout, generator=gen) < 0.2] = -1
    if own > 2:
        src[own // 2] = -1
    want = torch.zeros(own * fanout + 5, row_bytes, dtype=torch.uint8)
    for i in range(own):
        for d in dst[i * fanout:(i + 1) * fanout].tolist():
            if src[i] >= 0 and d >= 0:
                want[d] = rows[src[i]]
    rows_d, src_d, dst_d, gave_up = rows.cuda(), src.cuda(), dst.cuda(), torch.zeros(1, dtype=torch.int32, device="cuda")
    out = torch.zeros_like(want, device="cuda")
    assert ring(rows_d.data_ptr(), out.data_ptr(), row_bytes, own, fanout, src_d.data_ptr(), dst_d.data_ptr(), at, gave_up.data_ptr()) == 0
    piece = min(row_bytes if own > 1 else row_bytes // 32 * 16, 16384)
    units = [i for i in range(own) for _ in range(-(-row_bytes // piece))]             # own row of every unit; two warps take turns
    assert int(gave_up.item()) == sum(any(src[i] >= 0 for i in units[w::2][at:6]) for w in (0, 1))
    assert torch.equal(out.cpu(), want)
