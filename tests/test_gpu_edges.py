"""Kernels at the sizes where their work splits change: edges of tiles and
lists, remainders, the smallest and the largest of their ranges, against the
oracle (same bars as the other parity tests)."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


# head statistics: head blocks of 4, 7 and 8 with and without padded heads, one
# pair of blocks to several passes over them, 8 / 16 / 32 tokens a block, rows of
# A on 16 bytes and not, one query, queries that end inside a stage
@pytest.mark.parametrize("H,Hkv,T,gh,gw,B", [
    (1, 1, [1], 5, 7, 1), (3, 1, [33], 6, 6, 1), (5, 5, [9], 9, 9, 1), (28, 4, [31], 7, 9, 1),
    (32, 8, [65], 6, 10, 1), (56, 8, [17], 8, 8, 1), (9, 3, [5, 40], 33, 75, 2),
    (14, 2, [3, 12, 8, 1], 60, 44, 4)])
def test_head_statistics_sizes(H, Hkv, T, gh, gw, B):
    from paper_2608_02134_gb300 import workloads
    from tests.test_gpu_clients import _compare
    wl = workloads.make("qwen", B=B, T=T, gh=gh, gw=gw, D=64, d=32, H=H, Hkv=Hkv, K=9)
    _compare(wl, range(B))


# the query-weighted squares over many queries (whole lines of tokens, one lane a
# token): every head sees the same nearly even attention, so that neither the heads
# nor a few large terms hide how the sum over the queries was rounded.  Root mean
# square error over the tokens: the attention's, the probe's and the heads' fp32 leave
# 8.5e-8 and 6.1e-8; with one fp32 chain over the queries it is 1.5e-7 and 9.5e-8
@pytest.mark.parametrize("B,T,bar", [(8, 256, 1.1e-7), (8, 100, 7.5e-8)])
def test_message_energy_over_many_queries(B, T, bar):
    from paper_2608_02134_gb300 import gmc
    from tests import parity
    gh, gw, H, Hkv, d, D, K = 36, 36, 28, 4, 64, 64, 16
    N = gh * gw
    g = torch.Generator(device="cuda")
    g.manual_seed(T)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    hid = rnd(B, N + T, D).bfloat16()
    key = rnd(B, 1, N + T, 1, d).expand(-1, -1, -1, Hkv, -1)
    kv = torch.cat([key, rnd(B, 1, N + T, Hkv, d)], 1).bfloat16().contiguous()
    q = (0.5 * rnd(B, T, 1, d)).expand(-1, -1, H, -1).bfloat16().contiguous()
    pos = torch.zeros(B * 3 * (N + T), dtype=torch.int32, device="cuda")
    W = rnd(H, d, 4) / d ** 0.5
    comp = gmc.Compressor(B, gh, gw, T, H, Hkv, d, D, K, gmc.GMC_BF16, trace=True)
    out = comp.run(hid.view(-1, D), kv.view(-1), q.view(-1), pos, W)
    torch.cuda.synchronize()
    assert comp.status() == 0
    tr = parity.parse_trace(out.trace.cpu().numpy(), out.layout, B, K, H, N,
                            comp.params.max_head_clusters)
    nu = torch.ones(T, dtype=torch.float64, device="cuda")
    nu[-1] = comp.params.terminal_q_weight
    nu /= nu.sum()
    for b in {0, B - 1}:
        S = q[b, :, 0].double() @ kv[b, 0, :, 0].double().T / d ** 0.5
        S[:, N:] = S[:, N:].masked_fill(torch.ones(T, T, device="cuda").triu(1).bool(), -torch.inf)
        W2 = (nu[:, None] * torch.softmax(S, 1)[:, :N].square()).sum(0)
        V = kv[b, 1, :N].double().repeat_interleave(H // Hkv, 1)
        Z2 = torch.einsum("nhd,hdr->nhr", V, W.double()).square().sum(2)
        om = torch.tensor(tr[b].omega, dtype=torch.float64, device="cuda")
        e = ((Z2 + Z2.mean(0) / 4) @ om * W2).sqrt()
        got = torch.tensor(tr[b].ebar, dtype=torch.float64, device="cuda")
        rel = (got / (e / e.mean()) - 1).square().mean().sqrt()
        assert float(rel) <= bar, float(rel)


def _clients(kind, B, M, N, seed):
    r = np.random.default_rng(seed)
    if kind == "equal":      # every token its own row of one value: all gains tie in every round
        C = np.zeros((B, M, N), np.float32)
        C[:, np.arange(N) % M, np.arange(N)] = 0.01
        return C
    if kind == "close":      # the same with gains a few units in the last place apart
        C = np.zeros((B, M, N), np.float32)
        v = np.float32(0.01) * (1 + r.permutation(N).astype(np.float32) * np.float32(2.0 ** -22))
        C[:, np.arange(N) % M, np.arange(N)] = v
        return C
    from tests.test_gpu_stages import _structured_clients
    if kind == "dense":      # many survivors a round: lists that start in global memory
        C = r.exponential(size=(B, M, N)) ** 0.25
        return (C / C.sum(axis=(1, 2), keepdims=True)).astype(np.float32)
    return _structured_clients(B, M, N, seed)


# the cluster solver: more equal or nearly equal gains than a round lists exactly
# (the radix search and its ties), lists that are in global memory for its first rounds
# (23,700 and 21,300 entries a CTA where 19,200 fit) above and below N = 4,096, token
# counts that are no multiple of 32, the widest pool, pools that are no power of two, one to sixteen
# CTAs an image, a budget of one round, rounds left over by a fill
@pytest.mark.parametrize("kind,B,M,N,K,b,mult", [
    ("equal", 1, 1200, 1200, 100, 16, 4), ("close", 1, 1300, 1300, 90, 16, 4),
    ("dense", 4, 3000, 1100, 96, 16, 4), ("plain", 1, 500, 33, 20, 16, 4),
    ("plain", 1, 90, 1025, 300, 32, 4), ("plain", 2, 700, 500, 100, 3, 5),
    ("plain", 20, 300, 300, 60, 16, 4), ("plain", 90, 120, 200, 40, 16, 4),
    ("plain", 1, 400, 640, 16, 16, 4), ("plain", 1, 60, 7000, 200, 16, 4),
    ("equal", 1, 40, 700, 64, 16, 4), ("dense", 1, 3000, 4500, 60, 2, 4),
    ("dense", 1, 2500, 4501, 40, 2, 4), ("dense", 1, 3000, 1100, 40, 1, 4)])
def test_cluster_solver_sizes(kind, B, M, N, K, b, mult):
    from tests.test_gpu_stages import _check_select
    _check_select(_clients(kind, B, M, N, 5 + N), K, batch_b=b, pool_mult=mult)


# the hand-over to the cluster solver follows what its shared memory holds of the lists:
# at one token count more client rows take more rounds on the whole GPU (launches of a
# call: copy and sum, exponent, column sums, three of the dense round, three a sparse
# round, the cluster's), and never more than the budget has left
@pytest.mark.parametrize("B,M,N,K,sparse", [
    (1, 2000, 1296, 200, 1), (1, 8720, 1296, 200, 4), (1, 8720, 1296, 33, 2), (1, 8720, 1296, 16, 0),
    (4, 600, 900, 60, 1)])
def test_sparse_rounds_follow_the_client_rows(B, M, N, K, sparse):
    from paper_2608_02134_gb300 import gmc
    from tests.test_gpu_stages import _check_select
    n0 = gmc.launch_count()
    _check_select(_clients("plain", B, M, N, 11 + M), K)
    assert gmc.launch_count() - n0 == 7 + 3 * sparse


# the wide solver: one, four and eight pool slots a thread, rows on 16 bytes and not,
# the most tokens, all gains equal (the digits of the token decide) or nearly so, a
# batch that is the whole pool, more rows than blocks and fewer
@pytest.mark.parametrize("kind,B,M,N,K,b,mult", [
    ("equal", 1, 40, 9000, 700, 100, 4), ("close", 1, 200, 3001, 600, 300, 4),
    ("dense", 1, 300, 2050, 900, 700, 5), ("plain", 3, 50, 1000, 400, 130, 1),
    ("plain", 1, 30, 16384, 64, 256, 8), ("plain", 1, 2300, 501, 200, 40, 4),
    ("dense", 2, 170, 4096, 1500, 512, 4), ("equal", 1, 33, 2600, 2600, 1024, 2)])
def test_wide_solver_sizes(kind, B, M, N, K, b, mult):
    from tests.test_gpu_stages import _check_select
    _check_select(_clients(kind, B, M, N, 7 + N), K, batch_b=b, pool_mult=mult)


# the wide solver's window pool (at most 128 slots, beyond the cluster solver's
# bytes) at odd token counts, where the staged gains end on 8 bytes and not on 16,
# over enough rounds that the window is read: pools of 64 and 128, one
# image and two
@pytest.mark.parametrize("B,M,N,K,b", [(1, 4300, 8191, 200, 32), (1, 7700, 8191, 70, 16),
                                       (2, 4300, 8189, 100, 32)])
def test_window_pool_at_odd_token_counts(B, M, N, K, b):
    from paper_2608_02134_gb300 import gmc
    from tests.test_gpu_stages import _check_select
    n0 = gmc.launch_count()
    _check_select(_clients("plain", B, M, N, 3 + N), K, batch_b=b)
    # the whole-GPU solver ran (four launches a round)
    assert gmc.launch_count() - n0 == 3 + 4 * (-(-K // b)) + 1 + 1


# transport: fewer and more member rows than a thread has in flight, lists of more
# than 64 members (one carrier takes every token), one list for the block (N above
# 4,096), a row that is one CTA and one that is eight, more text rows than carriers,
# K/V rows wider than the threads, both types; from a caller's assignment
@pytest.mark.parametrize("B,gh,gw,T,K,D,Hkv,d,dtype,spread", [
    (1, 5, 7, 3, 4, 64, 2, 32, "bf16", "all"), (2, 9, 31, 40, 11, 1032, 1, 8, "f32", "even"),
    (1, 66, 64, 5, 700, 256, 2, 32, "bf16", "even"), (1, 128, 64, 9, 3, 8192, 32, 128, "bf16", "all"),
    (3, 20, 13, 17, 260, 3584, 4, 128, "bf16", "even"), (1, 64, 64, 2, 33, 4096, 16, 64, "f32", "skew")])
def test_transport_sizes(B, gh, gw, T, K, D, Hkv, d, dtype, spread):
    from paper_2608_02134_gb300 import gmc
    N = gh * gw
    g = torch.Generator(device="cuda")
    g.manual_seed(N + D)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    hid = torch.randn((B, N + T, D), generator=g, device="cuda").to(tdt)
    kv = torch.randn((B, 2, N + T, Hkv, d), generator=g, device="cuda").to(tdt)
    pos = torch.randint(0, 1000, (B, 3, N + T), generator=g, device="cuda", dtype=torch.int32)
    sup = torch.stack([torch.randperm(N, generator=g, device="cuda")[:K].sort().values
                       for _ in range(B)])
    u = torch.rand((B, N), generator=g, device="cuda")
    slot = {"all": torch.zeros_like(u), "even": u * K, "skew": u ** 3 * K}[spread].long().clamp(max=K - 1)
    slot.scatter_(1, sup, torch.arange(K, device="cuda").expand(B, K))
    pi = sup.gather(1, slot)
    w = 0.5 + torch.rand((B, N), generator=g, device="cuda")
    prob = gmc.problem(B, gh, gw, Hkv, gmc.GMC_BF16 if dtype == "bf16" else gmc.GMC_F32)
    ws = gmc.alloc_workspace(gmc.transport_workspace_size(prob, N, T, K))
    oi = torch.empty(B * K, dtype=torch.int32, device="cuda")
    oh = torch.empty((B, K + T, D), dtype=tdt, device="cuda")
    okv = torch.empty((B, 2, K + T, Hkv, d), dtype=tdt, device="cuda")
    op = torch.empty((B, 3, K + T), dtype=torch.int32, device="cuda")
    gmc.transport(prob, gmc.default_params(), hid, kv, pos, sup.int().contiguous(),
                  pi.int().contiguous(), w, N, T, d, D, K, oi, oh, okv, op, ws)
    torch.cuda.synchronize()
    assert gmc.read_status(ws) == 0
    assert torch.equal(oi.view(B, K).long(), sup)
    for b in range(B):
        rows = torch.cat([sup[b], N + torch.arange(T, device="cuda")])
        assert torch.equal(okv[b], kv[b][:, rows]) and torch.equal(op[b], pos[b][:, rows])
        assert torch.equal(oh[b, K:], hid[b, N:])
        h, m = hid[b, :N].double(), w[b].double()
        acc = torch.zeros((K, D), dtype=torch.float64, device="cuda").index_add_(0, slot[b], m[:, None] * h)
        cen = acc / torch.zeros(K, dtype=torch.float64, device="cuda").index_add_(0, slot[b], m)[:, None]
        rms = lambda v: v.square().mean(1, keepdim=True).sqrt()  # noqa: E731
        ref = cen * rms(h[sup[b]]) / (rms(cen) + 1e-6)
        # fp32 sums of up to N terms, each rounded once (N 2^-24 of the terms' magnitude), and
        # the cast of the output: half an ulp of bf16
        terms = torch.zeros_like(acc).index_add_(0, slot[b], m[:, None] * h.abs()) / (acc.abs() + 1e-300)
        bound = (N * 2.0 ** -24) * (terms * ref.abs()) + 2e-6 * ref.abs() + 1e-7
        if dtype == "bf16":
            bound = bound + ref.abs() * 2.0 ** -8
        assert bool(((oh[b, :K].double() - ref).abs() <= bound).all())


def _check_grounded(wl):
    """The grounded rows of the first and the last image, at the GPU's head weights."""
    from oracle import gmc_oracle as O
    from tests.test_gpu_clients import _gpu_clients
    C, traces, comp = _gpu_clients(wl)
    p = O.params()
    f = lambda a: np.asarray(a, dtype=np.float64)  # noqa: E731
    for b in {0, wl.B - 1}:
        im, tr = wl.image(b), traces[b]
        A = O.message_slice(f(im.queries), f(im.keys), wl.N)
        Z, sigma = O.probe_values(f(im.values)[:wl.N], f(wl.probe()), wl.H, p)
        P, _ = O.grounded_clients(O.atom_norms(A, Z, sigma))
        nu = O.query_weights(im.T, p)
        ref = 0.5 * f(tr.omega)[:, None, None] * nu[None, :, None] * P
        got = C[b, :wl.H * im.T].reshape(wl.H, im.T, wl.N)
        err = np.abs(got - ref).max(2) / ref.max(2)
        assert err.max() <= 1e-3, err.max()   # the bar of the client parity tests


# message slice: key splits that fill a cluster, exceed the portable cluster size and
# exceed the largest one (two launches); query tiles that are ragged; keys that end
# inside a tile, rows of A on 16 bytes and not
@pytest.mark.parametrize("gh,gw,T,H,Hkv,B", [
    (16, 8, [40], 4, 2, 1), (48, 54, [8], 4, 4, 1), (23, 41, [70, 3, 33], 6, 2, 3), (36, 37, [21], 28, 28, 12),
    (66, 64, [9], 4, 1, 1), (128, 64, [5], 2, 1, 1)])
def test_message_slice_splits(gh, gw, T, H, Hkv, B):
    from paper_2608_02134_gb300 import workloads
    wl = workloads.make("qwen", B=B, T=T * (B // len(T)), gh=gh, gw=gw, D=64, d=64, H=H, Hkv=Hkv, K=9)
    _check_grounded(wl)


# few query tiles of a large image run as two launches over many splits, more of them as
# one launch of clusters (a call of gmc_clients counts one launch less): both, at one
# grid each, against the oracle's rows
@pytest.mark.parametrize("gh,gw,few,many", [(48, 54, 8, 192), (64, 64, 64, 128)])
def test_message_slice_launches(gh, gw, few, many):
    from paper_2608_02134_gb300 import gmc, workloads
    count = []
    for T in (few, many):
        wl = workloads.make("qwen", B=1, T=T, gh=gh, gw=gw, D=64, d=64, H=28, Hkv=4, K=9)
        n0 = gmc.launch_count()
        _check_grounded(wl)
        count.append(gmc.launch_count() - n0)
    assert count[0] == count[1] + 1


# probe: one head a KV group, more heads than warps, value rows of an odd and an even
# number of 16-byte units, a last block that is not full, both types
@pytest.mark.parametrize("name,gh,gw,T,H,Hkv,d,B", [
    ("qwen", 5, 13, [3], 4, 4, 8, 1), ("qwen", 9, 9, [17, 2], 18, 1, 72, 2),
    ("tiny", 7, 11, [6], 12, 1, 20, 1), ("tiny", 4, 8, [9], 3, 3, 64, 1),
    ("qwen", 11, 12, [40], 28, 4, 128, 3)])
def test_probe_sizes(name, gh, gw, T, H, Hkv, d, B):
    from paper_2608_02134_gb300 import workloads
    _check_grounded(workloads.make(name, B=B, T=T * (B // len(T)), gh=gh, gw=gw, D=64, d=d, H=H,
                                   Hkv=Hkv, K=9))


# assignment: gates that leave every gap open, some and none, a weight that lets the
# spatial term outweigh any gap and one of zero, one carrier, duplicated tokens (gap
# zero), several images: the carrier of every discarded token has the largest kappa
@pytest.mark.parametrize("shape,K,gate_scale,weight,margin,twins", [
    (dict(gh=8, gw=8, D=32), 16, 0.08, 0.5, 0.05, False),
    (dict(gh=9, gw=23, D=64), 60, 1e-3, 0.5, 0.05, False),
    (dict(gh=9, gw=23, D=64), 60, 1e-3, 8.0, 1.0, False),
    (dict(gh=9, gw=23, D=64), 33, 1e9, 0.5, 0.05, True),
    (dict(gh=17, gw=31, D=32), 100, 1e-3, 0.0, 0.05, True),
    (dict(gh=5, gw=7, D=32), 1, 1e-3, 0.5, 0.05, False),
    (dict(gh=9, gw=11, D=64, I=3), 40, 1e-3, 0.5, 0.2, True)])
def test_assignment_gates(shape, K, gate_scale, weight, margin, twins):
    from oracle import gmc_oracle as O
    from paper_2608_02134_gb300 import gmc, workloads
    from tests import gpu_harness as GH
    wl = workloads.make("tiny", K=K, T=9, **shape)
    inp = GH.to_device(wl)
    ng = wl.gh * wl.gw
    if twins:  # tokens 2 and 3 of every image hold the same state
        h = inp["hidden"].view(-1, wl.D)
        h[torch.arange(0, wl.N, ng) + 3] = h[torch.arange(0, wl.N, ng) + 2]
    params = gmc.default_params(gate_scale=gate_scale, assign_spatial_w=weight,
                                ambig_margin=margin)
    run = GH.run(wl, params=params, inputs=inp)
    assert run.status == 0
    tr, S = run.traces[0], run.idx[:K]
    p = O.params(gate_scale=gate_scale, assign_spatial_w=weight, ambig_margin=margin)
    x = O.unit_states(inp["hidden"].view(-1, wl.D)[:wl.N].cpu().numpy().astype(np.float64), p)
    cos = x @ x[S].T
    tok = np.arange(wl.N)
    cos[(tok[:, None] // ng) != (S[None] // ng)] = -np.inf
    top = np.sort(cos, axis=1)[:, ::-1]
    with np.errstate(invalid="ignore"):
        delta = top[:, 0] - top[:, 1] if K > 1 else np.zeros(wl.N)
    delta = np.where(np.isfinite(delta), delta, 0.0)
    pos = O.grid_coords(wl.gh, wl.gw)[tok % ng]
    d2 = ((pos[:, None] - pos[S][None]) ** 2).sum(2)
    gate = np.exp(-((delta / margin) ** p["gate_pow"]))
    kappa = cos + weight * tr.s_x * gate[:, None] * np.exp(-d2 / p["tau_s"])
    got = kappa[tok, np.searchsorted(S, tr.pi)]
    # fp32 cosines of D terms are within D 2^-24 each; the gate's slope is below
    # 3.1 / margin, and it multiplies the spatial term
    eps = wl.D * 2.0 ** -24 + 1e-6
    tol = 2 * eps + weight * (3.1 / margin) * 2 * eps
    disc = np.ones(wl.N, bool)
    disc[S] = False
    assert np.isin(tr.pi, S).all() and np.array_equal(tr.pi[S], S)
    assert (got[disc] >= kappa.max(1)[disc] - tol).all(), (kappa.max(1) - got)[disc].max()


# tensor-core Gram: one tile a CTA and several (both accumulators, the stage ring over
# tile boundaries), tiles of 128 and of 256 columns, rows of C on 16 bytes and not, a last tile that is shifted inward,
# blocks on, above and mirrored below the diagonal, K that ends inside a slice
@pytest.mark.parametrize("B,gh,gw,D,T", [
    (80, 16, 16, 64, 3), (4, 36, 36, 200, 2), (14, 24, 24, 64, 5), (90, 17, 17, 136, 1), (31, 12, 25, 1000, 5), (12, 23, 31, 264, 2), (2, 47, 49, 72, 7),
    (1, 64, 65, 512, 1), (3, 36, 36, 3584, 9), (1, 79, 77, 136, 4)])
def test_cosine_gram_tiles(B, gh, gw, D, T):
    from paper_2608_02134_gb300 import gmc
    N = gh * gw
    g = torch.Generator(device="cuda")
    g.manual_seed(N + D)
    hid = torch.randn((B, N + T, D), generator=g, device="cuda").to(torch.bfloat16)
    out = torch.full((B, N, N), float("nan"), device="cuda")
    ws = gmc.cosine(gmc.problem(B, gh, gw, 1, gmc.GMC_BF16), gmc.default_params(), hid, N, T, D, out)
    torch.cuda.synchronize()
    assert gmc.read_status(ws) == 0
    for b in {0, B // 2, B - 1}:
        x = hid[b, :N].double()
        x = x / x.norm(dim=1, keepdim=True)
        # products exact in fp32, D of them summed in fp32 (truncating at worst), then two
        # scales of fp32 norms: (D + 8) 2^-23 of the terms' magnitudes, which sum to at most 1
        assert float((out[b].double() - x @ x.T).abs().max()) <= (D + 8) * 2.0 ** -23
