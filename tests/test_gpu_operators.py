"""Operator-level GPU parity (need a B200): the stand-alone tree-attention and small-M GEMM entry points of
the C ABI against the CPU oracle, plus the bitwise row-invariance the lossless guarantee rests on."""
import numpy as np
import pytest
import torch

import synth
import paper_2603_17942_b200 as P
from oracle import esp as O

pytestmark = pytest.mark.gpu

R = P.ESP_MAX_ROWS


# ------------------------------------------------------------------ small-M GEMM
def _gemm(impl, x, w, rows):
    n_out, k_in = w.shape
    xd = torch.zeros(R, k_in, dtype=torch.bfloat16, device="cuda")
    xd[:rows] = x.cuda()
    y = torch.full((R, n_out), float("nan"), dtype=torch.float32, device="cuda")
    nb = P.esp_gemm_scratch_bytes()
    scratch = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    P.esp_gemm_bf16(impl, rows, n_out, k_in, xd, w, y, scratch, nb)
    torch.cuda.synchronize()
    return y[:rows].cpu().numpy()


@pytest.mark.parametrize("rows,n_out,k_in", [(1, 128, 64), (68, 384, 512), (80, 1000, 688), (68, 6144, 4096),
                                             (5, 4096, 14336), (68, 20000, 4096)])
def test_gemm_bf16_against_oracle(rows, n_out, k_in):
    """y = x W^T for bf16 operands with fp32 accumulation.  Products of bf16 values are exact in fp32, so the
    only difference to the oracle's running sum is the order of the fp32 additions."""
    g = torch.Generator().manual_seed(rows * 7919 + n_out)
    x = torch.randn(rows, k_in, generator=g).bfloat16()
    w = (torch.randn(n_out, k_in, generator=g) * 0.05).bfloat16().cuda()
    ref = O.linear(x.float().numpy(), w.cpu())
    scale = np.abs(ref).max()
    for impl in (0, 1):
        got = _gemm(impl, x, w, rows)
        assert np.isfinite(got).all()
        assert np.abs(got - ref).max() <= 2e-5 * scale, f"impl {impl}"


def test_gemm_rows_do_not_depend_on_their_neighbours():
    """A row's result has the same bits whether it runs alone or among 79 others (the tensor-core kernel is
    launched with one fixed tile shape and one fixed k split for every row count)."""
    g = torch.Generator().manual_seed(5)
    k_in, n_out = 4096, 4096
    x = torch.randn(R, k_in, generator=g).bfloat16()
    w = (torch.randn(n_out, k_in, generator=g) * 0.05).bfloat16().cuda()
    full = _gemm(0, x, w, R)
    for r in (0, 37, 79):
        alone = _gemm(0, x[r:r + 1], w, 1)
        assert np.array_equal(alone[0], full[r])
    again = _gemm(0, x, w, R)
    assert np.array_equal(full, again)       # run-to-run deterministic (no arrival-order dependence)


@pytest.mark.parametrize("rows", [1, 7, 8, 9, 128])
def test_cuda_core_gemm_by_elements_equals_16_byte_copies(rows):
    """A matrix that does not start on 16 bytes goes through the element-wise loads of the CUDA-core kernel: the same
    sums in the same order, so the same bits, for every remainder of the kernel's groups of 8 rows and 64 k."""
    g = torch.Generator().manual_seed(rows)
    n_out, k_in = 200, 136
    x = torch.randn(rows, k_in, generator=g).bfloat16()
    flat = torch.zeros(n_out * k_in + 8, dtype=torch.bfloat16, device="cuda")
    w = (torch.randn(n_out, k_in, generator=g) * 0.05).bfloat16().cuda()
    odd = flat[1:1 + n_out * k_in].view(n_out, k_in)
    odd.copy_(w)
    assert w.data_ptr() % 16 == 0 and odd.data_ptr() % 16 == 2
    assert np.array_equal(_gemm(1, x, w, rows), _gemm(1, x, odd, rows))


# ------------------------------------------------------------------ tree attention (the stand-alone operator workload)
def _tree_block(n_nodes, n_probes, max_depth, seed):
    parents = synth.random_tree_parents(n_nodes, max_depth, seed)
    M = n_nodes + n_probes
    depth = np.zeros(M, np.int32)
    vis = np.zeros((M, M), np.uint8)
    for i in range(n_nodes):
        a = i
        while a >= 0:
            vis[i, a] = 1
            a = int(parents[a])
        depth[i] = vis[i].sum() - 1
    for j in range(n_probes):        # a mask-probe chain under the root
        r = n_nodes + j
        vis[r, 0] = 1
        vis[r, n_nodes:r + 1] = 1
        depth[r] = j + 1
    return parents, depth, vis


def _anc_words(vis):
    M = vis.shape[0]
    anc = np.zeros((R, 2), np.uint64)
    for r in range(M):
        for i in range(M):
            if vis[r, i]:
                anc[r, i // 64] |= np.uint64(1) << np.uint64(i % 64)
    for r in range(M, R):
        anc[r, r // 64] = np.uint64(1) << np.uint64(r % 64)
    return anc


def _run_attention(dtype, q, kc, vc, anc, depth, n_rows, L, Hq, Hkv, h, dcap=16):
    """q [b,R,Hq,h]; kc/vc [b,Hkv,cap,h] with block rows already at L+i; anc [b,R,2]; depth [b,R]."""
    b, cap = kc.shape[0], kc.shape[2]
    out = torch.zeros_like(q)
    nb = P.esp_tree_attention_scratch_bytes(b, Hq, h, cap)
    scratch = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    P.esp_tree_attention(dtype, b, n_rows, L, cap, Hq, Hkv, h, dcap, q, kc, vc,
                         torch.from_numpy(anc.view(np.int64)).cuda(), torch.from_numpy(depth).cuda(), out, scratch, nb)
    torch.cuda.synchronize()
    assert P.esp_tree_attention_status(scratch) == 0       # no bounded wait ran out, no index left its range
    return out


def test_tree_attention_status_reports_a_set_error_word():
    """The operator reports device-side problems through the first word of its scratch.  The read-back is checked
    from the host side: a word set by hand must come back as ESP_E_DEVICE, and the next call must clear it."""
    Hq, Hkv, h, L = 32, 8, 128, 300
    cap = L + R
    q, kc, vc, _, _ = synth.random_qkv((1, R, Hq, h), (1, Hkv, cap, h), (1, Hkv, 4, h), seed=1, device="cuda")
    anc = np.zeros((1, R, 2), np.uint64)
    for i in range(R):
        anc[0, i, i // 64] = np.uint64(1) << np.uint64(i % 64)
    nb = P.esp_tree_attention_scratch_bytes(1, Hq, h, cap)
    scratch = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    args = (1, 1, 4, L, cap, Hq, Hkv, h, 16, q, kc, vc, torch.from_numpy(anc.view(np.int64)).cuda(),
            torch.zeros((1, R), dtype=torch.int32, device="cuda"), torch.zeros_like(q), scratch, nb)
    P.esp_tree_attention(*args)
    assert P.esp_tree_attention_status(scratch) == 0
    scratch[:4] = torch.tensor([2, 0, 0, 0], dtype=torch.uint8, device="cuda")     # as a kernel would record DEV_E_INDEX
    with pytest.raises(P.EspError) as e:
        P.esp_tree_attention_status(scratch)
    assert e.value.code == -5                               # ESP_E_DEVICE
    P.esp_tree_attention(*args)
    assert P.esp_tree_attention_status(scratch) == 0


@pytest.mark.parametrize("batch,L,dt", [(1, 4096, "bf16"), (16, 4096, "bf16"), (4, 4096, "bf16"), (2, 777, "bf16"),
                                        (1, 0, "bf16"), (1, 5, "bf16"), (2, 300, "fp32")])
def test_tree_attention_against_oracle(batch, L, dt):
    """32 query heads / 8 KV heads of 128, N(0,1) cache, a 64-node random tree of depth <= 5 plus 4 mask-probe
    rows.  The split length follows the batch: 16 splits of 256 positions for one sequence at 4096, one split of
    4096 for 16 sequences, 4 splits of 1024 for 4 sequences (items of 8 chunks on the persistent kernel, merged
    over splits).  Tolerance: the output is a convex combination of N(0,1) values, bf16 rounding of the probabilities
    and of the output bounds the error by a few 2^-8 relative steps; 2e-2 absolute covers it."""
    Hq, Hkv, h, n_nodes, n_probes = 32, 8, 128, 64, 4
    M = n_nodes + n_probes
    cap = L + R
    tdt = torch.bfloat16 if dt == "bf16" else torch.float32
    q, kc, vc, kb, vb = synth.random_qkv((batch, R, Hq, h), (batch, Hkv, cap, h), (batch, Hkv, M, h), seed=L + batch,
                                         device="cuda", dtype=tdt)
    kc[:, :, L:L + M] = kb
    vc[:, :, L:L + M] = vb
    anc = np.zeros((batch, R, 2), np.uint64)
    depth = np.zeros((batch, R), np.int32)
    vis_all = []
    for s in range(batch):
        _, d, vis = _tree_block(n_nodes, n_probes, 5, seed=100 * L + s)
        anc[s] = _anc_words(vis)
        depth[s, :M] = d
        vis_all.append(vis)
    out = _run_attention(0 if dt == "fp32" else 1, q, kc, vc, anc, depth, M, L, Hq, Hkv, h)
    tol = 2e-2 if dt == "bf16" else 2e-5
    for s in sorted({0, batch // 2, batch - 1}):
        ref = O.tree_attention(q[s, :M].float().cpu().numpy(), kc[s, :, :L].float().permute(1, 0, 2).cpu().numpy(),
                               vc[s, :, :L].float().permute(1, 0, 2).cpu().numpy(),
                               kb[s].float().permute(1, 0, 2).cpu().numpy(), vb[s].float().permute(1, 0, 2).cpu().numpy(),
                               vis_all[s])
        got = out[s, :M].float().cpu().numpy()
        assert np.isfinite(got).all()
        assert np.abs(got - ref).max() <= tol, f"sequence {s}"


def test_tree_attention_rows_equal_decoding_each_path_alone():
    """Bitwise: a node verified inside the tree block gets the bits it would get if its ancestors had been
    accepted into the cache and it were decoded alone (what lossless verification needs)."""
    Hq, Hkv, h, n_nodes, n_probes, L = 32, 8, 128, 64, 4, 1500
    M = n_nodes + n_probes
    cap = L + R + 16                                  # room for the deepest path moved into the cache
    q, kc, vc, kb, vb = synth.random_qkv((1, R, Hq, h), (1, Hkv, cap, h), (1, Hkv, M, h), seed=9, device="cuda")
    kc[:, :, L:L + M] = kb
    vc[:, :, L:L + M] = vb
    _, depth_m, vis = _tree_block(n_nodes, n_probes, 5, seed=77)
    depth = np.zeros((1, R), np.int32)
    depth[0, :M] = depth_m
    tree_out = _run_attention(1, q, kc, vc, _anc_words(vis)[None], depth, M, L, Hq, Hkv, h)
    rng = np.random.default_rng(0)
    for r in [0, M - 1] + [int(x) for x in rng.choice(np.arange(1, M - 1), 6, replace=False)]:
        chain = [i for i in range(M) if vis[r, i]]
        d = len(chain) - 1
        kc1, vc1 = kc.clone(), vc.clone()
        for j, i in enumerate(chain):               # ancestors become cache entries L..L+d-1, the row itself sits at L+d
            kc1[0, :, L + j] = kb[0, :, i]
            vc1[0, :, L + j] = vb[0, :, i]
        q1 = torch.zeros_like(q)
        q1[0, 0] = q[0, r]
        anc1 = np.zeros((1, R, 2), np.uint64)
        for i in range(R):
            anc1[0, i, i // 64] = np.uint64(1) << np.uint64(i % 64)
        alone = _run_attention(1, q1, kc1, vc1, anc1, np.zeros((1, R), np.int32), 1, L + d, Hq, Hkv, h)
        assert torch.equal(alone[0, 0], tree_out[0, r]), f"row {r} (depth {d})"


@pytest.mark.parametrize("dt,h,group,n_rows,L", [("fp32", 64, 2, 35, 777), ("fp32", 128, 1, 17, 300), ("fp32", 32, 8, 3, 33),
                                                 ("bf16", 64, 4, 9, 1025), ("bf16", 32, 3, 128, 64)])
def test_cuda_core_attention_edges(dt, h, group, n_rows, L):
    """The CUDA-core attention against its definition in fp64 at the edges of its 16-pair CTAs, 32-key chunks and
    splits, with a cache that starts on 16 bytes and one that does not (same bits).  A chain of n_rows rows, so that
    row r sees positions 0..L+r.  fp32: sums of at most L + n_rows terms; bf16: the result's own rounding."""
    dtype = torch.float32 if dt == "fp32" else torch.bfloat16
    Hkv, cap, b = 2, L + R, 2
    Hq = Hkv * group
    g = torch.Generator().manual_seed(h + L)
    q = torch.randn(b, R, Hq, h, generator=g).to(dtype).cuda()
    kc, vc = (torch.randn(b, Hkv, cap, h, generator=g).to(dtype).cuda() for _ in range(2))
    vis = np.tril(np.ones((n_rows, n_rows), np.uint8))
    anc = np.stack([_anc_words(vis)] * b)
    depth = np.zeros((b, R), np.int32)
    depth[:, :n_rows] = np.arange(n_rows)
    dcap = (max(16, n_rows) + 15) // 16 * 16
    out = _run_attention(int(dt == "bf16"), q, kc, vc, anc, depth, n_rows, L, Hq, Hkv, h, dcap)[:, :n_rows]
    odd = []
    for t in (kc, vc):
        flat = torch.zeros(t.numel() + 8, dtype=dtype, device="cuda")
        odd.append(flat[1:1 + t.numel()].view(t.shape))
        odd[-1].copy_(t)
    assert torch.equal(out, _run_attention(int(dt == "bf16"), q, odd[0], odd[1], anc, depth, n_rows, L, Hq, Hkv, h, dcap)[:, :n_rows])
    s = torch.einsum("brhd,bhcd->bhrc", q[:, :n_rows].double(), kc.repeat_interleave(group, 1)[:, :, :L + n_rows].double()) / h ** 0.5
    hide = torch.arange(L + n_rows)[None] > L + torch.arange(n_rows)[:, None]
    s.masked_fill_(hide.cuda(), -float("inf"))
    ref = torch.einsum("bhrc,bhcd->brhd", s.softmax(-1), vc.repeat_interleave(group, 1)[:, :, :L + n_rows].double())
    tol = 2e-5 if dt == "fp32" else 2.0 ** -8 * float(ref.abs().max())
    assert (out.double() - ref).abs().max() <= tol


def test_tree_attention_one_item_and_persistent_kernels_agree_bitwise():
    """The cache below T0 is summed by one of two tensor-core kernels, picked by the number of (split, KV head,
    row tile, sequence) items in the launch.  The split length is a function of capacity, batch and head count, so
    the two are compared inside one batch: 12 sequences at KV 2048 get one split each; with 68 rows (3 row tiles)
    that is 288 items, above the switch, with the block cut to its first 20 rows (1 row tile, ancestors are
    earlier rows) 96 items, below it.  The 20 rows must come out bit for bit alike from both calls, every copy of
    a sequence like the others, and a different sequence in the same call must not disturb them."""
    Hq, Hkv, h, n_nodes, n_probes, L, few = 32, 8, 128, 64, 4, 2048, 20
    M = n_nodes + n_probes
    cap = L + R
    q, kc, vc, kb, vb = synth.random_qkv((1, R, Hq, h), (1, Hkv, cap, h), (1, Hkv, M, h), seed=77, device="cuda")
    kc[:, :, L:L + M] = kb
    vc[:, :, L:L + M] = vb
    _, d, vis = _tree_block(n_nodes, n_probes, 5, seed=5)
    assert not vis[:few, few:].any()
    anc = _anc_words(vis)[None]
    depth = np.zeros((1, R), np.int32)
    depth[0, :M] = d
    q2, kc2, vc2, _, _ = synth.random_qkv((1, R, Hq, h), (1, Hkv, cap, h), (1, Hkv, M, h), seed=78, device="cuda")
    order = [0, 1] + [0] * 10
    qq = torch.cat([(q, q2)[i] for i in order]).contiguous()
    kk = torch.cat([(kc, kc2)[i] for i in order]).contiguous()
    vv = torch.cat([(vc, vc2)[i] for i in order]).contiguous()
    ancs, depths = np.repeat(anc, len(order), 0), np.repeat(depth, len(order), 0)
    many = _run_attention(1, qq, kk, vv, ancs, depths, M, L, Hq, Hkv, h)
    anc_few = ancs.copy()
    for r in range(few, M):
        anc_few[:, r] = 0
        anc_few[:, r, r // 64] = np.uint64(1) << np.uint64(r % 64)
    fewer = _run_attention(1, qq, kk, vv, anc_few, depths, few, L, Hq, Hkv, h)
    for s in range(len(order)):
        assert torch.equal(many[s, :few], fewer[s, :few]), f"sequence {s}: the two kernels differ"
        if s >= 2:
            assert torch.equal(many[s, :M], many[0, :M]), f"copy {s}"
    assert not torch.equal(many[1, :M], many[0, :M])


def test_tree_attention_long_context_against_oracle():
    """KV length 32768 (the longest context of the batch sweep): the cache is cut in 32 splits of 1024; every
    row and head against the oracle."""
    Hq, Hkv, h, n_nodes, n_probes, L = 32, 8, 128, 64, 4, 32768
    M = n_nodes + n_probes
    cap = L + R
    q, kc, vc, kb, vb = synth.random_qkv((1, R, Hq, h), (1, Hkv, cap, h), (1, Hkv, M, h), seed=3, device="cuda")
    kc[:, :, L:L + M] = kb
    vc[:, :, L:L + M] = vb
    _, d, vis = _tree_block(n_nodes, n_probes, 5, seed=5)
    depth = np.zeros((1, R), np.int32)
    depth[0, :M] = d
    out = _run_attention(1, q, kc, vc, _anc_words(vis)[None], depth, M, L, Hq, Hkv, h)
    ref = O.tree_attention(q[0, :M].float().cpu().numpy(), kc[0, :, :L].float().permute(1, 0, 2).cpu().numpy(),
                           vc[0, :, :L].float().permute(1, 0, 2).cpu().numpy(), kb[0].float().permute(1, 0, 2).cpu().numpy(),
                           vb[0].float().permute(1, 0, 2).cpu().numpy(), vis)
    got = out[0, :M].float().cpu().numpy()
    assert np.isfinite(got).all()
    assert np.abs(got - ref).max() <= 2e-2


def test_bounded_wait_gives_up_and_leaves_the_context_usable():
    """A barrier that nothing signals: the kernel's wait must run out (about 50 ms), report the wait-timeout
    code through the error word and return; the next kernel on the same context works."""
    import time
    scratch = torch.zeros(256, dtype=torch.uint8, device="cuda")
    t0 = time.perf_counter()
    status = P.esp_debug_wait_selftest(scratch)
    dt = time.perf_counter() - t0
    assert status == 1                      # DEV_E_WAIT_TIMEOUT
    assert 0.03 < dt < 2.0
    g = torch.Generator().manual_seed(1)
    x = torch.randn(4, 64, generator=g).bfloat16()
    w = (torch.randn(128, 64, generator=g) * 0.05).bfloat16().cuda()
    got = _gemm(0, x, w, 4)
    ref = O.linear(x.float().numpy(), w.cpu())
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()


@pytest.mark.parametrize("dt,h", [("fp32", 64), ("bf16", 128)])
def test_tree_attention_with_room_for_the_block_only(dt, h):
    """cap = ESP_MAX_ROWS, L = 0: no cached position and no room for one, with several sequences."""
    dtype = torch.float32 if dt == "fp32" else torch.bfloat16
    b, Hq, Hkv, n_rows = 2, 4, 2, 9
    g = torch.Generator().manual_seed(3)
    q = torch.randn(b, R, Hq, h, generator=g).to(dtype).cuda()
    kc, vc = (torch.randn(b, Hkv, R, h, generator=g).to(dtype).cuda() for _ in range(2))
    _, depth1, vis = _tree_block(n_rows, 0, 4, 8)
    depth = np.zeros((b, R), np.int32)
    depth[:, :n_rows] = depth1
    out = _run_attention(int(dt == "bf16"), q, kc, vc, np.stack([_anc_words(vis)] * b), depth, n_rows, 0, Hq, Hkv, h)[:, :n_rows]
    s = torch.einsum("brhd,bhcd->bhrc", q[:, :n_rows].double(), kc.repeat_interleave(2, 1)[:, :, :n_rows].double()) / h ** 0.5
    s.masked_fill_(torch.from_numpy(vis == 0).cuda(), -float("inf"))
    ref = torch.einsum("bhrc,bhcd->brhd", s.softmax(-1), vc.repeat_interleave(2, 1)[:, :, :n_rows].double())
    tol = 2e-5 if dt == "fp32" else 2.0 ** -8 * float(ref.abs().max())      # sums of a few terms; the result's own rounding
    assert (out.double() - ref).abs().max() <= tol


@pytest.mark.parametrize("group,n_rows,L,dcap", [(1, 33, 5, 16), (2, 9, 0, 16), (4, 68, 15, 16), (8, 41, 16, 32), (16, 7, 40, 48), (4, 128, 16, 128)])
def test_tree_attention_tail_alone(group, n_rows, L, dcap):
    """No row has a position below its T0, so the tail kernel does it all: fewer heads per KV head than a warp takes together,
    as many, and several times as many; lists of one key, of 32 and one more, of several chunks; keys before, on and behind the
    end of the cache.  The bound is the result's own rounding; that the weights keep their bits is seen by
    test_tree_attention_tail_weights_keep_their_24_bits."""
    Hkv, h, b = 2, 128, 2
    Hq, cap = Hkv * group, L + R
    if dcap == 128:
        depth1, vis = np.arange(n_rows), np.tril(np.ones((n_rows, n_rows), np.uint8))
    else:
        _, depth1, vis = _tree_block(n_rows, 0, dcap, n_rows)
    assert (np.maximum(L + depth1 - dcap, 0) // 16 * 16).max() == 0
    g = torch.Generator().manual_seed(group)
    q = torch.randn(b, R, Hq, h, generator=g).bfloat16().cuda()
    kc, vc = (torch.randn(b, Hkv, cap, h, generator=g).bfloat16().cuda() for _ in range(2))
    depth = np.zeros((b, R), np.int32)
    depth[:, :n_rows] = depth1
    out = _run_attention(1, q, kc, vc, np.stack([_anc_words(vis)] * b), depth, n_rows, L, Hq, Hkv, h, dcap)[:, :n_rows]
    s = torch.einsum("brhd,bhcd->bhrc", q[:, :n_rows].double(), kc.repeat_interleave(group, 1)[:, :, :L + n_rows].double()) / h ** 0.5
    hide = torch.zeros(n_rows, L + n_rows, dtype=torch.bool)
    hide[:, L:] = torch.from_numpy(vis == 0)
    ref = torch.einsum("bhrc,bhcd->brhd", s.masked_fill_(hide.cuda(), -float("inf")).softmax(-1), vc.repeat_interleave(group, 1)[:, :, :L + n_rows].double())
    assert (out.double() - ref).abs().max() <= 2.0 ** -8 * float(ref.abs().max())


@pytest.mark.parametrize("dt,h,offset", [("bf16", 128, 4), ("bf16", 64, 1), ("fp32", 64, 1)])
def test_tree_attention_output_of_the_stores_own_alignment(dt, h, offset):
    """`out` may start on any 8 bytes (tensor-core path), or on any element (CUDA-core path): the same bits, and nothing beside
    them is written.  L = 200: the cache and the tail both take part."""
    dtype = torch.float32 if dt == "fp32" else torch.bfloat16
    b, Hq, Hkv, n_rows, L = 1, 8, 2, 21, 200
    g = torch.Generator().manual_seed(5)
    q = torch.randn(b, R, Hq, h, generator=g).to(dtype).cuda()
    kc, vc = (torch.randn(b, Hkv, L + R, h, generator=g).to(dtype).cuda() for _ in range(2))
    _, depth1, vis = _tree_block(n_rows, 0, 6, 8)
    depth = np.zeros((b, R), np.int32)
    depth[:, :n_rows] = depth1
    ref = _run_attention(int(dt == "bf16"), q, kc, vc, _anc_words(vis)[None], depth, n_rows, L, Hq, Hkv, h)
    flat = torch.full((q.numel() + 16,), 7.0, dtype=dtype, device="cuda")
    out = flat[offset:offset + q.numel()].view_as(q)
    nb = P.esp_tree_attention_scratch_bytes(b, Hq, h, L + R)
    scratch = torch.zeros(nb, dtype=torch.uint8, device="cuda")
    P.esp_tree_attention(int(dt == "bf16"), b, n_rows, L, L + R, Hq, Hkv, h, 16, q, kc, vc, torch.from_numpy(_anc_words(vis)[None].view(np.int64)).cuda(),
                         torch.from_numpy(depth).cuda(), out, scratch, nb)
    assert P.esp_tree_attention_status(scratch) == 0
    assert torch.equal(out[:, :n_rows], ref[:, :n_rows])
    assert (out[:, n_rows:] == 7).all() and (flat[:offset] == 7).all() and (flat[offset + q.numel():] == 7).all()


@pytest.mark.parametrize("group", [1, 2, 4])
@pytest.mark.parametrize("L,dcap", [(0, 16), (9, 48)])
def test_tree_attention_infinite_values_in_the_tail(group, L, dcap):
    """A value that is not finite reaches the dimensions of the rows that give its key a weight, as one product with the whole weight
    does: infinite where the sum is, NaN only where opposite infinities or a NaN meet; a key whose weight underflows leaves nothing
    behind.  Keys: the one with the largest weight, an ordinary one, one of weight 0, one that only some rows see."""
    Hkv, h, b, n_rows = 2, 128, 1, 40
    Hq, inf = Hkv * group, float("inf")
    _, depth1, vis = _tree_block(n_rows, 0, dcap, 3)
    g = torch.Generator().manual_seed(group)
    q = torch.randn(b, R, Hq, h, generator=g)
    kc, vc = (torch.randn(b, Hkv, L + R, h, generator=g) for _ in range(2))
    q[..., 0] = 8.0
    kc[..., 0] = 0.0
    kc[:, :, L, 0] = 40.0                     # the root: weight 1 in every row
    far = L + 1
    kc[:, :, far, 0] = -400.0                 # its weight underflows
    vc[:, :, L, 0], vc[:, :, L, 1] = inf, -inf
    vc[:, :, far, 2], vc[:, :, far, 3] = inf, float("nan")
    vc[:, :, L + 2, 4], vc[:, :, L + 2, 5] = inf, float("nan")
    vc[:, :, L + 5, 0], vc[:, :, L + 5, 1] = -inf, -inf       # meets the root's +inf where it is visible
    q, kc, vc = q.bfloat16().cuda(), kc.bfloat16().cuda(), vc.bfloat16().cuda()
    depth = np.zeros((b, R), np.int32)
    depth[:, :n_rows] = depth1
    assert (np.maximum(L + depth1 - dcap, 0) // 16 * 16).max() == 0        # the tail does it all
    out = _run_attention(1, q, kc, vc, _anc_words(vis)[None], depth, n_rows, L, Hq, Hkv, h, dcap)[0, :n_rows].double().cpu()
    k, v = (t[0].repeat_interleave(group, 0)[:, :L + n_rows].double().cpu() for t in (kc, vc))
    s = torch.einsum("rhd,hcd->rhc", q[0, :n_rows].double().cpu(), k) / h ** 0.5
    hide = torch.zeros(n_rows, 1, L + n_rows, dtype=torch.bool)
    hide[:, 0, L:] = torch.from_numpy(vis == 0)
    s = s.masked_fill(hide, -inf)
    p = torch.exp(s - s.max(-1, keepdim=True).values)
    p[p < 2.0 ** -140] = 0.0
    assert (p[..., far] == 0).all()
    terms = torch.where(p[..., None] > 0, p[..., None] * v[None], torch.zeros(()).double())
    ref = terms.sum(2) / p.sum(-1, keepdim=True)
    assert torch.equal(torch.isnan(out), torch.isnan(ref)) and torch.equal(torch.isinf(out), torch.isinf(ref))
    assert torch.isinf(ref[..., :2]).any() and torch.isnan(ref[..., 0]).any() and torch.isfinite(ref[:, :, 2:4]).all()
    odd = torch.isinf(ref)
    assert torch.equal(out[odd], ref[odd])
    fin = torch.isfinite(ref)
    assert (out[fin] - ref[fin]).abs().max() <= 2.0 ** -8 * float(ref[fin].abs().max())


@pytest.mark.parametrize("odd", [False, True])
@pytest.mark.parametrize("L", [33, 301, 1111])
@pytest.mark.parametrize("dt,h", [("fp32", 32), ("fp32", 64), ("fp32", 128), ("bf16", 32), ("bf16", 64)])
def test_cuda_core_attention_has_the_same_bits_in_launches_of_every_size(dt, h, L, odd):
    """The CUDA-core kernel over the cache takes one or four pairs to a warp and several groups of warps or one by the size of the launch;
    the first rows of a block have the same bits whichever runs, and with a cache that starts on any element.  Splits that end in the
    middle of a chunk, with fewer chunks than groups, and full ones."""
    dtype = torch.float32 if dt == "fp32" else torch.bfloat16
    Hq, Hkv, cap = 32, 8, L + R
    g = torch.Generator().manual_seed(h + L)
    q = torch.randn(1, R, Hq, h, generator=g).to(dtype).cuda()
    kc, vc = (torch.randn(1, Hkv, cap, h, generator=g).to(dtype).cuda() for _ in range(2))
    if odd:
        kc, vc = (torch.cat([t.new_zeros(1), t.flatten()])[1:].view_as(t) for t in (kc, vc))
        assert kc.data_ptr() % 16 == kc.element_size()
    _, depth1, vis = _tree_block(R, 0, 12, 5)
    outs = [_run_attention(int(dt == "bf16"), q, kc, vc, _anc_words(vis)[None], depth1[None], n, L, Hq, Hkv, h)[0] for n in (1, 5, 16, 44, R)]
    for n, o in zip((1, 5, 16, 44), outs):
        assert torch.equal(o[:n], outs[-1][:n])
    s = torch.einsum("rhd,hcd->rhc", q[0].double(), kc[0].repeat_interleave(4, 0).double()) / h ** 0.5
    hide = torch.zeros(R, 1, cap, dtype=torch.bool)
    hide[:, 0, L:] = torch.from_numpy(vis == 0)
    ref = torch.einsum("rhc,hcd->rhd", s.masked_fill_(hide.cuda(), -float("inf")).softmax(-1), vc[0].repeat_interleave(4, 0).double())
    # (fp32: sums of up to 1239 terms; bf16: the result's own rounding)
    assert (outs[-1].double() - ref).abs().max() <= (1e-5 if dt == "fp32" else 2.0 ** -8) * float(ref.abs().max())


@pytest.mark.parametrize("group,n_rows,L,dcap", [(1, 33, 5, 16), (2, 9, 0, 16), (4, 68, 15, 16), (8, 41, 16, 32), (16, 7, 40, 48), (4, 128, 3, 128)])
def test_tree_attention_tail_weights_keep_their_24_bits(group, n_rows, L, dcap):
    """Three keys have weight, and their values nearly cancel in a dimension of each (row, head): what is left is far below the result's
    bf16 rounding of any one product, so a weight that lost bits shows.  Scores are single products (exact), so a weight's error is
    that of its scaled exponent (below 4, 2^-22) and of the exponential: 2^-21 of sum(p |v|), twice that allowed beside the result's own
    rounding.  Weights of 16 bits, and of 8, must fail the same bound."""
    Hkv, h = 2, 128
    Hq, cap = Hkv * group, L + R
    parents = np.minimum(np.arange(n_rows) - 1, 2)                 # a trunk of three nodes, the others behind it
    vis = np.zeros((n_rows, n_rows), np.uint8)
    depth = np.zeros((1, R), np.int32)
    for r in range(n_rows):
        vis[r, r] = 1
        if r:
            vis[r] |= vis[parents[r]]
            depth[0, r] = depth[0, parents[r]] + 1
    rng = np.random.default_rng(group * 1000 + n_rows)

    def bf(x):
        return torch.from_numpy(np.asarray(x, np.float32)).bfloat16().double().numpy()

    c = bf(rng.uniform(1, 4, (n_rows, Hq)))                        # queries and keys: one dimension each
    key = np.full((Hkv, L + n_rows), -2048.0)                      # weight 0
    key[:, L:L + 3] = bf([[0.0, -2.7, -5.2], [-4.1, 0.0, -1.9]])
    head_kv = np.repeat(np.arange(Hkv), group)
    s = c[:, :, None] * key[head_kv][None] / h ** 0.5
    s = np.where(np.concatenate([np.ones((n_rows, L)), vis], 1)[:, None] > 0, s, -np.inf)
    p = np.exp(s - s.max(-1, keepdims=True))
    p[p < 2.0 ** -149] = 0.0
    assert np.array_equal((p[2:] > 0).sum(-1), np.full((n_rows - 2, Hq), 3))
    # dimension d of a KV head: values of the trunk that cancel for one (row, head)
    v = np.zeros((Hkv, L + n_rows, h))
    v[:, L] = bf(rng.uniform(500, 2000, (Hkv, h)))
    for kv in range(Hkv):
        for d in range(h):
            w = p[2 + d % (n_rows - 2), kv * group + d % group, L:L + 3]
            v[kv, L + 1, d] = bf(-v[kv, L, d] * w[0] / w[1])
            v[kv, L + 2, d] = bf(-(v[kv, L, d] * w[0] + v[kv, L + 1, d] * w[1]) / w[2])

    def out_of(pp):
        return np.einsum("rhc,hcd->rhd", pp, v[head_kv]) / p.sum(-1)[..., None]

    ref = out_of(p)
    tol = 2.0 ** -8 * np.abs(ref) + 2.0 ** -20 * np.einsum("rhc,hcd->rhd", p, np.abs(v[head_kv])) / p.sum(-1)[..., None]
    hi = bf(p)
    mid = bf(p - hi)
    assert (np.abs(out_of(hi) - ref) > tol).any() and (np.abs(out_of(hi + mid) - ref) > tol).any()
    assert (np.abs(out_of(hi + mid + bf(p - hi - mid)) - ref) <= tol / 4).all()
    q = torch.zeros(1, R, Hq, h)
    q[0, :n_rows, :, 7] = torch.from_numpy(c)
    kc, vc = torch.zeros(1, Hkv, cap, h), torch.zeros(1, Hkv, cap, h)
    kc[0, :, :L + n_rows, 7] = torch.from_numpy(key)
    vc[0, :, :L + n_rows] = torch.from_numpy(v)
    out = _run_attention(1, q.bfloat16().cuda(), kc.bfloat16().cuda(), vc.bfloat16().cuda(), _anc_words(vis)[None], depth, n_rows, L, Hq, Hkv, h, dcap)
    assert (np.abs(out[0, :n_rows].double().cpu().numpy() - ref) <= tol).all()
