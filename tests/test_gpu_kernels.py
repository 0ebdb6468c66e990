"""Kernel-level parity through the C ABI: the tcgen05 / fp32 linear and the paged
tree attention against the fp64 oracle's definitions, at ragged sizes."""
import numpy as np
import pytest
import torch

import paper_2402_15758_gb300 as pkg
from oracle import chimera_oracle as co

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2402_15758_gb300 import build
    build.build()
    pkg.load()


def _rel_rows(a, ref):
    return float(np.max(np.abs(a - ref) / np.maximum(np.max(np.abs(ref), axis=-1, keepdims=True), 1e-30)))


LINEAR_SHAPES = [(1, 128, 64), (5, 300, 72), (16, 256, 512), (17, 1000, 520), (64, 1536, 1024),
                 (100, 384, 1024), (256, 512, 2048), (300, 256, 256), (64, 4096, 4096), (8, 32000, 512),
                 (1, 4096, 12288)]


@pytest.mark.parametrize("M,N,K", LINEAR_SHAPES)
def test_linear_bf16_fp32_out(M, N, K):
    g = torch.Generator().manual_seed(M * 7 + N + K)
    X = torch.randn(M, K, generator=g).to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    Y = torch.full((M, N), float("nan"), dtype=torch.float32, device="cuda")
    pkg.op_linear(X.cuda(), W.cuda(), Y, epi=0, out_f32=True)
    torch.cuda.synchronize()
    ref = X.double().numpy() @ W.double().numpy().T
    assert _rel_rows(Y.cpu().numpy(), ref) <= 1e-4


@pytest.mark.parametrize("M,N,K", [(3, 640, 192), (64, 1408, 512), (33, 256, 1408)])
def test_linear_bf16_epilogues(M, N, K):
    g = torch.Generator().manual_seed(99 + M)
    X = torch.randn(M, K, generator=g).to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    ref = X.double().numpy() @ W.double().numpy().T
    # bf16 store: one rounding of the fp32 accumulator
    Y = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda")
    pkg.op_linear(X.cuda(), W.cuda(), Y, epi=0)
    assert _rel_rows(Y.float().cpu().numpy(), ref) <= 8e-3
    # SiLU
    pkg.op_linear(X.cuda(), W.cuda(), Y, epi=1)
    assert _rel_rows(Y.float().cpu().numpy(), co.silu(ref)) <= 8e-3
    # residual add into fp32
    R0 = torch.randn(M, N, generator=g)
    R = R0.clone().cuda()
    pkg.op_linear(X.cuda(), W.cuda(), R, epi=2)
    torch.cuda.synchronize()
    assert _rel_rows(R.cpu().numpy(), R0.double().numpy() + ref) <= 1e-5


@pytest.mark.parametrize("M,N,K", [(1, 256, 512), (64, 1536, 1024), (100, 384, 4096)])
def test_linear_bf16_split_operand(M, N, K):
    # X = hi + lo (two bf16 halves): W (hi + lo) reproduces the fp32 activation
    g = torch.Generator().manual_seed(3 * M + K)
    X32 = torch.randn(M, K, generator=g)
    hi = X32.to(torch.bfloat16)
    lo = (X32 - hi.float()).to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g) * 0.05).to(torch.bfloat16)
    Y = torch.zeros(M, N, dtype=torch.float32, device="cuda")
    pkg.op_linear(hi.cuda(), W.cuda(), Y, epi=0, out_f32=True, X_lo=lo.cuda())
    torch.cuda.synchronize()
    ref = X32.double().numpy() @ W.double().numpy().T
    assert _rel_rows(Y.cpu().numpy(), ref) <= 2e-5
    # without the lo half the error is the bf16 rounding of X
    pkg.op_linear(hi.cuda(), W.cuda(), Y, epi=0, out_f32=True)
    torch.cuda.synchronize()
    assert _rel_rows(Y.cpu().numpy(), ref) > 1e-4


# stored outputs: two whole tiles per CTA (160 tiles), one, two to eight parts of a tile; chains
# of one and of two stages, token tiles of 16, 32, 48 and 64 columns
@pytest.mark.parametrize("M,N,K", [(5, 20480, 520), (1, 300, 1400), (24, 2050, 4104), (40, 12288, 520), (40, 300, 9000),
                                   (64, 1000, 4096), (3, 4096, 11008)])
@pytest.mark.parametrize("epi,out_f32", [(0, True), (1, True), (1, False)])
def test_linear_stored_parts(M, N, K, epi, out_f32):
    g = torch.Generator().manual_seed(M + N + K)
    X32 = torch.randn(M, K, generator=g)
    hi = X32.to(torch.bfloat16)
    lo = (X32 - hi.float()).to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g) * 0.02).to(torch.bfloat16)
    ref = ((hi.cuda().double() + lo.cuda().double()) @ W.cuda().double().T).cpu().numpy()
    got = []
    for _ in range(2):
        Y = torch.full((M, N), float("nan"), dtype=torch.float32 if out_f32 else torch.bfloat16, device="cuda")
        pkg.op_linear(hi.cuda(), W.cuda(), Y, epi=epi, out_f32=out_f32, X_lo=lo.cuda())
        pkg.op_sync()
        got.append(Y.float().cpu().numpy())
    # chains of at most 16 truncated fp32 steps (2^-23 each, partly cancelling), or one rounding to bf16
    assert _rel_rows(got[1], co.silu(ref) if epi else ref) <= (2e-6 if out_f32 else 8e-3)
    assert np.array_equal(got[0], got[1])


# the CTA-pair kernel: split activations of more than 64 rows with at least 1000 stages x
# tokens per pair.  Ragged token tiles (1 of 80 and of 112 rows, 2 of 80, 3 of 96, 9 in two
# rounds of 5), an odd number of 128-feature halves, columns that are no multiple of 4, a
# ragged last K block
@pytest.mark.parametrize("M,N,K", [(65, 8200, 4096), (100, 6001, 4104), (129, 4224, 4096), (256, 2050, 8000), (257, 1000, 12296), (640, 1536, 5000),
                                   (1100, 1024, 3400)])
@pytest.mark.parametrize("epi,out_f32", [(0, True), (1, False), (2, True)])
def test_linear_pair_kernel(M, N, K, epi, out_f32):
    g = torch.Generator().manual_seed(M + N + K)
    X32 = torch.randn(M, K, generator=g)
    hi = X32.to(torch.bfloat16)
    lo = (X32 - hi.float()).to(torch.bfloat16)
    W = (torch.randn(N, K, generator=g) * 0.02).to(torch.bfloat16)
    Y0 = torch.randn(M, N, generator=g).to(torch.float32 if out_f32 else torch.bfloat16)
    ref = (hi.cuda().double() + lo.cuda().double()) @ W.cuda().double().T
    ref = {0: ref, 1: ref * torch.sigmoid(ref), 2: Y0.cuda().double() + ref}[epi].cpu().numpy()
    got = []
    for _ in range(2):
        Y = Y0.cuda()
        pkg.op_linear(hi.cuda(), W.cuda(), Y, epi=epi, out_f32=out_f32, X_lo=lo.cuda())
        pkg.op_sync()
        got.append(Y.float().cpu().numpy())
    # chains of at most 128 truncated fp32 steps (2^-23 each, partly cancelling), or one rounding to bf16
    assert _rel_rows(got[1], ref) <= (1.6e-5 if out_f32 else 8e-3)
    if epi != 2:  # stored outputs are summed in a fixed order
        assert np.array_equal(got[0], got[1])


# W written by the launch just before on the stream: 16 rows and 64 rows (linear_tc.cu), 100 rows
# (the CTA-pair kernel), and the allocation-free entry point
@pytest.mark.parametrize("M,split,noalloc", [(16, False, False), (64, True, False), (100, True, False), (16, True, True)])
def test_linear_weights_from_the_launch_before(M, split, noalloc):
    g = torch.Generator().manual_seed(M)
    D = 4096
    A = torch.randn(D, 2048, generator=g).to(torch.bfloat16).cuda()
    B = (torch.randn(D, 2048, generator=g) * 0.02).to(torch.bfloat16).cuda()
    X32 = torch.randn(M, D, generator=g)
    hi = X32.to(torch.bfloat16).cuda()
    lo = (X32 - hi.cpu().float()).to(torch.bfloat16).cuda() if split else None
    op = pkg.op_linear_noalloc if noalloc else pkg.op_linear
    for _ in range(3):
        W = torch.full((D, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        Y = torch.empty(M, D, device="cuda")
        pkg.op_linear(A, B, W, epi=0)
        op(hi, W, Y, epi=0, out_f32=True, X_lo=lo)
        pkg.op_sync()
        ref = (hi.double() + (lo.double() if split else 0.0)) @ W.double().T
        # fp32 sums of 4096 products, truncated at most every 16 K: 256 * 2^-23 at most
        assert _rel_rows(Y.cpu().numpy(), ref.cpu().numpy()) <= 3e-5


# launches that overlap: tiles cut between CTAs (fp32 output, summed in a fixed order) and a
# split fp32 attention, on more streams than have a workspace of their own, beside a graph
# captured on a stream without an earlier call
@pytest.mark.parametrize("n_streams", [2, 11])
def test_ops_on_several_streams(n_streams):
    g = torch.Generator().manual_seed(8)
    X = torch.randn(5, 9000, generator=g).to(torch.bfloat16).cuda()
    W = (torch.randn(300, 9000, generator=g) * 0.02).to(torch.bfloat16).cuda()
    kv = torch.randn(70, 2, 2, 16, 64, generator=g).cuda()
    q = torch.randn(1, 128, generator=g).cuda()
    pages = torch.arange(70, dtype=torch.int32, device="cuda").view(1, 70)
    n_ctx = torch.tensor([1100], dtype=torch.int32, device="cuda")
    anc = torch.ones(1, dtype=torch.int64, device="cuda")

    def call(y, o, stream):
        pkg.op_linear(X, W, y, epi=0, out_f32=True, stream=stream)
        pkg.op_attention(q, kv, pages, n_ctx, anc, o, 1, 0, 1, 1, 2, 64, splits=4, stream=stream)

    outs = [(torch.zeros(5, 300, device="cuda"), torch.zeros(1, 128, device="cuda")) for _ in range(n_streams + 2)]
    call(*outs[0], None)
    graph = torch.cuda.CUDAGraph()
    streams = [torch.cuda.Stream() for _ in range(n_streams)]
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        call(*outs[1], torch.cuda.current_stream())
        call(*outs[2], streams[0])  # an eager call beside the capture
    ref = tuple(t.clone() for t in outs[0])
    assert _rel_rows(ref[0].cpu().numpy(), (X.double() @ W.double().T).cpu().numpy()) <= 2e-6
    torch.cuda.synchronize()
    for rep in range(100):
        for st, out in zip(streams, outs[2:]):
            call(*out, st)
        graph.replay()
        if rep % 10 == 9:
            torch.cuda.synchronize()
            for y, o in outs:
                assert torch.equal(y, ref[0]) and torch.equal(o, ref[1])
                if rep < 90:
                    y.zero_(), o.zero_()
            call(*outs[0], None)
            torch.cuda.synchronize()
    pkg.op_sync()


def test_linear_deterministic():
    g = torch.Generator().manual_seed(5)
    X = torch.randn(64, 4096, generator=g).to(torch.bfloat16).cuda()
    W = (torch.randn(4096, 4096, generator=g) * 0.02).to(torch.bfloat16).cuda()
    a = torch.zeros(64, 4096, device="cuda")
    b = torch.zeros(64, 4096, device="cuda")
    pkg.op_linear(X, W, a, out_f32=True)
    pkg.op_linear(X, W, b, out_f32=True)
    torch.cuda.synchronize()
    assert torch.equal(a, b)


@pytest.mark.parametrize("M,N,K", [(1, 64, 8), (16, 1024, 768), (64, 688, 256)])
def test_linear_fp32(M, N, K):
    g = torch.Generator().manual_seed(N)
    X = torch.randn(M, K, generator=g)
    W = torch.randn(N, K, generator=g) * 0.05
    Y = torch.zeros(M, N, device="cuda")
    pkg.op_linear(X.cuda(), W.cuda(), Y, epi=0)
    torch.cuda.synchronize()
    assert _rel_rows(Y.cpu().numpy(), X.double().numpy() @ W.double().numpy().T) <= 1e-5


# one row / few rows / full and ragged 16-row tiles; K below, at and past the 512-wide chunk,
# with and without 16-byte rows; enough features that a warp takes two
@pytest.mark.parametrize("M,N,K", [(1, 7, 1), (1, 768, 359), (3, 130, 512), (5, 33, 516), (16, 256, 688),
                                   (17, 1001, 513), (64, 1300, 1028), (33, 2048, 30)])
@pytest.mark.parametrize("epi", [0, 1, 2])
def test_linear_fp32_edges(M, N, K, epi):
    g = torch.Generator().manual_seed(M * N + K)
    X = torch.randn(M, K, generator=g)
    W = torch.randn(N, K, generator=g) * 0.05
    Y0 = torch.randn(M, N, generator=g)
    Y = Y0.cuda()
    pkg.op_linear(X.cuda(), W.cuda(), Y, epi=epi)
    torch.cuda.synchronize()
    ref = X.double().numpy() @ W.double().numpy().T
    ref = {0: ref, 1: co.silu(ref), 2: Y0.double().numpy() + ref}[epi]
    # fp32 sums of K terms in at most K / 32 + 5 roundings of 2^-24 each, against a row maximum of
    # at least the sums' own size: 37 * 6e-8 = 2.2e-6 at K = 1028
    assert _rel_rows(Y.cpu().numpy(), ref) <= 1e-5


def _random_tree_anc(n, rng):
    parent = [-1] + [int(rng.integers(0, j)) for j in range(1, n)]
    anc = []
    for i in range(n):
        m, j = 0, i
        while j >= 0:
            m |= 1 << j
            j = parent[j]
        anc.append(m)
    return anc


ATT_CASES = [
    # B, H, hd, n_ctx per seq, n_local, nq, q_local0, splits
    (1, 4, 64, [77], 16, 16, 0, 1),
    (1, 4, 64, [77], 16, 16, 0, 5),
    (2, 3, 128, [0, 300], 64, 64, 0, 7),
    (3, 2, 128, [16, 1, 129], 5, 1, 4, 3),     # draft-style: one query, local rows 0..4
    (1, 2, 128, [1000], 64, 64, 0, 8),
    (2, 3, 128, [700, 3], 64, 64, 0, 4),     # a split whose key range is empty for b=1
    (1, 2, 128, [0], 3, 3, 0, 1),            # one tile: the odd-tile stream has none
    (2, 2, 128, [100, 63], 17, 17, 0, 1),    # two tiles (and a row in a second warp), 80 keys
    (1, 2, 128, [1500], 33, 33, 0, 2),       # many tiles per stream, row counts no multiple of 16
    (2, 40, 128, [2100, 330], 5, 1, 4, 2),   # one query, tiles around the ring, more CTAs than SMs
]


@pytest.mark.parametrize("dtype", ["fp32", "bf16", "bf16_split"])
@pytest.mark.parametrize("case", range(len(ATT_CASES)))
def test_attention_tree_masked_paged(dtype, case):
    B, H, hd, nctx, n_local, nq, q0, splits = ATT_CASES[case]
    rng = np.random.default_rng(case)
    max_pages = (max(nctx) + n_local + 15) // 16 + 1
    n_blocks = B * max_pages + 3
    perm = rng.permutation(n_blocks)[: B * max_pages].reshape(B, max_pages).astype(np.int32)
    assert perm.max() < n_blocks
    kv32 = torch.randn(n_blocks, H, 2, 16, hd, generator=torch.Generator().manual_seed(case))
    if dtype == "fp32":
        pool, Kref = kv32, kv32.double()
        odt = torch.float32
    elif dtype == "bf16":
        pool = kv32.to(torch.bfloat16)
        Kref = pool.double()
        odt = torch.bfloat16
    else:  # K_hi, K_lo, V_hi, V_lo planes; the reference uses the fp32 values
        hi = kv32.to(torch.bfloat16)
        lo = (kv32 - hi.float()).to(torch.bfloat16)
        pool = torch.stack([hi[:, :, 0], lo[:, :, 0], hi[:, :, 1], lo[:, :, 1]], dim=2).contiguous()
        Kref = kv32.double()
        odt = torch.bfloat16
    q = torch.randn(B * nq, H * hd, generator=torch.Generator().manual_seed(100 + case))
    anc = _random_tree_anc(n_local, rng) if q0 == 0 else [(1 << (i + 1)) - 1 for i in range(n_local)]
    out = torch.zeros(B * nq, H * hd, dtype=odt, device="cuda")
    out_lo = torch.zeros_like(out) if odt == torch.bfloat16 else None
    anc_t = torch.tensor(np.array(anc, dtype=np.uint64).view(np.int64), device="cuda")
    pkg.op_attention(q.cuda(), pool.cuda(), torch.tensor(perm, device="cuda"),
                     torch.tensor(nctx, dtype=torch.int32, device="cuda"), anc_t, out, nq=nq, q_local0=q0,
                     n_local=n_local, q_rows=nq, n_heads=H, head_dim=hd, splits=splits, out_lo=out_lo)
    torch.cuda.synchronize()
    got = out.float().cpu().numpy().reshape(B, nq, H, hd)
    if out_lo is not None:
        got = got + out_lo.float().cpu().numpy().reshape(B, nq, H, hd)
    P = Kref.numpy()
    Q = q.double().numpy().reshape(B, nq, H, hd)

    def kv(b, slot):
        blk = perm[b, slot // 16]
        return P[blk, :, 0, slot % 16], P[blk, :, 1, slot % 16]

    # fp32 path: fp32 arithmetic; tensor-core path (head_dim 128, bf16 model): bf16
    # split products of the fp32 query / probabilities (and of the split K/V planes),
    # which drop the lo*lo terms (~2^-16 relative)
    tol = 1e-5 if (dtype == "fp32" or hd != 128) else 5e-5
    for b in range(B):
        for i in range(nq):
            m = anc[q0 + i]
            slots = list(range(nctx[b])) + [nctx[b] + j for j in range(n_local) if (m >> j) & 1]
            Ks = np.array([kv(b, s)[0] for s in slots])
            Vs = np.array([kv(b, s)[1] for s in slots])
            ref = co.attend(Q[b, i], Ks, Vs)
            err = np.max(np.abs(got[b, i] - ref)) / np.max(np.abs(ref))
            assert err <= tol, (b, i, err)


# the SIMT kernel (fp32 models, head_dim 64): one query and query groups of 16 (8 at head_dim
# 128), contexts below, at and past a 64-key pass and a 256-key split, planes of both types,
# a pool that is not aligned for vectors
@pytest.mark.parametrize("dtype,hd", [("fp32", 64), ("fp32", 128), ("bf16", 64), ("bf16_split", 64)])
@pytest.mark.parametrize("nctx,nq,splits", [([0], 1, 1), ([64, 63], 1, 16), ([700, 5], 1, 3), ([130], 9, 2), ([300, 0], 64, 16)])
@pytest.mark.parametrize("offset", [0, 1])
def test_attention_simt(dtype, hd, nctx, nq, splits, offset):
    _attention_simt(dtype, hd, nctx, nq, splits, offset)


# groups of 8 queries, partly filled and full
@pytest.mark.parametrize("dtype,hd", [("fp32", 64), ("bf16", 64), ("bf16_split", 64)])
@pytest.mark.parametrize("nctx,nq,splits", [([0, 130], 2, 1), ([700, 5], 7, 3), ([300], 8, 16)])
@pytest.mark.parametrize("offset", [0, 1])
def test_attention_simt_few_queries(dtype, hd, nctx, nq, splits, offset):
    _attention_simt(dtype, hd, nctx, nq, splits, offset)


def _attention_simt(dtype, hd, nctx, nq, splits, offset):
    B, H, n_local = len(nctx), 3, max(nq, 2)
    rng = np.random.default_rng(nq + splits)
    max_pages = (max(nctx) + n_local + 15) // 16
    perm = rng.permutation(B * max_pages).reshape(B, max_pages).astype(np.int32)
    kv = torch.randn(B * max_pages, H, 2, 16, hd, generator=torch.Generator().manual_seed(nq))
    hi = kv.to(torch.bfloat16)
    pool = kv if dtype == "fp32" else hi
    ref_kv = pool.double().numpy()
    if dtype == "bf16_split":
        lo = (kv - hi.float()).to(torch.bfloat16)
        pool = torch.stack([hi[:, :, 0], lo[:, :, 0], hi[:, :, 1], lo[:, :, 1]], dim=2)
        ref_kv = np.stack([(hi + 0).double().numpy()[:, :, i] + lo.double().numpy()[:, :, i] for i in (0, 1)], 2)
    flat = torch.zeros(pool.numel() + 4, dtype=pool.dtype, device="cuda")
    flat[offset:offset + pool.numel()] = pool.reshape(-1).cuda()
    dev = flat[offset:offset + pool.numel()].view(pool.shape)
    q = torch.randn(B * nq, H * hd, generator=torch.Generator().manual_seed(9))
    q0 = n_local - nq  # the queries are the last local rows of a causal chain
    anc = np.array([(1 << (i + 1)) - 1 for i in range(n_local)], dtype=np.uint64)
    out = torch.zeros(B * nq, H * hd, dtype=torch.float32 if dtype == "fp32" else torch.bfloat16, device="cuda")
    out_lo = None if dtype == "fp32" else torch.zeros_like(out)
    for _ in range(2):  # the split counters are back at zero after a launch
        pkg.op_attention(q.cuda(), dev, torch.tensor(perm, device="cuda"),
                         torch.tensor(nctx, dtype=torch.int32, device="cuda"),
                         torch.tensor(anc.view(np.int64), device="cuda"), out, nq=nq, q_local0=q0, n_local=n_local,
                         q_rows=nq, n_heads=H, head_dim=hd, splits=splits, out_lo=out_lo)
        pkg.op_sync()
    got = out.double() + (0 if out_lo is None else out_lo.double())
    got = got.cpu().numpy().reshape(B, nq, H, hd)
    Q = q.double().numpy().reshape(B, nq, H, hd)
    for b in range(B):
        for i in range(nq):
            slots = range(nctx[b] + q0 + i + 1)
            K, V = (np.stack([ref_kv[perm[b, t // 16], :, j, t % 16] for t in slots]) for j in (0, 1))
            ref = co.attend(Q[b, i], K, V)
            # fp32 sums; a bf16 output is a hi + lo pair (2^-17)
            assert np.max(np.abs(got[b, i] - ref)) / np.max(np.abs(ref)) <= (1e-5 if dtype == "fp32" else 2e-5), (b, i)


@pytest.mark.parametrize("jump", [40.0, 150.0])
@pytest.mark.parametrize("splits", [1, 2])
def test_attention_rescale_after_one_sided_tile(jump, splits):
    """Online softmax with a far move of the running maximum. Every query row sees the 20
    context keys, local row 0 and itself, so row 50's first tile has visible keys in its
    first key half only; its own key (second tile) scores `jump` nats above zero, which
    moves the maximum by far more than the lazy-rescale threshold (the correction is
    about 2^-53 at 40 nats and underflows to 0 at 150). All 128 output columns of the
    row must then be rescaled, whichever key half saw keys before."""
    import math
    H, hd, nctx, n_local, nq = 2, 128, 20, 64, 64
    max_pages = (nctx + n_local + 15) // 16 + 1
    perm = np.arange(max_pages, dtype=np.int32).reshape(1, max_pages)
    kv32 = torch.randn(max_pages, H, 2, 16, hd, generator=torch.Generator().manual_seed(7))
    q = torch.randn(nq, H * hd, generator=torch.Generator().manual_seed(8))
    anc = [1 | (1 << i) for i in range(n_local)]
    r, slot = 50, nctx + 50
    for h in range(H):
        qv = q[r, h * hd:(h + 1) * hd]
        kv32[slot // 16, h, 0, slot % 16] = qv * (jump * math.sqrt(hd) / float(qv @ qv))
    hi = kv32.to(torch.bfloat16)
    lo = (kv32 - hi.float()).to(torch.bfloat16)
    pool = torch.stack([hi[:, :, 0], lo[:, :, 0], hi[:, :, 1], lo[:, :, 1]], dim=2).contiguous()
    out = torch.zeros(nq, H * hd, dtype=torch.bfloat16, device="cuda")
    out_lo = torch.zeros_like(out)
    anc_t = torch.tensor(np.array(anc, dtype=np.uint64).view(np.int64), device="cuda")
    pkg.op_attention(q.cuda(), pool.cuda(), torch.tensor(perm, device="cuda"),
                     torch.tensor([nctx], dtype=torch.int32, device="cuda"), anc_t, out, nq=nq, q_local0=0,
                     n_local=n_local, q_rows=nq, n_heads=H, head_dim=hd, splits=splits, out_lo=out_lo)
    torch.cuda.synchronize()
    got = (out.float() + out_lo.float()).cpu().numpy().reshape(nq, H, hd)
    P = kv32.double().numpy()
    Q = q.double().numpy().reshape(nq, H, hd)
    for i in range(nq):
        slots = list(range(nctx)) + [nctx + j for j in range(n_local) if (anc[i] >> j) & 1]
        Ks = np.array([P[s // 16, :, 0, s % 16] for s in slots])
        Vs = np.array([P[s // 16, :, 1, s % 16] for s in slots])
        ref = co.attend(Q[i], Ks, Vs)
        err = np.max(np.abs(got[i] - ref)) / np.max(np.abs(ref))
        assert err <= 5e-5, (i, err)
