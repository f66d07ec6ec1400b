"""Kernel-level parity: each CUDA kernel, called through the C ABI, against
the CPU oracle on the same seeded inputs."""
import threading

import numpy as np
import pytest

import oracle as O
from oracle import diffusion_head as HO
from oracle import fp8
import synth
from paper_2503_12450_gb300 import lazymar as lm
from _gpu import DT, TOL, dev, dev_int, empty, host, max_rel, sync, torch_cuda

pytestmark = pytest.mark.gpu


# --------------------------------------------------------------------------
# Selection (Eq. 8): indices bit-exact
# --------------------------------------------------------------------------

@pytest.mark.parametrize("rows,T,D,N,dtype", [
    (2, 80, 256, 20, "fp32"),      # tiny
    (64, 320, 768, 50, "bf16"),    # MAR-B
    (16, 320, 1024, 32, "bf16"),   # MAR-L, 10 %
    (8, 320, 1280, 50, "bf16"),    # MAR-H
    (32, 1088, 1024, 272, "bf16"),  # high resolution, 25 %
    (3, 320, 768, 0, "bf16"),
    (3, 320, 768, 320, "bf16"),
    (1, 1, 8, 1, "fp32"),
    (5, 100, 16, 37, "bf16"),
    (4, 513, 64, 129, "fp32"),     # T spans two scan chunks
])
def test_select_tokens_bit_exact(rows, T, D, N, dtype):
    torch = torch_cuda()
    cur, ref = synth.similarity_inputs(rows, T, D, seed=rows * 1000 + T, dtype=dtype)
    g_cur, g_ref = dev(cur, dtype), dev(ref, dtype)
    idx = torch.full((rows, max(N, 1)), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT[dtype], g_cur, g_ref, rows, T, D, N, idx)
    sync()
    got = idx.cpu().numpy()[:, :N]
    for r in range(rows):
        expect = O.select_compute(O.cosine_similarity(cur[r], ref[r]), N)
        assert got[r].tolist() == expect.tolist(), "row %d" % r
    # the reference now holds the current values, bit for bit
    assert torch.equal(g_ref, g_cur)


@pytest.mark.parametrize("rule", [lm.LAZYMAR_SELECT_LEAST_SIMILAR, lm.LAZYMAR_SELECT_MOST_SIMILAR,
                                  lm.LAZYMAR_SELECT_RANDOM])
@pytest.mark.parametrize("with_prio", [False, True])
@pytest.mark.parametrize("rows,T,D,N,dtype", [
    (64, 320, 768, 50, "bf16"),    # MAR-B
    (2, 80, 256, 20, "fp32"),      # tiny
    (5, 100, 16, 37, "bf16"),
    (3, 320, 768, 320, "bf16"),    # N = T
    (4, 513, 64, 129, "fp32"),
])
def test_select_rules_bit_exact(rule, with_prio, rows, T, D, N, dtype):
    """Selection strategies of Table 3 (V, IV, III) with and without priority
    classes (observation-based / type strategies) against the oracle on the
    same buffers: indices bit-exact, reference updated."""
    torch = torch_cuda()
    cur, ref = synth.similarity_inputs(rows, T, D, seed=rows * 1000 + T + rule, dtype=dtype)
    rng = np.random.default_rng(rows + T + 7 * rule + with_prio)
    prio = rng.integers(0, 3, size=(rows, T)).astype(np.uint8) if with_prio else None
    keys = rng.integers(0, 1 << 32, size=(rows, T), dtype=np.uint64).astype(np.uint32)
    keys[:, 1::7] = keys[:, 0:1]  # repeated keys: the index decides
    g_cur, g_ref = dev(cur, dtype), dev(ref, dtype)
    g_prio = torch.from_numpy(prio).cuda() if with_prio else None
    g_keys = torch.from_numpy(keys.view(np.int32)).cuda()
    idx = torch.full((rows, max(N, 1)), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens_ex(DT[dtype], g_cur, g_ref, rows, T, D, N, rule, g_prio, g_keys, idx)
    sync()
    got = idx.cpu().numpy()[:, :N]
    for r in range(rows):
        expect = O.select_by_rule(O.cosine_similarity(cur[r], ref[r]), N, rule,
                                  None if prio is None else prio[r], keys[r])
        assert got[r].tolist() == expect.tolist(), "row %d" % r
    assert torch.equal(g_ref, g_cur)


def _selection_edge_inputs(T, D, seed):
    """bf16 rows that exercise both similarity paths of the kernel.

    row 0: every element scaled by 2^u, u uniform in [-60, 60] (exponent span
           far beyond the exact integer sums: the fp64 path);
    row 1: per token either a narrow ([-4, 4]) or a wide ([-30, 30]) span;
    row 2: subnormal and near-subnormal values, zero tokens, cur = -ref;
    row 3: Inf / NaN elements in a few tokens (S is NaN, ranked as -inf).
    """
    rng = np.random.Generator(np.random.PCG64(seed))
    ref = rng.standard_normal((4, T, D)).astype(np.float32)
    cur = ref * (1 + 0.05 * rng.standard_normal((4, T, D))).astype(np.float32)
    big = rng.random((4, T)) < 0.2
    cur[big] = rng.standard_normal((int(big.sum()), D)).astype(np.float32)
    u = rng.integers(-60, 61, size=(T, D))
    cur[0] *= np.exp2(u).astype(np.float32)
    ref[0] *= np.exp2(u).astype(np.float32)
    span = np.where(rng.random(T) < 0.5, 4, 30)[:, None]
    u = rng.integers(-span, span + 1, size=(T, D))
    cur[1] *= np.exp2(u).astype(np.float32)
    ref[1] *= np.exp2(u).astype(np.float32)
    scale = np.where(rng.random((T, 1)) < 0.5, 2.0 ** -130, 2.0 ** -120).astype(np.float32)
    cur[2] *= scale
    ref[2] *= scale
    cur[2, :5] = 0.0
    ref[2, 3:8] = 0.0
    cur[2, 10:20] = -ref[2, 10:20]
    for t, v in [(0, np.inf), (7, -np.inf), (11, np.nan)]:
        cur[3, t, t % D] = v
    ref[3, 20, 5] = np.inf
    ref[3, 21, 6] = np.nan
    return synth.round_bf16(cur), synth.round_bf16(ref)


@pytest.mark.parametrize("D", [768, 1280, 64])
def test_select_tokens_exponent_range_and_specials(D):
    """Selections agree with the oracle on data whose exponent spans, subnormals
    and Inf/NaN elements steer tokens through both the exact integer sums and
    the fp64 fallback. (Where the spans exceed what fp64 sums exactly, both
    sides round; the random data has no near-ties for that to reorder.)"""
    torch = torch_cuda()
    T, N = 200, 60
    cur, ref = _selection_edge_inputs(T, D, seed=D)
    g_cur, g_ref = dev(cur, "bf16"), dev(ref, "bf16")
    idx = torch.full((4, N), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT["bf16"], g_cur, g_ref, 4, T, D, N, idx)
    sync()
    got = idx.cpu().numpy()
    with np.errstate(invalid="ignore", over="ignore"):
        for r in range(4):
            expect = O.select_compute(O.cosine_similarity(cur[r], ref[r]), N)
            assert got[r].tolist() == expect.tolist(), "row %d" % r
    # bit patterns: the copied NaNs compare unequal as values
    assert torch.equal(g_ref.view(torch.int16), g_cur.view(torch.int16))


@pytest.mark.parametrize("D", [1288, 2048])
def test_select_tokens_wide_bf16_vectors(D):
    """bf16 wider than 1280: sums in triples of floats, and in fp64 where exponents
    or Inf/NaN ask for it."""
    test_select_tokens_exponent_range_and_specials(D)


@pytest.mark.parametrize("D,octaves", [(8, 22), (8, 23), (256, 19), (256, 20), (768, 18), (768, 19), (1280, 18),
                                       (1280, 19), (1288, 18)])
@pytest.mark.parametrize("rows,T", [(1, 9), (1, 333), (20, 333)])
def test_select_tokens_fixed_point_span(D, octaves, rows, T):
    """Exponent spans at the limit of the fixed-point sums and one octave
    beyond (D = 8, 256, 768, 1280: spans of 22, 19, 18 and 18 octaves; D = 1288
    takes the fp64 sums), with zeros, whole-vector powers of two down to the
    limit of the scaling, and a top value on either side of the span."""
    torch = torch_cuda()
    rng = np.random.default_rng(1000 * octaves + D + T + rows)
    ref = rng.uniform(1, 2, (rows, T, D)) * rng.choice([-1.0, 1.0], (rows, T, D))
    cur = ref * (1 + 0.3 * rng.standard_normal((rows, T, 1)) * rng.standard_normal((rows, T, D)))
    u = rng.integers(-octaves, 1, (rows, T, D))
    u[..., 0], u[..., 1] = 0, -octaves
    whole = rng.choice([-100, -20, 0, 30], (rows, T, 1))  # -100: below the fixed-point tier's exponents
    cur, ref = cur * np.exp2(u + whole), ref * np.exp2(u)
    cur[rng.random((rows, T, D)) < 0.05] = 0
    cur, ref = synth.round_bf16(cur.astype(np.float32)), synth.round_bf16(ref.astype(np.float32))
    g_cur, g_ref = dev(cur, "bf16"), dev(ref, "bf16")
    N = T // 3
    idx = torch.full((rows, N), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT["bf16"], g_cur, g_ref, rows, T, D, N, idx)
    sync()
    got = idx.cpu().numpy()
    for r in range(rows):
        assert got[r].tolist() == O.select_compute(O.cosine_similarity(cur[r], ref[r]), N).tolist(), "row %d" % r
    assert torch.equal(g_ref, g_cur)


@pytest.mark.parametrize("magnitude", [1.5, 1.75, 1.9921875, None])
@pytest.mark.parametrize("rows,T,D", [(2, 120, 256), (1, 97, 512), (2, 120, 768), (1, 97, 1024), (1, 97, 1280),
                                      (1, 97, 1272)])
def test_select_tokens_nearly_constant_magnitudes(rows, T, D, magnitude):
    """Vectors whose elements are all of (nearly) the largest magnitude: the
    fixed-point sums of 32 lanes come close to 2^68, in the norms, and in dot
    products of both signs (cur = ref, cur = -ref, and some signs flipped).
    None: magnitudes of [1.5, 2), 1.9921875 is the largest bf16 below 2."""
    torch = torch_cuda()
    rng = np.random.default_rng(D + T)
    mag = magnitude or rng.uniform(1.5, 1.99, (rows, T, D))
    ref = mag * rng.choice([-1.0, 1.0], (rows, T, D)) * np.exp2(rng.choice([-3, 0, 5], (rows, T, 1)))
    flips = rng.choice([0.0, 0.02, 0.5, 0.98, 1.0], (rows, T, 1))
    cur = np.where(rng.random((rows, T, D)) < flips, -ref, ref)
    cur, ref = synth.round_bf16(cur.astype(np.float32)), synth.round_bf16(ref.astype(np.float32))
    g_cur, g_ref = dev(cur, "bf16"), dev(ref, "bf16")
    N = T // 2
    idx = torch.full((rows, N), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT["bf16"], g_cur, g_ref, rows, T, D, N, idx)
    sync()
    got = idx.cpu().numpy()
    for r in range(rows):
        assert got[r].tolist() == O.select_compute(O.cosine_similarity(cur[r], ref[r]), N).tolist(), "row %d" % r


@pytest.mark.parametrize("rows,T,D", [(1, 9, 8), (2, 333, 256), (21, 65, 768), (3, 130, 1288), (1, 700, 1280)])
def test_select_tokens_fp32_ranges(rows, T, D):
    """fp32 sums in triples of floats, and the fp64 sums of vectors whose products
    leave the floats' range: magnitudes on both sides of 2^52 and 2^-51, zeros, Inf
    and NaN. The similarities are random, so that their gaps exceed the roundings."""
    torch = torch_cuda()
    rng = np.random.default_rng(rows + T + D)
    cur, ref = rng.standard_normal((2, rows, T, D))
    ref += 0.5 * cur
    for t, x, y in [(0, 2.0**51, 1.0), (1, 2.0**54, 2.0**-54), (2, 2.0**-49, 2.0**-48), (3, 2.0**-60, 1.0)]:
        cur[:, t] *= x
        ref[:, t] *= y
    cur[:, 4, ::2] = 0.0
    cur[:, 5] = 0.0
    cur[:, 6, :] *= np.exp2(rng.integers(-40, 41, D))
    cur[:, 7, D // 2] = np.inf
    ref[:, 8, D - 1] = np.nan
    cur, ref = cur.astype(np.float32), ref.astype(np.float32)
    g_cur, g_ref = dev(cur), dev(ref)
    N = max(1, T // 3)
    idx = torch.full((rows, N), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT["fp32"], g_cur, g_ref, rows, T, D, N, idx)
    sync()
    got = idx.cpu().numpy()
    with np.errstate(invalid="ignore", over="ignore"):
        for r in range(rows):
            assert got[r].tolist() == O.select_compute(O.cosine_similarity(cur[r], ref[r]), N).tolist(), "row %d" % r
    assert torch.equal(g_ref.view(torch.int32), g_cur.view(torch.int32))


@pytest.mark.parametrize("T", [1, 7, 8, 9, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("D,dtype", [(768, "bf16"), (1280, "bf16"), (1288, "bf16"), (256, "fp32")])
def test_select_tokens_few_tokens(T, D, dtype):
    """Rows of at most 64 tokens, where the CTAs per row and the stages of the
    copy ring follow the number of tokens; many rows and one."""
    torch = torch_cuda()
    for rows in (1, 40):
        cur, ref = synth.similarity_inputs(rows, T, D, seed=rows * 1000 + T, dtype=dtype)
        for N in sorted({1, T // 2, T} - {0}):
            g_cur, g_ref = dev(cur, dtype), dev(ref, dtype)
            idx = torch.full((rows, N), -1, dtype=torch.int32, device="cuda")
            lm.lazymar_select_tokens(DT[dtype], g_cur, g_ref, rows, T, D, N, idx)
            sync()
            got = idx.cpu().numpy()
            for r in range(rows):
                assert got[r].tolist() == O.select_compute(O.cosine_similarity(cur[r], ref[r]), N).tolist()
            assert torch.equal(g_ref, g_cur)


@pytest.mark.parametrize("rows,T,D,dtype", [(1, 16384, 1280, "bf16"), (9, 16384, 64, "bf16"), (2, 16384, 64, "fp32"),
                                            (3, 5000, 768, "bf16")])
def test_select_tokens_many_tokens_of_few_rows(rows, T, D, dtype):
    """Clusters of 16 CTAs with up to the largest shared memory a selection takes."""
    torch = torch_cuda()
    cur, ref = synth.similarity_inputs(rows, T, D, seed=rows + T, dtype=dtype)
    g_cur, g_ref = dev(cur, dtype), dev(ref, dtype)
    N = T // 5
    idx = torch.full((rows, N), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT[dtype], g_cur, g_ref, rows, T, D, N, idx)
    sync()
    got = idx.cpu().numpy()
    for r in range(rows):
        assert got[r].tolist() == O.select_compute(O.cosine_similarity(cur[r], ref[r]), N).tolist(), "row %d" % r
    assert torch.equal(g_ref, g_cur)


def test_select_tokens_more_than_2_to_the_28_rows():
    """The CTAs of all rows are counted without overflow: every row is copied and
    selected (2^28 + 1 rows of one token of 8 elements)."""
    torch = torch_cuda()
    rows = 2 ** 28 + 1
    cur = torch.full((rows, 1, 8), 2.0, dtype=torch.bfloat16, device="cuda")
    cache = torch.ones_like(cur)
    idx = torch.full((rows, 1), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT["bf16"], cur, cache, rows, 1, 8, 1, idx)
    sync()
    assert (cache == 2.0).all() and (idx == 0).all()


def _in_threads(jobs):
    """Runs the jobs on host threads of their own, each on a CUDA stream of its
    own, at the same time; the first error any of them raised, or None."""
    torch = torch_cuda()
    errors, start = [], threading.Barrier(len(jobs))

    def go(job):
        try:
            stream = torch.cuda.Stream()
            start.wait()
            with torch.cuda.stream(stream):
                job()
            stream.synchronize()
        except Exception as e:  # raised again by the caller
            errors.append(e)

    threads = [threading.Thread(target=go, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors[0] if errors else None


def test_select_tokens_from_two_threads():
    """Selections of 320 and of 1088 tokens, which take different amounts of
    shared memory in one kernel, called from two host threads at once."""
    torch = torch_cuda()
    jobs, results = [], []
    for T, N in ((320, 50), (1088, 272)):
        cur, ref = (dev(x, "bf16") for x in synth.similarity_inputs(4, T, 768, seed=T, dtype="bf16"))
        first, idx = (torch.empty((4, N), dtype=torch.int32, device="cuda") for _ in range(2))
        cache = ref.clone()
        lm.lazymar_select_tokens(DT["bf16"], cur, cache, 4, T, 768, N, first)
        sync()

        def job(cur=cur, ref=ref, cache=cache, T=T, N=N, idx=idx):
            for _ in range(3000):
                lm.lazymar_select_tokens(DT["bf16"], cur, cache, 4, T, 768, N, idx)
            cache.copy_(ref)
            lm.lazymar_select_tokens(DT["bf16"], cur, cache, 4, T, 768, N, idx)

        jobs.append(job)
        results.append((idx, first))
    error = _in_threads(jobs)
    assert error is None, error
    sync()
    assert all(torch.equal(idx, first) for idx, first in results)


def test_select_tokens_fp32_near_ties():
    """fp32 similarities are fp64 sums rounded at every addition, in the
    kernel's order on the GPU and in numpy's on the CPU, so mathematically
    equal similarities may come out a few ulps apart on either side. Tokens
    t and t + 32 carry the same vectors with their elements permuted (equal
    exact sums, different rounding) and the budget N cuts through those
    pairs. The GPU's selection must be valid against the oracle's S up to
    8 ulps; every token outside that band is selected exactly as the oracle
    selects it."""
    torch = torch_cuda()
    rows, T, D, N = 4, 64, 256, 40
    rng = np.random.default_rng(31)
    ref = rng.standard_normal((rows, T, D)).astype(np.float32)
    cur = (ref + 0.3 * rng.standard_normal((rows, T, D))).astype(np.float32)
    perm = rng.permutation(D)
    cur[:, 32:], ref[:, 32:] = cur[:, :32][:, :, perm], ref[:, :32][:, :, perm]
    g_cur, g_ref = dev(cur), dev(ref)
    idx = torch.full((rows, N), -1, dtype=torch.int32, device="cuda")
    lm.lazymar_select_tokens(DT["fp32"], g_cur, g_ref, rows, T, D, N, idx)
    sync()
    got = idx.cpu().numpy()
    for r in range(rows):
        S = O.cosine_similarity(cur[r], ref[r])
        margin = 8 * np.spacing(np.abs(S).max())
        sel = set(got[r].tolist())
        assert len(sel) == N and got[r].tolist() == sorted(sel)
        for a in sel:
            for b in set(range(T)) - sel:
                assert S[a] <= S[b] + margin, (r, a, b)
        thr = np.sort(S)[N - 1]
        clear = np.abs(S - thr) > margin
        expect = set(O.select_compute(S, N).tolist())
        assert {t for t in range(T) if clear[t] and t in sel} == {t for t in range(T) if clear[t] and t in expect}


# --------------------------------------------------------------------------
# Condition cache / guidance (Eq. 7 reading, Eq. 10)
# --------------------------------------------------------------------------

@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("mode", [lm.LAZYMAR_CFG_GUIDE, lm.LAZYMAR_CFG_REFRESH, lm.LAZYMAR_CFG_REUSE])
@pytest.mark.parametrize("n", [8 * 1000 + 3, 32 * 256 * 768])
def test_cfg_combine(dtype, mode, n):
    gamma = 3.0
    c = synth.tensor((n,), 11, dtype=dtype)
    u = synth.tensor((n,), 12, dtype=dtype)
    d = synth.tensor((n,), 13, std=0.1, dtype=dtype)
    gc, gu, gd = dev(c, dtype), dev(u, dtype), dev(d, dtype)
    g, uo = empty((n,), dtype), empty((n,), dtype)
    lm.lazymar_cfg_combine(DT[dtype], mode, gc, gu, gd, gamma, n, uo, g)
    sync()
    tol = 8e-3 if dtype == "bf16" else 1e-6
    if mode == lm.LAZYMAR_CFG_REUSE:
        u_ref = O.cond_cache_reuse(c, d)
        assert max_rel(host(uo), u_ref) < tol
    else:
        u_ref = u
    if mode == lm.LAZYMAR_CFG_REFRESH:
        assert max_rel(host(gd), O.cond_cache_store(c, u)) < tol
    assert max_rel(host(g), O.guidance(c, u_ref, gamma)) < tol


# --------------------------------------------------------------------------
# GEMMs (tcgen05 for bf16, CUDA cores for fp32) with every epilogue
# --------------------------------------------------------------------------

GEMM_SHAPES = [
    (1, 384, 128), (40, 768, 256), (200, 2304, 768), (3200, 2304, 768), (3200, 768, 768),
    (3200, 3072, 768), (3200, 768, 3072), (777, 1280, 1280), (384, 3840, 1280),
    (100, 256, 192), (33, 384, 320),  # K not a multiple of 128: 64-deep stages at every width
]


def _linear_case(dtype, epi, M, N, K, flags, seed, scatter=True):
    torch = torch_cuda()
    a = synth.tensor((M, K), seed, dtype=dtype)
    w = synth.tensor((N, K), seed + 1, std=0.05, dtype=dtype)
    b = synth.tensor((N,), seed + 2, std=0.1, dtype=dtype)
    ga, gw, gb = dev(a, dtype), dev(w, dtype), dev(b, dtype)
    ref = O.linear(a, w, b)
    out_dtype_tol = 1e-2 if dtype == "bf16" else 1e-4
    if epi in (lm.LAZYMAR_EPI_BIAS, lm.LAZYMAR_EPI_GELU, lm.LAZYMAR_EPI_SILU):
        out = empty((M, N), dtype)
        lm.lazymar_linear(DT[dtype], epi, ga, gw, gb, M, N, K, out, N, flags=flags)
        sync()
        expect = {lm.LAZYMAR_EPI_BIAS: ref, lm.LAZYMAR_EPI_GELU: O.gelu(ref), lm.LAZYMAR_EPI_SILU: HO.silu(ref)}[epi]
        assert max_rel(host(out), expect) < out_dtype_tol
    elif epi == lm.LAZYMAR_EPI_RESIDUAL:
        r0 = synth.tensor((M, N), seed + 3)
        out = dev(r0, "fp32")
        lm.lazymar_linear(DT[dtype], epi, ga, gw, gb, M, N, K, out, N, flags=flags)
        sync()
        assert max_rel(host(out), r0 + ref) < 1e-4
    elif not scatter:
        D = N // 3
        q, gk, gv = empty((M, D), dtype), empty((M, D), dtype), empty((M, D), dtype)
        lm.lazymar_linear(DT[dtype], epi, ga, gw, gb, M, N, K, q, D, gk, gv, None, flags=flags)
        sync()
        assert max_rel(host(q), ref[:, :D]) < out_dtype_tol
        assert max_rel(host(gk), ref[:, D:2 * D]) < out_dtype_tol
        assert max_rel(host(gv), ref[:, 2 * D:]) < out_dtype_tol
    else:
        D = N // 3
        R = M + 17
        row_map = synth.distinct_rows(M, R, seed + 4)
        k0 = synth.tensor((R, D), seed + 5, dtype=dtype)
        v0 = synth.tensor((R, D), seed + 6, dtype=dtype)
        q, gk, gv = empty((M, D), dtype), dev(k0, dtype), dev(v0, dtype)
        lm.lazymar_linear(DT[dtype], epi, ga, gw, gb, M, N, K, q, D, gk, gv, dev_int(row_map), flags=flags)
        sync()
        assert max_rel(host(q), ref[:, :D]) < out_dtype_tol
        k, v = host(gk), host(gv)
        assert max_rel(k[row_map], ref[:, D:2 * D]) < out_dtype_tol
        assert max_rel(v[row_map], ref[:, 2 * D:]) < out_dtype_tol
        keep = np.setdiff1d(np.arange(R), row_map)
        assert np.array_equal(k[keep], k0[keep]) and np.array_equal(v[keep], v0[keep])


@pytest.mark.parametrize("M,N,K", GEMM_SHAPES)
@pytest.mark.parametrize("epi", [lm.LAZYMAR_EPI_BIAS, lm.LAZYMAR_EPI_GELU, lm.LAZYMAR_EPI_RESIDUAL,
                                 lm.LAZYMAR_EPI_QKV, lm.LAZYMAR_EPI_SILU])
def test_linear_bf16_tcgen05(M, N, K, epi):
    if epi == lm.LAZYMAR_EPI_QKV and (N % 3 or (N // 3) % 32):
        pytest.skip("not a QKV shape")
    for flags in [1, 4] + ([2] if N % 256 == 0 else []) + ([3] if N % 192 == 0 else []):
        _linear_case("bf16", epi, M, N, K, flags, seed=M + N + K + epi)


def _tiles(epi, M, N, K):
    """(rows, width, parts of a tile of the last round) of the automatic choice."""
    sms = torch_cuda().cuda.get_device_properties(0).multi_processor_count
    rows, width, _, parts = lm.lazymar_linear_tiles(epi, M, N, K, sms)
    return rows, width, parts


@pytest.mark.parametrize("M,N,K,epi,tiles", [
    (20480, 768, 768, lm.LAZYMAR_EPI_RESIDUAL, (128, 256, 4)),    # out-projection: three rounds, then 96 tiles 64 wide
    (20480, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 256, 4)),   # fc2: three rounds of CTA pairs, then 48 tiles 64 wide
    (20480, 2304, 768, lm.LAZYMAR_EPI_QKV, (256, 256, 2)),        # Q/K/V: nine rounds of pairs, then 72 tiles 128 wide
])
def test_linear_last_wave_split(M, N, K, epi, tiles):
    """Full layers, whose last round of tiles would leave most SMs idle: it runs
    as narrower tiles of the same launch."""
    assert _tiles(epi, M, N, K) == tiles
    _linear_case("bf16", epi, M, N, K, 0, seed=M + N + K + epi)
    if epi == lm.LAZYMAR_EPI_QKV:
        _linear_case("bf16", epi, M, N, K, 0, seed=M + N + K, scatter=False)


@pytest.mark.parametrize("M,N,K,epi,tiles", [
    (20353, 2304, 768, lm.LAZYMAR_EPI_QKV, (256, 256, 2)),        # one row in the even CTA's half of the last tile
    (20480, 2304, 768, lm.LAZYMAR_EPI_QKV, (256, 256, 2)),
    (6529, 4096, 1024, lm.LAZYMAR_EPI_GELU, (256, 256, 2)),       # one row in the odd CTA's half
    (20480, 3072, 832, lm.LAZYMAR_EPI_BIAS, (256, 256, 1)),       # 13 K steps: the ring wraps within a tile
    (9700, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 256, 2)),
    (12345, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 256, 1)),
    (20480, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 256, 4)),
    (7169, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 256, 4)),
    # 192-wide pairs: whole, and a last round of halves (96 wide, 48 rows of W in each CTA) or thirds
    (2049, 1152, 4608, lm.LAZYMAR_EPI_RESIDUAL, (256, 192, 1)),
    (6464, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 192, 2)),
    (7040, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 192, 2)),
    (7041, 768, 3072, lm.LAZYMAR_EPI_RESIDUAL, (256, 192, 2)),
    (3201, 1152, 4608, lm.LAZYMAR_EPI_RESIDUAL, (256, 192, 3)),
])
def test_linear_pairs_equal_single_ctas(M, N, K, epi, tiles):
    """At these sizes the automatic choice is 256-row tiles on CTA pairs. An
    accumulator sums the same products in the same order as a single CTA's, so
    the results equal the 128-wide tiles' bit for bit; rows past M and cache
    rows outside the row map stay as they were."""
    assert _tiles(epi, M, N, K) == tiles
    torch = torch_cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N + K)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    a, w, b = r(M, K).bfloat16(), (0.05 * r(N, K)).bfloat16(), r(N).bfloat16()
    D = N // 3
    maps = [None, torch.randperm(M + 40, generator=g, device="cuda")[:M].int()] if epi == lm.LAZYMAR_EPI_QKV else [None]
    for row_map in maps:
        res = []
        for flags in (1, 0):
            if epi == lm.LAZYMAR_EPI_QKV:
                outs = [torch.full((M + 40, D), 7.0, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
                lm.lazymar_linear(DT["bf16"], epi, a, w, b, M, N, K, outs[0], D, outs[1], outs[2], row_map, flags)
            else:
                dt = torch.float32 if epi == lm.LAZYMAR_EPI_RESIDUAL else torch.bfloat16
                outs = [torch.full((M + 40, N), 7.0, device="cuda", dtype=dt)]
                lm.lazymar_linear(DT["bf16"], epi, a, w, b, M, N, K, outs[0], N, flags=flags)
            sync()
            res.append(outs)
        assert all(torch.equal(x, y) for x, y in zip(*res))
        assert (res[1][0][M:] == 7.0).all()


@pytest.mark.parametrize("M,N,K,epi", [
    # on 152 SMs: one round of 256-wide tiles and 4 or 8 tiles in quarters, 64 in halves
    (1571, 3072, 128, lm.LAZYMAR_EPI_GELU),
    (1600, 3072, 832, lm.LAZYMAR_EPI_BIAS),
    (2500, 2048, 1024, lm.LAZYMAR_EPI_RESIDUAL),
    (3377, 2048, 64, lm.LAZYMAR_EPI_RESIDUAL),
    (2241, 3072, 256, lm.LAZYMAR_EPI_QKV),
    (20480, 768, 768, lm.LAZYMAR_EPI_RESIDUAL),     # four rounds, the last in quarters
])
def test_linear_split_round_equals_equal_tiles(M, N, K, epi):
    """256-wide tiles of single CTAs whose last round is split into narrower ones (by
    forced width, and in the automatic choice but for the Q/K/V case) give the
    128-wide tiles' results bit for bit."""
    assert epi == lm.LAZYMAR_EPI_QKV or _tiles(epi, M, N, K) in ((128, 256, 2), (128, 256, 4))
    torch = torch_cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N + K)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    a, w, b = r(M, K).bfloat16(), (0.05 * r(N, K)).bfloat16(), r(N).bfloat16()
    D = N // 3
    maps = [None, torch.randperm(M + 40, generator=g, device="cuda")[:M].int()] if epi == lm.LAZYMAR_EPI_QKV else [None]
    for row_map in maps:
        res = []
        for flags in (1, 2, 0):
            if epi == lm.LAZYMAR_EPI_QKV:
                outs = [torch.full((M + 40, D), 7.0, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
                lm.lazymar_linear(DT["bf16"], epi, a, w, b, M, N, K, outs[0], D, outs[1], outs[2], row_map, flags)
            else:
                dt = torch.float32 if epi == lm.LAZYMAR_EPI_RESIDUAL else torch.bfloat16
                outs = [torch.full((M + 40, N), 7.0, device="cuda", dtype=dt)]
                lm.lazymar_linear(DT["bf16"], epi, a, w, b, M, N, K, outs[0], N, flags=flags)
            sync()
            res.append(outs)
        for other in res[1:]:
            assert all(torch.equal(x, y) for x, y in zip(res[0], other))
        assert (res[1][0][M:] == 7.0).all()


@pytest.mark.parametrize("M,N,K", [(1, 384, 128), (63, 768, 256), (65, 768, 3072), (200, 2304, 768), (449, 1024, 1024),
                                   (320, 1536, 640), (1537, 768, 768), (1600, 768, 3072)])
@pytest.mark.parametrize("epi", [lm.LAZYMAR_EPI_BIAS, lm.LAZYMAR_EPI_GELU, lm.LAZYMAR_EPI_RESIDUAL,
                                 lm.LAZYMAR_EPI_QKV, lm.LAZYMAR_EPI_SILU])
def test_linear_few_rows_equal_128_row_tiles(M, N, K, epi):
    """Few rows take 64-row tiles (K % 128 == 0, one round of 64 x 64 tiles, or of
    64 x 128 ones in the residual kinds): bit for bit the 128-row tiles' results, rows past M untouched."""
    torch = torch_cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N + K + epi)
    r = lambda *s: torch.randn(s, generator=g, device="cuda")
    a, w, b = r(M, K).bfloat16(), (0.05 * r(N, K)).bfloat16(), r(N).bfloat16()
    D = N // 3
    if epi == lm.LAZYMAR_EPI_QKV and (N % 3 or D % 32):
        pytest.skip("not a QKV shape")
    if M < 1000:
        assert _tiles(epi, M, N, K)[:2] == (64, 64)
    elif epi == lm.LAZYMAR_EPI_RESIDUAL:
        assert _tiles(epi, M, N, K)[:2] == (64, 128)
    maps = [None, torch.randperm(M + 40, generator=g, device="cuda")[:M].int()] if epi == lm.LAZYMAR_EPI_QKV else [None]
    for row_map in maps:
        res = []
        for flags in (1, 0):
            if epi == lm.LAZYMAR_EPI_QKV:
                outs = [torch.full((M + 40, D), 7.0, device="cuda", dtype=torch.bfloat16) for _ in range(3)]
                lm.lazymar_linear(DT["bf16"], epi, a, w, b, M, N, K, outs[0], D, outs[1], outs[2], row_map, flags)
            else:
                dt = torch.float32 if epi == lm.LAZYMAR_EPI_RESIDUAL else torch.bfloat16
                outs = [torch.full((M + 40, N), 7.0, device="cuda", dtype=dt)]
                lm.lazymar_linear(DT["bf16"], epi, a, w, b, M, N, K, outs[0], N, flags=flags)
            sync()
            res.append(outs)
        assert all(torch.equal(x, y) for x, y in zip(*res))
        assert (res[1][0][M:] == 7.0).all()


@pytest.mark.parametrize("M,N,K", [(1, 12, 8), (40, 768, 256), (160, 1024, 256), (77, 256, 1024)])
@pytest.mark.parametrize("epi", [lm.LAZYMAR_EPI_BIAS, lm.LAZYMAR_EPI_GELU, lm.LAZYMAR_EPI_RESIDUAL,
                                 lm.LAZYMAR_EPI_QKV, lm.LAZYMAR_EPI_SILU])
def test_linear_fp32(M, N, K, epi):
    if epi == lm.LAZYMAR_EPI_QKV and (N % 3 or (N // 3) % 4):
        pytest.skip("not a QKV shape")
    _linear_case("fp32", epi, M, N, K, 0, seed=M + N + K + epi)


@pytest.mark.parametrize("M,N,K", [(1, 4, 4), (17, 36, 516), (33, 260, 1028), (160, 1024, 256), (300, 772, 260),
                                   (2561, 1028, 64), (40, 256, 1024), (9, 2048, 2052)])
@pytest.mark.parametrize("epi", [lm.LAZYMAR_EPI_GELU, lm.LAZYMAR_EPI_RESIDUAL])
def test_linear_fp32_tiles(M, N, K, epi):
    """Edges of the 16, 32 and 64 wide fp32 tiles, slices of K that are uneven,
    empty or not a multiple of the staged chunk."""
    _linear_case("fp32", epi, M, N, K, 0, seed=M + N + K + epi)


@pytest.mark.parametrize("M,N,K", [(641, 1028, 68), (641, 1028, 260), (2399, 772, 772), (161, 1028, 1028), (159, 772, 1028),
                                   (9, 20004, 64), (1279, 772, 128)])
def test_linear_fp32_tile_choice(M, N, K):
    """Sizes on either side of the lines between the fp32 tiles and splits of K."""
    _linear_case("fp32", lm.LAZYMAR_EPI_BIAS, M, N, K, 0, seed=M + N + K)


@pytest.mark.parametrize("rows,n_q,T,heads,dh", [(2, 5, 32, 2, 64), (1, 9, 33, 3, 30), (1, 4, 127, 1, 128), (2, 3, 128, 2, 64),
                                                 (1, 6, 129, 2, 64), (1, 2, 300, 2, 66), (3, 1, 1, 2, 1), (1, 5, 8192, 1, 8)])
def test_attention_fp32_chunks(rows, n_q, T, heads, dh):
    """fp32 attention at the edges of its key chunks (32 to 128 keys, one chunk
    or several) and at head widths that are not a multiple of 4."""
    D = heads * dh
    q, k, v = (synth.tensor((rows, n, D), 31 + i) for i, n in enumerate((n_q, T, T)))
    o = empty((rows, n_q, D))
    lm.lazymar_attention(DT["fp32"], dev(q), dev(k), dev(v), o, rows, n_q, T, heads, dh)
    sync()
    ref = np.stack([O.attention(q[r], k[r], v[r], heads) for r in range(rows)])
    assert max_rel(host(o), ref) < 1e-5


def test_attention_fp32_from_threads():
    """fp32 attention over 80 and over 128 keys, which takes different amounts of
    shared memory in one kernel, called from four host threads at once, for long
    enough to fill their streams."""
    torch = torch_cuda()
    jobs, results = [], []
    for T in (80, 128, 80, 128):
        q, k, v = (dev(synth.tensor((32, n, 256), T + i)) for i, n in enumerate((80, T, T)))
        first, o = empty((32, 80, 256)), empty((32, 80, 256))
        lm.lazymar_attention(DT["fp32"], q, k, v, first, 32, 80, T, 4, 64)
        sync()

        def job(q=q, k=k, v=v, o=o, T=T):
            for _ in range(4000):
                lm.lazymar_attention(DT["fp32"], q, k, v, o, 32, 80, T, 4, 64)

        jobs.append(job)
        results.append((o, first))
    error = _in_threads(jobs)
    assert error is None, error
    sync()
    assert all(torch.equal(o, first) for o, first in results)


# --------------------------------------------------------------------------
# E4M3 Q/K/V projection (qkv_e4m3): weight quantization, LayerNorm to E4M3,
# the kind::f8f6f4 GEMM
# --------------------------------------------------------------------------

def _e4m3_codes(shape, seed):
    """Random E4M3 bytes over the whole finite range (no NaN codes)."""
    c = np.random.default_rng(seed).integers(0, 256, size=shape).astype(np.uint8)
    c[(c & 0x7F) == 0x7F] = 0x38
    return c


@pytest.mark.parametrize("rows,cols", [(2304, 768), (3840, 1280), (5, 8), (130, 1024)])
def test_quantize_e4m3_bit_exact(rows, cols):
    """Per-row scales and E4M3 codes of a bf16 weight matrix. The rounding
    decision is taken in fp32 on both sides (the kernel's precision): scale =
    fp32(max|w|) / 448, code = E4M3(fp32(w) / scale); the oracle's rounding is
    the format's definition. Rows of zeros, a row with an exact tie and
    mixed magnitudes included."""
    torch = torch_cuda()
    w = synth.tensor((rows, cols), rows + cols, std=0.02, dtype="bf16")
    w[0] = 0.0
    if rows > 2:
        w[1] = synth.round_bf16(np.linspace(-3, 3, cols).astype(np.float32))
        w[2] = synth.round_bf16(w[2] * np.float32(1e4))
    gw = dev(w, "bf16")
    q = torch.zeros((rows, cols), dtype=torch.uint8, device="cuda")
    sc = torch.zeros(rows, dtype=torch.float32, device="cuda")
    lm.lazymar_quantize_e4m3(gw, rows, cols, q, sc)
    sync()
    amax = np.abs(w).max(axis=1).astype(np.float32)
    s32 = np.where(amax > 0, amax / np.float32(448.0), np.float32(1.0)).astype(np.float32)
    np.testing.assert_array_equal(sc.cpu().numpy(), s32)
    expect = fp8.e4m3_round((w.astype(np.float32) / s32[:, None]).astype(np.float32))
    got = fp8.e4m3_decode(q.cpu().numpy())
    np.testing.assert_array_equal(np.abs(got), np.abs(expect))
    nz = expect != 0
    assert (np.sign(got[nz]) == np.sign(expect[nz])).all()


def test_layernorm_e4m3_output():
    """LayerNorm rows to E4M3 (unit scale): every code is the E4M3 rounding of
    the oracle's LayerNorm, or its neighbour where the fp32 value lies within
    rounding distance of the midpoint between two codes."""
    torch = torch_cuda()
    M, D = 300, 768
    x = synth.tensor((M, D), 41, std=3.0, mean=0.5)
    g = synth.tensor((D,), 42, std=0.5, mean=1.0, dtype="bf16")
    b = synth.tensor((D,), 43, std=0.2, dtype="bf16")
    y = torch.zeros((M, D), dtype=torch.uint8, device="cuda")
    lm.lazymar_layernorm(lm.LAZYMAR_E4M3, dev(x), None, dev(g, "bf16"), dev(b, "bf16"), y, M, D, 1e-6)
    sync()
    ref = O.layer_norm(x, g, b, 1e-6)
    got = fp8.e4m3_decode(y.cpu().numpy())
    exact = fp8.e4m3_round(ref)
    bad = got != exact
    assert bad.mean() < 1e-3
    # where they differ, the oracle's value sits at a rounding midpoint of the two codes
    lo, hi = np.minimum(got[bad], exact[bad]), np.maximum(got[bad], exact[bad])
    mid = (lo + hi) / 2
    assert (np.abs(ref[bad] - mid) <= 1e-5 * np.maximum(np.abs(mid), 1.0)).all()
    assert (hi - lo <= np.maximum(np.abs(hi), np.abs(lo)) * 2.0 ** -3 + 2.0 ** -9).all()


@pytest.mark.parametrize("M,N,K", [(3200, 2304, 768), (1600, 2304, 768), (12800, 3840, 1280), (777, 3072, 1024),
                                   (1, 384, 128), (130, 256, 256)])
@pytest.mark.parametrize("epi", [lm.LAZYMAR_EPI_BIAS, lm.LAZYMAR_EPI_QKV])
def test_linear_e4m3(M, N, K, epi):
    """The kind::f8f6f4 GEMM on E4M3 operands with per-column weight scales
    against the oracle's product of the decoded operands (exact in fp64; the
    GPU accumulates in fp32 and writes bf16), every tile width."""
    if epi == lm.LAZYMAR_EPI_QKV and (N % 3 or (N // 3) % 32):
        pytest.skip("not a QKV shape")
    torch = torch_cuda()
    seed = M + N + K + epi
    ac, wc = _e4m3_codes((M, K), seed), _e4m3_codes((N, K), seed + 1)   # subnormals to +-448
    scale = (np.random.default_rng(seed + 2).uniform(0.5, 2.0, N) * 1e-3).astype(np.float32)
    bias = synth.tensor((N,), seed + 3, std=0.1, dtype="bf16")
    ref = fp8.e4m3_decode(ac) @ (fp8.e4m3_decode(wc) * scale[:, None].astype(np.float64)).T + bias
    ga = torch.from_numpy(ac).cuda()
    gw = torch.from_numpy(wc).cuda()
    gs = torch.from_numpy(scale).cuda()
    gb = dev(bias, "bf16")
    for flags in [1] + ([2] if N % 256 == 0 else []) + ([3] if N % 192 == 0 else []):
        if epi == lm.LAZYMAR_EPI_BIAS:
            out = empty((M, N), "bf16")
            lm.lazymar_linear_e4m3(epi, ga, gw, gs, gb, M, N, K, out, N, flags=flags)
            sync()
            assert max_rel(host(out), ref) < 1e-2, flags
        else:
            D = N // 3
            R = M + 17
            row_map = synth.distinct_rows(M, R, seed + 4)
            k0 = synth.tensor((R, D), seed + 5, dtype="bf16")
            v0 = synth.tensor((R, D), seed + 6, dtype="bf16")
            q, gk, gv = empty((M, D), "bf16"), dev(k0, "bf16"), dev(v0, "bf16")
            lm.lazymar_linear_e4m3(epi, ga, gw, gs, gb, M, N, K, q, D, gk, gv, dev_int(row_map), flags=flags)
            sync()
            assert max_rel(host(q), ref[:, :D]) < 1e-2
            k, v = host(gk), host(gv)
            assert max_rel(k[row_map], ref[:, D:2 * D]) < 1e-2 and max_rel(v[row_map], ref[:, 2 * D:]) < 1e-2
            keep = np.setdiff1d(np.arange(R), row_map)
            assert np.array_equal(k[keep], k0[keep]) and np.array_equal(v[keep], v0[keep])


# --------------------------------------------------------------------------
# Attention (Eq. 3 with a query subset)
# --------------------------------------------------------------------------

@pytest.mark.parametrize("rows,n_q,T,heads,dh,dtype,q_std", [
    (2, 50, 320, 12, 64, "bf16", 1.0),    # MAR-B cached layer
    (2, 320, 320, 4, 64, "bf16", 1.0),    # full layer
    (1, 272, 1088, 2, 64, "bf16", 1.0),   # high resolution cached layer
    (3, 50, 320, 4, 80, "bf16", 1.0),     # MAR-H head width, cached layer
    (2, 320, 320, 16, 80, "bf16", 1.0),   # MAR-H full layer (three query tiles)
    (2, 65, 130, 2, 80, "bf16", 1.0),     # ragged queries and keys
    (1, 129, 200, 3, 80, "bf16", 1.0),    # one query past a tile, a ragged key chunk
    (3, 256, 300, 5, 64, "bf16", 1.0),    # whole query tiles only (no shorter last tile)
    (1, 1, 1, 1, 80, "bf16", 1.0),
    (1, 1, 1, 1, 64, "bf16", 1.0),
    # scores of std ~6 (log2 units): the running maximum is raised mid-row
    # and O in tensor memory rescaled
    (2, 50, 320, 4, 64, "bf16", 4.0),
    (2, 50, 320, 4, 80, "bf16", 4.0),
    (2, 20, 80, 4, 64, "fp32", 1.0),      # tiny
    (1, 3, 5, 2, 32, "fp32", 1.0),
])
def test_attention(rows, n_q, T, heads, dh, dtype, q_std):
    D = heads * dh
    q = synth.tensor((rows, n_q, D), 21, std=q_std, dtype=dtype)
    k = synth.tensor((rows, T, D), 22, dtype=dtype)
    v = synth.tensor((rows, T, D), 23, dtype=dtype)
    o = empty((rows, n_q, D), dtype)
    lm.lazymar_attention(DT[dtype], dev(q, dtype), dev(k, dtype), dev(v, dtype), o, rows, n_q, T, heads, dh)
    sync()
    ref = np.stack([O.attention(q[r], k[r], v[r], heads) for r in range(rows)])
    assert max_rel(host(o), ref) < (1e-2 if dtype == "bf16" else 1e-5)


# --------------------------------------------------------------------------
# LayerNorm (gathering rows)
# --------------------------------------------------------------------------

@pytest.mark.parametrize("rows,n_q,T,heads,dh,q_std", [
    (64, 129, 320, 12, 64, 1.0),   # more CTAs than one wave: probabilities in tensor memory
    (46, 65, 65, 12, 64, 1.0),     # one query and one key past a tile and a chunk
    (40, 320, 63, 12, 64, 1.0),    # a single, partial key chunk
    (30, 300, 1088, 6, 64, 4.0),   # running maxima raised mid-row
    (26, 50, 320, 12, 80, 1.0),    # width 80: 48-key chunks, any number of queries
    (16, 129, 97, 16, 80, 1.0),
    (40, 1, 49, 16, 80, 1.0),
    (12, 300, 500, 16, 80, 4.0),
])
def test_attention_large_grids(rows, n_q, T, heads, dh, q_std):
    D = heads * dh
    q = synth.tensor((rows, n_q, D), 41, std=q_std, dtype="bf16")
    k = synth.tensor((rows, T, D), 42, dtype="bf16")
    v = synth.tensor((rows, T, D), 43, dtype="bf16")
    o = empty((rows, n_q, D), "bf16")
    lm.lazymar_attention(DT["bf16"], dev(q, "bf16"), dev(k, "bf16"), dev(v, "bf16"), o, rows, n_q, T, heads, dh)
    sync()
    got = host(o)
    for r in (0, rows // 2, rows - 1):
        assert max_rel(got[r], O.attention(q[r], k[r], v[r], heads)) < 1e-2, "row %d" % r
    torch = torch_cuda()
    split = [x.view(rows, -1, heads, dh).transpose(1, 2) for x in (dev(q), dev(k), dev(v))]
    ref = torch.nn.functional.scaled_dot_product_attention(*split).transpose(1, 2).reshape(rows, n_q, D)
    assert max_rel(got, host(ref)) < 1e-2


@pytest.mark.parametrize("T", [48, 49, 63, 64, 65, 97, 200, 320])
@pytest.mark.parametrize("heads,dh", [(16, 80), (16, 64)])
def test_attention_large_grid_equals_small(T, heads, dh):
    """A row computed in a large grid (attention_tm_kernel) and by itself
    (attention_tc_kernel): the probabilities are the same bf16 values, because
    both kernels take the first running maximum over 64 keys; only the fp32 row
    sums are in another order, 2^-24 against the 2^-9 of the results, so that
    about 1 result in 2^14 may fall on the other side of a rounding."""
    torch = torch_cuda()
    rows, n_q, D = 64, 65, heads * dh
    q = dev(synth.tensor((rows, n_q, D), 51, dtype="bf16"), "bf16")
    k = dev(synth.tensor((rows, T, D), 52, dtype="bf16"), "bf16")
    v = dev(synth.tensor((rows, T, D), 53, dtype="bf16"), "bf16")
    o = empty((rows, n_q, D), "bf16")
    lm.lazymar_attention(DT["bf16"], q, k, v, o, rows, n_q, T, heads, dh)
    sync()
    for r in (0, rows // 2, rows - 1):
        one = empty((1, n_q, D), "bf16")
        lm.lazymar_attention(DT["bf16"], q[r:r + 1], k[r:r + 1], v[r:r + 1], one, 1, n_q, T, heads, dh)
        sync()
        assert (one[0] != o[r]).sum().item() <= n_q * D * 2.0 ** -9, "row %d" % r


@pytest.mark.parametrize("rows,n_q,T,q_std", [
    (1, 1, 65, 1.0), (2, 31, 64, 1.0), (10, 33, 320, 1.0), (24, 63, 129, 1.0), (32, 64, 1, 1.0),
    (40, 64, 320, 1.0), (64, 32, 63, 1.0), (40, 50, 1088, 4.0),     # four CTAs per SM
])
def test_attention_up_to_64_queries(rows, n_q, T, q_std):
    """CTAs of 64 query rows, one to four per SM: the large grids' checks."""
    test_attention_large_grids(rows, n_q, T, 12, 64, q_std)


@pytest.mark.parametrize("M,D,gather,dtype", [(100, 768, False, "bf16"), (50, 1280, True, "bf16"),
                                              (80, 256, True, "fp32"), (3, 1024, False, "fp32")])
def test_layernorm(M, D, gather, dtype):
    R = M + 30
    x = synth.tensor((R, D), 31, std=2.0, mean=0.5)
    g = synth.tensor((D,), 32, std=0.1, mean=1.0, dtype=dtype)
    b = synth.tensor((D,), 33, std=0.1, dtype=dtype)
    rm = synth.distinct_rows(M, R, 34) if gather else None
    y = empty((M, D), dtype)
    lm.lazymar_layernorm(DT[dtype], dev(x), None if rm is None else dev_int(rm), dev(g, dtype), dev(b, dtype), y,
                         M, D, 1e-6)
    sync()
    src = x[rm] if gather else x[:M]
    assert max_rel(host(y), O.layer_norm(src, g, b, 1e-6)) < (1e-2 if dtype == "bf16" else 1e-5)


def test_gelu_epilogue_matches_erf_gelu():
    """The MLP epilogue's GELU (the normal tail as 2^P(|x|), P a fitted degree-5
    polynomial, within 2.8e-7 max(1, |x|) in fp32) against the oracle's fp64
    erf GELU. An fp32 GEMM with W = I makes the pre-activation exactly the
    input, on a dense grid over [-8, 8]."""
    M, K = 512, 64
    x = np.linspace(-8.0, 8.0, M * K, dtype=np.float32).reshape(M, K)
    out = empty((M, K), "fp32")
    lm.lazymar_linear(DT["fp32"], lm.LAZYMAR_EPI_GELU, dev(x), dev(np.eye(K, dtype=np.float32)), None, M, K, K,
                      out, K)
    sync()
    err = np.abs(host(out) - O.gelu(x.astype(np.float64)))
    assert (err <= 1e-6 * np.maximum(1.0, np.abs(x))).all(), float(err.max())


# --------------------------------------------------------------------------
# Failure detection: a bounded device wait that runs out
# --------------------------------------------------------------------------

def test_bounded_wait_expires_and_device_stays_usable():
    """The self-test kernel waits 50 ms on an mbarrier nothing completes: the
    wait gives up, the host reads LAZYMAR_ERR_TIMEOUT (then the word is clear),
    and kernels launched afterwards still run correctly."""
    import time
    lm.lazymar_device_check()
    t0 = time.perf_counter()
    lm.lazymar_selftest_wait(50000)
    with pytest.raises(lm.LazymarError) as e:
        lm.lazymar_device_check()
    assert e.value.status == 5                       # LAZYMAR_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 10
    lm.lazymar_device_check()                        # reported once, then clear
    _linear_case("bf16", lm.LAZYMAR_EPI_BIAS, 200, 256, 128, 1, seed=5)
    lm.lazymar_device_check()

