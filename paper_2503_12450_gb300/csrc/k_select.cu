// Token selection of Eq. 8: one kernel, one thread-block cluster per row.
//
// The CTAs of a cluster take equal ranges of the row's tokens, one warp per
// token: the cosine of its current and cached representation, whose current
// vector then replaces the cached one. Every CTA pushes its tokens'
// similarities, as order-preserving 64-bit integer keys, into the shared
// memory of all CTAs of the cluster; each CTA ranks its own tokens under the
// strict total order (priority descending, rule key ascending, index
// ascending), and with the counts of the lower CTAs writes its part of
// I_compute in ascending order with the gather/scatter row map r*T + t. No
// similarity reaches global memory, so a selection needs no scratch.
//
// Floor: streaming 3 x rows x T x D elements, 13.9 us at 64 rows x 320 tokens
// x 768 bf16 (94 MB). Measured there: 31.6 us a call, against
// 75.5 us for a similarity kernel (every token through the second tier below
// and its own fp64 division), a top-N kernel with one CTA per row and scratch
// allocated for the similarities in between. What is left above the floor is
// instruction issue (about 13 us) and the row's serial tail: fp64 divisions
// and square roots, ranks, three cluster barriers. Sums kept in registers
// instead of the shared-memory ring took 36.7 us, one division per warp
// instead of per CTA round 41.5 us.
//
// Similarities. bf16 x bf16 products are exact in fp64, and so are their sums
// for any realistic dynamic range, which makes S independent of the summation
// order: the oracle's fp64 sum gives bit-identical S, hence bit-identical
// selections. The kernel computes the three sums exactly on the integer pipe
// (GB300's fp64 rate is a small fraction of its integer rate) or, wider than 1280,
// in triples of floats, and rounds each once. fp32 x fp32 products are exact in fp64 too, but a sum of them is
// rounded at every addition: the kernel's sums (correctly rounded but for the
// last bit) and the oracle's pairwise ones can differ in the last bits of S (a
// relative 1e-15 or so). Two tokens whose similarities lie that close may then be
// ordered differently; every other fp32 selection is identical.
#include <atomic>
#include <cfloat>
#include <climits>

#include "lazymar_internal.cuh"

namespace lm {

// Order-preserving 64-bit key of a similarity: unsigned comparison of keys
// matches numeric comparison of the doubles, with NaN mapped to -inf and -0
// to +0 (so equal similarities give equal keys and the index decides). Keys
// are compared on the integer pipe; GB300's fp64 pipe is far slower.
__device__ __forceinline__ unsigned long long sim_key(double s) {
  if (s != s) s = -HUGE_VAL;
  if (s == 0.0) s = 0.0;
  const unsigned long long u = (unsigned long long)__double_as_longlong(s);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// The sums of one token: dot, |a|^2, |c|^2, as v[i] * 2^e[i] with integer v, as
// the bits of a double in v[i], or as the sum of three floats: the bits of two in
// v[i] and of one in e[i].
enum { SUMS_INT, SUMS_F64, SUMS_F32X3 };
struct SimSums {
  long long v[3];
  int e[3], kind;
};

__device__ __forceinline__ double sim_value(const SimSums& s) {
  double d[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float hi = __int_as_float((int)s.v[i]), mid = __int_as_float((int)(s.v[i] >> 32)), lo = __int_as_float(s.e[i]);
    d[i] = s.kind == SUMS_F64     ? __longlong_as_double(s.v[i])
           : s.kind == SUMS_F32X3 ? ((double)hi + (double)mid) + (double)lo
                                  : ldexp((double)s.v[i], s.e[i]);
  }
  const double eps = 1e-8;
  return d[0] / sqrt(fmax(d[1] * d[2], eps * eps));
}

// Sum of v * 2^e over the warp's lanes as an integer times a power of two
// that rounds to the same double as the exact sum. Three 22-, 22- and 20-bit
// pieces go through the warp's integer reduction. A total, below 2^68 in
// magnitude, that has reached 2^62 is shifted right by 6 with its lost bits kept as a
// sticky lowest bit: at least 56 bits are left, of which a double holds 53.
__device__ __forceinline__ void warp_sum64(long long v, int e, long long& out_v, int& out_e) {
  const unsigned p0 = __reduce_add_sync(0xffffffffu, (unsigned)(v & 0x3FFFFF));
  const unsigned p1 = __reduce_add_sync(0xffffffffu, (unsigned)((v >> 22) & 0x3FFFFF));
  const int p2 = __reduce_add_sync(0xffffffffu, (int)(v >> 44));
  const long long hi = (long long)p2 * (1ll << 22) + (long long)p1 + (long long)(p0 >> 22);  // total = hi 2^22 + lo
  const long long lo = (long long)(p0 & 0x3FFFFFu);
  const bool wide = hi >= (1ll << 40) || hi < -(1ll << 40);
  out_v = wide ? (hi * (1ll << 16)) | (lo >> 6) | ((lo & 63) != 0) : hi * (1ll << 22) + lo;
  out_e = wide ? e + 6 : e;
}

// fp64 sums of one token in lane-strided order; no copy.
template <typename T>
__device__ __forceinline__ void sums_fp64(const T* a, const T* c, int D, int lane, SimSums& s) {
  constexpr int V = 16 / sizeof(T);
  double dot = 0.0, na = 0.0, nc = 0.0;
#pragma unroll 1
  for (int i = lane * V; i < D; i += 32 * V) {
    float av[V], cv[V];
    Vec<T, V>::load(a + i, av);
    Vec<T, V>::load(c + i, cv);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const double x = (double)av[k], y = (double)cv[k];
      dot = fma(x, y, dot);
      na = fma(x, x, na);
      nc = fma(y, y, nc);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    dot += __shfl_xor_sync(0xffffffffu, dot, o);
    na += __shfl_xor_sync(0xffffffffu, na, o);
    nc += __shfl_xor_sync(0xffffffffu, nc, o);
  }
  s.v[0] = __double_as_longlong(dot);
  s.v[1] = __double_as_longlong(na);
  s.v[2] = __double_as_longlong(nc);
  s.kind = SUMS_F64;
}

// Two running sums, one per half of the packed registers, each the unevaluated
// sum of three floats, of which each is about 2^-24 of the one before.
struct F32x3 {
  unsigned long long s, c, d;
};
__device__ __forceinline__ unsigned long long f32x2_sub(unsigned long long a, unsigned long long b) {
  return f32x2_fma(b, 0xBF800000BF800000ull, a);  // a - 1 b
}
// a + b = s + e exactly (Knuth's two-sum)
__device__ __forceinline__ void two_sum(unsigned long long a, unsigned long long b, unsigned long long& s,
                                        unsigned long long& e) {
  const unsigned long long t = f32x2_add(a, b), bb = f32x2_sub(t, a);
  e = f32x2_add(f32x2_sub(a, f32x2_sub(t, bb)), f32x2_sub(b, bb));
  s = t;
}
// x y = p + e exactly; both join the sum.
__device__ __forceinline__ void add_product(F32x3& t, unsigned long long x, unsigned long long y) {
  const unsigned long long p = f32x2_fma(x, y, 0ull);
  const unsigned long long e = f32x2_fma(x, y, p ^ 0x8000000080000000ull);
  unsigned long long q, r, u;
  two_sum(t.s, p, t.s, q);
  two_sum(t.c, q, t.c, r);
  two_sum(t.c, e, t.c, u);
  t.d = f32x2_add(t.d, f32x2_add(r, u));
}
__device__ __forceinline__ void add_sum(F32x3& t, const F32x3& o) {
  unsigned long long q, r, u;
  two_sum(t.s, o.s, t.s, q);
  two_sum(t.c, o.c, t.c, r);
  two_sum(t.c, q, t.c, u);
  t.d = f32x2_add(f32x2_add(t.d, o.d), f32x2_add(r, u));
}

// 16 bytes of elements as pairs of floats.
__device__ __forceinline__ void load_pairs(const float* p, unsigned long long (&w)[2]) {
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
  w[0] = q.x;
  w[1] = q.y;
}
__device__ __forceinline__ void load_pairs(const bf16* p, unsigned long long (&w)[4]) {
  const uint4 q = *reinterpret_cast<const uint4*>(p);
  const uint32_t v[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) w[i] = (unsigned long long)(v[i] << 16) | ((unsigned long long)(v[i] & 0xFFFF0000u) << 32);
}

// Sums of one token in triples of floats (Ogita, Rump and Oishi's compensated
// dot product with one more level): products and the errors of the first two
// levels are exact, and the third's roundings lie 2^-72 below the sum of the
// terms' magnitudes, so the sums are rounded to double once, where an fp64 sum
// rounds at every addition. GB300 has about two fp64 lanes per SM, and an element
// pair costs five fp64 instructions, 320 issue cycles of a scheduler, against about
// 45 here with two elements per instruction. Measured, fp64 sums -> this (us a
// call): 64 rows x 320 tokens x 768 200 -> 74, 26 x 320 x 1024 132 -> 51, 1 x 1088 x
// 1280 146 -> 63 (84 with fp64 sums spread over all SMs), 8 x 320 x 1280 83 -> 32.
// Largest error of the sums of 60 vectors of 256 to 1280 normal elements: 1.1e-16 of
// the sum, of fp64 sums 1.2e-14. bf16 vectors wider than 1280 (whose products are exact
// in a float): 1 row x 320 x 2048 66 -> 26, 1024 x 65 x 2048 1509 -> 467.
// Vectors with an element of magnitude from 2^52 or (nonzero) below 2^-51, whose
// products could overflow or lose bits, and ones with Inf or NaN take fp64 sums.
template <typename T>
__device__ __forceinline__ void sums_f32x3(const T* a, const T* c, int D, int lane, SimSums& s) {
  constexpr int V = 16 / sizeof(T);
  F32x3 dot{}, na{}, nc{};
  uint32_t most = 0, least = 0xFFFFFFFFu;  // of the magnitudes' bits; of those - 1, in which zeros are the largest
#pragma unroll 2
  for (int i = lane * V; i < D; i += 32 * V) {
    unsigned long long x[V / 2], y[V / 2];  // two elements each
    load_pairs(a + i, x);
    load_pairs(c + i, y);
#pragma unroll
    for (int h = 0; h < V / 2; ++h) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const unsigned long long w = j ? y[h] : x[h];
        const uint32_t m0 = (uint32_t)w & 0x7FFFFFFFu, m1 = (uint32_t)(w >> 32) & 0x7FFFFFFFu;
        most = max(most, max(m0, m1));
        least = min(least, min(m0 - 1u, m1 - 1u));
      }
      add_product(dot, x[h], y[h]);
      add_product(na, x[h], x[h]);
      add_product(nc, y[h], y[h]);
    }
  }
  most = __reduce_max_sync(0xffffffffu, most);
  least = __reduce_min_sync(0xffffffffu, least);
  if (most >= (179u << 23) || least < (76u << 23) - 1u) {
    sums_fp64(a, c, D, lane, s);
    return;
  }
  // (dot, |a|^2) and (|c|^2, 0): the halves of each, then the lanes
  auto low = [](unsigned long long x, unsigned long long y) { return (x & 0xFFFFFFFFull) | (y << 32); };
  auto high = [](unsigned long long x, unsigned long long y) { return (x >> 32) | (y & 0xFFFFFFFF00000000ull); };
  F32x3 u{low(dot.s, na.s), low(dot.c, na.c), low(dot.d, na.d)}, w{low(nc.s, 0), low(nc.c, 0), low(nc.d, 0)};
  add_sum(u, F32x3{high(dot.s, na.s), high(dot.c, na.c), high(dot.d, na.d)});
  add_sum(w, F32x3{high(nc.s, 0), high(nc.c, 0), high(nc.d, 0)});
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    auto other = [&](unsigned long long x) { return __shfl_xor_sync(0xffffffffu, x, o); };
    auto first = [&](unsigned long long x) { return (unsigned long long)__shfl_xor_sync(0xffffffffu, (uint32_t)x, o); };
    add_sum(u, F32x3{other(u.s), other(u.c), other(u.d)});
    add_sum(w, F32x3{first(w.s), first(w.c), first(w.d)});
  }
  s.v[0] = (long long)low(u.s, u.c);
  s.v[1] = (long long)high(u.s, u.c);
  s.v[2] = (long long)low(w.s, w.c);
  s.e[0] = (int)(uint32_t)u.d;
  s.e[1] = (int)(u.d >> 32);
  s.e[2] = (int)(uint32_t)w.d;
  s.kind = SUMS_F32X3;
}

// Exact sums of a bf16 token of which each lane has NCH 16-byte chunks of
// both vectors (zero beyond D) at sa[32 j] and sc[32 j], in two tiers of
// integer arithmetic:
//
// 1. Fixed point. Scaled by a power of two (k below) so that its largest
//    element stays below 2^bits, every element of a vector whose nonzero
//    exponents span at most bits - 8 octaves is an integer of the int32 range,
//    and the three sums are one 32 x 32 -> 64 multiply-add per product. A
//    lane's 8 NCH products stay within an int64: bits = 30, 29, 29, 29, 28 for
//    NCH = 1..5. About 1 in 400 tokens of normally distributed elements
//    exceeds the 21 octaves of widths 264 to 1024. About 14 issue slots per
//    element pair against 55 for the second tier.
// 2. Shifted products. A bf16 value is M * 2^(E - 134) with an 8-bit integer
//    significand M (hidden bit included) and E = max(biased exponent, 1), so a
//    product of two is (Ma Mb) * 2^(Ea + Eb - 268) with Ma Mb < 2^16. Each sum
//    is taken relative to a base exponent span = 62 - 16 - ceil(log2 D) below
//    its largest possible term exponent (from the vectors' largest exponents):
//    shifted to the base, every term is an integer below 2^(16 + span) and the
//    D-term sum is exact in an int64.
//
// A token with a nonzero term below that base, or with an Inf/NaN element,
// takes the fp64 sums instead. An integer sum converts to double with one
// rounding of the exact value, whatever the tier: it equals the fp64 sum of
// the same products whenever that sum is exact.
template <int NCH>
__device__ __forceinline__ void sums_bf16(const uint4* sa, const uint4* sc, const bf16* a, const bf16* c, int D,
                                          int span, int lane, SimSums& s) {
  constexpr int bits = NCH == 1 ? 30 : NCH <= 4 ? 29 : 28;
  static_assert(NCH >= 1 && NCH <= 5, "8 NCH products below 2^(2 bits) in an int64");
  // per vector: the largest magnitude (two bf16 per word, unsigned), and the
  // smallest nonzero one. (w | sign) - 1 per half is 0x7FFF for a zero and
  // 0x8000 + magnitude - 1 otherwise, so a signed minimum skips the zeros.
  uint32_t xa = 0, xc = 0, na = 0x7FFF7FFFu, nc = 0x7FFF7FFFu;
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    const uint4 qa = sa[32 * j], qc = sc[32 * j];
    const uint32_t wa[4] = {qa.x, qa.y, qa.z, qa.w}, wc[4] = {qc.x, qc.y, qc.z, qc.w};
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      xa = __vmaxu2(xa, wa[h] & 0x7FFF7FFFu);
      xc = __vmaxu2(xc, wc[h] & 0x7FFF7FFFu);
      na = __vmins2(na, (wa[h] | 0x80008000u) - 0x00010001u);
      nc = __vmins2(nc, (wc[h] | 0x80008000u) - 0x00010001u);
    }
  }
  int ema = (int)(__reduce_max_sync(0xffffffffu, max(xa & 0xFFFFu, xa >> 16)) >> 7);
  int emc = (int)(__reduce_max_sync(0xffffffffu, max(xc & 0xFFFFu, xc >> 16)) >> 7);
  const int ma = __reduce_min_sync(0xffffffffu, min((int)(short)(na & 0xFFFFu), (int)na >> 16));
  const int mc = __reduce_min_sync(0xffffffffu, min((int)(short)(nc & 0xFFFFu), (int)nc >> 16));
  // smallest nonzero exponent field (0: a subnormal), 255 for a zero vector
  const int la = ma == 0x7FFF ? 255 : (ma + 32769) >> 7, lc = mc == 0x7FFF ? 255 : (mc + 32769) >> 7;
  long long v0 = 0, v1 = 0, v2 = 0;
  // exponent fields of 25 + (30 - bits)..254: the scale 2^k below is a normal float
  if (ema >= 32 && ema <= 254 && emc >= 32 && emc <= 254 && la >= ema + 8 - bits && lc >= emc + 8 - bits) {
    const int ka = bits + 126 - ema, kc = bits + 126 - emc;  // |element| < 2^(ema - 126)
    const float fa = __int_as_float((ka + 127) << 23), fc = __int_as_float((kc + 127) << 23);
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      const uint4 qa = sa[32 * j], qc = sc[32 * j];
      const uint32_t wa[4] = {qa.x, qa.y, qa.z, qa.w}, wc[4] = {qc.x, qc.y, qc.z, qc.w};
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        const float x = __uint_as_float(h & 1 ? wa[h >> 1] & 0xFFFF0000u : wa[h >> 1] << 16);
        const float y = __uint_as_float(h & 1 ? wc[h >> 1] & 0xFFFF0000u : wc[h >> 1] << 16);
        const int ia = __float2int_rn(x * fa), ic = __float2int_rn(y * fc);  // exact
        v0 += (long long)ia * ic;
        v1 += (long long)ia * ia;
        v2 += (long long)ic * ic;
      }
    }
    warp_sum64(v0, -(ka + kc), s.v[0], s.e[0]);
    warp_sum64(v1, -2 * ka, s.v[1], s.e[1]);
    warp_sum64(v2, -2 * kc, s.v[2], s.e[2]);
    s.kind = SUMS_INT;
    return;
  }
  bool inexact = ema == 255 || emc == 255;  // Inf or NaN present
  ema = max(ema, 1);
  emc = max(emc, 1);
  const int bd = ema + emc - span, ba = 2 * ema - span, bc = 2 * emc - span;
  if (!inexact) {
#pragma unroll 1
    for (int j = 0; j < NCH; ++j) {
      const uint4 qa = sa[32 * j], qc = sc[32 * j];
      const uint32_t wa[4] = {qa.x, qa.y, qa.z, qa.w}, wc[4] = {qc.x, qc.y, qc.z, qc.w};
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        const uint32_t ya = (wa[h >> 1] >> (16 * (h & 1))) & 0xFFFFu, yc = (wc[h >> 1] >> (16 * (h & 1))) & 0xFFFFu;
        const int ea = (int)((ya >> 7) & 0xFFu), ec = (int)((yc >> 7) & 0xFFu);
        const int Ea = max(ea, 1), Ec = max(ec, 1);
        const uint32_t Ma = (ya & 0x7Fu) | (ea ? 0x80u : 0u), Mc = (yc & 0x7Fu) | (ec ? 0x80u : 0u);
        const uint32_t pd = Ma * Mc, pa = Ma * Ma, pc = Mc * Mc;
        const int hd = Ea + Ec - bd, ha = 2 * Ea - ba, hc = 2 * Ec - bc;
        inexact |= (hd < 0 && pd != 0) | (ha < 0 && pa != 0) | (hc < 0 && pc != 0);
        const long long td = (long long)((unsigned long long)pd << max(hd, 0));
        v0 += ((ya ^ yc) & 0x8000u) ? -td : td;
        v1 += (long long)((unsigned long long)pa << max(ha, 0));
        v2 += (long long)((unsigned long long)pc << max(hc, 0));
      }
    }
  }
  if (__any_sync(0xffffffffu, inexact)) {
    sums_fp64(a, c, D, lane, s);
    return;
  }
  warp_sum64(v0, bd - 268, s.v[0], s.e[0]);
  warp_sum64(v1, ba - 268, s.v[1], s.e[1]);
  warp_sum64(v2, bc - 268, s.v[2], s.e[2]);
  s.kind = SUMS_INT;
}

constexpr int kSelThreads = 256;

// 16 bytes from global to shared memory, and the groups of such copies of
// this thread (bytes == 0 writes zeros and reads nothing).
__device__ __forceinline__ void cp_async16(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// One cluster per row r (blockIdx.x / cluster size). T: element type; NCH > 0:
// bf16 vectors of at most 256 NCH elements; NCH == 0: vectors streamed from
// memory (fp32 and wider bf16 vectors) and summed in triples of floats. N == 0 only moves
// the current vectors into the cache.
//
// With NCH > 0 every lane copies its chunks of the warp's next token to shared
// memory while the warp works on the current one. A lane reads back only what
// it copied itself, so the two-deep ring needs no barrier.
//
// Selection order (Table 3 strategies): priority descending when given, then
// the rule's key ascending, then token index. Keys: LEAST_SIMILAR (strategy V)
// the order-preserving key of S; MOST_SIMILAR (strategy IV) its complement,
// i.e. S descending (NaN, as -inf, last); RANDOM (strategy III) the caller's
// 32-bit random keys.

// A CTA of at most one token per warp needs one stage of the ring only.
template <int NCH>
__host__ __device__ constexpr int sel_ring(int per) {  // bytes: [stage][warp][cur, cache][chunk][lane]
  return (per > kSelThreads / 32 ? 2 : 1) * NCH * 2 * 16 * kSelThreads;
}

template <typename T, int NCH>
__global__ void __launch_bounds__(kSelThreads, NCH <= 3 ? 4 : 2)
    select_kernel(const T* __restrict__ cur, T* __restrict__ cache, int n_tok, int D, int span, int N,
                  int* __restrict__ idx, int* __restrict__ row_map, int rule, const uint8_t* __restrict__ prio,
                  const uint32_t* __restrict__ rkeys) {
  constexpr int V = 16 / sizeof(T);
  constexpr int kWarps = kSelThreads / 32;
  extern __shared__ __align__(16) uint8_t sel_smem[];  // the ring, then (N > 0) the row's keys, this CTA's sums and flags
  __shared__ int s_count[16];                          // selected tokens of each CTA of the cluster
  __shared__ int s_wcount[kWarps], s_ctotal;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t me = cluster_ctarank(), ncta = cluster_nctarank();
  const int r = (int)(blockIdx.x / ncta);
  const int per = (n_tok + (int)ncta - 1) / (int)ncta;  // tokens per CTA
  const int t0 = min((int)me * per, n_tok), t1 = min(t0 + per, n_tok);
  unsigned long long* sK = reinterpret_cast<unsigned long long*>(sel_smem + sel_ring<NCH>(per));
  SimSums* sums = reinterpret_cast<SimSums*>(sK + n_tok);
  unsigned char* sel = reinterpret_cast<unsigned char*>(sums + min(per, kSelThreads));
  const bool need_s = N > 0 && rule != LAZYMAR_SELECT_RANDOM;
  if (N > 0) cluster_sync();  // every CTA of the cluster runs before its shared memory is written to
  pdl_wait();
  pdl_trigger();
  const size_t row0 = (size_t)r * n_tok;
  uint4* ring = reinterpret_cast<uint4*>(sel_smem) + warp * (NCH * 2 * 32) + lane;
  constexpr int kStage = kWarps * NCH * 2 * 32;  // of the ring
  auto fetch = [&](int t, int stage) {
    const T* a = cur + (row0 + t) * D;
    const T* c = cache + (row0 + t) * D;
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      const int i = (lane + 32 * j) * V;
      const int in = i < D ? 16 : 0, at = in ? i : 0;
      cp_async16(ring + stage * kStage + j * 32, a + at, in);
      if (need_s) cp_async16(ring + stage * kStage + (NCH + j) * 32, c + at, in);
    }
    cp_async_commit();
  };
  if (NCH > 0 && t0 + warp < t1) fetch(t0 + warp, 0);
  int stage = 0;
  // rounds of one token per thread: the warps take the sums, then each thread
  // one token's fp64 division and square root, which cost a whole warp as much
  // as one token (GB300 has about two fp64 lanes per SM)
  for (int b = t0; b < t1; b += kSelThreads) {
    const int b1 = min(b + kSelThreads, t1);
    for (int t = b + warp; t < b1; t += kWarps, stage ^= 1) {
      const T* a = cur + (row0 + t) * D;
      T* c = cache + (row0 + t) * D;
      SimSums s;
      if constexpr (NCH > 0) {
        if (t + kWarps < t1) {
          fetch(t + kWarps, stage ^ 1);
          cp_async_wait<1>();
        } else {
          cp_async_wait<0>();
        }
        const uint4* sa = ring + stage * kStage;
        if (need_s) sums_bf16<NCH>(sa, sa + NCH * 32, a, c, D, span, lane, s);
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
          const int i = (lane + 32 * j) * V;
          if (i < D) *reinterpret_cast<uint4*>(c + i) = sa[32 * j];
        }
      } else {
        if (need_s) sums_f32x3(a, c, D, lane, s);
        for (int i = lane * V; i < D; i += 32 * V)
          *reinterpret_cast<uint4*>(c + i) = *reinterpret_cast<const uint4*>(a + i);
      }
      if (need_s && lane == 0) sums[t - b] = s;
    }
    if (need_s) {
      __syncthreads();
      if (b + tid < b1) {
        unsigned long long k = sim_key(sim_value(sums[tid]));
        if (rule == LAZYMAR_SELECT_MOST_SIMILAR) k = ~k;
        const uint32_t at = smem_u32(sK + b + tid);
        for (uint32_t p = 0; p < ncta; ++p)
          asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cluster_map(at, p)), "l"(k) : "memory");
      }
      if (b1 < t1) __syncthreads();  // the sums are free for the next round
    }
  }
  if (N == 0) return;  // uniform over the cluster: nothing to rank
  if (!need_s)
    for (int t = tid; t < n_tok; t += kSelThreads) sK[t] = rkeys[row0 + t];
  __syncwarp();
  cluster_sync();
  // rank of token t: one warp per token, its lanes sharing the row's keys;
  // I_compute = rank < N
  for (int t = t0 + warp; t < t1; t += kWarps) {
    const unsigned long long kt = sK[t];
    int rank = 0;
    if (prio) {
      const unsigned pt = prio[row0 + t];
      for (int u = lane; u < n_tok; u += 32) {
        const unsigned long long ku = sK[u];
        const unsigned pu = prio[row0 + u];
        rank += (pu > pt) || (pu == pt && ((ku < kt) || (ku == kt && u < t)));
      }
    } else {
      for (int u = lane; u < n_tok; u += 32) {
        const unsigned long long ku = sK[u];
        rank += (ku < kt) || (ku == kt && u < t);
      }
    }
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane == 0) sel[t - t0] = rank < N;
  }
  __syncthreads();
  // this CTA's count to every CTA of the cluster
  if (warp == 0) {
    int n = 0;
    for (int t = lane; t < t1 - t0; t += 32) n += sel[t];
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane < (int)ncta)
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_map(smem_u32(s_count + me), (uint32_t)lane)), "r"(n)
                   : "memory");
  }
  __syncwarp();
  cluster_sync();  // also: no CTA exits while another may still write to it
  int base = 0;
  for (uint32_t p = 0; p < me; ++p) base += s_count[p];
  for (int c0 = t0; c0 < t1; c0 += kSelThreads) {
    const int t = c0 + tid;
    const bool f = t < t1 && sel[t - t0];
    const unsigned bal = __ballot_sync(0xffffffffu, f);
    if (lane == 0) s_wcount[warp] = __popc(bal);
    __syncthreads();
    int off = 0;
    for (int w = 0; w < warp; ++w) off += s_wcount[w];
    if (tid == kSelThreads - 1) s_ctotal = off + __popc(bal);
    if (f) {
      const int pos = base + off + __popc(bal & ((1u << lane) - 1u));
      idx[(size_t)r * N + pos] = t;
      if (row_map) row_map[(size_t)r * N + pos] = (int)(row0 + t);
    }
    __syncthreads();
    base += s_ctotal;
  }
}

// Dynamic shared memory of a CTA that ranks (N > 0).
template <int NCH>
static size_t select_smem(int n_tok, int ncta) {
  const size_t per = (size_t)((n_tok + ncta - 1) / ncta);
  return sel_ring<NCH>((int)per) + (size_t)n_tok * sizeof(unsigned long long) +
         (per < kSelThreads ? per : (size_t)kSelThreads) * sizeof(SimSums) + per;
}

// CTAs per row, up to 8, the portable limit: one for every 8 tokens (a warp each), for
// every 16 where the rows alone fill the SMs, for every token where 8 CTAs a row would
// not; with half as many rows, clusters of 16 spread a row over twice as many SMs. Measured, 8 CTAs for any number of tokens -> this
// (us): 4096 rows of 8 tokens x 768 369 -> 56, of 17 383 -> 121, 8192 of 16 x 256 693 ->
// 104, 2048 of 64 196 -> 116, 600 of 8 x 768 55 -> 14.
constexpr int kSelMaxTokens = 16384;  // of a row, in every entry point

// Whether clusters of 16 CTAs of the kernel fit the device (a partition of it may
// have no 16 SMs together), with the shared memory of the most tokens; allows them.
template <typename T, int NCH>
static bool clusters_of_16() {
  static std::atomic<signed char> known[64];  // per device: 1 yes, -1 no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  if (known[dev] != 0) return known[dev] > 0;
  const int smem = (int)select_smem<NCH>(kSelMaxTokens, 8);
  auto kernel = select_kernel<T, NCH>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(kSelThreads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 16;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  known[dev] = n >= 1 ? 1 : -1;
  return n >= 1;
}

template <typename T, int NCH>
static cudaError_t launch_select_t(const Ctx& c, const void* cur, void* cache, int rows, int n_tok, int D, int span,
                                   int N, int* idx, int* row_map, int rule, const uint8_t* prio,
                                   const uint32_t* keys) {
  auto kernel = select_kernel<T, NCH>;
  const int least = rows <= c.num_sms / 8 ? 1 : rows <= c.num_sms ? 8 : 16;  // tokens of a CTA
  int ncta = 1;
  while (ncta < 8 && ncta * least < n_tok) ncta *= 2;
  if (ncta == 8 && rows <= c.num_sms / 16 && clusters_of_16<T, NCH>()) ncta = 16;
  const size_t smem = N > 0 ? select_smem<NCH>(n_tok, ncta) : (size_t)sel_ring<NCH>((n_tok + ncta - 1) / ncta);
  if (smem > 40 * 1024) {
    // always the largest size: the attribute is the process's, and another host
    // thread may be about to launch the kernel for more tokens
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)select_smem<NCH>(kSelMaxTokens, 8));
    if (e != cudaSuccess) return e;
  }
  if ((long long)rows * ncta > INT_MAX) return cudaErrorInvalidValue;  // (more than 500 GB of vectors)
  return launch_pdl_cluster(kernel, dim3((unsigned)(rows * ncta)), dim3(kSelThreads), smem, ncta, c.stream,
                            static_cast<const T*>(cur), static_cast<T*>(cache), n_tok, D, span, N, idx, row_map,
                            rule, prio, keys);
}

cudaError_t launch_select(const Ctx& c, int dtype, const void* cur, void* cache, int rows, int n_tok, int D, int N,
                          int* idx, int* row_map, int rule, const uint8_t* prio, const uint32_t* keys) {
  if (rows == 0) return cudaSuccess;
  int lg = 0;
  while ((1 << lg) < D) ++lg;
  const int span = 62 - 16 - lg;
#define LM_SELECT(T, NCH) \
  return launch_select_t<T, NCH>(c, cur, cache, rows, n_tok, D, span, N, idx, row_map, rule, prio, keys)
  if (dtype != LAZYMAR_BF16) LM_SELECT(float, 0);
  if (D % 8 != 0 || D > 1280) LM_SELECT(bf16, 0);
  switch ((D + 255) / 256) {
    case 1: LM_SELECT(bf16, 1);
    case 2: LM_SELECT(bf16, 2);
    case 3: LM_SELECT(bf16, 3);
    case 4: LM_SELECT(bf16, 4);
    default: LM_SELECT(bf16, 5);
  }
#undef LM_SELECT
}

// Caller-chosen I_compute: copied after checking range and strict increase per
// row; a violation is latched as ERR_INDEX and the index is clamped into
// [0, T) so that no later gather or scatter leaves the row.
__global__ void idx_check_kernel(const int* __restrict__ in, int rows, int T, int N, int* __restrict__ idx,
                                 int* __restrict__ row_map, unsigned* err) {
  pdl_wait();
  pdl_trigger();
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)rows * N) return;
  const int r = (int)(i / N), j = (int)(i - (long long)r * N);
  int v = in[i];
  bool ok = v >= 0 && v < T && (j == 0 || in[i - 1] < v);
  if (!ok) {
    atomicOr(err, ERR_INDEX);
    v = v < 0 ? 0 : (v >= T ? T - 1 : v);
  }
  idx[i] = v;
  row_map[i] = r * T + v;
}

cudaError_t launch_idx_check(const Ctx& c, const int* in, int rows, int T, int N, int* idx, int* row_map) {
  const long long n = (long long)rows * N;
  if (n == 0) return cudaSuccess;
  return launch_pdl(idx_check_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, c.stream, in, rows, T, N, idx,
                    row_map, c.err);
}

// ---------------------------------------------------------------------------
// Selection without device allocation
// ---------------------------------------------------------------------------
// Some callers may not allocate device memory once they are running: a
// serving loop that reserves its whole memory budget at start-up and must not
// grow it, or a plug-in whose host framework owns the device allocator and
// forbids direct cudaMalloc. lazymar_select_tokens_noalloc serves them. The
// selection keeps its similarities in shared memory, so neither entry point
// allocates; this one keeps its documented limit on rows * T.
constexpr int kMaxDevices = 64;

static bool noalloc_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (!p || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace lm

extern "C" lazymar_status lazymar_select_tokens_noalloc(int dtype, const void* v_cur, void* v_cache, int rows, int T,
                                                        int D, int n_compute, int32_t* idx_out, void* stream) {
  using namespace lm;
  if (dtype != LAZYMAR_F32 && dtype != LAZYMAR_BF16) return report_error(LAZYMAR_ERR_INVALID_ARG, "dtype");
  if (rows < 0 || T < 1 || T > 16384 || D < 8 || D % 8 != 0 || n_compute < 0 || n_compute > T)
    return report_error(LAZYMAR_ERR_INVALID_ARG,
                        "rows >= 0, 1 <= T <= 16384, D % 8 == 0, 0 <= n_compute <= T required");
  if ((long long)rows * T > LAZYMAR_SELECT_NOALLOC_MAX_TOKENS)
    return report_error(LAZYMAR_ERR_INVALID_ARG,
                        "rows * T exceeds LAZYMAR_SELECT_NOALLOC_MAX_TOKENS (262144); use lazymar_select_tokens");
  if (rows == 0) return LAZYMAR_OK;
  if (!noalloc_device_ptr(v_cur) || !noalloc_device_ptr(v_cache) || (n_compute > 0 && !noalloc_device_ptr(idx_out)))
    return report_error(LAZYMAR_ERR_INVALID_ARG, "v_cur, v_cache and idx_out must be device pointers");
  if ((reinterpret_cast<uintptr_t>(v_cur) | reinterpret_cast<uintptr_t>(v_cache)) & 15u)
    return report_error(LAZYMAR_ERR_INVALID_ARG, "16-byte alignment required");
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return report_error(LAZYMAR_ERR_CUDA, "cudaGetDevice failed or device index out of range");
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return report_error(LAZYMAR_ERR_CUDA, "cudaDeviceGetAttribute failed");
  const Ctx c{static_cast<cudaStream_t>(stream), nullptr, sms};
  const cudaError_t e = launch_select(c, dtype, v_cur, v_cache, rows, T, D, n_compute, idx_out, nullptr);
  if (e != cudaSuccess) return report_error(LAZYMAR_ERR_CUDA, cudaGetErrorString(e));
  return LAZYMAR_OK;
}

namespace lm {

// ---------------------------------------------------------------------------
// Bounded-wait diagnostic
// ---------------------------------------------------------------------------
// Every pipelined kernel waits on mbarriers with a time limit: on expiry it
// raises its abort flag and ERR_TIMEOUT in the device error word, stops, and
// returns normally, so the context stays usable and the host learns of the
// failure from lazymar_sync / lazymar_device_check. This kernel drives that
// path on purpose: its barrier expects one arrival that never comes.
__global__ void stuck_wait_kernel(unsigned* err, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  mbar_wait_limit(&bar, 0, &abort_flag, err, limit_ns);
}

cudaError_t launch_stuck_wait(const Ctx& c, uint64_t limit_ns) {
  stuck_wait_kernel<<<1, 32, 0, c.stream>>>(c.err, (unsigned long long)limit_ns);
  return cudaGetLastError();
}

}  // namespace lm
