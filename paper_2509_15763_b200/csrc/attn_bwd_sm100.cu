// Backward gist-masked attention on Blackwell tensor cores (tcgen05 + TMEM + TMA) on the SHIFTED sequence
// [sinks (s) | raw (T) | gists (n)]; a tile never straddles two of these segments.
//   bwd_prep_kernel            Delta = rowsum(dO o O) (fp32) and, for an fp32 dO, its bf16 copy; zeroes the fp32
//                              dQ accumulator of the fused kernel.
// head_dim 128: attn_bwd_fused_sm100_kernel (described where it is defined) and dq_convert_kernel.
// head_dim 64: two kernels (a 64-row dQ^T accumulator would halve the fused kernel's tensor throughput):
//   attn_bwd_dkdv_sm100_kernel one thread block owns a 128-key tile of one KV head (where a walk would be the tail, two
//                              blocks of a cluster share a sink or gist key tile) and walks every
//                              128-query tile of every query head of the group that can see it:
//                              S^T = K Q^T and dP^T = V dO^T (TMEM), P^T = exp2(S^T c - LSE),
//                              dS^T = P^T o (dP^T - Delta), dV += P^T dO, dK += dS^T Q.  dK and dV
//                              live in TMEM for the whole block: no atomics, deterministic.
//   attn_bwd_dq_sm100_kernel   beside the tail of the other: one thread block owns a 128-query tile of one query head and walks
//                              the visible 64-key tiles: S, dP, dS as above, dQ += dS K in TMEM.
// Tiles without a visible pair are never loaded; only "partial" tiles evaluate the mask.
#include <algorithm>
#include <vector>

#include "sm100_ptx.cuh"
#include "ug_common.cuh"

namespace ug {
namespace {

using namespace sm100;

constexpr float kLog2e = 1.4426950408889634f;
__device__ unsigned int g_bwd_timeout = 0;

// ------------------------------------------------------------------------------------------------
// A run of equal sequences as the per-token kernels see it: its geometry, its first packed token and its
// [batch, Hq, N] block of Delta.  One problem is one run; a packed sample (cross-document masking) has several
// and a warp finds its token's run by scanning the (at most twelve) first-token indices.
struct TokRun {
  Geom g;
  GeomDiv div;
  long long tok_begin;
  float* delta;
};
TokRun make_tok_run(const Geom& g, long long tok_begin, float* delta) {
  return {g, make_geom_div(g), tok_begin, delta};
}
template <int kRuns>
struct TokRuns {
  TokRun run[kRuns];
  int n;
};


// Delta and dO conversion: one warp per token.  Bound by HBM: reads dO and O, writes zeros for the dQ accumulator, which
// is 8 bytes an element in all.  The token's batch index and shifted position are worked out once, by multiplication;
// its Hq rows then go by in 16-byte pieces, D / 8 lanes to a row, kSteps rows (times the rows a warp covers at once) of dO
// and O in flight before the first use.
template <bool kF32, int kRuns, int D>
__global__ void __launch_bounds__(256)
bwd_prep_kernel(const __grid_constant__ TokRuns<kRuns> P, int interleaved, int Hq, int tokens, const void* __restrict__ d_o,
                const __nv_bfloat16* __restrict__ o, __nv_bfloat16* __restrict__ d_o_bf16, float* __restrict__ dq32) {
  pdl_wait();
  constexpr int kLanes = D / 8, kRows = 32 / kLanes, kSteps = 4;  // lanes of a row, rows of a warp access
  const int lane = threadIdx.x & 31, sub = lane / kLanes, col = (lane % kLanes) * 8;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
  for (long long tk = warp; tk < tokens; tk += nwarps) {  // tk = packed token index (run's first token + b * N + t)
    int ri = 0;
    if constexpr (kRuns > 1)
      while (ri + 1 < P.n && tk >= P.run[ri + 1].tok_begin) ++ri;
    const TokRun& R = P.run[ri];
    const int N = R.g.N, local = (int)(tk - R.tok_begin);
    const int b = fdiv(R.div.n, local), t = local - b * N;
    // Delta is kept in shifted order, whatever the order of dO and O
    float* delta_tok = R.delta + (long long)b * Hq * N + (interleaved ? unshift_perm(R.g, R.div, t) : t);
    const long long row0 = tk * Hq;
    for (int h0 = 0; h0 < Hq; h0 += kRows * kSteps) {
      uint4 db[kSteps], ob[kSteps];  // 8 bf16 of dO and of O
#pragma unroll
      for (int u = 0; u < kSteps; ++u) {
        const int h = h0 + u * kRows + sub;
        if (h >= Hq) continue;
        const long long at = (row0 + h) * D + col;
        if (kF32) {
          const float4 x = __ldcs(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(d_o) + at));
          const float4 y = __ldcs(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(d_o) + at) + 1);
          db[u] = make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w), pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
        } else {
          db[u] = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(d_o) + at);
        }
        ob[u] = *reinterpret_cast<const uint4*>(o + at);
      }
      // the fused backward accumulates dQ into this fp32 buffer: start it at zero
      if (dq32) {
        const int n4 = min(kRows * kSteps, Hq - h0) * (D / 4);
        float4* z = reinterpret_cast<float4*>(dq32 + (row0 + h0) * D);
#pragma unroll
        for (int i = 0; i < kRows * kSteps * (D / 4) / 32; ++i)
          if (i * 32 + lane < n4) __stcs(z + i * 32 + lane, make_float4(0.f, 0.f, 0.f, 0.f));
      }
#pragma unroll
      for (int u = 0; u < kSteps; ++u) {
        const int h = h0 + u * kRows + sub;
        float acc = 0.f;
        if (h < Hq) {
          if (kF32) *reinterpret_cast<uint4*>(d_o_bf16 + (row0 + h) * D + col) = db[u];
          const uint32_t x[4] = {db[u].x, db[u].y, db[u].z, db[u].w}, y[4] = {ob[u].x, ob[u].y, ob[u].z, ob[u].w};
#pragma unroll
          for (int e = 0; e < 4; ++e)  // a bf16 is the high half of an fp32
            acc += __uint_as_float(x[e] << 16) * __uint_as_float(y[e] << 16) +
                   __uint_as_float(x[e] & 0xffff0000u) * __uint_as_float(y[e] & 0xffff0000u);
        }
#pragma unroll
        for (int off = kLanes / 2; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (h < Hq && lane % kLanes == 0) delta_tok[(long long)h * N] = acc;
      }
    }
  }
}

// Query rows (numbered inside the raw or the gist segment, inclusive) that see a given key:
// Eq. 3 read column-wise.  An empty interval has lo > hi.
__host__ __device__ __forceinline__ void key_q_interval(const Geom& g, const FastDiv& rdiv, bool key_is_raw, int key, bool key_valid,
                                               bool q_is_raw, int& lo, int& hi) {
  if (!key_valid) {
    lo = 1;
    hi = 0;
    return;
  }
  if (key_is_raw) {
    const int u = fdiv(rdiv, key);
    if (q_is_raw) {
      lo = key;
      hi = min(g.T - 1, (u + g.k + 1) * g.r - 1);
    } else {
      lo = u;
      hi = min(g.n - 1, u + g.k);
    }
  } else {
    if (q_is_raw) {
      lo = (key + 1) * g.r;
      hi = g.T - 1;
    } else {
      lo = key;
      hi = g.n - 1;
    }
  }
}

// Query rows of segment qseg (numbered inside it, inclusive) that see key `key` of segment kseg:
// Eq. 3 read column-wise, sinks included.  An empty interval has lo > hi.
__host__ __device__ __forceinline__ void key_q_interval3(const Geom& g, const FastDiv& rdiv, int kseg, int key, bool key_valid, int qseg, int& lo,
                                                int& hi) {
  lo = 1;
  hi = 0;
  if (!key_valid) return;
  if (kseg == kSegSink) {  // a sink is seen by the sinks from itself on and by every raw and gist query
    lo = qseg == kSegSink ? key : 0;
    hi = seg_len(g, qseg) - 1;
    return;
  }
  if (qseg == kSegSink) return;  // sink queries see sinks only
  key_q_interval(g, rdiv, kseg == kSegRaw, key, true, qseg == kSegRaw, lo, hi);
}

// One 32-query chunk of P^T for one key: p = 2^(s * c + nl[q]), nl = -LSE in log2 units; kMasked: bit e of `bits` says
// query e sees the key.  Two queries at a time (packed fp32).
template <bool kMasked>
__device__ __forceinline__ void p_chunk(const uint32_t (&v)[32], const float* __restrict__ nl, uint64_t scale2, uint32_t bits,
                                        float* __restrict__ p, uint32_t (&pk)[16]) {
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    const ulonglong2 l4 = *reinterpret_cast<const ulonglong2*>(nl + i);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = i + 2 * h;
      float x0, x1;
      f32x2_split(fma2(f32x2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])), scale2, h ? l4.y : l4.x), x0, x1);
      if (kMasked) {
        x0 = (bits >> e) & 1u ? x0 : -INFINITY;
        x1 = (bits >> (e + 1)) & 1u ? x1 : -INFINITY;
      }
      p[e] = ex2(x0);
      p[e + 1] = ex2(x1);
      pk[e / 2] = pack_bf16(p[e], p[e + 1]);
    }
  }
}
// dS = p (dP - Delta) of two neighbours, rounded to bf16; nd = -Delta of both.
__device__ __forceinline__ uint32_t ds_pair(float p0, float p1, uint32_t dp0, uint32_t dp1, uint64_t nd) {
  float x0, x1;
  f32x2_split(mul2(f32x2(p0, p1), add2(f32x2(__uint_as_float(dp0), __uint_as_float(dp1)), nd)), x0, x1);
  return pack_bf16(x0, x1);
}
// Bit e: column e of 32 lies inside [lo, hi].
__device__ __forceinline__ uint32_t piece_bits(int lo, int hi) {
  const int a = max(lo, 0), b = min(hi, 31);
  return a > b ? 0u : ((0xffffffffu >> (31 - b)) & (0xffffffffu << a));
}

// ------------------------------------------------------------------------------------------------
// dK / dV kernel.  Bound by the chain scores -> P -> dP -> dS of one step, not by the tensor pipe: with head_dim 64
// tensor memory has room for a second S buffer and shared memory for four Q / dO stages, which take the scores and the
// loads off that chain (two sequences of 8190 raw tokens, ratio 7, 16 / 4 heads: 0.70 -> 0.45 ms, heavy tiles first over
// all heads included); shared heavy tiles, 16 compute warps and packed arithmetic brought it to 0.32.
constexpr int KV_BM = 128;       // keys per block (TMEM lanes)
constexpr int KV_BN = 128;       // queries per step
// 16 compute warps (four per TMEM lane quarter, 32 query columns each: half the columns per thread shorten the chain of a
// step), 1 TMA warp, 1 MMA warp
constexpr int kKvCompute = 16, kKvThreads = (kKvCompute + 2) * 32;

template <int D>
struct KvSmem {
  static constexpr int kSlab = 128 * 128;
  static constexpr int kTile = kSlab * (D / 64);
  static constexpr int kStages = D == 64 ? 4 : 2;              // of Q, dO, LSE and Delta
  static constexpr int kSBufs = D == 64 ? 2 : 1;               // buffers of S^T / P^T in tensor memory
  static constexpr int kOffStats = (2 + 2 * kStages) * kTile;  // [stage][lse2 | delta][128] fp32
  static constexpr int kOffBars = kOffStats + kStages * 2 * KV_BN * 4;
  static constexpr int kBytes = kOffBars + 256 + 1024;
};

template <int D>
__global__ void __launch_bounds__(kKvThreads, 1)
attn_bwd_dkdv_sm100_kernel(const __grid_constant__ CUtensorMap tm_q_sink, const __grid_constant__ CUtensorMap tm_q_raw,
                           const __grid_constant__ CUtensorMap tm_q_gist, const __grid_constant__ CUtensorMap tm_do_sink,
                           const __grid_constant__ CUtensorMap tm_do_raw, const __grid_constant__ CUtensorMap tm_do_gist,
                           const __grid_constant__ CUtensorMap tm_k_sink, const __grid_constant__ CUtensorMap tm_k_raw,
                           const __grid_constant__ CUtensorMap tm_k_gist, const __grid_constant__ CUtensorMap tm_v_sink,
                           const __grid_constant__ CUtensorMap tm_v_raw, const __grid_constant__ CUtensorMap tm_v_gist,
                           Geom g, int Hq, int Hkv, float scale, const float* __restrict__ lse,
                           const float* __restrict__ delta, __nv_bfloat16* __restrict__ dk,
                           __nv_bfloat16* __restrict__ dv, int n_sink_kt, int n_gist_kt, int n_raw_kt, int pairs, int shared,
                           FastDiv heavy_div, FastDiv raw_div, FastDiv hkv_div, FastDiv rdiv) {
  using SM = KvSmem<D>;
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* gen = smem_dyn + (base - smem_u32(smem_dyn));
  const uint32_t sK = base, sV = base + SM::kTile;
  constexpr int kSt = SM::kStages;
  const uint32_t sQ0 = base + 2 * SM::kTile, sDO0 = sQ0 + kSt * SM::kTile;  // stage st at + st * kTile
  float* stats = reinterpret_cast<float*>(gen + SM::kOffStats);             // [stage][2][128]
  const uint32_t bars = base + SM::kOffBars;
  // (two barriers per S buffer: a buffer's next phase cannot complete before everyone has seen the one before)
  const uint32_t bar_kv = bars, bar_S = bars + 8 /* + 8 * buffer */, bar_dP = bars + 24,
                 bar_P = bars + 32 /* + 8 * buffer */, bar_dS = bars + 48, bar_final = bars + 56, tmem_slot = bars + 64;
  const uint32_t bar_full = bars + 72, bar_empty = bars + 72 + 8 * kSt;  // + 8 * stage
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(gen + SM::kOffBars + 64);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = Hq / Hkv;
  // Sink and gist key tiles are seen by every later query: heaviest, and first over ALL heads and batch indices (a long walk
  // that starts late is the kernel's tail).  Where even that leaves a long walk as the tail (dkdv_shares), blocks come in
  // clusters of two: they share ONE such key tile, each walks half of its queries, and they add their dK and dV through
  // distributed shared memory; of the raw key tiles either block of a cluster takes one of its own.  The tiles of one KV
  // head are neighbours and share its Q and dO.
  const int n_heavy = n_sink_kt + n_gist_kt, crank = shared ? blockIdx.x & 1 : 0, unit = blockIdx.x >> shared;
  const bool split = shared && unit < n_heavy * pairs;
  int pair, rank;  // pair = batch index * Hkv + KV head
  if (unit < n_heavy * pairs) {
    pair = fdiv(heavy_div, unit);
    rank = unit - pair * n_heavy;
  } else {
    const int y = unit - n_heavy * pairs;
    pair = fdiv(raw_div, y);
    rank = n_heavy + ((y - pair * ((n_raw_kt + shared) >> shared)) << shared) + crank;
    if (rank >= n_heavy + n_raw_kt) return;  // an odd number of raw key tiles (its cluster never meets)
  }
  const int b = fdiv(hkv_div, pair), hk = pair - b * Hkv;
  const int kseg = rank < n_sink_kt ? kSegSink : (rank < n_heavy ? kSegGist : kSegRaw);
  const int kt = rank - (kseg == kSegSink ? 0 : (kseg == kSegGist ? n_sink_kt : n_heavy));
  const int key_seg_len = seg_len(g, kseg);
  const int key_seg_base = seg_base(g, kseg);
  const int key_a = kt * KV_BM, key_b = min(key_a + KV_BM - 1, key_seg_len - 1);
  const bool key_tile_whole = key_a + KV_BM - 1 <= key_seg_len - 1;

  // query tiles that see this key tile, per query segment: first tile and count, and the bounds inside which a
  // tile is "full" (seen by the last key from t_lo on, by the first key up to t_hi)
  int lo_a, hi_a, lo_b, hi_b;
  key_q_interval3(g, rdiv, kseg, key_a, true, kSegRaw, lo_a, hi_a);
  key_q_interval3(g, rdiv, kseg, key_b, true, kSegRaw, lo_b, hi_b);
  const int n_raw_q = hi_b >= lo_a ? hi_b / KV_BN - lo_a / KV_BN + 1 : 0, rq_lo = lo_a / KV_BN, raw_t_lo = lo_b, raw_t_hi = hi_a;
  key_q_interval3(g, rdiv, kseg, key_a, true, kSegGist, lo_a, hi_a);
  key_q_interval3(g, rdiv, kseg, key_b, true, kSegGist, lo_b, hi_b);
  const int n_gist_q = hi_b >= lo_a ? hi_b / KV_BN - lo_a / KV_BN + 1 : 0, gq_lo = lo_a / KV_BN, gist_t_lo = lo_b, gist_t_hi = hi_a;
  key_q_interval3(g, rdiv, kseg, key_a, true, kSegSink, lo_a, hi_a);
  key_q_interval3(g, rdiv, kseg, key_b, true, kSegSink, lo_b, hi_b);
  const int n_sink_q = hi_b >= lo_a ? hi_b / KV_BN - lo_a / KV_BN + 1 : 0, sq_lo = lo_a / KV_BN, sink_t_lo = lo_b, sink_t_hi = hi_a;
  // this block's part of the walk: query tiles [t_begin, t_end) in the order of the steps below
  const int n_tiles = n_raw_q + n_gist_q + n_sink_q, t_half = (n_tiles + 1) / 2;
  const int t_begin = split && crank ? t_half : 0, t_end = split && !crank ? t_half : n_tiles;
  const int n_iter = (t_end - t_begin) * G;

  if (threadIdx.x == 0) {
    mbar_init(bar_kv, 1);
    for (int i = 0; i < kSt; ++i) {
      mbar_init(bar_full + 8 * i, 1);
      mbar_init(bar_empty + 8 * i, 1);
    }
    mbar_init(bar_S, 1);
    mbar_init(bar_S + 8, 1);
    mbar_init(bar_dP, 1);
    mbar_init(bar_P, kKvCompute);
    mbar_init(bar_P + 8, kKvCompute);
    mbar_init(bar_dS, kKvCompute);
    mbar_init(bar_final, 1);
    mbar_fence_init();
  }
  if (warp == kKvCompute + 1) tmem_alloc(tmem_slot, 512);
  pdl_wait();
  // The dQ kernel reads nothing that this one writes: its blocks take the SMs that this one's tail leaves idle, or never used
  // (backward of 2 x 8190 raw tokens, ratio 7, 16 / 4 heads: 581 -> 560 us; of 1 x 448, one head: 22.5 -> 13.8).
  pdl_release();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;
  const uint32_t t_dK = tmem, t_dV = tmem + D, t_A0 = tmem + 2 * D /* + 128 * S buffer */, t_B = t_A0 + 128 * SM::kSBufs;
  static_assert(2 * D + 128 * (SM::kSBufs + 1) <= 512, "tensor memory");
  bool ok = true;

  // steps: query tiles (raw, gist, sink) from the first one up, the G heads of a tile back to back
  struct StepIter {
    int t, hd;
  };
  auto advance = [&](StepIter& x) {
    if (++x.hd == G) x.hd = 0, ++x.t;
  };
  auto tile_of = [&](const StepIter& x, int& qseg, int& qt, int& head) {
    const int t = x.t;
    head = hk * G + x.hd;
    if (t < n_raw_q) {
      qseg = kSegRaw;
      qt = rq_lo + t;
    } else if (t < n_raw_q + n_gist_q) {
      qseg = kSegGist;
      qt = gq_lo + (t - n_raw_q);
    } else {
      qseg = kSegSink;
      qt = sq_lo + (t - n_raw_q - n_gist_q);
    }
  };

  if (warp == kKvCompute) {
    // ------------------------------------------------------------ producer: K, V once; Q, dO, LSE, Delta per step
    if (lane == 0) {
      mbar_arrive_expect_tx(bar_kv, 2 * SM::kTile);
      const CUtensorMap* mk = kseg == kSegRaw ? &tm_k_raw : (kseg == kSegGist ? &tm_k_gist : &tm_k_sink);
      const CUtensorMap* mv = kseg == kSegRaw ? &tm_v_raw : (kseg == kSegGist ? &tm_v_gist : &tm_v_sink);
#pragma unroll
      for (int sl = 0; sl < D / 64; ++sl) {
        tma_load_4d(sK + sl * SM::kSlab, mk, bar_kv, sl * 64, hk, key_a, b);
        tma_load_4d(sV + sl * SM::kSlab, mv, bar_kv, sl * 64, hk, key_a, b);
      }
    }
    // LSE (in log2 units) and Delta of a step's 128 query rows, 4 rows per lane, fetched one step ahead
    float st_l[KV_BN / 32], st_d[KV_BN / 32];
    auto fetch_stats = [&](const StepIter& at) {
      int qseg, qt, head;
      tile_of(at, qseg, qt, head);
      const int q_seg_len = seg_len(g, qseg);
      const long long row_base = ((long long)b * Hq + head) * g.N + seg_base(g, qseg);
#pragma unroll
      for (int i = 0; i < KV_BN / 32; ++i) {
        const int row = qt * KV_BN + lane + 32 * i;
        const bool valid = row < q_seg_len;
        // both negated, so that they are added; rows past the segment get LSE = +inf, so their P is exactly zero
        st_l[i] = valid ? -(lse[row_base + row] * kLog2e) : -INFINITY;
        st_d[i] = valid ? -delta[row_base + row] : 0.f;
      }
    };
    StepIter cur{t_begin, 0}, ahead{t_begin, 0};
    if (n_iter > 0) fetch_stats(ahead);
    for (int it = 0; it < n_iter; ++it, advance(cur)) {
      const int st = it % kSt;
      int qseg, qt, head;
      tile_of(cur, qseg, qt, head);
      if (it >= kSt) ok = mbar_wait_warp(bar_empty + 8 * st, (it / kSt - 1) & 1);
      if (!ok) break;
      float* ls = stats + st * 2 * KV_BN;
#pragma unroll
      for (int i = 0; i < KV_BN / 32; ++i) {
        ls[lane + 32 * i] = st_l[i];
        ls[KV_BN + lane + 32 * i] = st_d[i];
      }
      __syncwarp();
      if (lane == 0) {
        mbar_arrive_expect_tx(bar_full + 8 * st, 2 * SM::kTile);
        const CUtensorMap* mq = qseg == kSegRaw ? &tm_q_raw : (qseg == kSegGist ? &tm_q_gist : &tm_q_sink);
        const CUtensorMap* md = qseg == kSegRaw ? &tm_do_raw : (qseg == kSegGist ? &tm_do_gist : &tm_do_sink);
#pragma unroll
        for (int sl = 0; sl < D / 64; ++sl) {
          tma_load_4d(sQ0 + st * SM::kTile + sl * SM::kSlab, mq, bar_full + 8 * st, sl * 64, head, qt * KV_BN, b);
          tma_load_4d(sDO0 + st * SM::kTile + sl * SM::kSlab, md, bar_full + 8 * st, sl * 64, head, qt * KV_BN, b);
        }
      }
      __syncwarp();
      advance(ahead);
      if (it + 1 < n_iter) fetch_stats(ahead);
    }
    if (!ok) atomicExch(&g_bwd_timeout, 1u);
  } else if (warp == kKvCompute + 1) {
    // ------------------------------------------------------------ MMA issuer
    {
      const uint32_t leader = elect_one();
      constexpr uint32_t idesc_s = make_idesc_bf16(KV_BM, KV_BN, false, false);
      constexpr uint32_t idesc_acc = make_idesc_bf16(KV_BM, D, false, true);
      // A operand of the accumulating MMAs: bf16 pairs in TMEM; query columns [32 h, 32 h + 32) are packed at
      // columns [32 h, 32 h + 16) of the buffer
      auto a_col = [](int kk) { return (kk / 2) * 32 + (kk % 2) * 8; };
      auto issue_S = [&](int it) {  // S^T of step it, once its Q (and dO) have arrived
        const int st = it % kSt, sb = it % SM::kSBufs;
        if (!mbar_wait_warp(bar_full + 8 * st, (it / kSt) & 1)) return false;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t off = (kk / 4) * SM::kSlab + (kk % 4) * 32;
          umma_ss(leader, t_A0 + 128 * sb, make_smem_desc(sK + off, 16, 1024),
                  make_smem_desc(sQ0 + st * SM::kTile + off, 16, 1024), idesc_s, kk > 0);
        }
        umma_commit(leader, bar_S + 8 * sb);
        return true;
      };
      auto issue_dP = [&](int it) {
        const int st = it % kSt;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t off = (kk / 4) * SM::kSlab + (kk % 4) * 32;
          umma_ss(leader, t_B, make_smem_desc(sV + off, 16, 1024), make_smem_desc(sDO0 + st * SM::kTile + off, 16, 1024),
                  idesc_s, kk > 0);
        }
        umma_commit(leader, bar_dP);
      };
      ok = mbar_wait_warp(bar_kv, 0);
      if (ok && n_iter > 0) ok = issue_S(0);
      if (ok && n_iter > 0) issue_dP(0);
      for (int it = 0; it < n_iter && ok; ++it) {
        const int st = it % kSt, sb = it % SM::kSBufs;
        // With two S buffers the next scores do not wait for this step's P^T: the exponentials of step it + 1 follow
        // dS of step it at once, and dP(it + 1) runs under them.
        if (SM::kSBufs == 2 && it + 1 < n_iter) ok = issue_S(it + 1);
        ok = ok && mbar_wait_warp(bar_P + 8 * sb, (it / SM::kSBufs) & 1);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < KV_BN / 16; ++kk)
          umma_ts(leader, t_dV, t_A0 + 128 * sb + a_col(kk), make_smem_desc(sDO0 + st * SM::kTile + kk * 2048, SM::kSlab, 1024),
                  idesc_acc, (it > 0 || kk > 0) ? 1u : 0u);
        if (SM::kSBufs == 1 && it + 1 < n_iter) ok = issue_S(it + 1);
        ok = ok && mbar_wait_warp(bar_dS, it & 1);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < KV_BN / 16; ++kk)
          umma_ts(leader, t_dK, t_B + a_col(kk), make_smem_desc(sQ0 + st * SM::kTile + kk * 2048, SM::kSlab, 1024), idesc_acc,
                  (it > 0 || kk > 0) ? 1u : 0u);
        umma_commit(leader, bar_empty + 8 * st);
        if (it + 1 < n_iter) issue_dP(it + 1);
      }
      if (ok && n_iter > 0) umma_commit(leader, bar_final);
      if (!ok && leader) atomicExch(&g_bwd_timeout, 1u);
    }
  } else {
    // ------------------------------------------------------------ compute: thread = key (TMEM lane), 32 query columns
    const int qd = warp & 3, hf = warp >> 2;
    const int key = key_a + qd * 32 + lane;
    const bool key_valid = key <= key_b;
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    const uint64_t scale2 = f32x2(scale * kLog2e, scale * kLog2e);
    int my_lo_r, my_hi_r, my_lo_g, my_hi_g, my_lo_s, my_hi_s;  // queries that see this key, per query segment
    key_q_interval3(g, rdiv, kseg, key, key_valid, kSegRaw, my_lo_r, my_hi_r);
    key_q_interval3(g, rdiv, kseg, key, key_valid, kSegGist, my_lo_g, my_hi_g);
    key_q_interval3(g, rdiv, kseg, key, key_valid, kSegSink, my_lo_s, my_hi_s);

    StepIter cur{t_begin, 0};
    for (int it = 0; it < n_iter && ok; ++it, advance(cur)) {
      const int st = it % kSt, sb = it % SM::kSBufs;
      const uint32_t t_A = t_A0 + 128 * sb;
      int qseg, qt, head;
      tile_of(cur, qseg, qt, head);
      const int q0 = qt * KV_BN, q_seg_len = seg_len(g, qseg);
      const int qb = min(q0 + KV_BN - 1, q_seg_len - 1);
      // full: every (query, key) pair of the tile is visible -> no mask arithmetic
      const int t_lo = qseg == kSegRaw ? raw_t_lo : (qseg == kSegGist ? gist_t_lo : sink_t_lo);
      const int t_hi = qseg == kSegRaw ? raw_t_hi : (qseg == kSegGist ? gist_t_hi : sink_t_hi);
      const bool full = key_tile_whole && q0 >= t_lo && qb <= t_hi;
      const int lo = (qseg == kSegRaw ? my_lo_r : (qseg == kSegGist ? my_lo_g : my_lo_s)) - q0 - 32 * hf;
      const int hi = (qseg == kSegRaw ? my_hi_r : (qseg == kSegGist ? my_hi_g : my_hi_s)) - q0 - 32 * hf;
      const float* ls = stats + st * 2 * KV_BN + 32 * hf;
      const float* dl = ls + KV_BN;
      ok = mbar_wait_warp(bar_full + 8 * st, (it / kSt) & 1) && mbar_wait_warp(bar_S + 8 * sb, (it / SM::kSBufs) & 1);
      if (!ok) break;
      tc_fence_after();
      float p[32];
      {
        uint32_t v[32];
        tmem_ld(t_A + lane_base + 32 * hf, v);
        tmem_wait_ld();
        uint32_t pk[16];
        // a partly visible tile: most of its 32 x 32 pieces are wholly visible all the same
        uint32_t bits = 0xffffffffu;
        if (!full) bits = piece_bits(lo, hi);
        if (full || __all_sync(0xffffffffu, bits == 0xffffffffu))
          p_chunk<false>(v, ls, scale2, 0u, p, pk);
        else
          p_chunk<true>(v, ls, scale2, bits, p, pk);
        tmem_st(t_A + lane_base + 32 * hf, pk);
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive_warp(bar_P + 8 * sb);
      ok = mbar_wait_warp(bar_dP, it & 1);
      if (!ok) break;
      tc_fence_after();
      {
        uint32_t v[32];
        tmem_ld(t_B + lane_base + 32 * hf, v);
        tmem_wait_ld();
        uint32_t pk[16];
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const ulonglong2 d4 = *reinterpret_cast<const ulonglong2*>(dl + i);
          pk[i / 2] = ds_pair(p[i], p[i + 1], v[i], v[i + 1], d4.x);
          pk[i / 2 + 1] = ds_pair(p[i + 2], p[i + 3], v[i + 2], v[i + 3], d4.y);
        }
        tmem_st(t_B + lane_base + 32 * hf, pk);
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive_warp(bar_dS);
    }
    if (ok && n_iter > 0) ok = mbar_wait_warp(bar_final, 0);
    if (!ok) atomicExch(&g_bwd_timeout, 1u);
  }

  // dK and dV leave: a compute warp has its 32 keys and 32 columns of one of them (D = 64) or of both (D = 128).  Where
  // two blocks share the key tile, block 0 finishes dK and block 1 dV: each puts its part of the other one into its
  // (consumed) Q ring, rows of D floats with the 16-byte pieces permuted by row.
  const int hf = warp >> 2, krow = (warp & 3) * 32 + lane;
  const bool compute = warp < kKvCompute;
  constexpr int kWhich = D == 128 ? 2 : 1;
  auto is_dk_of = [&](int which) { return D == 128 ? which == 0 : hf < 2; };
  const int col0 = D == 128 ? 32 * hf : 32 * (hf & 1);
  auto load = [&](bool is_dk, uint32_t (&v)[32]) {
    if (n_iter > 0) {
      tmem_ld((is_dk ? t_dK : t_dV) + (static_cast<uint32_t>((warp & 3) * 32) << 16) + col0, v);
      tmem_wait_ld();
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = 0u;
    }
  };
  auto piece = [&](int i) { return sQ0 + krow * D * 4 + ((((col0 + i) / 4) ^ (krow & 7)) << 4); };
  if (compute) tc_fence_after();
  if (split) {
    if (compute && ok) {
#pragma unroll
      for (int which = 0; which < kWhich; ++which) {
        if (is_dk_of(which) == (crank == 0)) continue;
        uint32_t v[32];
        load(is_dk_of(which), v);
#pragma unroll
        for (int i = 0; i < 32; i += 4) st_shared_v4(piece(i), make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]));
      }
    }
    cluster_sync();
  }
  if (compute && ok) {
    const int key = key_a + krow;
    const long long tok = (long long)b * g.N + key_seg_base + key;
#pragma unroll
    for (int which = 0; which < kWhich; ++which) {
      const bool is_dk = is_dk_of(which);
      if (split && is_dk != (crank == 0)) continue;
      uint32_t v[32];
      load(is_dk, v);
      if (split) {
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float4 x = ld_cluster_v4(piece(i), crank ^ 1);
          v[i] = __float_as_uint(__uint_as_float(v[i]) + x.x);
          v[i + 1] = __float_as_uint(__uint_as_float(v[i + 1]) + x.y);
          v[i + 2] = __float_as_uint(__uint_as_float(v[i + 2]) + x.z);
          v[i + 3] = __float_as_uint(__uint_as_float(v[i + 3]) + x.w);
        }
      }
      __nv_bfloat16* dst = (is_dk ? dk : dv) + (tok * Hkv + hk) * D + col0;
      const float mul = is_dk ? scale : 1.f;
      if (key <= key_b) {
#pragma unroll
        for (int i = 0; i < 32; i += 8) {
          uint4 pk;
          pk.x = pack_bf16(__uint_as_float(v[i]) * mul, __uint_as_float(v[i + 1]) * mul);
          pk.y = pack_bf16(__uint_as_float(v[i + 2]) * mul, __uint_as_float(v[i + 3]) * mul);
          pk.z = pack_bf16(__uint_as_float(v[i + 4]) * mul, __uint_as_float(v[i + 5]) * mul);
          pk.w = pack_bf16(__uint_as_float(v[i + 6]) * mul, __uint_as_float(v[i + 7]) * mul);
          *reinterpret_cast<uint4*>(dst + i) = pk;
        }
      }
    }
  }
  if (split) cluster_sync();  // the other block has read this one's shared memory
  tc_fence_before();
  __syncthreads();
  if (warp == kKvCompute + 1) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------------------------------------
// dQ kernel.  Two blocks per SM cover each other's softmax; with head_dim 64 a ring of four K / V stages and a second S
// buffer leave only dP and dS on the chain of a step (the problem above: 0.38 ms -> 0.285; 0.27 with a row's operands loaded in
// one go and packed arithmetic; eight compute warps of 32 keys were slower, 0.31).  dP of the next step is issued as soon as
// this step's operands are in registers, so that the chain of a step is the softmax alone (0.261 -> 0.240; fetching dP under
// the exponentials instead of with the scores lost all of it again; the dK / dV kernel, whose four compute warps per
// scheduler overlap by themselves, became 2 % slower the same way).
constexpr int DQ_BM = 128;  // query rows per block
constexpr int DQ_BN = 64;   // keys per step
constexpr int kDqThreads = 192;

template <int D>
struct DqSmem {
  static constexpr int kQSlab = DQ_BM * 128, kQTile = kQSlab * (D / 64);
  static constexpr int kKSlab = DQ_BN * 128, kKTile = kKSlab * (D / 64);
  // Two blocks share an SM (its shared memory, and 256 tensor-memory columns each); with head_dim 64 that leaves room
  // for a ring of K / V tiles and a second S buffer.
  static constexpr int kStages = D == 64 ? 4 : 1;
  static constexpr int kSBufs = D == 64 ? 2 : 1;
  static constexpr int kOffBars = 2 * kQTile + 2 * kStages * kKTile;
  static constexpr int kBytes = kOffBars + 256 + 1024;
};

template <int D>
__global__ void __launch_bounds__(kDqThreads, 2)
attn_bwd_dq_sm100_kernel(const __grid_constant__ CUtensorMap tm_q_sink, const __grid_constant__ CUtensorMap tm_q_raw,
                         const __grid_constant__ CUtensorMap tm_q_gist, const __grid_constant__ CUtensorMap tm_do_sink,
                         const __grid_constant__ CUtensorMap tm_do_raw, const __grid_constant__ CUtensorMap tm_do_gist,
                         const __grid_constant__ CUtensorMap tm_k_sink, const __grid_constant__ CUtensorMap tm_k_raw,
                         const __grid_constant__ CUtensorMap tm_k_gist, const __grid_constant__ CUtensorMap tm_v_sink,
                         const __grid_constant__ CUtensorMap tm_v_raw, const __grid_constant__ CUtensorMap tm_v_gist,
                         Geom g, int Hq, int Hkv, float scale, const float* __restrict__ lse,
                         const float* __restrict__ delta, __nv_bfloat16* __restrict__ dq, int n_sink_qt, int n_raw_qt,
                         int after_dkdv, FastDiv rdiv) {
  using SM = DqSmem<D>;
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* gen = smem_dyn + (base - smem_u32(smem_dyn));
  constexpr int kSt = SM::kStages;
  const uint32_t sQ = base, sDO = base + SM::kQTile, sK0 = base + 2 * SM::kQTile /* + stage * kKTile */, sV0 = sK0 + kSt * SM::kKTile;
  const uint32_t bars = base + SM::kOffBars;
  const uint32_t bar_q = bars, bar_s = bars + 8, bar_fin = bars + 24, tmem_slot = bars + 32;
  const uint32_t full_k = bars + 40, full_v = full_k + 8 * kSt, empty_k = full_v + 8 * kSt, empty_v = empty_k + 8 * kSt;
  const uint32_t bar_read = empty_v + 8 * kSt;  // S and dP of the step have been read: dP may be overwritten
  const uint32_t bar_p = bar_read + 8;          // dS is stored (+ 8 * S buffer: step j + 1's may come before the issuer looks for step j's)
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(gen + SM::kOffBars + 32);

  const int warp = threadIdx.x >> 5;
  const int h = blockIdx.y, b = blockIdx.z, hk = h / (Hq / Hkv);
  // heaviest tiles first: gist query tiles from the end, then raw query tiles from the end, sink tiles last
  const int qt_lin = gridDim.x - 1 - blockIdx.x;
  const int qseg = qt_lin < n_sink_qt ? kSegSink : (qt_lin < n_sink_qt + n_raw_qt ? kSegRaw : kSegGist);
  const int qt = qt_lin - (qseg == kSegSink ? 0 : (qseg == kSegRaw ? n_sink_qt : n_sink_qt + n_raw_qt));
  const int q_len = seg_len(g, qseg);
  const int q_base = seg_base(g, qseg);
  const int row_a = qt * DQ_BM, row_b = min(row_a + DQ_BM - 1, q_len - 1);
  auto div_r = [&](int x) { return fdiv(rdiv, x); };
  const RowIv iv_a = row_intervals_with(g, q_base + row_a, div_r), iv_b = row_intervals_with(g, q_base + row_b, div_r);
  // visible 64-key tiles: sink tiles [0, n_sink), raw tiles [raw_lo, raw_lo + n_raw), gist tiles [0, n_gist)
  const int n_sink = iv_b.hi_sink >= 0 ? iv_b.hi_sink / DQ_BN + 1 : 0;
  const int raw_lo = iv_a.lo_raw / DQ_BN, n_raw = iv_b.hi_raw >= iv_a.lo_raw ? iv_b.hi_raw / DQ_BN - raw_lo + 1 : 0;
  const int n_gist = iv_b.hi_gist >= 0 ? iv_b.hi_gist / DQ_BN + 1 : 0;
  const int nt = n_sink + n_raw + n_gist;
  // step j: its key segment and 64-key tile
  auto key_tile = [&](int j, int& sg, int& idx) {
    if (j < n_raw) {
      sg = kSegRaw;
      idx = raw_lo + j;
    } else if (j < n_raw + n_gist) {
      sg = kSegGist;
      idx = j - n_raw;
    } else {
      sg = kSegSink;
      idx = j - n_raw - n_gist;
    }
  };

  if (threadIdx.x == 0) {
    mbar_init(bar_q, 1);
    for (int i = 0; i < 4 * kSt; ++i) mbar_init(full_k + 8 * i, 1);
    mbar_init(bar_s, 1);
    mbar_init(bar_p, 4);
    mbar_init(bar_p + 8, 4);
    mbar_init(bar_read, 4);
    mbar_init(bar_fin, 1);
    mbar_fence_init();
  }
  if (warp == 5) tmem_alloc(tmem_slot, 256);
  // The dK / dV kernel lets this one in once all of its blocks have seen the end of what went before them, Delta included,
  // and hands nothing on to it.  (Delta and LSE are read past the L1, which may hold an earlier call's.)
  if (after_dkdv) pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;
  const uint32_t t_S0 = tmem /* + 64 * S buffer */, t_dP = tmem + 64 * SM::kSBufs, t_dQ = t_dP + 64;
  static_assert(64 * (SM::kSBufs + 1) + D <= 256, "tensor memory of a block");
  bool ok = true;

  if (warp == 4) {
    if (elect_one()) {
      mbar_arrive_expect_tx(bar_q, 2 * SM::kQTile);
      const CUtensorMap* mq = qseg == kSegRaw ? &tm_q_raw : (qseg == kSegGist ? &tm_q_gist : &tm_q_sink);
      const CUtensorMap* md = qseg == kSegRaw ? &tm_do_raw : (qseg == kSegGist ? &tm_do_gist : &tm_do_sink);
#pragma unroll
      for (int sl = 0; sl < D / 64; ++sl) {
        tma_load_4d(sQ + sl * SM::kQSlab, mq, bar_q, sl * 64, h, row_a, b);
        tma_load_4d(sDO + sl * SM::kQSlab, md, bar_q, sl * 64, h, row_a, b);
      }
      for (int j = 0; j < nt && ok; ++j) {
        int sg, idx;
        key_tile(j, sg, idx);
        const CUtensorMap* mk = sg == kSegRaw ? &tm_k_raw : (sg == kSegGist ? &tm_k_gist : &tm_k_sink);
        const CUtensorMap* mv = sg == kSegRaw ? &tm_v_raw : (sg == kSegGist ? &tm_v_gist : &tm_v_sink);
        const int st = j % kSt, ph = (j / kSt - 1) & 1;
        if (j >= kSt) ok = mbar_wait(empty_v + 8 * st, ph);  // dP of step j - kSt done
        if (!ok) break;
        mbar_arrive_expect_tx(full_v + 8 * st, SM::kKTile);
#pragma unroll
        for (int sl = 0; sl < D / 64; ++sl)
          tma_load_4d(sV0 + st * SM::kKTile + sl * SM::kKSlab, mv, full_v + 8 * st, sl * 64, hk, idx * DQ_BN, b);
        if (j >= kSt) ok = mbar_wait(empty_k + 8 * st, ph);  // dQ of step j - kSt done
        if (!ok) break;
        mbar_arrive_expect_tx(full_k + 8 * st, SM::kKTile);
#pragma unroll
        for (int sl = 0; sl < D / 64; ++sl)
          tma_load_4d(sK0 + st * SM::kKTile + sl * SM::kKSlab, mk, full_k + 8 * st, sl * 64, hk, idx * DQ_BN, b);
      }
      if (!ok) atomicExch(&g_bwd_timeout, 1u);
    }
  } else if (warp == 5) {
    {
      const uint32_t leader = elect_one();
      constexpr uint32_t idesc_s = make_idesc_bf16(DQ_BM, DQ_BN, false, false);
      constexpr uint32_t idesc_dq = make_idesc_bf16(DQ_BM, D, false, true);
      auto issue_S = [&](int j) {
        const int st = j % kSt;
        if (!mbar_wait_warp(full_k + 8 * st, (j / kSt) & 1)) return false;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t qoff = (kk / 4) * SM::kQSlab + (kk % 4) * 32, koff = (kk / 4) * SM::kKSlab + (kk % 4) * 32;
          umma_ss(leader, t_S0 + 64 * (j % SM::kSBufs), make_smem_desc(sQ + qoff, 16, 1024),
                  make_smem_desc(sK0 + st * SM::kKTile + koff, 16, 1024), idesc_s, kk > 0);
        }
        return true;
      };
      auto issue_dP = [&](int j) {  // completes the step's inputs: its S went before
        const int st = j % kSt;
        if (!mbar_wait_warp(full_v + 8 * st, (j / kSt) & 1)) return false;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t qoff = (kk / 4) * SM::kQSlab + (kk % 4) * 32, koff = (kk / 4) * SM::kKSlab + (kk % 4) * 32;
          umma_ss(leader, t_dP, make_smem_desc(sDO + qoff, 16, 1024), make_smem_desc(sV0 + st * SM::kKTile + koff, 16, 1024),
                  idesc_s, kk > 0);
        }
        umma_commit(leader, bar_s);
        umma_commit(leader, empty_v + 8 * st);
        return true;
      };
      ok = mbar_wait_warp(bar_q, 0) && issue_S(0);  // (every query row sees a key: nt > 0)
      ok = ok && issue_dP(0);
      for (int j = 0; j < nt && ok; ++j) {
        const int st = j % kSt;
        const bool has_next = j + 1 < nt;
        if (SM::kSBufs == 2 && has_next) {  // the next step's scores and dP run under the softmax of step j
          ok = issue_S(j + 1) && mbar_wait_warp(bar_read, j & 1);
          if (!ok) break;
          tc_fence_after();
          ok = issue_dP(j + 1);
        }
        ok = ok && mbar_wait_warp(bar_p + 8 * (j % SM::kSBufs), (j / SM::kSBufs) & 1);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < DQ_BN / 16; ++kk)
          umma_ts(leader, t_dQ, t_S0 + 64 * (j % SM::kSBufs) + kk * 8,
                  make_smem_desc(sK0 + st * SM::kKTile + kk * 2048, SM::kKSlab, 1024), idesc_dq, (j > 0 || kk > 0) ? 1u : 0u);
        umma_commit(leader, empty_k + 8 * st);
        if (SM::kSBufs == 1 && has_next) {
          ok = issue_S(j + 1);
          ok = ok && issue_dP(j + 1);
        }
      }
      if (ok) umma_commit(leader, bar_fin);
      if (!ok && leader) atomicExch(&g_bwd_timeout, 1u);
    }
  } else {
    const int r_in_tile = threadIdx.x;
    const int row = min(row_a + r_in_tile, row_b);
    const bool valid = row_a + r_in_tile <= row_b;
    const RowIv my = row_intervals_with(g, q_base + row, div_r);
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
    const uint64_t scale2 = f32x2(scale * kLog2e, scale * kLog2e);
    const long long stat_idx = ((long long)b * Hq + h) * g.N + q_base + row;
    const float nl = -(__ldcg(lse + stat_idx) * kLog2e), nd = -__ldcg(delta + stat_idx);
    const uint64_t nl2 = f32x2(nl, nl), nd2 = f32x2(nd, nd);
    for (int j = 0; j < nt && ok; ++j) {
      int sg, idx;
      key_tile(j, sg, idx);
      const int col0 = idx * DQ_BN;
      bool full;
      int lo, hi;
      if (sg == kSegRaw) {
        full = col0 >= iv_b.lo_raw && col0 + DQ_BN - 1 <= iv_a.hi_raw;
        lo = my.lo_raw - col0;
        hi = my.hi_raw - col0;
      } else if (sg == kSegGist) {
        full = col0 + DQ_BN - 1 <= iv_a.hi_gist;
        lo = 0;
        hi = my.hi_gist - col0;
      } else {
        full = col0 + DQ_BN - 1 <= iv_a.hi_sink;
        lo = 0;
        hi = my.hi_sink - col0;
      }
      ok = mbar_wait_warp(bar_s, j & 1);
      if (!ok) break;
      tc_fence_after();
      const uint32_t t_S = t_S0 + 64 * (j % SM::kSBufs);
      // both operands of the whole row in one go (a block's 192 threads leave 168 registers each)
      uint32_t sv[DQ_BN], dv_[DQ_BN];
#pragma unroll
      for (int c = 0; c < DQ_BN / 32; ++c) {
        tmem_ld32(t_S + lane_base + 32 * c, sv + 32 * c);
        tmem_ld32(t_dP + lane_base + 32 * c, dv_ + 32 * c);
      }
      tmem_wait_ld();
      if (SM::kSBufs == 2) {
        tc_fence_before();
        mbar_arrive_warp(bar_read);
      }
#pragma unroll
      for (int c = 0; c < DQ_BN / 32; ++c) {
        uint32_t pk[16];
        uint32_t bits = 0xffffffffu;
        if (!full) bits = piece_bits(lo - 32 * c, hi - 32 * c);
        auto piece = [&](bool masked) {
#pragma unroll
          for (int i = 0; i < 32; i += 2) {
            const int e = 32 * c + i;
            float x0, x1;
            f32x2_split(fma2(f32x2(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1])), scale2, nl2), x0, x1);
            if (masked) {
              x0 = (bits >> i) & 1u ? x0 : -INFINITY;
              x1 = (bits >> (i + 1)) & 1u ? x1 : -INFINITY;
            }
            pk[i / 2] = ds_pair(ex2(x0), ex2(x1), dv_[e], dv_[e + 1], nd2);
          }
        };
        if (full || __all_sync(0xffffffffu, bits == 0xffffffffu)) piece(false); else piece(true);
        tmem_st(t_S + lane_base + 16 * c, pk);
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive_warp(bar_p + 8 * (j % SM::kSBufs));
    }
    if (ok) ok = mbar_wait_warp(bar_fin, 0);
    if (ok) {
      tc_fence_after();
      const long long tok = (long long)b * g.N + q_base + row_a + r_in_tile;
      __nv_bfloat16* drow = dq + (tok * Hq + h) * D;
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t v[32];
        tmem_ld(t_dQ + lane_base + 32 * c, v);
        tmem_wait_ld();
        if (valid) {
#pragma unroll
          for (int i = 0; i < 32; i += 8) {
            uint4 pk;
            pk.x = pack_bf16(__uint_as_float(v[i]) * scale, __uint_as_float(v[i + 1]) * scale);
            pk.y = pack_bf16(__uint_as_float(v[i + 2]) * scale, __uint_as_float(v[i + 3]) * scale);
            pk.z = pack_bf16(__uint_as_float(v[i + 4]) * scale, __uint_as_float(v[i + 5]) * scale);
            pk.w = pack_bf16(__uint_as_float(v[i + 6]) * scale, __uint_as_float(v[i + 7]) * scale);
            *reinterpret_cast<uint4*>(drow + 32 * c + i) = pk;
          }
        }
      }
    } else {
      atomicExch(&g_bwd_timeout, 1u);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    __syncwarp();
    tmem_dealloc(tmem, 256);
  }
  // whoever comes after this kernel counts on dK and dV too: its last block waits for them
  if (blockIdx.x == gridDim.x - 1 && blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1) pdl_wait();
}

// ------------------------------------------------------------------------------------------------
// Fused backward for head_dim 128: one kernel, five matrix products per (key tile, query tile) pair.
//
// A thread block owns a 128-key tile of one KV head (dK, dV in TMEM for its lifetime: no atomics,
// deterministic) and walks every 128-query tile of every query head of the group that sees it:
//   S^T = K Q^T, dP^T = V dO^T        (both operands in shared memory)          -> TMEM
//   P^T = exp2(S^T c - LSE)            bf16, written over S^T in TMEM
//   dV += P^T dO                       (P^T read from TMEM)
//   dS^T = P^T o (dP^T - Delta)        bf16, written to shared memory [key][query]
//   dK += dS^T Q                       (dS^T from shared memory, query-contiguous = K-major A)
//   dQ^T = K^T dS^T                    (K tile as MN-major A, dS^T as MN-major B) -> TMEM, over dP^T
// dQ^T (head_dim x queries, fp32) is then added into an fp32 dQ buffer in global memory by TMA
// reductions from small staging buffers, since several key tiles contribute to one query tile; a
// small kernel scales and rounds that buffer to bf16 afterwards.
// MMA issue order per step i:  dV(i), S(i+1), dQ(i), dK(i), dP(i+1)  so that the exponentials of
// step i+1 and the dQ read-out of step i run under matrix products.
// Warps: 0-7 compute (thread = key, 64 query columns each), 8-15 dQ read-out (two warps per TMEM lane
// quarter, 64 query columns each, so the dQ^T columns are free again after two TMEM loads), 16 TMA, 17 MMA.
constexpr int kFuThreads = 640;
constexpr int kFuTmaWarp = 16, kFuMmaWarp = 17;
constexpr int kFuRegsLaunch = 96, kFuRegsCompute = 128, kFuRegsReadout = 80, kFuRegsOther = 64;
static_assert(kFuThreads * kFuRegsLaunch <= 65536 && kFuThreads * (kFuRegsLaunch + 8) > 65536,
              "launch register count is stale");
static_assert(2 * kFuRegsCompute + 2 * kFuRegsReadout + kFuRegsOther <= 5 * kFuRegsLaunch,
              "register split exceeds the block's allocation");

struct FuSmem {
  static constexpr int kSlab = 128 * 128;    // [128 rows x 64 bf16]
  static constexpr int kTile = 2 * kSlab;    // [128 x 128] bf16
  static constexpr int kOffK = 0, kOffV = kTile, kOffQ = 2 * kTile /* 2 stages */, kOffDO = 4 * kTile, kOffDS = 5 * kTile;
  static constexpr int kOffStage = 6 * kTile;             // dQ staging: [8 warps][32 queries][32 floats]
  static constexpr int kOffStats = 7 * kTile;             // [stage][lse2 | delta][128] fp32
  static constexpr int kOffBars = kOffStats + 2 * 2 * 128 * 4;
  static constexpr int kUsed = kOffBars + 192;
  static constexpr int kBytes = 232448;  // all a block may have; the 1024-byte alignment slack comes out of it
};

// One launch unit of the fused backward: a batch of sequences of one geometry with its own tensor maps (one per
// segment) and output pointers.  A call on one problem is one unit with a (blocks, 1, batch) grid; a packed
// sample under cross-document masking is several units in ONE launch with a flat grid, and a block finds its
// unit from the units' first block indices.
struct alignas(64) BwdRun {
  CUtensorMap q[3], dout[3], k[3], v[3], dq[3];
  Geom g;
  const float* lse;
  const float* delta;
  __nv_bfloat16* dk;
  __nv_bfloat16* dv;
  int n_sink_kt, n_gist_kt, n_raw_kt;
  int plane;  // blocks per batch index
  // flat grid (several units in one launch): the sink / gist blocks of ALL units come first, then the raw blocks;
  // the unit's first block in each of the two ranges, and its blocks per batch index there
  int heavy_begin, raw_begin, heavy_plane, raw_plane;
  FastDiv heavy_plane_div, raw_plane_div;
  // A sink or gist key tile's walk over its query tiles is cut into n_chunks chunks of chunk_tiles tiles, one
  // block each; `partial` receives the fp32 dK / dV of the chunks of key tiles that have more than one
  // ([batch][KV head][heavy key tile][chunk][dK | dV][128 keys][128]).
  int n_chunks, chunk_tiles;
  float* partial;
  FastDiv heavy_div /* by n_chunks * heavy tiles */, tile_div /* by heavy tiles */, raw_div;
};
template <int kRuns>
struct BwdRuns {
  BwdRun run[kRuns];
  int n;
  int total_heavy;  // flat grid: blocks of the sink / gist range
};
static_assert(sizeof(BwdRuns<kMaxRunsPerLaunch>) + 256 <= 32764, "the launch units must fit the kernel parameter space");

template <int kRuns>
__global__ void __launch_bounds__(kFuThreads, 1)
attn_bwd_fused_sm100_kernel(const __grid_constant__ BwdRuns<kRuns> P, int Hq, int Hkv, float scale, int interleaved,
                            FastDiv rdiv) {
  int ri = 0, bx, b;
  if constexpr (kRuns == 1) {
    bx = blockIdx.x, b = blockIdx.z;
  } else {
    const int c = blockIdx.x;
    if (c < P.total_heavy) {
      while (ri + 1 < P.n && c >= P.run[ri + 1].heavy_begin) ++ri;
      const int local = c - P.run[ri].heavy_begin;
      b = fdiv(P.run[ri].heavy_plane_div, local);
      bx = local - b * P.run[ri].heavy_plane;  // < heavy_plane: a sink / gist block of the unit
    } else {
      while (ri + 1 < P.n && c >= P.run[ri + 1].raw_begin) ++ri;
      const int local = c - P.run[ri].raw_begin;
      b = fdiv(P.run[ri].raw_plane_div, local);
      bx = P.run[ri].heavy_plane + (local - b * P.run[ri].raw_plane);
    }
  }
  const BwdRun& R = P.run[ri];
  const Geom g = R.g;
  const float* __restrict__ lse = R.lse;
  const float* __restrict__ delta = R.delta;
  __nv_bfloat16* __restrict__ dk = R.dk;
  __nv_bfloat16* __restrict__ dv = R.dv;
  const int n_sink_kt = R.n_sink_kt, n_gist_kt = R.n_gist_kt, n_raw_kt = R.n_raw_kt;
  using SM = FuSmem;
  constexpr int D = 128;
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t raw_base = smem_u32(smem_dyn);
  const uint32_t base = (raw_base + 1023u) & ~1023u;
  if (base - raw_base + SM::kUsed > SM::kBytes) {  // cannot happen with a 1024-aligned window; never run past it
    if (threadIdx.x == 0) atomicExch(&g_bwd_timeout, 1u);
    return;
  }
  unsigned char* gen = smem_dyn + (base - raw_base);
  const uint32_t sK = base + SM::kOffK, sV = base + SM::kOffV, sDS = base + SM::kOffDS;
  const uint32_t sQ0 = base + SM::kOffQ /* stage st at + st * kTile */, sDO = base + SM::kOffDO;
  float* stats = reinterpret_cast<float*>(gen + SM::kOffStats);
  const uint32_t bars = base + SM::kOffBars;
  const uint32_t bar_kv = bars, bar_S = bars + 8, bar_dP = bars + 16, bar_P = bars + 24, bar_dS = bars + 32,
                 bar_dSfree = bars + 40, bar_dQ = bars + 48, bar_dQfree = bars + 56, bar_final = bars + 64;
  const uint32_t full_q0 = bars + 72, empty_q0 = bars + 88 /* + 8 * st */, full_do = bars + 104, empty_do = bars + 120;
  const uint32_t tmem_slot = bars + 136;
  volatile uint32_t* tmem_slot_ptr = reinterpret_cast<volatile uint32_t*>(gen + SM::kOffBars + 136);
  // number of Q tiles whose load the producer has issued so far (a scheduling hint for the dQ read-out, see there)
  volatile int* q_issued = reinterpret_cast<volatile int*>(gen + SM::kOffBars + 144);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Block order (the hardware starts blocks in the order of their index).  Sink and gist key tiles are seen by
  // every later query: they are the heaviest and come first, before any raw key tile.  Their walk over the query
  // tiles (which starts at the last query tile for every one of them) is cut into chunks of the same query tiles,
  // one block per (key tile, chunk), ordered KV head, chunk, key tile: the blocks that run side by side are the key
  // tiles of ONE KV head over ONE chunk of queries, they start together, take the same time and read the same
  // Q / dO / dQ tiles, which therefore come from DRAM once and from L2 for every other block.  (One block per
  // key tile over all its queries had blocks of very different lengths start whenever an SM fell free, each
  // sweeping the head's queries on its own: 7 times the algorithmic DRAM traffic.)  The raw key tiles of one KV
  // head are consecutive too; their windows of query tiles overlap.
  const int G = Hq / Hkv;
  const int n_heavy_kt = n_sink_kt + n_gist_kt;
  int hk, rank, chunk = 0;
  if (bx < n_heavy_kt * R.n_chunks * Hkv) {
    hk = fdiv(R.heavy_div, bx);
    const int rem = bx - hk * n_heavy_kt * R.n_chunks;
    chunk = fdiv(R.tile_div, rem);
    rank = rem - chunk * n_heavy_kt;
  } else {
    const int y = bx - n_heavy_kt * R.n_chunks * Hkv;
    hk = fdiv(R.raw_div, y);
    rank = n_heavy_kt + (y - hk * n_raw_kt);
  }
  const int kseg = rank < n_sink_kt ? kSegSink : (rank < n_sink_kt + n_gist_kt ? kSegGist : kSegRaw);
  const int kt = rank - (kseg == kSegSink ? 0 : (kseg == kSegGist ? n_sink_kt : n_sink_kt + n_gist_kt));
  const int key_seg_len = seg_len(g, kseg);
  const int key_a = kt * 128, key_b = min(key_a + 127, key_seg_len - 1);
  const bool key_tile_whole = key_a + 127 <= key_seg_len - 1;

  // query tiles that see this key tile, per query segment: [first tile, count], and the bounds inside
  // which a tile is "full" (seen by the last key from t_lo on, by the first key up to t_hi)
  int lo_a, hi_a, lo_b, hi_b;
  key_q_interval3(g, rdiv, kseg, key_a, true, kSegRaw, lo_a, hi_a);
  key_q_interval3(g, rdiv, kseg, key_b, true, kSegRaw, lo_b, hi_b);
  const int n_raw_q = hi_b >= lo_a ? hi_b / 128 - lo_a / 128 + 1 : 0, rq_lo = lo_a / 128, raw_t_lo = lo_b, raw_t_hi = hi_a;
  key_q_interval3(g, rdiv, kseg, key_a, true, kSegGist, lo_a, hi_a);
  key_q_interval3(g, rdiv, kseg, key_b, true, kSegGist, lo_b, hi_b);
  const int n_gist_q = hi_b >= lo_a ? hi_b / 128 - lo_a / 128 + 1 : 0, gq_lo = lo_a / 128, gist_t_lo = lo_b, gist_t_hi = hi_a;
  key_q_interval3(g, rdiv, kseg, key_a, true, kSegSink, lo_a, hi_a);
  key_q_interval3(g, rdiv, kseg, key_b, true, kSegSink, lo_b, hi_b);
  const int n_sink_q = hi_b >= lo_a ? hi_b / 128 - lo_a / 128 + 1 : 0, sq_lo = lo_a / 128, sink_t_lo = lo_b, sink_t_hi = hi_a;
  // this block's part of the walk: tiles [t_begin, t_end) of the order below (all of them for a raw key tile)
  const int n_tiles = n_raw_q + n_gist_q + n_sink_q;
  const bool heavy = kseg != kSegRaw;
  const int t_begin = heavy ? chunk * R.chunk_tiles : 0;
  const int t_end = heavy ? min(t_begin + R.chunk_tiles, n_tiles) : n_tiles;
  if (chunk > 0 && t_begin >= n_tiles) return;  // this key tile has no such chunk (whole block, before any barrier)
  const bool to_partial = heavy && n_tiles > R.chunk_tiles;  // several chunks: fp32 partial sums, reduced afterwards
  const int n_iter = (t_end - t_begin) * G;

  if (threadIdx.x == 0) {
    mbar_init(bar_kv, 1);
    mbar_init(bar_S, 1);
    mbar_init(bar_dP, 1);
    mbar_init(bar_P, 8);
    mbar_init(bar_dS, 8);
    mbar_init(bar_dSfree, 1);
    mbar_init(bar_dQ, 1);
    mbar_init(bar_dQfree, 8);
    mbar_init(bar_final, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(full_q0 + 8 * i, 1);
      mbar_init(empty_q0 + 8 * i, 1);
    }
    mbar_init(full_do, 1);
    mbar_init(empty_do, 1);
    *q_issued = 0;
    mbar_fence_init();
  }
  if (warp == kFuMmaWarp) tmem_alloc(tmem_slot, 512);
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot_ptr;
  const uint32_t t_dK = tmem, t_dV = tmem + 128, t_S = tmem + 256, t_dP = tmem + 384;
  bool ok = true;

  // Step order.  Tiles: raw query tiles from the last one down, then gist query tiles, then sink query tiles.
  // A sink or gist key tile is seen up to the last tile of every segment, so the blocks of one KV head that start
  // together walk the same tiles: with the G heads of a tile back to back they stay in step until each runs out,
  // and share Q / dO / dQ lines in L2.  A raw key tile sees a window of query tiles that moves with the key tile:
  // its neighbour is one tile behind, i.e. G steps with the heads innermost but a single step with the tiles
  // innermost (head by head), which keeps the shared lines in L2 between the two uses.
  const bool tiles_inner = kseg == kSegRaw;
  struct StepIter {
    int t, hd;  // tile index in the order above, head of the group
  };
  auto advance = [&](StepIter& x) {  // no division: the walk is sequential for every role
    if (tiles_inner) {
      if (++x.t == n_tiles) x.t = 0, ++x.hd;
    } else {
      if (++x.hd == G) x.hd = 0, ++x.t;
    }
  };
  auto tile_of = [&](const StepIter& x, int& qseg, int& qt, int& head) {
    const int t = x.t;
    head = hk * G + x.hd;
    if (t < n_raw_q) {
      qseg = kSegRaw;
      qt = rq_lo + (n_raw_q - 1 - t);
    } else if (t < n_raw_q + n_gist_q) {
      qseg = kSegGist;
      qt = gq_lo + (n_gist_q - 1 - (t - n_raw_q));
    } else {
      qseg = kSegSink;
      qt = sq_lo + (n_sink_q - 1 - (t - n_raw_q - n_gist_q));
    }
  };

  if (warp >= 16) {
    reg_dealloc<kFuRegsOther>();
    if (warp == kFuTmaWarp) {
      // ---------------------------------------------------------- producer: K, V once; Q, dO, LSE, Delta per step
      // tile coordinate: its first unit (a raw tile of an interleaved tensor spans 128 / r gist units)
      auto first_unit = [&](int sg, int row0) { return interleaved && sg == kSegRaw ? fdiv(rdiv, row0) : row0; };
      if (lane == 0) {
        mbar_arrive_expect_tx(bar_kv, 2 * SM::kTile);
        const CUtensorMap* mk = &R.k[kseg];
        const CUtensorMap* mv = &R.v[kseg];
#pragma unroll
        for (int sl = 0; sl < 2; ++sl) {
          tma_load_5d(sK + sl * SM::kSlab, mk, bar_kv, sl * 64, hk, 0, first_unit(kseg, key_a), b);
          tma_load_5d(sV + sl * SM::kSlab, mv, bar_kv, sl * 64, hk, 0, first_unit(kseg, key_a), b);
        }
      }
      // LSE (in log2 units) and Delta of the step's 128 query rows, 4 rows per lane, fetched one step ahead
      float st_l[4], st_d[4];
      auto fetch_stats = [&](const StepIter& at) {
        int qseg, qt, head;
        tile_of(at, qseg, qt, head);
        const int q_seg_len = seg_len(g, qseg), q_seg_base = seg_base(g, qseg);
        const long long row_base = ((long long)b * Hq + head) * g.N + q_seg_base;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int row = qt * 128 + lane + 32 * i;
          const bool valid = row < q_seg_len;
          // both negated, so that they are added; rows past the segment get LSE = +inf, so their P is exactly zero
          st_l[i] = valid ? -(lse[row_base + row] * kLog2e) : -INFINITY;
          st_d[i] = valid ? -delta[row_base + row] : 0.f;
        }
      };
      StepIter cur{t_begin, 0}, ahead{t_begin, 0};
      if (n_iter > 0) fetch_stats(ahead);
      for (int it = 0; it < n_iter; ++it, advance(cur)) {
        const int st = it & 1;
        int qseg, qt, head;
        tile_of(cur, qseg, qt, head);
        if (it >= 2) ok = mbar_wait_warp(empty_q0 + 8 * st, ((it >> 1) - 1) & 1);
        if (!ok) break;
        float* ls = stats + st * 256;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          ls[lane + 32 * i] = st_l[i];
          ls[128 + lane + 32 * i] = st_d[i];
        }
        __syncwarp();
        if (lane == 0) {
          mbar_arrive_expect_tx(full_q0 + 8 * st, SM::kTile);
          const CUtensorMap* mq = &R.q[qseg];
#pragma unroll
          for (int sl = 0; sl < 2; ++sl)
            tma_load_5d(sQ0 + st * SM::kTile + sl * SM::kSlab, mq, full_q0 + 8 * st, sl * 64, head, 0,
                        first_unit(qseg, qt * 128), b);
          *q_issued = it + 1;
        }
        advance(ahead);
        if (it + 1 < n_iter) fetch_stats(ahead);
        if (it >= 1) ok = mbar_wait_warp(empty_do, (it - 1) & 1);  // one dO buffer: free once dV of the step before is done
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(full_do, SM::kTile);
          const CUtensorMap* md = &R.dout[qseg];
#pragma unroll
          for (int sl = 0; sl < 2; ++sl)
            tma_load_5d(sDO + sl * SM::kSlab, md, full_do, sl * 64, head, 0, first_unit(qseg, qt * 128), b);
        }
        __syncwarp();
      }
      if (!ok && lane == 0) atomicExch(&g_bwd_timeout, 1u);
    } else if (warp == kFuMmaWarp) {
      // ---------------------------------------------------------- MMA issuer
      {
      const uint32_t leader = elect_one();
        constexpr uint32_t idesc_s = make_idesc_bf16(128, 128, false, false);   // K-major A and B
        constexpr uint32_t idesc_acc = make_idesc_bf16(128, 128, false, true);  // K-major A, MN-major B
        constexpr uint32_t idesc_dq = make_idesc_bf16(128, 128, true, true);    // MN-major A and B
        constexpr uint32_t kHi = smem_desc_hi(1024);
        constexpr uint32_t kStage = SM::kTile >> 4;  // stage st of Q / dO: + st * kStage on the low word
        const uint32_t k_lo = smem_desc_lo(sK, 16), v_lo = smem_desc_lo(sV, 16);
        const uint32_t kT_lo = smem_desc_lo(sK, SM::kSlab);    // K tile read as MN-major A (head_dim contiguous)
        const uint32_t ds_lo = smem_desc_lo(sDS, 16);          // dS^T as K-major A (queries contiguous)
        const uint32_t dsT_lo = smem_desc_lo(sDS, SM::kSlab);  // dS^T as MN-major B
        const uint32_t q_lo = smem_desc_lo(sQ0, 16), qT_lo = smem_desc_lo(sQ0, SM::kSlab);
        const uint32_t do_lo = smem_desc_lo(sDO, 16), doT_lo = smem_desc_lo(sDO, SM::kSlab);
        // K-major operands step 32 B per 16 elements inside a 64-element slab; MN-major ones 2048 B
        auto koff = [](int kk) { return (uint32_t)(((kk / 4) * SM::kSlab + (kk % 4) * 32) >> 4); };
        auto moff = [](int kk) { return (uint32_t)((kk * 2048) >> 4); };
        // bf16 pairs of P^T in TMEM: query columns [0,64) packed at [0,32), [64,128) at [64,96)
        auto a_col = [](int kk) { return (uint32_t)((kk / 4) * 64 + (kk % 4) * 8); };
        auto issue_S = [&](int st) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            umma_ss(leader, t_S, smem_desc_join(k_lo + koff(kk), kHi), smem_desc_join(q_lo + st * kStage + koff(kk), kHi),
                    idesc_s, kk > 0);
          umma_commit(leader, bar_S);
        };
        auto issue_dP = [&]() {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            umma_ss(leader, t_dP, smem_desc_join(v_lo + koff(kk), kHi), smem_desc_join(do_lo + koff(kk), kHi), idesc_s, kk > 0);
          umma_commit(leader, bar_dP);
        };
        ok = mbar_wait_warp(bar_kv, 0);
        if (ok && n_iter > 0) {
          ok = mbar_wait_warp(full_q0, 0);
          if (ok) {
            tc_fence_after();
            issue_S(0);
            ok = mbar_wait_warp(full_do, 0);
          }
          if (ok) {
            tc_fence_after();
            issue_dP();
          }
        }
        for (int it = 0; it < n_iter && ok; ++it) {
          const int st = it & 1, ph = it & 1;
          const bool has_next = it + 1 < n_iter;
          ok = mbar_wait_warp(bar_P, ph);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)  // dV += P^T dO
            umma_ts(leader, t_dV, t_S + a_col(kk), smem_desc_join(doT_lo + moff(kk), kHi), idesc_acc,
                    (it > 0 || kk > 0) ? 1u : 0u);
          umma_commit(leader, empty_do);
          if (has_next) {
            ok = mbar_wait_warp(full_q0 + 8 * (st ^ 1), ((it + 1) >> 1) & 1);
            if (!ok) break;
            tc_fence_after();
            issue_S(st ^ 1);
          }
          ok = mbar_wait_warp(bar_dS, ph);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)  // dQ^T = K^T dS^T  (contraction over the 128 keys)
            umma_ss(leader, t_dP, smem_desc_join(kT_lo + moff(kk), kHi), smem_desc_join(dsT_lo + moff(kk), kHi), idesc_dq,
                    kk > 0);
          umma_commit(leader, bar_dQ);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)  // dK += dS^T Q  (contraction over the 128 queries)
            umma_ss(leader, t_dK, smem_desc_join(ds_lo + koff(kk), kHi), smem_desc_join(qT_lo + st * kStage + moff(kk), kHi),
                    idesc_acc, (it > 0 || kk > 0) ? 1u : 0u);
          umma_commit(leader, empty_q0 + 8 * st);
          umma_commit(leader, bar_dSfree);
          if (has_next) {
            ok = mbar_wait_warp(bar_dQfree, ph) && mbar_wait_warp(full_do, (it + 1) & 1);
            if (!ok) break;
            tc_fence_after();
            issue_dP();
          }
        }
        if (ok) umma_commit(leader, bar_final);
        if (!ok && leader) atomicExch(&g_bwd_timeout, 1u);
      }
    }
  } else if (warp >= 8) {
    // ------------------------------------------------------------ dQ read-out: lane = head_dim index
    // Each warp moves its 32 head_dim rows x 64 queries of dQ^T, 32 queries at a time, through its own
    // staging buffer ([32 queries][32 floats]) and has the TMA unit add them into the fp32 dQ tensor.
    reg_dealloc<kFuRegsReadout>();
    const int qd = warp & 3, half = (warp >> 2) & 1;
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    float* stage_gen = reinterpret_cast<float*>(gen + SM::kOffStage) + (warp - 8) * 1024 + lane;
    const uint32_t stage_sh = base + SM::kOffStage + (warp - 8) * 4096;
    StepIter cur{t_begin, 0};
    for (int it = 0; it < n_iter && ok; ++it, advance(cur)) {
      int qseg, qt, head;
      tile_of(cur, qseg, qt, head);
      const CUtensorMap* mdq = &R.dq[qseg];
      const int nq = seg_len(g, qseg) - qt * 128;  // rows of this tile inside the segment (may exceed 128)
      ok = mbar_wait_warp(bar_dQ, it & 1);
      if (!ok) break;
      tc_fence_after();
      // both halves of this warp's 64 query columns into registers, then the dQ^T columns are free again: the
      // MMA warp never waits for the staging buffer or for the TMA unit
      uint32_t v0[32], v1[32];
      const int col0 = 64 * half;
      tmem_ld32(t_dP + lane_base + col0, v0);
      tmem_ld32(t_dP + lane_base + col0 + 32, v1);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_relaxed(bar_dQfree);
      auto stage_rows = [&](const uint32_t (&v)[32]) {  // the reduction issued before has finished reading the staging buffer
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 32; ++e) stage_gen[e * 32] = __uint_as_float(v[e]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
      };
      auto reduce_rows = [&](int c0) {
        if (lane == 0 && c0 < nq) {  // rows past the segment's end are clipped by the tensor map
          tma_reduce_add_4d(mdq, stage_sh, qd * 32, head, qt * 128 + c0, b);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      };
      stage_rows(v0);
      // The TMA unit takes its work in order, and a step's 16 reduce-adds keep it busy for about 1200 clocks.
      // The Q tile of step it + 2 can be loaded once dK of this step is done, a few hundred clocks from now, and
      // S of that step waits for it: let that load go first.  A hint only: bounded, and no error if it runs out.
      if (lane == 0 && it + 2 < n_iter)
        for (int spin = 0; spin < 4096 && *q_issued < it + 3; ++spin) __nanosleep(20);
      __syncwarp();
      reduce_rows(col0);
      stage_rows(v1);
      reduce_rows(col0 + 32);
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok && lane == 0) atomicExch(&g_bwd_timeout, 1u);
  } else {
    // ------------------------------------------------------------ compute: thread = key (TMEM lane), 64 query columns
    reg_alloc<kFuRegsCompute>();
    const int qd = warp & 3, hf = warp >> 2;
    const int krow = qd * 32 + lane;
    const int key = key_a + krow;
    const bool key_valid = key <= key_b;
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    const uint64_t scale2 = f32x2(scale * kLog2e, scale * kLog2e);
    int my_lo_r, my_hi_r, my_lo_g, my_hi_g, my_lo_s, my_hi_s;  // queries that see this key, per query segment
    key_q_interval3(g, rdiv, kseg, key, key_valid, kSegRaw, my_lo_r, my_hi_r);
    key_q_interval3(g, rdiv, kseg, key, key_valid, kSegGist, my_lo_g, my_hi_g);
    key_q_interval3(g, rdiv, kseg, key, key_valid, kSegSink, my_lo_s, my_hi_s);
    // this thread's row of the dS^T tile in shared memory: slab hf, row krow, 16-byte chunks swizzled by row
    unsigned char* ds_row = gen + SM::kOffDS + hf * SM::kSlab + krow * 128;
    const int swz = krow & 7;

    StepIter cur{t_begin, 0};
    for (int it = 0; it < n_iter && ok; ++it, advance(cur)) {
      const int st = it & 1;
      int qseg, qt, head;
      tile_of(cur, qseg, qt, head);
      const int q0 = qt * 128, q_seg_len = seg_len(g, qseg);
      const int qb = min(q0 + 127, q_seg_len - 1);
      // full: every (query, key) pair of the tile is visible -> no mask arithmetic
      const int t_lo = qseg == kSegRaw ? raw_t_lo : (qseg == kSegGist ? gist_t_lo : sink_t_lo);
      const int t_hi = qseg == kSegRaw ? raw_t_hi : (qseg == kSegGist ? gist_t_hi : sink_t_hi);
      const bool full = key_tile_whole && q0 >= t_lo && qb <= t_hi;
      const int lo = (qseg == kSegRaw ? my_lo_r : (qseg == kSegGist ? my_lo_g : my_lo_s)) - q0 - 64 * hf;
      const int hi = (qseg == kSegRaw ? my_hi_r : (qseg == kSegGist ? my_hi_g : my_hi_s)) - q0 - 64 * hf;
      const float* ls = stats + st * 256 + 64 * hf;
      const float* dl = ls + 128;
      ok = mbar_wait_warp(full_q0 + 8 * st, (it >> 1) & 1) && mbar_wait_warp(bar_S, it & 1);
      if (!ok) break;
      tc_fence_after();
      float p[64];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t v[32];
        tmem_ld32(t_S + lane_base + 64 * hf + 32 * c, v);
        tmem_wait_ld();
        uint32_t pk[16];
        if (full) {
          p_chunk<false>(v, ls + 32 * c, scale2, 0u, p + 32 * c, pk);
        } else {
          p_chunk<true>(v, ls + 32 * c, scale2, piece_bits(lo - 32 * c, hi - 32 * c), p + 32 * c, pk);
        }
        tmem_st(t_S + lane_base + 64 * hf + 16 * c, pk);
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive_warp(bar_P);
      ok = mbar_wait_warp(bar_dP, it & 1);
      if (ok && it > 0) ok = mbar_wait_warp(bar_dSfree, (it - 1) & 1);  // the previous dS^T has been consumed
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        uint32_t v[32];
        tmem_ld32(t_dP + lane_base + 64 * hf + 32 * c, v);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; i += 8) {  // 8 queries = one 16-byte chunk of this key's dS^T row
          const ulonglong2 d0 = *reinterpret_cast<const ulonglong2*>(dl + 32 * c + i);
          const ulonglong2 d1 = *reinterpret_cast<const ulonglong2*>(dl + 32 * c + i + 4);
          const float* pp = p + 32 * c + i;
          uint4 w;
          w.x = ds_pair(pp[0], pp[1], v[i], v[i + 1], d0.x);
          w.y = ds_pair(pp[2], pp[3], v[i + 2], v[i + 3], d0.y);
          w.z = ds_pair(pp[4], pp[5], v[i + 4], v[i + 5], d1.x);
          w.w = ds_pair(pp[6], pp[7], v[i + 6], v[i + 7], d1.y);
          const int chunk = 4 * c + i / 8;
          *reinterpret_cast<uint4*>(ds_row + ((chunk ^ swz) << 4)) = w;
        }
      }
      tc_fence_before();  // the dP^T columns may be overwritten (by dQ^T) once every thread has arrived
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // dS^T visible to the tensor core's reads
      mbar_arrive_warp(bar_dS);
    }
    if (ok && n_iter > 0) ok = mbar_wait_warp(bar_final, 0);
    if (ok) {
      tc_fence_after();
      const long long tok = (long long)b * g.N + seg_row_to_token(g, interleaved != 0, kseg, key_valid ? key : key_a);
      // where this key's row of the chunk's fp32 partial sums goes when the key tile has several chunks
      float* part_row = R.partial + (((((long long)b * Hkv + hk) * n_heavy_kt + rank) * R.n_chunks + chunk) * 2 * 128 + krow) * 128 + 64 * hf;
      // this warp stores columns [64 hf, 64 hf + 64) of dK and of dV
#pragma unroll
      for (int which = 0; which < 2; ++which) {
        const bool is_dk = which == 0;
        const uint32_t tsrc = (is_dk ? t_dK : t_dV) + lane_base + 64 * hf;
        __nv_bfloat16* dst = (is_dk ? dk : dv) + (tok * Hkv + hk) * D + 64 * hf;
        const float mul = is_dk ? scale : 1.f;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t v[32];
          if (n_iter > 0) {
            tmem_ld32(tsrc + 32 * c, v);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = 0u;
          }
          if (to_partial) {
            if (key_valid) {
              float4* pd = reinterpret_cast<float4*>(part_row + which * 128 * 128 + 32 * c);
#pragma unroll
              for (int i = 0; i < 32; i += 4)
                pd[i / 4] = make_float4(__uint_as_float(v[i]), __uint_as_float(v[i + 1]), __uint_as_float(v[i + 2]),
                                        __uint_as_float(v[i + 3]));
            }
          } else if (key_valid) {
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
              uint4 pk;
              pk.x = pack_bf16(__uint_as_float(v[i]) * mul, __uint_as_float(v[i + 1]) * mul);
              pk.y = pack_bf16(__uint_as_float(v[i + 2]) * mul, __uint_as_float(v[i + 3]) * mul);
              pk.z = pack_bf16(__uint_as_float(v[i + 4]) * mul, __uint_as_float(v[i + 5]) * mul);
              pk.w = pack_bf16(__uint_as_float(v[i + 6]) * mul, __uint_as_float(v[i + 7]) * mul);
              *reinterpret_cast<uint4*>(dst + 32 * c + i) = pk;
            }
          }
        }
      }
    } else {
      atomicExch(&g_bwd_timeout, 1u);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kFuMmaWarp) {
    __syncwarp();
    tmem_dealloc(tmem, 512);
  }
}

// Number of 128-query tiles that see a key tile [key_a, key_b] of segment kseg (all query segments).
__host__ __device__ __forceinline__ int count_q_tiles(const Geom& g, const FastDiv& rdiv, int kseg, int key_a, int key_b) {
  int n = 0;
#pragma unroll
  for (int qseg = 0; qseg < 3; ++qseg) {
    int lo_a, hi_a, lo_b, hi_b;
    key_q_interval3(g, rdiv, kseg, key_a, true, qseg, lo_a, hi_a);
    key_q_interval3(g, rdiv, kseg, key_b, true, qseg, lo_b, hi_b);
    n += hi_b >= lo_a ? hi_b / 128 - lo_a / 128 + 1 : 0;
  }
  return n;
}

// The launch units of a fused backward whose walks were cut, for the kernel below.
struct ReduceRun {
  Geom g;
  const float* partial;
  __nv_bfloat16 *dk, *dv;
  int n_sink_kt, n_gist_kt, n_chunks, chunk_tiles;
  int begin;  // first block of this unit (flat grid)
};
template <int kRuns>
struct ReduceRuns {
  ReduceRun run[kRuns];
  int n;
};

// dK, dV of the sink and gist key tiles whose walk was cut into several chunks: the chunks' fp32 partial sums
// added in chunk order (the same bits on every run), scaled, rounded to bf16 and stored at the keys' rows.
// The units of a packed sample go in one launch (each by itself cost 5 - 7 us a unit: twelve documents of about 500 tokens, 16 / 2
// heads, 226 -> 147 us for the whole backward).  Bound by the latency of the chunks' loads: a warp takes one key row, four chunks
// of dK and dV in flight (with four rows a warp 11264 raw tokens, 19 chunks, took 288 us instead of 261).
constexpr int kReduceBlocks = 32;  // per heavy key tile, KV head and sequence
template <int kRuns>
__global__ void __launch_bounds__(128)
dkdv_reduce_kernel(const __grid_constant__ ReduceRuns<kRuns> P, int interleaved, int Hkv, float scale, FastDiv rdiv) {
  pdl_wait();
  int ri = 0, bx = blockIdx.x, hk = blockIdx.y, b = blockIdx.z;
  if constexpr (kRuns > 1) {
    while (ri + 1 < P.n && (int)blockIdx.x >= P.run[ri + 1].begin) ++ri;
    const int heavy = (P.run[ri].n_sink_kt + P.run[ri].n_gist_kt) * kReduceBlocks, plane = heavy * Hkv;
    bx -= P.run[ri].begin;
    b = bx / plane;
    bx -= b * plane;
    hk = bx / heavy;
    bx -= hk * heavy;
  }
  const ReduceRun& R = P.run[ri];
  const Geom& g = R.g;
  const int n_sink_kt = R.n_sink_kt, n_gist_kt = R.n_gist_kt, n_chunks = R.n_chunks, chunk_tiles = R.chunk_tiles;
  const int rank = bx / kReduceBlocks, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int krow = bx % kReduceBlocks * 4 + warp;
  const int n_heavy_kt = n_sink_kt + n_gist_kt;
  const int kseg = rank < n_sink_kt ? kSegSink : kSegGist;
  const int kt = rank - (kseg == kSegSink ? 0 : n_sink_kt);
  const int key_a = kt * 128, key_b = min(key_a + 127, seg_len(g, kseg) - 1);
  const int n_tiles = count_q_tiles(g, rdiv, kseg, key_a, key_b);
  if (n_tiles <= chunk_tiles || key_a + krow > key_b) return;  // a single chunk: the fused kernel stored dK, dV itself
  const int chunks = (n_tiles + chunk_tiles - 1) / chunk_tiles;
  const float* base = R.partial + ((((long long)b * Hkv + hk) * n_heavy_kt + rank) * n_chunks) * 2 * 128 * 128;
  const long long tok = (long long)b * g.N + seg_row_to_token(g, interleaved != 0, kseg, key_a + krow);
  float4 acc[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
#pragma unroll 4
  for (int c = 0; c < chunks; ++c) {
#pragma unroll
    for (int which = 0; which < 2; ++which) {
      const float4 x = __ldcs(reinterpret_cast<const float4*>(base + ((long long)(c * 2 + which) * 128 + krow) * 128) + lane);
      acc[which].x += x.x, acc[which].y += x.y, acc[which].z += x.z, acc[which].w += x.w;
    }
  }
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    const float mul = which == 0 ? scale : 1.f;
    __nv_bfloat16* dst = (which == 0 ? R.dk : R.dv) + (tok * Hkv + hk) * 128 + lane * 4;
    *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16(acc[which].x * mul, acc[which].y * mul),
                                                pack_bf16(acc[which].z * mul, acc[which].w * mul));
  }
}

// dQ (bf16) = scale * dQ accumulated in fp32 (shifted order, head_dim 128).  One warp per token: Hq rows of
// 128 floats, 4 per lane; the bf16 row goes to the token's shifted or interleaved position.
template <int kRuns>
__global__ void __launch_bounds__(256)
dq_convert_kernel(const __grid_constant__ TokRuns<kRuns> P, int interleaved, int Hq, long long tokens,
                  const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, float scale) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long tk = warp; tk < tokens; tk += nwarps) {  // tk = packed token index, shifted order inside a sequence
    int ri = 0;
    if constexpr (kRuns > 1)
      while (ri + 1 < P.n && tk >= P.run[ri + 1].tok_begin) ++ri;
    const TokRun& R = P.run[ri];
    const Geom& g = R.g;
    const int local = (int)(tk - R.tok_begin), b = fdiv(R.div.n, local), sigma = local - b * g.N;
    const long long out_tk = R.tok_begin + (long long)b * g.N + (interleaved ? shift_perm(g, R.div, sigma) : sigma);
    const float4* s4 = reinterpret_cast<const float4*>(src + tk * Hq * 128) + lane;
    uint2* d2 = reinterpret_cast<uint2*>(dst + out_tk * Hq * 128) + lane;
    for (int h0 = 0; h0 < Hq; h0 += 4) {
      float4 a[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (h0 + u < Hq) a[u] = __ldcs(s4 + (h0 + u) * 32);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (h0 + u < Hq)
          d2[(h0 + u) * 32] = make_uint2(pack_bf16(a[u].x * scale, a[u].y * scale), pack_bf16(a[u].z * scale, a[u].w * scale));
    }
  }
}

}  // namespace

namespace {

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// The backward's scratch for `tokens` packed tokens: Delta (fp32, per run a [batch, Hq, N] block that starts at
// float Hq * first token), the bf16 copy of an fp32 dO, and for the fused backward the fp32 dQ accumulator.
struct BwdScratch {
  float* delta;
  __nv_bfloat16* do_bf16;
  float* dq32;
};
BwdScratch carve_scratch(void* workspace, long long tokens, int Hq, int D, bool f32, bool fused) {
  char* ws = static_cast<char*>(workspace);
  BwdScratch sc;
  sc.delta = reinterpret_cast<float*>(ws);
  ws += align256((size_t)tokens * Hq * sizeof(float));
  sc.do_bf16 = f32 ? reinterpret_cast<__nv_bfloat16*>(ws) : nullptr;
  if (f32) ws += align256((size_t)tokens * Hq * D * 2);
  sc.dq32 = fused ? reinterpret_cast<float*>(ws) : nullptr;
  return sc;
}

template <int kRuns>
int32_t launch_prep(const TokRuns<kRuns>& T, const unigist_problem& p, long long tokens, const void* d_o, const void* o,
                    const BwdScratch& sc, cudaStream_t st) {
  const bool f32 = (p.flags & UNIGIST_FLAG_DOUT_FP32) != 0;
  const int il = (p.flags & UNIGIST_FLAG_INTERLEAVED) ? 1 : 0;
  const int blocks = (int)((tokens + 7) / 8 < sm_count() * 16 ? (tokens + 7) / 8 : sm_count() * 16);
  {
    KernelScope ks("bwd_prep_kernel", st);
    const auto kern = p.head_dim == 128 ? (f32 ? bwd_prep_kernel<true, kRuns, 128> : bwd_prep_kernel<false, kRuns, 128>)
                                        : (f32 ? bwd_prep_kernel<true, kRuns, 64> : bwd_prep_kernel<false, kRuns, 64>);
    launch_chained(kern, dim3(blocks), 256, 0, st, 1, T, il, p.num_q_heads, (int)tokens, d_o, (const __nv_bfloat16*)o,
                   sc.do_bf16, sc.dq32);
  }
  return check_launch("backward prep kernel");
}

template <int kRuns>
int32_t launch_convert(const TokRuns<kRuns>& T, const unigist_problem& p, long long tokens, const BwdScratch& sc, void* dq,
                       float scale, cudaStream_t st) {
  const int blocks = (int)((tokens + 7) / 8 < sm_count() * 16 ? (tokens + 7) / 8 : sm_count() * 16);
  {
    KernelScope ks("dq_convert_kernel", st);
    launch_chained(dq_convert_kernel<kRuns>, dim3(blocks), 256, 0, st, 1, T, (p.flags & UNIGIST_FLAG_INTERLEAVED) ? 1 : 0, p.num_q_heads, tokens,
                                                     sc.dq32, (__nv_bfloat16*)dq, scale);
  }
  return check_launch("dQ convert kernel");
}

int tiles(long long rows) { return (int)((rows + 127) / 128); }
// The walks of one sequence's key tiles for one query head: steps (key tile, query tile) of all, steps of the longest raw key
// tile's, and how many blocks they take if the sink and gist ones are cut into two at least.
struct Walks {
  long long steps;
  int longest_raw, blocks;
};
Walks count_walks(const Geom& g) {
  const FastDiv rdiv = make_fastdiv(g.r);
  const int all = tiles(g.s) + tiles(g.T) + tiles(g.n);
  Walks w = {0, 0, 0};
  for (int kseg = 0; kseg < 3; ++kseg)
    for (int key = 0; key < seg_len(g, kseg); key += 128) {
      const int n = count_q_tiles(g, rdiv, kseg, key, std::min(key + 127, seg_len(g, kseg) - 1));
      w.steps += n;
      w.blocks += kseg != kSegRaw && n > (all + 1) / 2 ? 2 : 1;
      if (kseg == kSegRaw) w.longest_raw = std::max(w.longest_raw, n);
    }
  return w;
}

// What a launch of the fused backward holds besides its longest walk, in steps (key tile, query tile, query head).
struct LaunchLoad {
  long long end;       // when the SMs would be through if no walk outlasted the others and the long ones were cut
  long long late;      // when the last sink and gist key tiles start
  long long raw_walk;  // longest walk of a raw key tile
};
// in_turn: one problem, whose sequences' blocks follow each other; otherwise all sink and gist key tiles come first.
constexpr int kBlockSteps = 2;  // the fixed part of a block, in steps
LaunchLoad launch_load(const SeqRun* runs, int n_runs, int Hq, int Hkv, bool in_turn) {
  const long long G = Hq / Hkv, sms = sm_count();
  long long steps = 0, raw_walk = 0, blocks = 0, before_last = 0;
  for (int i = 0; i < n_runs; ++i) {
    const Geom& g = runs[i].g;
    const Walks w = count_walks(g);
    const long long n_heavy = tiles(g.s) + tiles(g.n), n_raw = tiles(g.T);
    steps += w.steps * Hq * runs[i].batch;
    blocks += (long long)w.blocks * Hkv * runs[i].batch;
    raw_walk = std::max(raw_walk, w.longest_raw * G);
    before_last = ((n_heavy + n_raw) * (runs[i].batch - 1) + n_heavy) * Hkv;
  }
  LaunchLoad load;
  load.raw_walk = raw_walk;
  load.end = (steps + kBlockSteps * blocks) / sms;
  load.late = in_turn && before_last > sms ? std::max(0ll, load.end - load.end / runs[0].batch - raw_walk / 2) : 0;
  if (blocks > sms) load.end += raw_walk / 2;  // blocks that start when others end do not end together
  return load;
}

// How the walk of a sink or gist key tile over its query tiles is cut (head_dim 128).  Not at all while the rows
// one KV head's blocks sweep (Q, dO and the fp32 dQ of its G query heads: 1 KB per token and head) fit in three
// quarters of the L2: however the blocks start, what one has read is still there for the next.  Otherwise into at
// most four chunks of at least 16 query tiles, fewer where the chunks' fp32 partial sums would take more than
// half the room of the dQ accumulator.
// Where the longest sink or gist walk, or chunk of one, would outlast the rest of the launch by eight steps or more (a step is
// about 2 us), the walks are cut further, if the workspace has room (load != nullptr): into chunks of half of the time the rest
// takes, no shorter than the longest raw key tile's walk; the second kernel and the partial sums cost about 5 us.  Whole
// backward, us, uncut and cut; steps of the longest walk / of the rest: 512 raw tokens, ratio 4, window 64, 32 / 8 heads 61 and
// 50, 22 / 4; 1024, ratio 8, window 128, 16 / 4 heads 91 and 47, 38 / 4; 4096, ratio 16, 16 / 2 heads 597 and 107, 274 / 16; 9000,
// ratio 8, 32 / 8 heads 805 and 509, 322 / 150; 4096, window 1024 378 and 310, 146 / 112; 16384 578 / 598, not cut; 4 x 384,
// ratio 16, window 128, 128 sinks, 64 / 8 heads 147 and 167, 42 / 44, not cut; 11520, ratio 16, 16 / 2 heads, past the L2, 497 in
// the four chunks of 192 steps that the L2 asks for and 271 in chunks of 48 (chunks are cut again only if they outlast the rest by
// an eighth: 33012, ratio 4, window 64, 8 / 1 heads, in 4 and 9 chunks, 1770 and 1931).  Over 1367 problems that it cuts, of 128 - 24000
// tokens: half the uncut time on average, 3 % above the best number of chunks, one slower than uncut by more than 3 %.
// -> tiles per chunk, number of chunks of the longest walk (1 = no cutting, no partial sums).
void bwd_chunking(const Geom& g, int batch, int Hq, int Hkv, const LaunchLoad* load, int* n_chunks, int* chunk_tiles) {
  const int n_raw = tiles(g.T), n_gist = tiles(g.n), n_heavy = tiles(g.s) + n_gist;
  const int max_tiles = n_heavy + n_raw;  // the first sink / gist key tile is seen by every query tile
  const size_t dq_bytes = (size_t)batch * g.N * Hq * 128 * sizeof(float);
  const size_t sweep_bytes = (size_t)g.N * (Hq / Hkv) * 1024;
  int C = sweep_bytes > l2_bytes() / 4 * 3 ? 4 : 1;
  while (C > 1 && ((max_tiles + C - 1) / C < 16 ||
                   (size_t)batch * Hkv * n_heavy * C * 2 * 128 * 128 * sizeof(float) > dq_bytes / 2))
    --C;
  if (load && n_heavy > 0) {
    const long long G = Hq / Hkv, longest = (max_tiles + C - 1) / C * G, target = std::max(load->raw_walk, load->end / 2);
    const long long start = load->late + kBlockSteps, least = C > 1 ? std::max(8ll, load->end / 8) : 8;
    int more = start + longest - std::max(start + target, load->end) >= least ? (int)((max_tiles * G + target - 1) / target) : C;
    while (more > C && (size_t)batch * Hkv * n_heavy * more * 2 * 128 * 128 * sizeof(float) > dq_bytes / 2) --more;
    C = std::max(C, more);
  }
  *chunk_tiles = (max_tiles + C - 1) / C;
  *n_chunks = (max_tiles + *chunk_tiles - 1) / *chunk_tiles;
}

// Tensor maps and tile counts of one launch unit of the fused backward: `batch` sequences of geometry g whose
// first rows are the given pointers.  128-row tile maps per segment (sinks, raw, gists) that read shifted or
// interleaved tensors, and reduction maps over the fp32 dQ tensor (always shifted).
int32_t fill_bwd_run(BwdRun* R, const Geom& g, const unigist_problem& p, int batch, const void* q, const void* do_src,
                     const void* k, const void* v, float* dq32, const float* lse, const float* delta, void* dk, void* dv,
                     float* partial, const LaunchLoad* load) {
  const int D = p.head_dim, Hq = p.num_q_heads, Hkv = p.num_kv_heads;
  const bool il = (p.flags & UNIGIST_FLAG_INTERLEAVED) != 0;
  for (int sg = 0; sg < 3; ++sg) {
    if (int32_t rc = encode_tile_map(&R->q[sg], q, D, Hq, batch, g.s, g.T, g.r, g.n, il, sg)) return rc;
    if (int32_t rc = encode_tile_map(&R->dout[sg], do_src, D, Hq, batch, g.s, g.T, g.r, g.n, il, sg)) return rc;
    if (int32_t rc = encode_tile_map(&R->k[sg], k, D, Hkv, batch, g.s, g.T, g.r, g.n, il, sg)) return rc;
    if (int32_t rc = encode_tile_map(&R->v[sg], v, D, Hkv, batch, g.s, g.T, g.r, g.n, il, sg)) return rc;
    const int rows = seg_len(g, sg) > 0 ? seg_len(g, sg) : 1;  // a tensor map cannot be empty
    if (int32_t rc = encode_segment_map_f32(&R->dq[sg], dq32, D, Hq, g.N, batch, seg_base(g, sg), rows, 32, 32)) return rc;
  }
  R->g = g;
  R->lse = lse;
  R->delta = delta;
  R->dk = static_cast<__nv_bfloat16*>(dk);
  R->dv = static_cast<__nv_bfloat16*>(dv);
  R->n_sink_kt = (g.s + 127) / 128;
  R->n_gist_kt = (g.n + 127) / 128;
  R->n_raw_kt = (g.T + 127) / 128;
  bwd_chunking(g, batch, Hq, Hkv, load, &R->n_chunks, &R->chunk_tiles);
  R->partial = partial;
  const int n_heavy = R->n_sink_kt + R->n_gist_kt;
  R->heavy_plane = n_heavy * R->n_chunks * Hkv;
  R->raw_plane = R->n_raw_kt * Hkv;
  R->plane = R->heavy_plane + R->raw_plane;
  R->heavy_begin = R->raw_begin = 0;
  R->heavy_plane_div = make_fastdiv(R->heavy_plane);
  R->raw_plane_div = make_fastdiv(R->raw_plane);
  R->heavy_div = make_fastdiv(n_heavy * R->n_chunks);
  R->tile_div = make_fastdiv(n_heavy);
  R->raw_div = make_fastdiv(R->n_raw_kt);
  return UNIGIST_OK;
}

template <int kRuns>
int32_t launch_fused(const BwdRuns<kRuns>& P, dim3 grid, const unigist_problem& p, float scale, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(attn_bwd_fused_sm100_kernel<kRuns>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       FuSmem::kBytes);
  if (e != cudaSuccess) return fail(UNIGIST_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
  {
    KernelScope ks("attn_bwd_fused_sm100_kernel", st);
    launch_chained(attn_bwd_fused_sm100_kernel<kRuns>, grid, kFuThreads, FuSmem::kBytes, st, 1, P, p.num_q_heads, p.num_kv_heads, scale, (p.flags & UNIGIST_FLAG_INTERLEAVED) ? 1 : 0, make_fastdiv(p.ratio));
  }
  return check_launch("tcgen05 fused backward kernel");
}

// Adds a unit to the reduce kernel's, from block `begin` on, if its walks were cut.  -> its blocks per KV head and sequence.
template <int kRuns>
int add_reduce_run(ReduceRuns<kRuns>* P, const BwdRun& R, int begin) {
  if (R.n_chunks <= 1) return 0;
  P->run[P->n++] = {R.g, R.partial, R.dk, R.dv, R.n_sink_kt, R.n_gist_kt, R.n_chunks, R.chunk_tiles, begin};
  return (R.n_sink_kt + R.n_gist_kt) * kReduceBlocks;
}

// Adds up the chunks' partial dK / dV of the units that were cut (nothing to do where no key tile has several chunks).
template <int kRuns>
int32_t launch_dkdv_reduce(const ReduceRuns<kRuns>& P, dim3 grid, const unigist_problem& p, float scale, cudaStream_t st) {
  if (P.n == 0) return UNIGIST_OK;
  {
    KernelScope ks("dkdv_reduce_kernel", st);
    launch_chained(dkdv_reduce_kernel<kRuns>, grid, 128, 0, st, 1, P, (p.flags & UNIGIST_FLAG_INTERLEAVED) ? 1 : 0, p.num_kv_heads,
                   scale, make_fastdiv(p.ratio));
  }
  return check_launch("dK/dV reduce kernel");
}

// Bytes of a unit's partial sums.
size_t unit_partial_bytes(const SeqRun& r, int Hq, int Hkv, const LaunchLoad* load) {
  int C, chunk_tiles;
  bwd_chunking(r.g, r.batch, Hq, Hkv, load, &C, &chunk_tiles);
  if (C <= 1) return 0;
  return align256((size_t)r.batch * Hkv * (tiles(r.g.s) + tiles(r.g.n)) * C * 2 * 128 * 128 * sizeof(float));
}

// Whether two blocks share each sink or gist key tile of the dK / dV kernel: where the longest walk (the first sink or gist key
// tile's) would otherwise be the time.  The dQ blocks fill the SMs that the tail of that kernel leaves idle, and they are about as
// much work again: up to twice the steps of an SM, and eight, a walk is hidden, and sharing it only costs blocks (us of the whole
// backward, shared and not; steps of the longest walk / of an SM: 1 x 8190 raw tokens, ratio 7, window 700, 16 / 4 heads, 296 / 100:
// 252 and 325; 2 x 8190, 296 / 201: 494 and 487; 4 x 8190, 296 / 400: 1043 and 1022; 2 x 12288, ratio 3, 512 / 658: 1577 and 1548;
// 8 x 2048, ratio 8, 72 / 121: 363 and 352; 256 x 128, 8 / 111: 612 and 422; 1 x 592, 32 / 8 heads, 24 / 4: 28.1 and 36.9; 1 x 448,
// one head, 5 / 0: 15.9 and 14.1).  Over 1931 problems of 128 - 24000 tokens 0.3 % above the better of the two.
bool dkdv_shares(const Geom& g, int batch, int Hq, int Hkv) {
  const long long longest = (long long)(tiles(g.s) + tiles(g.T) + tiles(g.n)) * (Hq / Hkv);
  return longest > 2 * (count_walks(g).steps * Hq * batch / sm_count()) + 8;
}

// The two-kernel backward (head_dim 64; head_dim 128 when dQ has to be the same bit for bit from run to run): a
// block of the first kernel owns a key tile (dK, dV), a block of the second a query tile (dQ, over 64-key tiles).
template <int D>
int32_t launch_two_kernels(const Geom& g, const unigist_problem& p, float scale, const void* q, const void* do_src,
                           const void* k, const void* v, const float* lse, const float* delta, void* dq, void* dk,
                           void* dv, cudaStream_t st) {
  const int Hq = p.num_q_heads, Hkv = p.num_kv_heads, B = p.batch;
  const int n_sink_t = (g.s + 127) / 128, n_raw_t = (g.T + 127) / 128, n_gist_t = (g.n + 127) / 128;
  // one map per segment (sinks, raw, gists; a tensor map cannot be empty) with 128-row boxes, and 64-row boxes
  // over K and V for the dQ kernel
  CUtensorMap mq[3], md[3], mk[3], mv[3], mk64[3], mv64[3];
  for (int sg = 0; sg < 3; ++sg) {
    const long long first = seg_base(g, sg), len = seg_len(g, sg) > 0 ? seg_len(g, sg) : 1;
    if (int32_t rc = encode_segment_map(&mq[sg], q, D, Hq, g.N, B, first, len, 128)) return rc;
    if (int32_t rc = encode_segment_map(&md[sg], do_src, D, Hq, g.N, B, first, len, 128)) return rc;
    if (int32_t rc = encode_segment_map(&mk[sg], k, D, Hkv, g.N, B, first, len, 128)) return rc;
    if (int32_t rc = encode_segment_map(&mv[sg], v, D, Hkv, g.N, B, first, len, 128)) return rc;
    if (int32_t rc = encode_segment_map(&mk64[sg], k, D, Hkv, g.N, B, first, len, DQ_BN)) return rc;
    if (int32_t rc = encode_segment_map(&mv64[sg], v, D, Hkv, g.N, B, first, len, DQ_BN)) return rc;
  }
  const int n_tiles = n_sink_t + n_raw_t + n_gist_t;
  cudaError_t e = cudaFuncSetAttribute(attn_bwd_dkdv_sm100_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       KvSmem<D>::kBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_bwd_dq_sm100_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, DqSmem<D>::kBytes);
  if (e != cudaSuccess) return fail(UNIGIST_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
  {
    KernelScope ks("attn_bwd_dkdv_sm100_kernel", st);
    const int pairs = B * Hkv, n_heavy = n_sink_t + n_gist_t;
    const int shared = dkdv_shares(g, B, Hq, Hkv) ? 1 : 0, raw_units = (n_raw_t + shared) >> shared;
    launch_chained(attn_bwd_dkdv_sm100_kernel<D>, dim3(((n_heavy + raw_units) * pairs) << shared), kKvThreads, KvSmem<D>::kBytes,
                   st, 1 << shared, mq[0], mq[1], mq[2], md[0], md[1], md[2], mk[0], mk[1], mk[2], mv[0], mv[1], mv[2], g, Hq, Hkv, scale,
                   lse, delta, (__nv_bfloat16*)dk, (__nv_bfloat16*)dv, n_sink_t, n_gist_t, n_raw_t, pairs, shared,
                   make_fastdiv(n_heavy), make_fastdiv(raw_units), make_fastdiv(Hkv), make_fastdiv(g.r));
  }
  if (int32_t rc = check_launch("tcgen05 dK/dV kernel")) return rc;
  {
    // dQ over Q or dO in place: not before the dK / dV kernel has read them
    const char *at = (const char*)dq, *end = at + (size_t)B * g.N * Hq * D * 2;
    auto apart = [&](const void* x) { return end <= (const char*)x || (const char*)x + (end - at) <= at; };
    KernelScope ks("attn_bwd_dq_sm100_kernel", st);
    launch_chained(attn_bwd_dq_sm100_kernel<D>, dim3(n_tiles, Hq, B), kDqThreads, DqSmem<D>::kBytes, st, 1, mq[0], mq[1], mq[2], md[0], md[1], md[2], mk64[0], mk64[1], mk64[2], mv64[0], mv64[1], mv64[2], g, Hq, Hkv, scale,
        lse, delta, (__nv_bfloat16*)dq, n_sink_t, n_raw_t, apart(q) && apart(do_src) ? 0 : 1, make_fastdiv(g.r));
  }
  return check_launch("tcgen05 dQ kernel");
}

}  // namespace

size_t bwd_scratch_bytes(long long tokens, int Hq, int D, bool dout_fp32, bool fused) {
  size_t b = align256((size_t)tokens * Hq * sizeof(float));
  if (dout_fp32) b += align256((size_t)tokens * Hq * D * 2);
  if (fused) b += align256((size_t)tokens * Hq * D * sizeof(float));
  return b;
}

size_t bwd_partial_bytes(const SeqRun* runs, int n_runs, int Hq, int Hkv, bool in_turn, bool spread) {
  LaunchLoad load;
  if (spread) load = launch_load(runs, n_runs, Hq, Hkv, in_turn);
  size_t b = 0;
  for (int i = 0; i < n_runs; ++i) b += unit_partial_bytes(runs[i], Hq, Hkv, spread ? &load : nullptr);
  return b;
}

int32_t launch_bwd_sm100(const Geom& g, const unigist_problem& p, float scale, const void* q, const void* k,
                         const void* v, const void* o, const float* lse, const void* d_o, void* dq, void* dk,
                         void* dv, void* workspace, bool spread, cudaStream_t st) {
  const int D = p.head_dim, Hq = p.num_q_heads, Hkv = p.num_kv_heads, B = p.batch;
  const bool f32 = (p.flags & UNIGIST_FLAG_DOUT_FP32) != 0;
  const long long tokens = (long long)B * g.N;
  // head_dim 64 takes the two-kernel path, and so does head_dim 128 when dQ must not depend on the order in which
  // blocks arrive
  const bool fused = bwd_is_fused(D, p.flags);
  const BwdScratch sc = carve_scratch(workspace, tokens, Hq, D, f32, fused);
  float* delta = sc.delta;
  const void* do_src = f32 ? static_cast<const void*>(sc.do_bf16) : d_o;
  TokRuns<1> T;
  T.n = 1;
  T.run[0] = make_tok_run(g, 0, delta);
  if (int32_t rc = launch_prep(T, p, tokens, d_o, o, sc, st)) return rc;

  if (!fused)
    return D == 64 ? launch_two_kernels<64>(g, p, scale, q, do_src, k, v, lse, delta, dq, dk, dv, st)
                   : launch_two_kernels<128>(g, p, scale, q, do_src, k, v, lse, delta, dq, dk, dv, st);
  BwdRuns<1> P;
  P.n = 1;
  P.total_heavy = 0;  // not used with the (blocks, 1, batch) grid
  float* partial = reinterpret_cast<float*>(static_cast<char*>(workspace) + bwd_scratch_bytes(tokens, Hq, D, f32, true));
  const SeqRun unit = {g, B, 0};
  LaunchLoad load;
  if (spread) load = launch_load(&unit, 1, Hq, Hkv, true);
  if (int32_t rc = fill_bwd_run(&P.run[0], g, p, B, q, do_src, k, v, sc.dq32, lse, delta, dk, dv, partial, spread ? &load : nullptr))
    return rc;
  if (int32_t rc = launch_fused(P, dim3(P.run[0].plane, 1, B), p, scale, st)) return rc;
  ReduceRuns<1> C;
  C.n = 0;
  const int reduce_blocks = add_reduce_run(&C, P.run[0], 0);
  if (int32_t rc = launch_dkdv_reduce(C, dim3(reduce_blocks, Hkv, B), p, scale, st)) return rc;
  return launch_convert(T, p, tokens, sc, dq, scale, st);
}

// Backward over a packed sample (head_dim 128): every run of equal documents is a launch unit; up to twelve
// units share one launch of the prep, fused and convert kernels.
int32_t launch_bwd_sm100_runs(const SeqRun* runs, int n_runs, long long tokens, const unigist_problem& p, float scale,
                              const void* q, const void* k, const void* v, const void* o, const float* lse,
                              const void* d_o, void* dq, void* dk, void* dv, void* workspace, bool spread, cudaStream_t st) {
  const int D = p.head_dim, Hq = p.num_q_heads, Hkv = p.num_kv_heads;
  const bool f32 = (p.flags & UNIGIST_FLAG_DOUT_FP32) != 0;
  const BwdScratch sc = carve_scratch(workspace, tokens, Hq, D, f32, true);
  const void* do_src = f32 ? static_cast<const void*>(sc.do_bf16) : d_o;
  const size_t rq = (size_t)Hq * D * 2, rk = (size_t)Hkv * D * 2;
  // the chunks' partial dK / dV: one slice per run, in token order, behind the scratch of the packed tokens
  char* partial_at = static_cast<char*>(workspace) + bwd_scratch_bytes(tokens, Hq, D, f32, true);
  for (int first = 0; first < n_runs; first += kMaxRunsPerLaunch) {
    const int n = n_runs - first < kMaxRunsPerLaunch ? n_runs - first : kMaxRunsPerLaunch;
    // the launches run one after the other: what one SM has to do in each goes by its own units
    LaunchLoad launch;
    if (spread) launch = launch_load(runs + first, n, Hq, Hkv, false);
    const LaunchLoad* load = spread ? &launch : nullptr;
    float* partial_of[kMaxRunsPerLaunch];
    for (int i = 0; i < n; ++i) {
      partial_of[i] = reinterpret_cast<float*>(partial_at);
      partial_at += unit_partial_bytes(runs[first + i], Hq, Hkv, load);
    }
    // the runs of one launch hold consecutive packed tokens [tok_lo, tok_hi)
    const long long tok_lo = runs[first].first_row;
    const long long tok_hi = runs[first + n - 1].first_row + (long long)runs[first + n - 1].g.N * runs[first + n - 1].batch;
    TokRuns<kMaxRunsPerLaunch> T;
    BwdRuns<kMaxRunsPerLaunch> P;
    T.n = P.n = n;
    // the per-token kernels scan the runs in token order; the fused kernel starts the longest run's blocks first
    int order[kMaxRunsPerLaunch];
    for (int i = 0; i < n; ++i) order[i] = i;
    std::stable_sort(order, order + n, [&](int a, int b) {
      return (long long)runs[first + a].g.N * runs[first + a].batch > (long long)runs[first + b].g.N * runs[first + b].batch;
    });
    long long ctas = 0;
    for (int i = 0; i < n; ++i) {
      const SeqRun& t = runs[first + i];
      T.run[i] = make_tok_run(t.g, t.first_row - tok_lo, sc.delta + t.first_row * Hq);
      const SeqRun& r = runs[first + order[i]];
      if (int32_t rc = fill_bwd_run(&P.run[i], r.g, p, r.batch, (const char*)q + r.first_row * rq,
                                    (const char*)do_src + r.first_row * rq, (const char*)k + r.first_row * rk,
                                    (const char*)v + r.first_row * rk, sc.dq32 + r.first_row * Hq * D,
                                    lse + r.first_row * Hq, sc.delta + r.first_row * Hq, (char*)dk + r.first_row * rk,
                                    (char*)dv + r.first_row * rk, partial_of[order[i]], load))
        return rc;
      ctas += (long long)P.run[i].plane * r.batch;
      if (ctas > 0x7fffffffLL) return fail(UNIGIST_ERR_SHAPE, "packed sample too large for one grid");
    }
    // block ranges: every unit's sink / gist blocks (the long ones) before any unit's raw blocks
    int at = 0;
    for (int i = 0; i < n; ++i) {
      P.run[i].heavy_begin = at;
      at += P.run[i].heavy_plane * runs[first + order[i]].batch;
    }
    P.total_heavy = at;
    for (int i = 0; i < n; ++i) {
      P.run[i].raw_begin = at;
      at += P.run[i].raw_plane * runs[first + order[i]].batch;
    }
    ReduceRuns<kMaxRunsPerLaunch> C;
    C.n = 0;
    long long reduce_ctas = 0;
    for (int i = 0; i < n; ++i) {
      reduce_ctas += (long long)add_reduce_run(&C, P.run[i], (int)reduce_ctas) * Hkv * runs[first + order[i]].batch;
      if (reduce_ctas > 0x7fffffffLL) return fail(UNIGIST_ERR_SHAPE, "packed sample too large for one grid");
    }
    for (int i = n; i < kMaxRunsPerLaunch; ++i) T.run[i] = T.run[0], P.run[i] = P.run[0];  // never selected
    for (int i = C.n; i < kMaxRunsPerLaunch; ++i) C.run[i] = ReduceRun();
    // the per-token kernels of this launch see the tensors from packed token tok_lo on
    BwdScratch part = sc;
    if (part.do_bf16) part.do_bf16 += tok_lo * Hq * D;
    part.dq32 += tok_lo * Hq * D;
    const size_t rdo = f32 ? 2 * rq : rq;
    if (int32_t rc = launch_prep(T, p, tok_hi - tok_lo, (const char*)d_o + tok_lo * rdo, (const char*)o + tok_lo * rq, part, st))
      return rc;
    if (int32_t rc = launch_fused(P, dim3((unsigned)ctas, 1, 1), p, scale, st)) return rc;
    if (int32_t rc = launch_dkdv_reduce(C, dim3((unsigned)reduce_ctas, 1, 1), p, scale, st)) return rc;
    if (int32_t rc = launch_convert(T, p, tok_hi - tok_lo, part, (char*)dq + tok_lo * rq, scale, st)) return rc;
  }
  return UNIGIST_OK;
}

int32_t bwd_sm100_take_timeout(bool* timed_out) {
  unsigned int flag = 0, zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&flag, g_bwd_timeout, sizeof(flag));
  if (e == cudaSuccess && flag) e = cudaMemcpyToSymbol(g_bwd_timeout, &zero, sizeof(zero));
  if (e != cudaSuccess) return fail(UNIGIST_ERR_CUDA, "reading the device status: %s", cudaGetErrorString(e));
  *timed_out = flag != 0;
  return UNIGIST_OK;
}

}  // namespace ug
