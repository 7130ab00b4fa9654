// Decode attention over the compacted, paged KV cache (Section 4.3): one query per sequence,
// every cache entry visible.  Split over keys: each thread block streams contiguous ranges of 64-token
// pages through a ring in shared memory.  A short walk is shared by a cluster of blocks that merge through
// distributed shared memory; otherwise the pages of all sequences are dealt out evenly and a second kernel adds
// up the sequences that were cut.  HBM-bound: K and V are read exactly once (64 sequences of 9216 tokens, 2.4 GB:
// 6.9 TB/s, the copy rate of the chip being 6.5; one of 1337 tokens: 5.7 us in a graph, 8.5 with two kernels).
//   producer warp:  per page one K and one V tile (64 tokens x 128 dims, 16 KB each) by TMA, 128-byte
//                   swizzle, into a 3-stage ring guarded by full / empty mbarriers; two thread blocks
//                   per SM keep about 128 KB of loads in flight.
//   consumer warps: three warps, one per ring stage, each takes every third page on its own and keeps a running
//                   (max, sum, output) for the G query heads of the KV head: S = Q K^T and O += P V
//                   with warp-level mma (m16n8k16, query heads padded to 16 rows), fragments
//                   fetched with ldmatrix.  The warps merge once, at the end.
#include <algorithm>
#include <cmath>

#include "sm100_ptx.cuh"
#include "ug_common.cuh"

namespace ug {
namespace {

using namespace sm100;

constexpr int PG = UNIGIST_PAGE_TOKENS;
constexpr int DD = 128;                     // head_dim
constexpr int STAGES = 3;
constexpr int PAGE_BYTES = PG * DD * 2;     // one K (or V) page of one KV head
constexpr int SLAB_BYTES = PAGE_BYTES / 2;  // [64 tokens x 64 dims], rows of 128 bytes
constexpr int STAGE_BYTES = 2 * PAGE_BYTES;
constexpr int kConsumers = STAGES;  // page i lives in stage i % STAGES and belongs to warp i % STAGES: every barrier
                                    // has one waiter, which sees each of its phases in turn
constexpr int THREADS = (kConsumers + 1) * 32;
constexpr float LOG2E = 1.4426950408889634f;

__device__ unsigned int g_decode_timeout = 0;

__device__ __forceinline__ void tma_load_2d(uint32_t smem_dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
// D (16x8 fp32) += A (16x16 bf16, row) * B (16x8 bf16, col)
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// x, or the largest finite number for an infinity or NaN (min of the magnitudes; the operand that is a number wins).
__device__ __forceinline__ float to_finite(float x) {
  float y;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(y) : "f"(x), "f"(3.402823466e38f));
  return y;
}

// Shared memory of a block: the ring, the barriers, the warps' results and, for the flat walk, the sequences'
// running page counts.  Two blocks share an SM (233,472 bytes with 1 KB of the system's own per block).
constexpr int kMaxFlatSeqs = 768;
struct DecSmem {
  static constexpr int kOffBars = STAGES * STAGE_BYTES;
  static constexpr int kOffMerge = kOffBars + 64;                              // [warps][8 heads][128 + 2] fp32
  static constexpr int kOffFirst = kOffMerge + kConsumers * 8 * (DD + 2) * 4;  // [S + 1] int
  static constexpr int kBytes = kOffFirst + (kMaxFlatSeqs + 1) * 4 + 1024 /*align*/;
};
static_assert(2 * (DecSmem::kBytes + 1024) <= 233472, "two blocks per SM");

struct DecParams {
  const __nv_bfloat16* q;
  const int32_t* table;
  const int32_t* seq_lens;
  const int32_t* holes;  // per sequence: [2] number of freed slots, [holes_off ..] the slots; or null
  __nv_bfloat16* o;
  float* lse;
  float* part_o;    // flat walk: [slots][Hq][128] unnormalised partial outputs
  float2* part_ml;  // [slots][Hq] (maximum in log2 units, sum)
  int S, Hq, Hkv, G, num_blocks, max_blocks, holes_stride, holes_off;
  float scale_log2;
};

// One element of O, and with it (d = 0) the row's LSE.  A sequence with nothing to attend to (length 0, or every
// slot freed) has O = 0 and LSE = -inf, not 0 / 0.
__device__ __forceinline__ void write_row(const DecParams& P, long long row, int d, float acc, float M, float L) {
  P.o[row * DD + d] = __float2bfloat16_rn(L > 0.f ? acc / L : 0.f);
  if (P.lse && d == 0) P.lse[row] = L > 0.f ? (M + log2f(L)) * 0.6931471805599453f : -INFINITY;
}

// Pages a sequence occupies, as far as its row of the block table names them.
__device__ __forceinline__ int pages_of(int len, int max_blocks) {
  return len > 0 ? min((len - 1) / PG + 1, max_blocks) : 0;
}

// first[i] = pages of the sequences before i (first[S] = all): every block works it out for itself, each thread
// adding up a run of neighbouring sequences.  `tmp`: 4 ints of shared memory.  Ends with a barrier.
__device__ __forceinline__ void page_prefix(const DecParams& P, int* first, int* tmp) {
  constexpr int kPer = kMaxFlatSeqs / THREADS;
  const int per = (P.S + THREADS - 1) / THREADS, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int n[kPer], sum = 0;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int s = threadIdx.x * per + i;
    n[i] = i < per && s < P.S ? pages_of(P.seq_lens[s], P.max_blocks) : 0;
  }
#pragma unroll
  for (int i = 0; i < kPer; ++i) sum += n[i];
  int incl = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += x;
  }
  if (lane == 31) tmp[warp] = incl;
  __syncthreads();
  int at = incl - sum;
  for (int w = 0; w < warp; ++w) at += tmp[w];
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int s = threadIdx.x * per + i;
    if (i < per && s <= P.S) first[s] = at;
    at += n[i];
  }
  // (where the runs end exactly at S, the last entry belongs to no thread's run)
  if (threadIdx.x == THREADS - 1 && THREADS * per == P.S) first[P.S] = at;
  __syncthreads();
}

// First page of share c when `total` pages are cut into n equal shares.
__device__ __forceinline__ int share_begin(int total, int n, int c) { return (int)((long long)total * c / n); }
// Shares of the flat walk: none may be empty, or a cut sequence would count a slot that nobody writes.
__device__ __forceinline__ int flat_shares(int total, int n) { return min(total, n); }

// What a block walks: runs of consecutive pages of one sequence.  Split by rank: one run, the rank's share of
// sequence blockIdx.z.  Flat: the block's share of all sequences' pages laid end to end, cut at the sequences' ends.
template <bool kFlat>
struct Walk {
  int seq, len, first, count;  // the current run: pages [first, first + count) of sequence seq
  bool whole;                  // ... which is all of the sequence
  int page, end;               // flat: position in the end-to-end order
  __device__ __forceinline__ bool next(const DecParams& P, const int* prefix) {
    if (page >= end) return false;
    if constexpr (kFlat) {
      while (prefix[seq + 1] <= page) ++seq;
      first = page - prefix[seq];
      count = min(prefix[seq + 1], end) - page;
      whole = first == 0 && page + count == prefix[seq + 1];
      len = P.seq_lens[seq];
      page += count;
    } else {
      page = end;
    }
    return true;
  }
};

// kFlat = false: grid (c, Hkv, S) in clusters of c blocks; the c blocks of a (sequence, KV head) share its pages
// evenly, merge through distributed shared memory and write O.  No scratch, one launch.
// kFlat = true: grid (n, Hkv); block x takes the x-th of n equal shares of all sequences' pages laid end to end, so
// that sequences of any lengths keep every block equally busy; a sequence that lies inside one share is finished
// there, one that is cut leaves a partial result per share in slot seq + share, for decode_combine_kernel.
template <bool kFlat>
__global__ void __launch_bounds__(THREADS, 2)
decode_split_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                    const __grid_constant__ DecParams P) {
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* gen = smem_dyn + (base - smem_u32(smem_dyn));
  const uint32_t bars = base + DecSmem::kOffBars;  // full[s] at + 8 s, empty[s] at + 8 (STAGES + s)
  float* merge = reinterpret_cast<float*>(gen + DecSmem::kOffMerge);
  int* prefix = reinterpret_cast<int*>(gen + DecSmem::kOffFirst);
  const int hk = blockIdx.y, G = P.G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(bars + 8 * i, 1);
      mbar_init(bars + 8 * (STAGES + i), 1);
    }
    mbar_fence_init();
  }
  pdl_wait();  // nothing above touches global memory
  Walk<kFlat> start;
  if constexpr (kFlat) {
    page_prefix(P, prefix, reinterpret_cast<int*>(merge));
    const int total = prefix[P.S], n = flat_shares(total, gridDim.x);
    const bool busy = (int)blockIdx.x < n;
    start.page = busy ? share_begin(total, n, blockIdx.x) : 0;
    start.end = busy ? share_begin(total, n, blockIdx.x + 1) : 0;
    int lo = 0, hi = P.S - 1;  // the sequence that holds the first page
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (prefix[mid] <= start.page) lo = mid; else hi = mid - 1;
    }
    start.seq = lo;
  } else {
    start.seq = blockIdx.z;
    start.len = P.seq_lens[start.seq];
    const int n = pages_of(start.len, P.max_blocks);
    start.first = share_begin(n, gridDim.x, blockIdx.x);
    start.count = share_begin(n, gridDim.x, blockIdx.x + 1) - start.first;
    start.whole = gridDim.x == 1;
    start.page = 0;
    start.end = 1;
    __syncthreads();
  }
  bool ok = true;

  if (warp == kConsumers) {
    // ------------------------------------------------------------ producer
    Walk<kFlat> w = start;
    int i = 0;  // pages loaded so far
    while (ok && w.next(P, prefix)) {
      const int32_t* row = P.table + (long long)w.seq * P.max_blocks;
      int32_t phys_mine = 0;
      for (int j = 0; j < w.count; ++j, ++i) {
        if ((j & 31) == 0) {  // the next 32 block-table entries, one per lane
          phys_mine = j + lane < w.count ? row[w.first + j + lane] : 0;
          phys_mine = min(max(phys_mine, 0), P.num_blocks - 1);  // never read outside the cache
        }
        const int phys = __shfl_sync(0xffffffffu, phys_mine, j & 31);
        const int st = i % STAGES, use = i / STAGES;
        if (use > 0) ok = mbar_wait_warp(bars + 8 * (STAGES + st), (use - 1) & 1);
        if (!ok) break;
        if (lane == 0) {
          const uint32_t full = bars + 8 * st, dst = base + st * STAGE_BYTES;
          const int row0 = (phys * P.Hkv + hk) * PG;
          mbar_arrive_expect_tx(full, STAGE_BYTES);
          tma_load_2d(dst, &tm_k, full, 0, row0);
          tma_load_2d(dst + SLAB_BYTES, &tm_k, full, 64, row0);
          tma_load_2d(dst + PAGE_BYTES, &tm_v, full, 0, row0);
          tma_load_2d(dst + PAGE_BYTES + SLAB_BYTES, &tm_v, full, 64, row0);
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) atomicExch(&g_decode_timeout, 1u);
  } else {
    // ------------------------------------------------------------ consumer: pages warp, warp + 3, ...
    const int g = lane >> 2, qc = lane & 3;   // query head (row of the padded 16 x 128 Q), column pair
    const int lr = lane & 7, lj = lane >> 3;  // ldmatrix: this lane supplies row lr of matrix lj
    Walk<kFlat> w = start;
    int i0 = 0;  // ring position of the run's first page
    while (w.next(P, prefix)) {
      // A fragments of Q for the 8 k-steps of 16 dims: rows 8..15 are padding (zero)
      uint32_t qa0[8], qa2[8];
      {
        const __nv_bfloat16* qp = P.q + ((long long)w.seq * P.Hq + hk * G + min(g, G - 1)) * DD;
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
          const uint32_t lo = *reinterpret_cast<const uint32_t*>(qp + 16 * ks + 2 * qc);
          const uint32_t hi = *reinterpret_cast<const uint32_t*>(qp + 16 * ks + 8 + 2 * qc);
          qa0[ks] = g < G ? lo : 0u;
          qa2[ks] = g < G ? hi : 0u;
        }
      }
      // cache slots that were freed and not yet reused (a decoding loop's eviction list) hold stale tokens
      const int32_t* hs = P.holes ? P.holes + (long long)w.seq * P.holes_stride : nullptr;
      const int n_holes = hs ? hs[2] : 0;
      const int hole_mine = lane < n_holes ? hs[P.holes_off + lane] : -1;  // (the first 32 stay in registers)
      float o[16][2];  // row g, dims 8 i + 2 qc + {0, 1}
#pragma unroll
      for (int i = 0; i < 16; ++i) o[i][0] = o[i][1] = 0.f;
      float m_run = -INFINITY, l_run = 0.f;  // of row g (the 4 lanes of a quad hold the same values)

      int j = warp - i0 % STAGES;
      if (j < 0) j += STAGES;
      for (; j < w.count && ok; j += kConsumers) {
        const int i = i0 + j, st = i % STAGES, use = i / STAGES;
        ok = mbar_wait_warp(bars + 8 * st, use & 1);
        if (!ok) break;
        const uint32_t sK = base + st * STAGE_BYTES, sV = sK + PAGE_BYTES;
        const int tok0 = (w.first + j) * PG;
        const int nvalid = min(PG, w.len - tok0);
        unsigned long long hole_bits = 0ull;
        for (int h0 = 0; h0 < n_holes; h0 += 32) {
          const int pos = (h0 == 0 ? hole_mine : (h0 + lane < n_holes ? hs[P.holes_off + h0 + lane] : -1)) - tok0;
          const bool mine = h0 + lane < n_holes && pos >= 0 && pos < PG;
          hole_bits |= (unsigned long long)__reduce_or_sync(0xffffffffu, mine && pos < 32 ? 1u << pos : 0u) |
                       (unsigned long long)__reduce_or_sync(0xffffffffu, mine && pos >= 32 ? 1u << (pos - 32) : 0u) << 32;
        }
        // S = Q K^T: 8 token tiles of 8, fp32
        float s[8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
#pragma unroll
          for (int e = 0; e < 4; ++e) s[nt][e] = 0.f;
          const int t = 8 * nt + lr;  // token whose row address this lane supplies
#pragma unroll
          for (int kq = 0; kq < 4; ++kq) {  // 32 dims = 4 chunks of 16 bytes per ldmatrix.x4
            const int chunk = (kq & 1) * 4 + lj;
            uint32_t k0, k1, k2, k3;
            ldsm_x4(sK + (kq >> 1) * SLAB_BYTES + t * 128 + ((chunk ^ (t & 7)) << 4), k0, k1, k2, k3);
            mma_bf16(s[nt], qa0[2 * kq], 0u, qa2[2 * kq], 0u, k0, k1);
            mma_bf16(s[nt], qa0[2 * kq + 1], 0u, qa2[2 * kq + 1], 0u, k2, k3);
          }
        }
        // running softmax of row g over the page's 64 tokens (this lane: tokens 8 nt + 2 qc + {0, 1})
        float mx = -INFINITY;
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const int tok = 8 * nt + 2 * qc;
          s[nt][0] = (tok < nvalid && !((hole_bits >> tok) & 1ull)) ? s[nt][0] * P.scale_log2 : -INFINITY;
          s[nt][1] = (tok + 1 < nvalid && !((hole_bits >> (tok + 1)) & 1ull)) ? s[nt][1] * P.scale_log2 : -INFINITY;
          mx = fmaxf(mx, fmaxf(s[nt][0], s[nt][1]));
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        const float m_new = fmaxf(m_run, mx);
        // (a page of nothing but freed slots leaves the maximum at -inf: keep the exponent arguments finite)
        const float f = m_new == -INFINITY ? 1.f : ex2(m_run - m_new);
        m_run = m_new;
        float ps = 0.f;
        // P as bf16 pairs, pa[nt] = tokens 8 nt + 2 qc + {0, 1} of row g, and what the rounding left over: it goes into
        // the padding rows 8 .. 15 of the same products, so that O sees P to 16 bits at no cost.  (Times an infinite V
        // a rest of zero gives NaN and one below zero the opposite infinity; the product with P alone is what counts there,
        // and it stays what it is when something finite is added.)
        uint32_t pa[8], pb[8];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
          const float p0 = m_new == -INFINITY ? 0.f : ex2(s[nt][0] - m_new);
          const float p1 = m_new == -INFINITY ? 0.f : ex2(s[nt][1] - m_new);
          ps += p0 + p1;
          pa[nt] = pack_bf16(p0, p1);
          pb[nt] = pack_bf16(p0 - __uint_as_float(pa[nt] << 16), p1 - __uint_as_float(pa[nt] & 0xffff0000u));
        }
        ps += __shfl_xor_sync(0xffffffffu, ps, 1);
        ps += __shfl_xor_sync(0xffffffffu, ps, 2);
        l_run = l_run * f + ps;
        // O = O f + P V, 4 k-steps of 16 tokens per pair of 8-dim tiles
#pragma unroll
        for (int np = 0; np < 8; ++np) {  // dim tiles 2 np, 2 np + 1
          float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
          const int chunk = 2 * np + (lj >> 1);  // 16-byte chunk of the 256-byte V row
#pragma unroll
          for (int ks = 0; ks < 4; ++ks) {
            const int t = 16 * ks + (lj & 1) * 8 + lr;
            uint32_t v0, v1, v2, v3;
            ldsm_x4_trans(sV + (chunk >> 3) * SLAB_BYTES + t * 128 + (((chunk & 7) ^ (t & 7)) << 4), v0, v1, v2, v3);
            mma_bf16(c0, pa[2 * ks], pb[2 * ks], pa[2 * ks + 1], pb[2 * ks + 1], v0, v1);
            mma_bf16(c1, pa[2 * ks], pb[2 * ks], pa[2 * ks + 1], pb[2 * ks + 1], v2, v3);
          }
          o[2 * np][0] = fmaf(o[2 * np][0], f, c0[0] + to_finite(c0[2]));
          o[2 * np][1] = fmaf(o[2 * np][1], f, c0[1] + to_finite(c0[3]));
          o[2 * np + 1][0] = fmaf(o[2 * np + 1][0], f, c1[0] + to_finite(c1[2]));
          o[2 * np + 1][1] = fmaf(o[2 * np + 1][1], f, c1[1] + to_finite(c1[3]));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bars + 8 * (STAGES + st));  // the stage may be refilled
      }
      i0 += w.count;
      // the warps' results for this run meet in shared memory
      if (g < G) {
        float* mrow = merge + (warp * 8 + g) * (DD + 2);
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) {
          mrow[8 * nt + 2 * qc] = o[nt][0];
          mrow[8 * nt + 2 * qc + 1] = o[nt][1];
        }
        if (qc == 0) {
          mrow[DD] = m_run;
          mrow[DD + 1] = l_run;
        }
      }
      named_barrier_sync(1, kConsumers * 32);
      const bool alone = kFlat ? w.whole : gridDim.x == 1;
      // split by rank: this block's result goes over the (consumed) first stage of the ring, for its peers to read
      float* mine = reinterpret_cast<float*>(gen);
      for (int idx = threadIdx.x; idx < G * DD; idx += kConsumers * 32) {
        const int h = idx / DD, d = idx % DD;
        float M = -INFINITY;
#pragma unroll
        for (int u = 0; u < kConsumers; ++u) M = fmaxf(M, merge[(u * 8 + h) * (DD + 2) + DD]);
        float acc = 0.f, L = 0.f;
#pragma unroll
        for (int u = 0; u < kConsumers; ++u) {
          const float* mrow = merge + (u * 8 + h) * (DD + 2);
          const float wgt = mrow[DD] == -INFINITY ? 0.f : ex2(mrow[DD] - M);
          acc += wgt * mrow[d];
          L += wgt * mrow[DD + 1];
        }
        if (alone) {
          write_row(P, (long long)w.seq * P.Hq + hk * G + h, d, acc, M, L);
        } else if (kFlat) {
          const long long slot = ((long long)w.seq + blockIdx.x) * P.Hq + hk * G + h;
          P.part_o[slot * DD + d] = acc;
          if (d == 0) P.part_ml[slot] = make_float2(M, L);
        } else {
          mine[h * (DD + 2) + d] = acc;
          if (d == 0) {
            mine[h * (DD + 2) + DD] = M;
            mine[h * (DD + 2) + DD + 1] = L;
          }
        }
      }
      if (kFlat) named_barrier_sync(1, kConsumers * 32);  // `merge` is free for the next run
    }
    if (!ok && lane == 0) atomicExch(&g_decode_timeout, 1u);
  }
  if constexpr (!kFlat) {
    if (gridDim.x == 1) return;
    // each block of the cluster merges its share of the G * 128 outputs over all the blocks' results
    cluster_sync();
    const int c = gridDim.x, per = (G * DD + c - 1) / c;
    const int lo = blockIdx.x * per, hi = min(lo + per, G * DD);
    for (int idx = lo + threadIdx.x; idx < hi; idx += THREADS) {
      const int h = idx / DD, d = idx % DD;
      const uint32_t ml_at = base + (h * (DD + 2) + DD) * 4, o_at = base + (h * (DD + 2) + d) * 4;
      float M = -INFINITY;
#pragma unroll 8
      for (int r = 0; r < c; ++r) M = fmaxf(M, ld_cluster_f32(ml_at, r));
      float acc = 0.f, L = 0.f;
#pragma unroll 8
      for (int r = 0; r < c; ++r) {
        const float m = ld_cluster_f32(ml_at, r);
        const float wgt = m == -INFINITY ? 0.f : ex2(m - M);
        acc += wgt * ld_cluster_f32(o_at, r);
        L += wgt * ld_cluster_f32(ml_at + 4, r);
      }
      write_row(P, (long long)blockIdx.z * P.Hq + hk * G + h, d, acc, M, L);
    }
    cluster_sync();  // the peers have read this block's shared memory
  }
}

// Flat walk: one block per (sequence, KV head) adds up the partial results of a sequence that was cut; a warp
// takes a query head, a lane four dims.  A sequence inside one share is finished already; an empty one has O = 0.
__global__ void __launch_bounds__(THREADS)
decode_combine_kernel(const __grid_constant__ DecParams P, int max_shares) {
  __shared__ int first[kMaxFlatSeqs + 1];
  __shared__ int tmp[THREADS / 32];
  pdl_wait();
  page_prefix(P, first, tmp);
  const int seq = blockIdx.x, hk = blockIdx.y, total = first[P.S], warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int a = first[seq], b = first[seq + 1], n = flat_shares(total, max_shares);
  // the shares that hold the sequence's first and last page
  const int c0 = b > a ? (int)((((long long)a + 1) * n - 1) / total) : 0;
  const int c1 = b > a ? (int)(((long long)b * n - 1) / total) : 0;
  if (b > a && c0 == c1) return;
  for (int h = warp; h < P.G; h += THREADS / 32) {
    const long long row = (long long)seq * P.Hq + hk * P.G + h;
    float M = -INFINITY, L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (b > a) {
      const long long slot0 = ((long long)seq + c0) * P.Hq + hk * P.G + h;
      const int cnt = c1 - c0 + 1;
      for (int i = lane; i < cnt; i += 32) M = fmaxf(M, P.part_ml[slot0 + (long long)i * P.Hq].x);
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
#pragma unroll 8
      for (int i = 0; i < cnt; ++i) {
        const long long slot = slot0 + (long long)i * P.Hq;
        const float2 ml = P.part_ml[slot];
        const float4 x = reinterpret_cast<const float4*>(P.part_o + slot * DD)[lane];
        const float wgt = ml.x == -INFINITY ? 0.f : ex2(ml.x - M);
        acc.x += wgt * x.x, acc.y += wgt * x.y, acc.z += wgt * x.z, acc.w += wgt * x.w;
        L += wgt * ml.y;
      }
    }
    reinterpret_cast<uint2*>(P.o + row * DD)[lane] =
        L > 0.f ? make_uint2(pack_bf16(acc.x / L, acc.y / L), pack_bf16(acc.z / L, acc.w / L)) : make_uint2(0u, 0u);
    if (P.lse && lane == 0) P.lse[row] = L > 0.f ? (M + log2f(L)) * 0.6931471805599453f : -INFINITY;
  }
}

}  // namespace

// Splits per sequence of the smallest scratch a call accepts: whole waves of 2 blocks per SM.
static int decode_num_splits(int S, int Hkv, int max_blocks) {
  constexpr int kMaxSplits = 32;
  const long long slots = (long long)sm_count() * 2;
  const long long base = (long long)S * Hkv;
  int best = 1;
  double best_eff = -1.0;
  for (int sp = 1; sp <= kMaxSplits; ++sp) {
    const int bps = (max_blocks + sp - 1) / sp;
    if (sp > 1 && bps < 4) break;
    if ((max_blocks + bps - 1) / bps != sp) continue;  // this count leaves an empty split
    const double waves = (double)(base * sp) / (double)slots;
    const double eff = waves / ceil(waves);
    if (eff > best_eff + 1e-9) {
      best_eff = eff;
      best = sp;
    }
  }
  return best;
}

namespace {
constexpr size_t kSlotBytes = (DD + 2) * sizeof(float);  // per query head

// How a decode call is cut.  flat = 0: clusters of `c` blocks per (sequence, KV head).  flat > 0: that many shares.
struct DecPlan {
  int c, flat;
};
DecPlan decode_plan(int S, int Hq, int Hkv, int max_blocks) {
  const long long slots = (long long)sm_count() * 2, pairs = (long long)S * Hkv;
  // few (sequence, KV head) pairs: enough blocks per pair to fill the chip, no more than shorten the walk of the
  // longest possible sequence (a block's three consumer warps take three pages at a time)
  auto rounds = [&](int c) { return ((max_blocks + c - 1) / c + kConsumers - 1) / kConsumers; };
  int best = 1;
  for (int c = 2; c <= 16 && pairs * c <= slots; c *= 2)
    if (rounds(c) < rounds(best)) best = c;
  // Up to four rounds a block stay with the clusters: a walk that short is all latency, and the flat walk pays for its
  // page counts, the cut sequences' second kernel and a merge at every sequence's end (64 sequences of 20 to 500
  // tokens: 33 us flat, 24 one block each).  Longer walks are bound by the memory system, and there an even share of
  // the pages per block wins, the more so the more the lengths differ (17 sequences of 150 to 6000 tokens: 52 -> 44 us).
  if (rounds(best) <= 4) return {best, 0};
  const long long n = slots / Hkv;
  const size_t need = (size_t)(S - 1 + n) * Hq * kSlotBytes;
  // the flat walk's page counts have to fit (shared memory, 31 bits), and its partial results the built-in scratch
  if (S > kMaxFlatSeqs || (long long)S * max_blocks > 0x7fffffffLL || n < 2 ||
      need > (size_t)UNIGIST_DECODE_STATIC_SCRATCH_BYTES)
    return {best, 0};
  return {1, (int)n};
}
}  // namespace

size_t decode_min_scratch_bytes(int S, int Hq, int Hkv, int D, int max_blocks) {
  return ((size_t)S * Hq * decode_num_splits(S, Hkv, max_blocks) * (D + 2) * sizeof(float) + 255) / 256 * 256;
}

size_t decode_scratch_bytes(int S, int Hq, int Hkv, int D, int max_blocks) {
  const DecPlan plan = decode_plan(S, Hq, Hkv, max_blocks);
  const size_t flat = plan.flat ? ((size_t)(S - 1 + plan.flat) * Hq * kSlotBytes + 255) / 256 * 256 : 0;
  return std::max(decode_min_scratch_bytes(S, Hq, Hkv, D, max_blocks), flat);
}

int32_t launch_decode(int S, int Hq, int Hkv, int D, float scale, const void* q, const void* kc,
                      const void* vc, int num_blocks, const int32_t* table, int max_blocks,
                      const int32_t* seq_lens, void* o, float* lse, void* ws, size_t ws_bytes, cudaStream_t st,
                      const int32_t* holes, int holes_stride, int holes_off) {
  (void)D;
  const int G = Hq / Hkv;
  if (G < 1 || G > 8) return fail(UNIGIST_ERR_UNSUPPORTED, "decode supports 1 to 8 query heads per KV head, got %d", G);
  DecPlan plan = decode_plan(S, Hq, Hkv, max_blocks);
  if (plan.flat) {  // a caller with the least accepted scratch gets as many shares as it holds
    const long long fit = (long long)(ws_bytes / ((size_t)Hq * kSlotBytes)) - S + 1;
    if (fit < plan.flat) plan.flat = fit >= 2 ? (int)fit : 0;
  }
  // the caches as 2-D tensors [num_blocks * Hkv * 64 tokens, 128 dims], tiles of 64 tokens x 64 dims
  CUtensorMap mk, mv;
  const long long rows = (long long)num_blocks * Hkv * PG;
  if (int32_t rc = encode_map_2d_bf16(&mk, kc, rows, DD, PG, 64)) return rc;
  if (int32_t rc = encode_map_2d_bf16(&mv, vc, rows, DD, PG, 64)) return rc;
  DecParams P;
  P.q = (const __nv_bfloat16*)q;
  P.table = table;
  P.seq_lens = seq_lens;
  P.holes = holes;
  P.o = (__nv_bfloat16*)o;
  P.lse = lse;
  P.part_o = (float*)ws;
  P.part_ml = reinterpret_cast<float2*>((float*)ws + (size_t)(plan.flat ? S - 1 + plan.flat : 0) * Hq * DD);
  P.S = S, P.Hq = Hq, P.Hkv = Hkv, P.G = G, P.num_blocks = num_blocks, P.max_blocks = max_blocks;
  P.holes_stride = holes_stride, P.holes_off = holes_off;
  P.scale_log2 = scale * LOG2E;
  const auto kern = plan.flat ? decode_split_kernel<true> : decode_split_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, DecSmem::kBytes);
  if (e == cudaSuccess && plan.c > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return fail(UNIGIST_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
  {
    KernelScope ks("decode_split_kernel", st);
    launch_chained(kern, plan.flat ? dim3(plan.flat, Hkv) : dim3(plan.c, Hkv, S), THREADS, DecSmem::kBytes, st,
                   plan.flat ? 1 : plan.c, mk, mv, P);
  }
  if (int32_t rc = check_launch("decode split kernel")) return rc;
  if (!plan.flat) return UNIGIST_OK;
  {
    KernelScope ks("decode_combine_kernel", st);
    launch_chained(decode_combine_kernel, dim3(S, Hkv), THREADS, 0, st, 1, P, plan.flat);
  }
  return check_launch("decode combine kernel");
}

int32_t decode_take_timeout(bool* timed_out) {
  unsigned int flag = 0, zero = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&flag, g_decode_timeout, sizeof(flag));
  if (e == cudaSuccess && flag) e = cudaMemcpyToSymbol(g_decode_timeout, &zero, sizeof(zero));
  if (e != cudaSuccess) return fail(UNIGIST_ERR_CUDA, "reading the device status: %s", cudaGetErrorString(e));
  *timed_out = flag != 0;
  return UNIGIST_OK;
}

}  // namespace ug

// ------------------------------------------------------------------------------------------------
// Decode without caller-provided scratch.  The split-KV partial results go to a fixed array that
// is part of the library image, so this entry point needs no allocation from anyone.
#include <cmath>
#include <mutex>

namespace {

// Lives in the global memory of every GPU that loads the library, from load until process exit.
static __device__ __align__(256) unsigned char g_decode_static_scratch[UNIGIST_DECODE_STATIC_SCRATCH_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
void* g_static_scratch_ptr[kMaxDevices] = {};

// In host code the array's name is only a handle; the device address has to be asked for, once
// per device, with that device current.
int32_t static_scratch_address(void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return ug::fail(UNIGIST_ERR_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return ug::fail(UNIGIST_ERR_UNSUPPORTED, "device ordinal %d out of range", dev);
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_scratch_ptr[dev]) {
    void* ptr = nullptr;
    e = cudaGetSymbolAddress(&ptr, g_decode_static_scratch);
    if (e != cudaSuccess || !ptr)
      return ug::fail(UNIGIST_ERR_CUDA, "cudaGetSymbolAddress(static decode scratch): %s", cudaGetErrorString(e));
    g_static_scratch_ptr[dev] = ptr;
  }
  *out = g_static_scratch_ptr[dev];
  return UNIGIST_OK;
}

}  // namespace

extern "C" int32_t unigist_decode_static(int32_t S, int32_t Hq, int32_t Hkv, int32_t D, float softmax_scale,
                                         const void* q, const void* kc, const void* vc, int32_t num_blocks,
                                         const int32_t* table, int32_t max_blocks, const int32_t* seq_lens,
                                         void* o, float* lse, void* stream) {
  using namespace ug;
  if (S < 1 || Hq < 1 || Hkv < 1 || max_blocks < 1 || num_blocks < 1)
    return fail(UNIGIST_ERR_INVALID_ARG, "decode has a non-positive size");
  if (Hq % Hkv) return fail(UNIGIST_ERR_SHAPE, "num_q_heads %d is not a multiple of num_kv_heads %d", Hq, Hkv);
  if (D != 128) return fail(UNIGIST_ERR_SHAPE, "decode supports head_dim 128, got %d", D);
  if (Hq / Hkv > 8) return fail(UNIGIST_ERR_UNSUPPORTED, "decode supports at most 8 query heads per KV head");
  if (!q || !kc || !vc || !table || !seq_lens || !o) return fail(UNIGIST_ERR_INVALID_ARG, "a pointer is NULL");
  if (!aligned16(q) || !aligned16(kc) || !aligned16(vc) || !aligned16(o))
    return fail(UNIGIST_ERR_ALIGNMENT, "tensor pointers must be 16-byte aligned");
  if (!(softmax_scale >= 0.f) || std::isinf(softmax_scale))
    return fail(UNIGIST_ERR_INVALID_ARG, "softmax_scale must be finite and >= 0");
  const size_t need = unigist_decode_workspace_bytes(S, Hq, Hkv, D, max_blocks);
  if (need > (size_t)UNIGIST_DECODE_STATIC_SCRATCH_BYTES)
    return fail(UNIGIST_ERR_WORKSPACE,
                "this decode needs %zu bytes of scratch but the built-in array holds %zu: use unigist_decode "
                "with a caller-provided workspace, or decode fewer sequences per call",
                need, (size_t)UNIGIST_DECODE_STATIC_SCRATCH_BYTES);
  void* scratch = nullptr;
  if (int32_t rc = static_scratch_address(&scratch)) return rc;
  const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)D);
  return launch_decode(S, Hq, Hkv, D, scale, q, kc, vc, num_blocks, table, max_blocks, seq_lens, o, lse, scratch,
                       UNIGIST_DECODE_STATIC_SCRATCH_BYTES, (cudaStream_t)stream);
}
