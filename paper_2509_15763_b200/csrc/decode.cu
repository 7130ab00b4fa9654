// Decode attention over the compacted, paged KV cache (Section 4.3): one query per sequence,
// every cache entry visible.  Split over keys: each thread block streams contiguous ranges of 64-token
// pages through a ring in shared memory.  A short walk is shared by a cluster of blocks that merge through
// distributed shared memory, or by more blocks whose results a second kernel adds up; otherwise the pages of all
// sequences are dealt out evenly, and the second kernel adds up the sequences that were cut (decode_plan).  HBM-bound:
// K and V are read exactly once (64 sequences of 9216 tokens, 2.4 GB: 6.9 TB/s, the copy rate of the chip being 6.5;
// one of 1337 tokens: 5.7 us in a graph, 8.5 with two kernels).
//   producer warp:  per page one K and one V tile (64 tokens x 128 dims, 16 KB each) by TMA, 128-byte
//                   swizzle, into a 3-stage ring guarded by mbarriers (full / free); two thread blocks
//                   per SM keep about 128 KB of loads in flight.
//   consumer warps: three warps, one per ring stage, each takes every third page on its own and keeps a running
//                   (max, sum, output) for the G query heads of the KV head: S = Q K^T and O += P V
//                   with warp-level mma (m16n8k16, query heads padded to 16 rows), fragments
//                   fetched with ldmatrix.  The warps merge once, at the end.
#include <algorithm>
#include <atomic>
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

// Shared memory of a block: the ring, the barriers, the warps' results and, for the flat walk, the running page
// counts.  Two blocks share an SM (233,472 bytes with 1 KB of the system's own per block).
constexpr int kRow = DD + 4;  // a head's result: 128 sums, maximum, sum of the weights (rows of whole 16-byte pieces)
struct DecSmem {
  static constexpr int kOffBars = STAGES * STAGE_BYTES;
  static constexpr int kOffMerge = kOffBars + 128;                             // [warps][8 heads][kRow] fp32
  static constexpr int kOffFirst = kOffMerge + kConsumers * 8 * kRow * 4;  // [THREADS + 1] 64-bit
  static constexpr int kBytes = kOffFirst + (THREADS + 1) * 8 + 1024 /*align*/;
};
static_assert(2 * (DecSmem::kBytes + 1024) <= 233472, "two blocks per SM");

struct DecParams {
  const __nv_bfloat16* q;
  const int32_t* table;
  const int32_t* seq_lens;
  const int32_t* holes;  // per sequence: [2] number of freed slots, [holes_off ..] the slots; or null
  __nv_bfloat16* o;
  float* lse;
  long long* pages_before;  // flat walk: [S + 1] pages of the sequences before each, left by the first kernel for the second
  int splits;               // even split: blocks per (sequence, KV head) whose partial results the second kernel adds, or 0
  float* part_o;            // [slots][Hq][128] unnormalised partial outputs
  float2* part_ml;          // [slots][Hq] (maximum in log2 units, sum)
  int S, Hq, Hkv, G, num_blocks, max_blocks, holes_stride, holes_off;
  float scale_log2;
};

__device__ __forceinline__ void add_weighted(float4& acc, float& L, float weight, float4 x, float l) {
  acc.x += weight * x.x, acc.y += weight * x.y, acc.z += weight * x.z, acc.w += weight * x.w;
  L += weight * l;
}
// Four elements of O, and with them (d = 0) the row's LSE.  A sequence with nothing to attend to (length 0, or every
// slot freed) has O = 0 and LSE = -inf, not 0 / 0.
__device__ __forceinline__ void write_row(const DecParams& P, long long row, int d, float4 acc, float M, float L) {
  *reinterpret_cast<uint2*>(P.o + row * DD + d) =
      L > 0.f ? make_uint2(pack_bf16(acc.x / L, acc.y / L), pack_bf16(acc.z / L, acc.w / L)) : make_uint2(0u, 0u);
  if (P.lse && d == 0) P.lse[row] = L > 0.f ? (M + log2f(L)) * 0.6931471805599453f : -INFINITY;
}

// Pages a sequence occupies, as far as its row of the block table names them.
__device__ __forceinline__ int pages_of(int len, int max_blocks) {
  return len > 0 ? min((len - 1) / PG + 1, max_blocks) : 0;
}

// The sequences are taken in groups of `per` neighbours, one group a thread: first[t] = pages of the groups before t
// (first[THREADS] = all).  Every block works it out for itself.  `tmp`: one number per warp.  Ends with a barrier.
__device__ __forceinline__ void page_prefix(const DecParams& P, int per, long long* first, long long* tmp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int s0 = min((int)threadIdx.x * per, P.S), s1 = min(s0 + per, P.S);
  long long sum = 0;
  for (int i = s0; i < s1; i += 8) {
    int n[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) n[u] = i + u < s1 ? pages_of(P.seq_lens[i + u], P.max_blocks) : 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) sum += n[u];
  }
  long long incl = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const long long x = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += x;
  }
  if (lane == 31) tmp[warp] = incl;
  __syncthreads();
  long long at = incl - sum;
  for (int w = 0; w < warp; ++w) at += tmp[w];
  first[threadIdx.x] = at;
  if (threadIdx.x == THREADS - 1) first[THREADS] = at + sum;
  __syncthreads();
}

// P.pages_before from the groups' counts: a warp of every block of the first KV head takes some of the groups.
__device__ __forceinline__ void leave_pages_before(const DecParams& P, int per, const long long* first) {
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.x; t < THREADS; t += gridDim.x) {
    const int s1 = min((t + 1) * per, P.S);
    long long at = first[t];
    for (int s = t * per + lane; s - lane < s1; s += 32) {
      const int n = s < s1 ? pages_of(P.seq_lens[s], P.max_blocks) : 0;
      long long incl = n;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const long long x = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += x;
      }
      if (s < s1) P.pages_before[s] = at + incl - n;
      at += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  if (blockIdx.x == 0 && lane == 0) P.pages_before[P.S] = first[THREADS];
}

// First page of share c when `total` pages are cut into n equal shares.
__device__ __forceinline__ long long share_begin(long long total, int n, int c) { return total * c / n; }
// Shares of the flat walk: a page for each of a block's warps where there are enough (and none may be empty, or a cut
// sequence would count a slot that nobody writes).
__device__ __forceinline__ int flat_shares(long long total, int n) {
  return (int)min((total + kConsumers - 1) / kConsumers, (long long)n);
}
// Slots for the partial results of S sequences cut into n shares, and the slot of a share's part of a sequence.  Along the
// walk sequence and share never fall and one of them rises from one part to the next, so their sum tells the parts apart;
// and a share holds at most two parts, the end of a sequence and the beginning of one.  Whichever takes less room.
__host__ __device__ __forceinline__ int flat_slots(int S, int n) { return n + (S - 1 < n ? S - 1 : n); }
__device__ __forceinline__ long long flat_slot(int S, int n, int seq, int share, bool begins) {
  return S - 1 < n ? seq + share : 2 * share + (begins ? 1 : 0);
}

// What a block walks: runs of consecutive pages of one sequence.  Split by rank: one run, the rank's share of
// sequence blockIdx.z.  Flat: the block's share of all sequences' pages laid end to end, cut at the sequences' ends.
template <bool kFlat>
struct Walk {
  int seq, len, first, count;  // the current run: pages [first, first + count) of sequence seq
  bool whole;                  // ... which is all of the sequence
  long long page, end;         // flat: position in the end-to-end order
  long long before;            // flat: pages before sequence seq
  __device__ __forceinline__ bool next(const DecParams& P) {
    if (page >= end) return false;
    if constexpr (kFlat) {
      int n;
      for (;; ++seq) {
        if (seq >= P.S) return false;
        len = P.seq_lens[seq];
        n = pages_of(len, P.max_blocks);
        if (before + n > page) break;
        before += n;
      }
      first = (int)(page - before);
      count = (int)(min(before + n, end) - page);
      whole = count == n;
      page += count;
    } else {
      page = end;
    }
    return true;
  }
};

// kFlat = false: grid (c, Hkv, S); the c blocks of a (sequence, KV head) share its pages evenly.  They are a cluster, merge
// through distributed shared memory and write O (no scratch, one launch), or (P.splits = c) leave partial results.
// kFlat = true: grid (n, Hkv); block x takes the x-th of n equal shares of all sequences' pages laid end to end, so
// that sequences of any lengths keep every block equally busy; a sequence that lies inside one share is finished
// there, one that is cut leaves a partial result per share in its flat_slot, for decode_combine_kernel.
// kApart: a stage's K and V arrive and are free again each by itself, instead of together (full_k, free_v).  A warp has one
// stage; with barriers of its own the K of its next page comes under this one's softmax and P V.  That pays where walks are
// short and bound by latency and a warp takes more than one page (8 sequences of 2112 tokens: 11.3 -> 10.6 us); with one page
// a warp it only costs (one of 1337: 5.39 -> 5.41), and a long walk is bound by the memory system, which takes K and V apart
// badly (past six rounds of pages: one of 65536, 44.5 -> 45.3 us; flat, 64 of 9216: 345 -> 357).
template <bool kFlat, bool kApart>
__global__ void __launch_bounds__(THREADS, 2)
decode_split_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                    const __grid_constant__ DecParams P) {
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* gen = smem_dyn + (base - smem_u32(smem_dyn));
  // barriers, + 8 * stage; together, a stage's K and V use full_k and free_v only, which come first
  const uint32_t full_k = base + DecSmem::kOffBars, free_v = full_k + 8 * STAGES, full_v = free_v + 8 * STAGES,
                 free_k = full_v + 8 * STAGES;
  float* merge = reinterpret_cast<float*>(gen + DecSmem::kOffMerge);
  long long* first = reinterpret_cast<long long*>(gen + DecSmem::kOffFirst);
  const int hk = blockIdx.y, G = P.G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < (kApart ? 4 : 2) * STAGES; ++i) mbar_init(full_k + 8 * i, 1);
    mbar_fence_init();
  }
  pdl_wait();  // nothing above touches global memory
  Walk<kFlat> start;
  const int per = (P.S + THREADS - 1) / THREADS;  // flat: sequences per group of the page counts
  if constexpr (kFlat) {
    page_prefix(P, per, first, reinterpret_cast<long long*>(merge));
    const long long total = first[THREADS];
    const int n = flat_shares(total, gridDim.x);
    const bool busy = (int)blockIdx.x < n;
    start.page = busy ? share_begin(total, n, blockIdx.x) : 0;
    start.end = busy ? share_begin(total, n, blockIdx.x + 1) : 0;
    int lo = 0, hi = THREADS - 1;  // the group that holds the first page
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (first[mid] <= start.page) lo = mid; else hi = mid - 1;
    }
    start.seq = lo * per;
    start.before = first[lo];
  } else {
    start.seq = blockIdx.z;
    start.len = P.seq_lens[start.seq];
    const int n = pages_of(start.len, P.max_blocks);
    start.first = (uint32_t)n * blockIdx.x / gridDim.x;  // (at most 2^25 pages, 32 blocks)
    start.count = (uint32_t)n * (blockIdx.x + 1) / gridDim.x - start.first;
    start.whole = gridDim.x == 1;
    start.page = 0;
    start.end = 1;
    __syncthreads();
  }
  bool ok = true;

  if (warp == kConsumers) {
    // ------------------------------------------------------------ producer
    Walk<kFlat> w = start;
    int i0 = 0;  // ring position of the run's first page
    while (ok && w.next(P)) {
      const int32_t* row = P.table + (long long)w.seq * P.max_blocks;
      int32_t phys_mine = 0;
      auto entries = [&](int j) {  // the next 32 block-table entries, one per lane
        if (j & 31) return;
        phys_mine = j + lane < w.count ? row[w.first + j + lane] : 0;
        phys_mine = min(max(phys_mine, 0), P.num_blocks - 1);  // never read outside the cache
      };
      auto row_of = [&](int j) { return (__shfl_sync(0xffffffffu, phys_mine, j & 31) * P.Hkv + hk) * PG; };
      if constexpr (!kApart) {
        for (int j = 0; j < w.count; ++j) {
          entries(j);
          const int row0 = row_of(j), i = i0 + j, st = i % STAGES, use = i / STAGES;
          if (use > 0) ok = mbar_wait_warp(free_v + 8 * st, (use - 1) & 1);
          if (!ok) break;
          if (lane == 0) {
            const uint32_t full = full_k + 8 * st, dst = base + st * STAGE_BYTES;
            mbar_arrive_expect_tx(full, STAGE_BYTES);
            tma_load_2d(dst, &tm_k, full, 0, row0);
            tma_load_2d(dst + SLAB_BYTES, &tm_k, full, 64, row0);
            tma_load_2d(dst + PAGE_BYTES, &tm_v, full, 0, row0);
            tma_load_2d(dst + PAGE_BYTES + SLAB_BYTES, &tm_v, full, 64, row0);
          }
          __syncwarp();
        }
      } else {
        for (int j0 = 0; j0 < w.count && ok; j0 += STAGES) {  // the K of a round of pages, then their V
          int row0[STAGES];
#pragma unroll
          for (int u = 0; u < STAGES; ++u) {
            if (j0 + u >= w.count) break;
            entries(j0 + u);
            row0[u] = row_of(j0 + u);
          }
#pragma unroll
          for (int v = 0; v < 2; ++v) {
#pragma unroll
            for (int u = 0; u < STAGES; ++u) {
              const int i = i0 + j0 + u, st = i % STAGES, use = i / STAGES;
              if (j0 + u >= w.count || !ok) break;
              if (use > 0) ok = mbar_wait_warp((v ? free_v : free_k) + 8 * st, (use - 1) & 1);
              if (!ok) break;
              if (lane == 0) {
                const uint32_t full = (v ? full_v : full_k) + 8 * st, dst = base + st * STAGE_BYTES + v * PAGE_BYTES;
                mbar_arrive_expect_tx(full, PAGE_BYTES);
                tma_load_2d(dst, v ? &tm_v : &tm_k, full, 0, row0[u]);
                tma_load_2d(dst + SLAB_BYTES, v ? &tm_v : &tm_k, full, 64, row0[u]);
              }
              __syncwarp();
            }
          }
        }
      }
      i0 += w.count;
    }
    if (!ok && lane == 0) atomicExch(&g_decode_timeout, 1u);
  } else {
    // ------------------------------------------------------------ consumer: pages warp, warp + 3, ...
    const int g = lane >> 2, qc = lane & 3;   // query head (row of the padded 16 x 128 Q), column pair
    const int lr = lane & 7, lj = lane >> 3;  // ldmatrix: this lane supplies row lr of matrix lj
    Walk<kFlat> w = start;
    int i0 = 0;  // ring position of the run's first page
    while (w.next(P)) {
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
        ok = mbar_wait_warp(full_k + 8 * st, use & 1);
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
        if (kApart) {  // the next K may come
          __syncwarp();
          if (lane == 0) mbar_arrive(free_k + 8 * st);
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
        if (kApart) ok = mbar_wait_warp(full_v + 8 * st, use & 1);
        if (!ok) break;
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
        if (lane == 0) mbar_arrive(free_v + 8 * st);
      }
      i0 += w.count;
      // the warps' results for this run meet in shared memory
      if (g < G) {
        float* mrow = merge + (warp * 8 + g) * kRow;
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
      const long long part = kFlat ? flat_slot(P.S, gridDim.x, w.seq, blockIdx.x, w.first == 0)
                                   : (long long)w.seq * P.splits + blockIdx.x;
      for (int idx = threadIdx.x; idx < G * (DD / 4); idx += kConsumers * 32) {
        const int h = idx / (DD / 4), d = idx % (DD / 4) * 4;
        float M = -INFINITY;
#pragma unroll
        for (int u = 0; u < kConsumers; ++u) M = fmaxf(M, merge[(u * 8 + h) * kRow + DD]);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float L = 0.f;
#pragma unroll
        for (int u = 0; u < kConsumers; ++u) {
          const float* mrow = merge + (u * 8 + h) * kRow;
          add_weighted(acc, L, mrow[DD] == -INFINITY ? 0.f : ex2(mrow[DD] - M), *reinterpret_cast<const float4*>(mrow + d), mrow[DD + 1]);
        }
        if (alone) {
          write_row(P, (long long)w.seq * P.Hq + hk * G + h, d, acc, M, L);
        } else if (kFlat || P.splits) {
          const long long slot = part * P.Hq + hk * G + h;
          *reinterpret_cast<float4*>(P.part_o + slot * DD + d) = acc;
          if (d == 0) P.part_ml[slot] = make_float2(M, L);
        } else {
          *reinterpret_cast<float4*>(mine + h * kRow + d) = acc;
          if (d == 0) {
            mine[h * kRow + DD] = M;
            mine[h * kRow + DD + 1] = L;
          }
        }
      }
      if (kFlat) named_barrier_sync(1, kConsumers * 32);  // `merge` is free for the next run
    }
    if (!ok && lane == 0) atomicExch(&g_decode_timeout, 1u);
    if (kFlat && warp == 0 && blockIdx.y == 0) leave_pages_before(P, per, first);
  }
  if constexpr (!kFlat) {
    if (gridDim.x == 1 || P.splits) return;
    // each block of the cluster merges its share of the G * 128 outputs over all the blocks' results
    cluster_sync();
    const int c = gridDim.x, per = (G * (DD / 4) + c - 1) / c;
    const int lo = blockIdx.x * per, hi = min(lo + per, G * (DD / 4));
    for (int idx = lo + threadIdx.x; idx < hi; idx += THREADS) {
      const int h = idx / (DD / 4), d = idx % (DD / 4) * 4;
      const uint32_t ml_at = base + (h * kRow + DD) * 4, o_at = base + (h * kRow + d) * 4;
      float M = -INFINITY;
#pragma unroll 8
      for (int r = 0; r < c; ++r) M = fmaxf(M, ld_cluster_f32(ml_at, r));
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float L = 0.f;
#pragma unroll 8
      for (int r = 0; r < c; ++r) {
        const float m = ld_cluster_f32(ml_at, r);
        add_weighted(acc, L, m == -INFINITY ? 0.f : ex2(m - M), ld_cluster_v4(o_at, r), ld_cluster_f32(ml_at + 4, r));
      }
      write_row(P, (long long)blockIdx.z * P.Hq + hk * G + h, d, acc, M, L);
    }
    cluster_sync();  // the peers have read this block's shared memory
  }
}

// Adds up the partial results of sequences that were cut.  kWide: a block per (sequence, query head), whose warps share the
// parts; otherwise a block per (sequence, KV head), a warp per query head.  A lane takes four dims.  In the flat walk a
// sequence inside one share is finished already; an empty one has O = 0.
template <bool kWide>
__global__ void __launch_bounds__(THREADS)
decode_combine_kernel(const __grid_constant__ DecParams P, int max_shares) {
  constexpr int kWarps = THREADS / 32, kStep = kWide ? kWarps : 1, kLoads = 8;  // parts in flight per warp
  __shared__ float4 sums[kWide ? kWarps : 1][32];
  __shared__ float2 stats[kWide ? kWarps : 1];
  pdl_wait();
  const int seq = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int c0 = 0, cnt = P.splits;  // the shares that hold the sequence: the first, and how many
  if (!P.splits) {
    const long long a = P.pages_before[seq], b = P.pages_before[seq + 1], total = P.pages_before[P.S];
    const int n = flat_shares(total, max_shares);
    if (b > a) {
      c0 = (int)(((a + 1) * n - 1) / total);
      cnt = (int)((b * n - 1) / total) - c0 + 1;
      if (cnt == 1) return;
    }
  }
  const int h_begin = kWide ? blockIdx.y : blockIdx.y * P.G + warp, h_end = kWide ? h_begin + 1 : (blockIdx.y + 1) * P.G;
  for (int h = h_begin; h < h_end; h += kWarps) {
    auto slot_of = [&](int i) {
      return (P.splits ? (long long)seq * P.splits + i : flat_slot(P.S, max_shares, seq, c0 + i, i == 0)) * P.Hq + h;
    };
    float M = -INFINITY, L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i0 = kWide ? warp : 0; i0 < cnt; i0 += kLoads * kStep) {
      float2 ml[kLoads];
      float4 x[kLoads];
#pragma unroll
      for (int u = 0; u < kLoads; ++u) {
        const int i = i0 + u * kStep;
        const long long slot = slot_of(min(i, cnt - 1));
        ml[u] = P.part_ml[slot];
        x[u] = reinterpret_cast<const float4*>(P.part_o + slot * DD)[lane];
        if (i >= cnt) ml[u].x = -INFINITY;
      }
      const float before = M;
#pragma unroll
      for (int u = 0; u < kLoads; ++u) M = fmaxf(M, ml[u].x);
      const float f = before == -INFINITY ? 0.f : ex2(before - M);
      acc.x *= f, acc.y *= f, acc.z *= f, acc.w *= f, L *= f;
#pragma unroll
      for (int u = 0; u < kLoads; ++u)
        if (ml[u].x != -INFINITY) add_weighted(acc, L, ex2(ml[u].x - M), x[u], ml[u].y);
    }
    if constexpr (kWide) {
      sums[warp][lane] = acc;
      if (lane == 0) stats[warp] = make_float2(M, L);
      __syncthreads();
      if (warp > 0) return;
      M = -INFINITY, L = 0.f, acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int w = 0; w < kWarps; ++w) M = fmaxf(M, stats[w].x);
#pragma unroll
      for (int w = 0; w < kWarps; ++w)
        if (stats[w].x != -INFINITY) add_weighted(acc, L, ex2(stats[w].x - M), sums[w][lane], stats[w].y);
    }
    write_row(P, (long long)seq * P.Hq + h, lane * 4, acc, M, L);
  }
}

}  // namespace

// Blocks per (sequence, KV head) of the even split: whole waves of 2 blocks per SM.
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
// Workspace of the flat walk: the sequences' page counts, then n shares' slots.
size_t flat_counts_bytes(int S) { return ((size_t)S + 1) * sizeof(long long) / 16 * 16 + 16; }
size_t flat_slot_bytes(int Hq) { return (size_t)Hq * (DD + 2) * sizeof(float); }
size_t flat_bytes(int S, int Hq, int n) { return flat_counts_bytes(S) + (size_t)flat_slots(S, n) * flat_slot_bytes(Hq); }

// Clusters of c = 2, 4, 8 or 16 blocks that the current device holds at once (asked once per device): fewer than its SMs
// have room for, since a cluster does not leave its group of SMs.  Without a device, what the B200 says.
int max_clusters(int c) {
  constexpr int kMaxDevices = 64, kB200[4] = {148, 71, 33, 14};
  static std::atomic<int> cached[kMaxDevices][4];  // 0 = not asked yet
  const int i = c == 2 ? 0 : c == 4 ? 1 : c == 8 ? 2 : 3;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return kB200[i];
  }
  int n = cached[dev][i].load(std::memory_order_relaxed);
  if (n > 0) return n;
  const auto kern = decode_split_kernel<false, false>;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = c;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = DecSmem::kBytes;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, DecSmem::kBytes) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    return kB200[i];
  }
  cached[dev][i].store(n, std::memory_order_relaxed);
  return n;
}

// How a decode call is cut: into `flat` shares of all pages, or (flat = 0) every (sequence, KV head) into `c` blocks, a
// cluster or (split) with partial results.  By sizes alone: the lengths are on the device.
struct DecPlan {
  int c, flat;
  bool split;
};
constexpr int kMaxShortRounds = 4;  // the longest walk that more blocks than fit at once still take as one block each
DecPlan decode_plan(int S, int Hq, int Hkv, int max_blocks, size_t ws_bytes) {
  const long long slots = (long long)sm_count() * 2, pairs = (long long)S * Hkv, n = slots / Hkv;
  // rounds of three pages (one for each consumer warp) that a block takes for `pages`, and for its share of one sequence
  auto rounds_of = [](long long pages) { return (pages + kConsumers - 1) / kConsumers; };
  auto rounds = [&](int c) { return rounds_of((max_blocks + c - 1) / c); };
  // Few (sequence, KV head) pairs: a cluster for each, no larger than shortens the walk of the longest possible sequence
  // and than the chip holds for all pairs at once (two sequences of 5120 tokens, 8 KV heads: 15.3 us in 16 clusters of 16
  // of which 14 fit, 9.3 as below).
  int best = 1;
  for (int c = 2; c <= 16 && pairs <= max_clusters(c); c *= 2)
    if (rounds(c) < rounds(best)) best = c;
  // Very few pairs and a longer walk: the even split puts more blocks on it than clusters can, which pays for its second
  // kernel (1.5 us) from three rounds on where it saves one (one sequence, 8 KV heads: 9216 tokens 11.0 -> 9.1 us; 6400
  // 10.1 -> 8.4).  Past six rounds the flat walk's even shares are worth their page counts and merges (4 sequences of 9216:
  // 19.3 us in six rounds, 21.4 flat; 8: 40.7 flat), for one sequence, which has no other to even out, past two more than it
  // takes (65536 tokens, 8 KV heads: 35.7 us split, 37.8 flat; one of 131072, 1 KV head: 35 and 21).
  if (rounds(best) >= 3) {
    const int even = decode_num_splits(S, Hkv, max_blocks);
    const long long most = S == 1 && n >= 2 ? std::max(6ll, rounds_of((max_blocks + n - 1) / n) + 2) : 6;
    if (pairs * even <= slots && rounds(even) < rounds(best) && rounds(even) <= most) return {even, 0, true};
  }
  // Short walks stay with the clusters: they are all latency, and the flat walk pays for its page counts, the cut sequences'
  // second kernel and a merge at every sequence's end (64 sequences of 20 to 500 tokens: 33 us flat, 21 one block each; 18
  // of up to 2304 in clusters of two: 17.1 flat, 14.8).
  if (rounds(best) <= (pairs * best <= slots ? 6 : kMaxShortRounds)) return {best, 0, false};
  // Longer walks are bound by the memory system, and there an even share of the pages per block wins, the more so the more
  // the lengths differ (17 sequences of 150 to 6000 tokens: 41 -> 32 us; 127 of 800 and one of 131072, 16 KV heads: 480 us
  // in equal parts of every sequence, 1190 one block each, 287 flat; 800 of 4096, 1 KV head: 260, 233, 246).
  if (n >= 2 && flat_bytes(S, Hq, (int)n) <= ws_bytes) return {1, (int)n, false};
  // more KV heads than SMs, or less scratch than the flat walk takes: the even split, whose scratch every call brings
  const int even = decode_num_splits(S, Hkv, max_blocks);
  return {even, 0, even > 1};
}
}  // namespace

size_t decode_min_scratch_bytes(int S, int Hq, int Hkv, int D, int max_blocks) {
  return ((size_t)S * Hq * decode_num_splits(S, Hkv, max_blocks) * (D + 2) * sizeof(float) + 255) / 256 * 256;
}

// What the plan may use, whichever it is on the device of the call: a size query asks no more of a device than its SM count
// (the clusters it holds cannot be asked for without making a context on it).
size_t decode_scratch_bytes(int S, int Hq, int Hkv, int D, int max_blocks) {
  const int n = sm_count() * 2 / Hkv;
  const size_t flat = n >= 2 && max_blocks > kMaxShortRounds * kConsumers ? (flat_bytes(S, Hq, n) + 255) / 256 * 256 : 0;
  return std::max(decode_min_scratch_bytes(S, Hq, Hkv, D, max_blocks), flat);
}

int32_t launch_decode(int S, int Hq, int Hkv, int D, float scale, const void* q, const void* kc,
                      const void* vc, int num_blocks, const int32_t* table, int max_blocks,
                      const int32_t* seq_lens, void* o, float* lse, void* ws, size_t ws_bytes, cudaStream_t st,
                      const int32_t* holes, int holes_stride, int holes_off) {
  (void)D;
  const int G = Hq / Hkv;
  if (G < 1 || G > 8) return fail(UNIGIST_ERR_UNSUPPORTED, "decode supports 1 to 8 query heads per KV head, got %d", G);
  const DecPlan plan = decode_plan(S, Hq, Hkv, max_blocks, ws_bytes);
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
  P.pages_before = (long long*)ws;
  P.splits = plan.split ? plan.c : 0;
  P.part_o = reinterpret_cast<float*>((char*)ws + (plan.flat ? flat_counts_bytes(S) : 0));
  const size_t parts = plan.flat ? flat_slots(S, plan.flat) : (size_t)S * P.splits;
  P.part_ml = reinterpret_cast<float2*>(P.part_o + parts * Hq * DD);
  P.S = S, P.Hq = Hq, P.Hkv = Hkv, P.G = G, P.num_blocks = num_blocks, P.max_blocks = max_blocks;
  P.holes_stride = holes_stride, P.holes_off = holes_off;
  P.scale_log2 = scale * LOG2E;
  const int walk = (max_blocks + plan.c - 1) / plan.c;  // pages a block takes of the longest possible sequence
  const bool apart = !plan.flat && walk > kConsumers && walk <= 6 * kConsumers;
  const auto kern = plan.flat ? decode_split_kernel<true, false> : apart ? decode_split_kernel<false, true> : decode_split_kernel<false, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, DecSmem::kBytes);
  const int cluster = plan.flat || plan.split ? 1 : plan.c;
  if (e == cudaSuccess && cluster > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return fail(UNIGIST_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
  {
    KernelScope ks("decode_split_kernel", st);
    launch_chained(kern, plan.flat ? dim3(plan.flat, Hkv) : dim3(plan.c, Hkv, S), THREADS, DecSmem::kBytes, st, cluster, mk, mv,
                   P);
  }
  if (int32_t rc = check_launch("decode split kernel")) return rc;
  if (!plan.flat && !plan.split) return UNIGIST_OK;
  {
    KernelScope ks("decode_combine_kernel", st);
    // a block per query head while they are few: with many sequences a sequence has few parts
    const bool wide = (long long)S * Hq <= 4ll * sm_count();
    launch_chained(wide ? decode_combine_kernel<true> : decode_combine_kernel<false>, dim3(S, wide ? Hq : Hkv), THREADS, 0, st, 1, P,
                   plan.flat);
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
