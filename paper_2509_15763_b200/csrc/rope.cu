// Rotary position embedding with the aligned position ids of Section 4.1 (step 3: a gist token takes
// the position id of the raw token right after it), optionally fused with the gist shift of Section 4.2.
// HBM-bound: every element is read once and written once.  The position id and the destination row are
// closed forms of the interleaved token index; no index table is read.
#include "ug_common.cuh"

namespace ug {

namespace {

// One warp per token.  A lane owns 8 consecutive rotary frequencies j .. j + 7 of one head row (features j and j + D / 2
// pair up; 16-byte accesses), D / 16 lanes cover a row and the warp takes 512 / D rows at once, two of those in flight.
// The angles are computed once per token, D / 64 a lane, in fp64 (a position times a frequency reaches 1e5 rad), handed
// to the lanes that need them and reused for every head.
template <int D>
__global__ void __launch_bounds__(256)
rope_kernel(Geom g, GeomDiv div, int tokens, int heads, double log2_theta, int to_shifted, int from_shifted, int inverse,
            const __nv_bfloat16* __restrict__ src, __nv_bfloat16* __restrict__ dst) {
  constexpr int kLanesPerRow = D / 16, kRowsPerPass = 32 / kLanesPerRow, kMine = D / 64;
  const int lane = threadIdx.x & 31;
  const int j0 = (lane % kLanesPerRow) * 8, sub = lane / kLanesPerRow;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
  double inv_freq[kMine];  // of frequencies lane, lane + 32
#pragma unroll
  for (int e = 0; e < kMine; ++e) inv_freq[e] = exp2(-2.0 * (lane + 32 * e) / D * log2_theta);
  pdl_wait();
  for (long long tk = warp; tk < tokens; tk += nwarps) {  // tk = b * N + t, t interleaved
    const int b = fdiv(div.n, (int)tk), t = (int)tk - b * g.N;
    const int sigma = unshift_perm(g, div, t);  // the token's shifted position
    // position id: sinks and raw tokens count up, gist u gets s + (u + 1) r
    const double pos = sigma < g.s + g.T ? sigma : g.s + (sigma - g.s - g.T + 1) * g.r;
    float my_cs[kMine], my_sn[kMine], cs[8], sn[8];
#pragma unroll
    for (int e = 0; e < kMine; ++e) {
      double a = pos * inv_freq[e];
      a -= 6.283185307179586476925 * rint(a * 0.15915494309189533577);  // into [-pi, pi]
      sincosf((float)a, &my_sn[e], &my_cs[e]);
      if (inverse) my_sn[e] = -my_sn[e];  // the transpose of the rotation: what the backward pass applies to a gradient
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {  // frequency j0 + e is lane (j0 + e) % 32's; a lane's eight lie in one half
      const float c0 = __shfl_sync(0xffffffffu, my_cs[0], j0 + e), s0 = __shfl_sync(0xffffffffu, my_sn[0], j0 + e);
      cs[e] = c0, sn[e] = s0;
      if (kMine == 2) {
        const float c1 = __shfl_sync(0xffffffffu, my_cs[kMine - 1], j0 + e), s1 = __shfl_sync(0xffffffffu, my_sn[kMine - 1], j0 + e);
        if (j0 >= 32) cs[e] = c1, sn[e] = s1;
      }
    }
    const __nv_bfloat16* s_tok = src + ((long long)b * g.N + (from_shifted ? sigma : t)) * heads * D;
    __nv_bfloat16* d_tok = dst + ((long long)b * g.N + (to_shifted ? sigma : t)) * heads * D;
    for (int h0 = 0; h0 < heads; h0 += 2 * kRowsPerPass) {  // two passes in flight
      uint4 lo[2], hi[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int h = h0 + u * kRowsPerPass + sub;
        if (h < heads) {
          lo[u] = *reinterpret_cast<const uint4*>(s_tok + h * D + j0);
          hi[u] = *reinterpret_cast<const uint4*>(s_tok + h * D + D / 2 + j0);
        }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int h = h0 + u * kRowsPerPass + sub;
        if (h < heads) {
          uint32_t x[4] = {lo[u].x, lo[u].y, lo[u].z, lo[u].w}, y[4] = {hi[u].x, hi[u].y, hi[u].z, hi[u].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {  // a bf16 is the high half of an fp32
            const float x0 = __uint_as_float(x[e] << 16), x1 = __uint_as_float(x[e] & 0xffff0000u);
            const float y0 = __uint_as_float(y[e] << 16), y1 = __uint_as_float(y[e] & 0xffff0000u);
            const __nv_bfloat162 a = __floats2bfloat162_rn(x0 * cs[2 * e] - y0 * sn[2 * e], x1 * cs[2 * e + 1] - y1 * sn[2 * e + 1]);
            const __nv_bfloat162 c = __floats2bfloat162_rn(y0 * cs[2 * e] + x0 * sn[2 * e], y1 * cs[2 * e + 1] + x1 * sn[2 * e + 1]);
            x[e] = *reinterpret_cast<const uint32_t*>(&a);
            y[e] = *reinterpret_cast<const uint32_t*>(&c);
          }
          *reinterpret_cast<uint4*>(d_tok + h * D + j0) = make_uint4(x[0], x[1], x[2], x[3]);
          *reinterpret_cast<uint4*>(d_tok + h * D + D / 2 + j0) = make_uint4(y[0], y[1], y[2], y[3]);
        }
      }
    }
  }
}

}  // namespace

int32_t launch_rope(const Geom& g, int B, int heads, int D, float theta_base, bool to_shifted, bool from_shifted,
                    bool inverse, const void* src, void* dst, cudaStream_t st) {
  const long long tokens = (long long)B * g.N;
  const long long want = (tokens + 7) / 8;  // 8 warps per block
  const long long cap = (long long)sm_count() * 8;
  const int blocks = (int)(want < cap ? (want > 0 ? want : 1) : cap);
  const double log2_theta = log2((double)theta_base);
  {
    KernelScope ks("rope_kernel", st);
    launch_chained(D == 128 ? rope_kernel<128> : rope_kernel<64>, dim3(blocks), 256, 0, st, 1, g, make_geom_div(g), (int)tokens, heads, log2_theta,
                   to_shifted ? 1 : 0, from_shifted ? 1 : 0, inverse ? 1 : 0, (const __nv_bfloat16*)src, (__nv_bfloat16*)dst);
  }
  return check_launch("rope kernel");
}

}  // namespace ug
