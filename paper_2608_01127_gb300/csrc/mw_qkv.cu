// QKV split with the temporal rotary embedding applied on the way (the input
// side of block-causal attention, Sec. 3.2; RoPE positions as in Sec. 3.5).
// The fused QKV projection leaves each token's heads interleaved as
// [B, N, 3, H, d]; the attention kernels read head-major [B, H, N, d] rows.
// One pass moves every element once and rotates the first rope_dims channels
// of Q and K: token t sits at frame first_frame + t / per_frame, and channel
// pair (2i, 2i+1) turns by frame * base^(-2i / rope_dims).  HBM-bound: each
// element is read and written once, 16 bytes per thread access.
#include "mw_internal.h"
#include "mw_ptx.cuh"

namespace mw {
namespace {

constexpr int kQkvTokens = 32;  // at most, per CTA
constexpr int kMaxPairs = kMaxRopePairs;
constexpr int kMaxUnroll = 6;

// grid.x: (b, block of `tokens` tokens); grid.y: groups of heads_per_block
// heads.  A thread owns one (token, 16-byte piece) of the block, fixed for
// the whole kernel, and walks Q, K, V and the group's heads with plain
// strides, UNROLL heads' pieces in flight at once; each warp reads whole row
// segments and writes contiguous bytes.
template <int UNROLL>
__global__ void __launch_bounds__(256) qkv_rope_kernel(const __nv_bfloat16* __restrict__ qkv,
                                                       __nv_bfloat16* __restrict__ q,
                                                       __nv_bfloat16* __restrict__ k,
                                                       __nv_bfloat16* __restrict__ v, int N, int H,
                                                       int d, int tokens, int rope_dims,
                                                       int heads_per_block,
                                                       const RopeFreq omega, int per_frame,
                                                       int first_frame) {
  __shared__ float2 table[kQkvTokens * kMaxPairs];  // (cos, sin) per (frame, pair)
  const int n_tb = (N + tokens - 1) / tokens;
  const int b = blockIdx.x / n_tb;
  const int t0 = (blockIdx.x % n_tb) * tokens;
  const int nt = min(tokens, N - t0);
  const int h0 = blockIdx.y * heads_per_block;
  const int h1 = min(H, h0 + heads_per_block);
  const int pairs = rope_dims / 2;
  const int f_lo = first_frame + t0 / per_frame;
  if (pairs > 0) {
    // frames of this token block: at most one per token
    const int nf = first_frame + (t0 + nt - 1) / per_frame - f_lo + 1;
    for (int e = threadIdx.x; e < nf * pairs; e += blockDim.x)
      table[e] = rope_cos_sin(f_lo + e / pairs, omega.hi[e % pairs], omega.lo[e % pairs]);
    __syncthreads();
  }
  const int pieces = d / 8;
  const int rot_pieces = (pairs + 3) / 4;  // pieces holding at least one rotated pair
  const size_t head_out = static_cast<size_t>(N) * d;  // output elements per head
  for (int r = threadIdx.x; r < nt * pieces; r += blockDim.x) {
    const int t = t0 + r / pieces;
    const int pc = r % pieces;
    // the piece's (cos, sin) pairs: index 4 pc + u < pairs turns
    const int np = pc < rot_pieces ? min(4, pairs - 4 * pc) : 0;
    float2 cs[4];
    if (np > 0) {
      const float2* row = table + (first_frame + t / per_frame - f_lo) * pairs + 4 * pc;
#pragma unroll
      for (int u = 0; u < 4; ++u) cs[u] = u < np ? row[u] : make_float2(1.f, 0.f);
    }
    const __nv_bfloat16* src = qkv + (static_cast<size_t>(b) * N + t) * 3 * H * d + pc * 8;
    const size_t dst0 = (static_cast<size_t>(b) * H * N + t) * d + pc * 8;
    for (int which = 0; which < 3; ++which) {
      __nv_bfloat16* out = which == 0 ? q : which == 1 ? k : v;
      const bool turn = which < 2 && np > 0;
      for (int h = h0; h < h1; h += UNROLL) {
        uint4 x[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
          if (h + u < h1)
            x[u] = *reinterpret_cast<const uint4*>(src + static_cast<size_t>(which * H + h + u) * d);
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
          if (h + u >= h1) continue;
          if (turn) {
            x[u].x = rope_turn(x[u].x, cs[0]);
            if (np > 1) x[u].y = rope_turn(x[u].y, cs[1]);
            if (np > 2) x[u].z = rope_turn(x[u].z, cs[2]);
            if (np > 3) x[u].w = rope_turn(x[u].w, cs[3]);
          }
          *reinterpret_cast<uint4*>(out + dst0 + (h + u) * head_out) = x[u];
        }
      }
    }
  }
}

}  // namespace

cudaError_t launch_qkv_rope(const __nv_bfloat16* qkv, __nv_bfloat16* q, __nv_bfloat16* k,
                            __nv_bfloat16* v, int B, int N, int H, int d, int rope_dims,
                            const RopeFreq& omega, int per_frame, int first_frame,
                            cudaStream_t s) {
  if (B == 0 || N == 0 || H == 0) return cudaSuccess;
  // as many tokens as fill the 256 threads (d = 128: twice), so that no pass
  // over the block is mostly idle: 32 tokens of 72 channels are 288 pieces
  const int pieces = d / 8;
  const int tokens = pieces == 16 ? kQkvTokens : 256 / pieces;
  const long long tb = static_cast<long long>(B) * ((N + tokens - 1) / tokens);
  // halve the heads per CTA until the grid holds enough CTAs to fill every SM
  // a few times over (the per-CTA (cos, sin) table is then amortised over as
  // many heads as the size allows)
  int hb = H;
  while (hb > 1 && tb * ((H + hb - 1) / hb) < 1216) hb = (hb + 1) / 2;
  // heads in flight: the fewest equal batches of up to six (12 heads of 64,
  // 2 x 14080 tokens, six heads a CTA: one batch of six 41.7 us, four and two
  // 42.8; 16 heads of 128, eight a CTA: four and four 73 us, six and two 79).
  // With both rules, a call of 16 heads of 72: 41.8 -> 35.9 us, 7 heads of 80:
  // 23.1 -> 16.8 us, 24 heads of 64: 66.3 -> 61.4 us
  const int batches = (hb + kMaxUnroll - 1) / kMaxUnroll;
  const int unroll = (hb + batches - 1) / batches;
  const dim3 grid(static_cast<unsigned>(tb), static_cast<unsigned>((H + hb - 1) / hb));
  auto launch = [&](auto kernel) {
    kernel<<<grid, 256, 0, s>>>(qkv, q, k, v, N, H, d, tokens, rope_dims, hb, omega, per_frame,
                                first_frame);
  };
  switch (unroll) {
    case 1: launch(qkv_rope_kernel<1>); break;
    case 2: launch(qkv_rope_kernel<2>); break;
    case 3: launch(qkv_rope_kernel<3>); break;
    case 4: launch(qkv_rope_kernel<4>); break;
    case 5: launch(qkv_rope_kernel<5>); break;
    default: launch(qkv_rope_kernel<6>); break;
  }
  return cudaGetLastError();
}

}  // namespace mw
