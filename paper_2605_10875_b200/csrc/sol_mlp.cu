// Per-token top-k over the intermediate channels of the SwiGLU MLP.
//
// For token i keep the m = ceil((1 - p_i) * ff) channels with the largest
// |t_j| = |silu(g_j) * u_j| (the count mirrors the paper's m = ceil(rho * d),
// "Per-token channel selection", with rho = 1 - p; ties: lower index).
//
// The gate/up projection leaves, per token, a 4096-bin histogram of |t| and
// the largest |g|, |u|.  channel_select_multi spreads every token over
// ff/1024 CTAs: each finds the histogram bin that holds the m-th largest |t|,
// keeps what lies above that bin (by more than the float32 error bound of t),
// drops what lies below, and lists the channels in between; the last CTA of a
// token ranks those candidates within their error bounds and patches the
// surely kept ones in; the few that the bounds leave open are recomputed
// exactly from the weight rows (many of a small batch by channel_select_rest,
// whose CTAs share them).  Outputs: the masked activations as two bf16
// parts (hi + lo) for the tensor-core down projection, a keep mask, and the
// "granule is live" flags that let the down projection skip weight rows
// nobody keeps.  A token with more candidates than the list holds (massive
// ties) is redone by one CTA of channel_select_rest, which is exact for
// any input; channel_list turns the mask into the ascending index list when a
// caller asks for it.
#include <math.h>

#include "sol_common.cuh"
#include "sol_internal.h"
#include "sol_select.cuh"

namespace sol {

struct ChanDev {
  int d, ff;
  const int32_t* p_permille;
  const float* g;
  const float* u;
  const float* t;
  const unsigned char* a_op;  // packed operand, Mpad rows
  const float* scale;
  const unsigned char* w_gu;  // packed gate/up weights: rows alternate gate_c, up_c
  int R, chunks, Mpad;        // rows per tile and 64-wide chunks of the packed weights; rows of the operand blocks
  uint32_t* sel;
  double* cand_val;
  int32_t* cand_idx;
  unsigned char* keep;
  int32_t* kept_ch;
  int32_t* kept_cnt;
  unsigned char* t_op;  // packed operand of the down projection: 2 Mpad rows (high parts, then low parts)
  int32_t* live;
  int* status;
  int hand_over;        // elements of open candidates above which the next kernel recomputes them; 0: never
};

// Running sum held as an unevaluated pair of floats (hi + lo): adds x with the rounding error of
// hi + x captured exactly (two-sum) and gathered in lo.  With terms that are exact float32 numbers the
// pair follows the exact sum to about 2^-45, on the float32 pipes instead of the scarce float64 ones.
__device__ __forceinline__ void pair_add(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
  hi = s;
  lo = __fadd_rn(lo, e);
}

// bf16 numbers as float64 by their bits (a conversion instruction runs at a small fraction of this rate).
// Operand elements, the number in the high half of a word: exact, whatever the number.
__device__ __forceinline__ double operand_to_f64(uint32_t high_half) {
  const uint32_t mag = (high_half >> 3) & 0x0fffe000u, sign = high_half & 0x80000000u;
  if (mag - 1u < 0x000fffffu || mag >= 0x0ff00000u) return (double)__uint_as_float(high_half & 0xffff0000u);  // denormal, infinite, NaN
  return __hiloint2double((int)((mag ? mag + 0x38000000u : 0u) | sign), 0);
}
// Weights: times 2^-896, so that no bias is added and zeros and denormals need no case of their own (they come out as
// zeros and float64 denormals; a product is good to 2^-178 at least).  A channel with an infinite or NaN weight has an
// infinite or NaN |t| and is never a candidate.
__device__ __forceinline__ double weight_to_f64(uint32_t high_half) {
  return __hiloint2double((int)(((high_half >> 3) & 0x0fffe000u) | (high_half & 0x80000000u)), 0);
}

// From the exact sums of a candidate's gate and up products (weights times 2^-896, see weight_to_f64) to its exact |t|.
__device__ __forceinline__ double exact_score(double g, double u, double scale) {
  const double unit = __hiloint2double((1023 + 896) << 20, 0);  // 2^896
  const double ag = g * unit * scale, au = u * unit * scale;
  return fabs(ag / (1.0 + exp(-ag)) * au);
}
// Patches a kept candidate into the masked activations, the mask and the live flags.
__device__ __forceinline__ void keep_channel(const ChanDev& p, int b, int j) {
  const float tv = p.t[(size_t)b * p.ff + j];
  const uint16_t hv = f2bf(tv);
  uint16_t* dst = reinterpret_cast<uint16_t*>(p.t_op + act_piece_offset(2 * p.Mpad, b, j >> 3) + (j & 7) * 2);
  dst[0] = hv;
  dst[(size_t)p.Mpad * 64] = f2bf(tv - bf2f(hv));
  p.keep[(size_t)b * p.ff + j] = 1;
  p.live[j >> 5] = 1;
}

// ============================================================================
// channel_select_rest: what channel_select_multi leaves to it
// ============================================================================
constexpr int CR_THREADS = 512;

// The open candidates of a token: their exact |t| in float64 (g_j = scale * sum_e x_e w_je with x the quantizer codes or the
// bf16 row), shared out over the token's CTAs; the last of them keeps the `need` best (ties: lower index).  Four warps per
// candidate, eight elements of both rows per thread and step, the next step's on their way.
// live == 0: a rehearsal on one made-up candidate, which reads weights only and writes nothing outside the CTA.
__device__ __forceinline__ void settle_open(const ChanDev& p, SelectSmem& sm, int b, int n_open, int need, int live) {
  constexpr int GROUPS = CR_THREADS / 128;
  __shared__ double2 part[GROUPS][4];
  __shared__ int s_last;
  const int tid = threadIdx.x, group = tid >> 7, gt = tid & 127, lane = tid & 31, d = p.d, X = gridDim.x;
  const uint32_t chunk_bytes = (uint32_t)p.R * 128;
  const int32_t* idx = p.cand_idx + (size_t)b * CH_CAND_CAP;
  double* val = p.cand_val + (size_t)b * CH_CAND_CAP;
#pragma unroll 1
  for (int i0 = live ? blockIdx.x * GROUPS : 0; i0 < n_open; i0 += GROUPS * X) {
    const int i = i0 + group;
    double g = 0.0, u = 0.0;
    if (i < n_open) {
      const int n = live ? 2 * __ldcg(idx + i) : 0, tile = n / p.R, r = n - tile * p.R;
      const unsigned char* row = p.w_gu + ((size_t)tile * p.chunks * p.R + r) * 128;  // the gate row; the up row follows
      const int swz = r & 7;                                                          // even: a gate row is an even row
      uint4 gn = make_uint4(0u, 0u, 0u, 0u), un = gn, xn = gn;
      auto load = [&](int e0) {
        if (e0 < d) {
          const int piece = (e0 >> 3) & 7;
          const unsigned char* src = row + (size_t)(e0 >> 6) * chunk_bytes;
          gn = *reinterpret_cast<const uint4*>(src + ((piece ^ swz) * 16));
          un = *reinterpret_cast<const uint4*>(src + 128 + ((piece ^ (swz + 1)) * 16));
          if (live) xn = *reinterpret_cast<const uint4*>(p.a_op + act_piece_offset(p.Mpad, b, e0 >> 3));
        }
      };
      load(gt * 8);
#pragma unroll 1
      for (int e0 = gt * 8; e0 < d; e0 += 1024) {
        const uint32_t ga[4] = {gn.x, gn.y, gn.z, gn.w}, ua[4] = {un.x, un.y, un.z, un.w}, xa[4] = {xn.x, xn.y, xn.z, xn.w};
        load(e0 + 1024);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const double x0 = operand_to_f64(xa[e] << 16), x1 = operand_to_f64(xa[e]);
          g = fma(x0, weight_to_f64(ga[e] << 16), g);
          u = fma(x0, weight_to_f64(ua[e] << 16), u);
          g = fma(x1, weight_to_f64(ga[e]), g);
          u = fma(x1, weight_to_f64(ua[e]), u);
        }
      }
    }
    g = warp_sum_d(g);
    u = warp_sum_d(u);
    if (lane == 0) part[group][gt >> 5] = make_double2(g, u);
    __syncthreads();
    if (gt == 0 && i < n_open) {
      const double2 a = part[group][0], b2 = part[group][1], c = part[group][2], e = part[group][3];
      const double v = exact_score((a.x + b2.x) + (c.x + e.x), (a.y + b2.y) + (c.y + e.y), live ? (double)p.scale[b] : 1.0);
      if (live) val[i] = v;
    }
    __syncthreads();
  }
  if (live && X > 1) {  // the token's last CTA goes on
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(p.sel + (size_t)b * CH_SEL_WORDS + CH_DONE_OPEN, 1u) == (uint32_t)(X - 1) ? 1 : 0;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
  }
  for (int c = tid; c < n_open; c += CR_THREADS) {
    sm.cand_val[c] = live ? __ldcg(val + c) : 0.0;
    sm.cand_idx[c] = live ? __ldcg(idx + c) : c;
  }
  __syncthreads();
  rank_candidates<CR_THREADS>(n_open, need, sm);
  for (int c = tid; c < n_open; c += CR_THREADS)
    if (live && sm.cand_keep[c]) keep_channel(p, b, sm.cand_idx[c]);
  if (live && tid == 0) atomicAdd(p.status + ST_CH_REFINED, n_open);
}

// A token whose candidates did not fit the list (long runs of equal scores), from the beginning and for any input, by one
// CTA: the m-th largest |t| by a radix select, the channels within the error bound of it by their exact scores, or, where
// those do not fit the list either, in float32 order with ties to the lower index.  Its loops over the row are short and read it
// from L2 each time, so the loads are 16 bytes wide and several in flight; a padding row's scores are all equal and need no radix
// select (128 rows of a Llama-8B MLP, half of them zeros: 222 us with single floats and the select, this 188; with the row in the
// registers of 1024 threads, a kernel of 124 registers in every layer's way, 202).
__device__ __noinline__ void redo_token(const ChanDev& p, SelectSmem& sm, int b) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int WARPS = CR_THREADS / 32;
  const int ff = p.ff, d = p.d;
  const float* tt = p.t + (size_t)b * ff;
  const int m = (int)(((long long)(1000 - p.p_permille[b]) * ff + 999) / 1000);
  if (tid < 4) sm.counts[tid] = 0;
  float gmax = 0.f, umax = 0.f;  // for the error window
  uint32_t key_max = 0u, key_min = 0xffffffffu;
#pragma unroll 4
  for (int j = tid * 4; j < ff; j += CR_THREADS * 4) {  // ff is a multiple of 4
    const float4 g4 = *reinterpret_cast<const float4*>(p.g + (size_t)b * ff + j), u4 = *reinterpret_cast<const float4*>(p.u + (size_t)b * ff + j),
                 t4 = *reinterpret_cast<const float4*>(tt + j);
    gmax = fmaxf(fmaxf(gmax, fmaxf(fabsf(g4.x), fabsf(g4.y))), fmaxf(fabsf(g4.z), fabsf(g4.w)));
    umax = fmaxf(fmaxf(umax, fmaxf(fabsf(u4.x), fabsf(u4.y))), fmaxf(fabsf(u4.z), fabsf(u4.w)));
    const uint32_t k0 = float_key(fabsf(t4.x)), k1 = float_key(fabsf(t4.y)), k2 = float_key(fabsf(t4.z)), k3 = float_key(fabsf(t4.w));
    key_max = max(max(key_max, max(k0, k1)), max(k2, k3));
    key_min = min(min(key_min, min(k0, k1)), min(k2, k3));
  }
  gmax = block_max<CR_THREADS>(gmax, 0, sm);
  umax = block_max<CR_THREADS>(umax, 1, sm);
  key_max = __reduce_max_sync(0xffffffffu, key_max);
  key_min = __reduce_min_sync(0xffffffffu, key_min);
  if (lane == 0) {
    sm.rank_key[warp] = key_max;
    sm.rank_key[WARPS + warp] = key_min;
  }
  __syncthreads();
  key_max = __reduce_max_sync(0xffffffffu, sm.rank_key[lane % WARPS]);
  key_min = __reduce_min_sync(0xffffffffu, sm.rank_key[WARPS + lane % WARPS]);
  __syncthreads();  // the scratch is taken by the selection
  uint32_t key_thr = key_max;
  int tie_need = m;
  if (key_min != key_max) {  // not all equal, as the scores of a padding row are
    auto key = [&](int i) -> uint32_t {
      const int j = i * CR_THREADS + tid;
      return j < ff ? float_key(fabsf(tt[j])) : 0u;
    };
    key_thr = select_kth<CR_THREADS, 0>(key, m, tie_need, sm, (ff + CR_THREADS - 1) / CR_THREADS);
  }
  const float thr32 = key_to_float(key_thr);
  // error taken for g_j, u_j: the tensor cores add each 16-long slice of the dot product to the running
  // float32 sum with truncation, so the error grows with the d/16 steps: (d/16) * 2^-24 of the largest
  // magnitude, and never less than 2^-18 of it
  const float eps = fmaxf(3.814697265625e-06f, (float)(d / 16) * 5.9604644775390625e-08f) * fmaxf(gmax, umax);
  const float delta = 2.0f * eps * (1.1f * umax + gmax) + 1e-6f * thr32;  // |silu'| <= 1.1, |silu(g)| <= |g|
  const float hi = thr32 + delta, lo = thr32 - delta;
  int n_in = 0;
#pragma unroll 2
  for (int j0 = 0; j0 < ff; j0 += CR_THREADS * 4) {
    const int j = j0 + tid * 4;
    float4 t4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j < ff) t4 = *reinterpret_cast<const float4*>(tt + j);
    const float vv[4] = {t4.x, t4.y, t4.z, t4.w};
    uint32_t in = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float sv = fabsf(vv[e]);
      if (j >= ff) continue;
      if (sv > hi) ++n_in;
      else if (sv >= lo) in |= 1u << e;
    }
    int incl = __popc(in);  // the candidates' places: one request per warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    int slot = 0;
    if (lane == 31 && incl) slot = atomicAdd(&sm.counts[0], incl);
    slot = __shfl_sync(0xffffffffu, slot, 31) + incl - __popc(in);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if ((in >> e) & 1u) {
        if (slot < SEL_CAND_CAP) sm.cand_idx[slot] = j + e;
        ++slot;
      }
  }
  n_in = block_count<CR_THREADS>(n_in, 0, sm);
  int n_cand = sm.counts[0];
  const int need = m - n_in;
  const bool by_window = n_cand <= SEL_CAND_CAP;  // else float32 order
  if (!by_window) {
    if (tid == 0) atomicAdd(p.status + ST_CH_OVERFLOW, 1);
    n_cand = 0;
  } else if (n_cand != need) {
    if (tid == 0) atomicAdd(p.status + ST_CH_REFINED, n_cand);
    // every product of two bf16 numbers is an exact float32, so the sums are gathered exactly in float pairs
    const double sc = (double)p.scale[b];
#pragma unroll 1
    for (int c = warp; c < n_cand; c += WARPS) {
      const int j = sm.cand_idx[c];
      float gh = 0.f, gl = 0.f, uh = 0.f, ul = 0.f;
#pragma unroll 1
      for (int e = lane * 8; e < d; e += 256) {  // the piece of elements e .. e + 7 of the operand row and of the channel's rows
        const uint4 xv = *reinterpret_cast<const uint4*>(p.a_op + act_piece_offset(p.Mpad, b, e >> 3));
        const uint4 gv = *reinterpret_cast<const uint4*>(p.w_gu + nk_piece_offset(p.R, p.chunks, 2 * j, e >> 6, (e >> 3) & 7));
        const uint4 uv = *reinterpret_cast<const uint4*>(p.w_gu + nk_piece_offset(p.R, p.chunks, 2 * j + 1, e >> 6, (e >> 3) & 7));
        const uint32_t xa[4] = {xv.x, xv.y, xv.z, xv.w}, ga[4] = {gv.x, gv.y, gv.z, gv.w}, ua[4] = {uv.x, uv.y, uv.z, uv.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float x0 = bf16_lo(xa[q]), x1 = bf16_hi(xa[q]);
          pair_add(gh, gl, __fmul_rn(x0, bf16_lo(ga[q])));
          pair_add(gh, gl, __fmul_rn(x1, bf16_hi(ga[q])));
          pair_add(uh, ul, __fmul_rn(x0, bf16_lo(ua[q])));
          pair_add(uh, ul, __fmul_rn(x1, bf16_hi(ua[q])));
        }
      }
      const double ag = warp_sum_d((double)gh + (double)gl) * sc;
      const double au = warp_sum_d((double)uh + (double)ul) * sc;
      if (lane == 0) sm.cand_val[c] = fabs(ag / (1.0 + exp(-ag)) * au);
    }
    __syncthreads();
    rank_candidates<CR_THREADS>(n_cand, need, sm);
  } else {
    for (int c = tid; c < n_cand; c += CR_THREADS) sm.cand_keep[c] = 1;
  }
  __syncthreads();

  // the masked activations as bf16 high and low parts, eight channels (one piece of the packed operand) per thread and round,
  // in index order: ties are kept until tie_need runs out
  int total = 0, ties_taken = 0;
#pragma unroll 1
  for (int base0 = 0; base0 < ff; base0 += CR_THREADS * 8) {
    const int j0 = base0 + tid * 8;  // ff is a multiple of 32, so eight are present or absent as a whole
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (j0 < ff) {
      const float4 v0 = *reinterpret_cast<const float4*>(tt + j0), v1 = *reinterpret_cast<const float4*>(tt + j0 + 4);
      v[0] = v0.x; v[1] = v0.y; v[2] = v0.z; v[3] = v0.w; v[4] = v1.x; v[5] = v1.y; v[6] = v1.z; v[7] = v1.w;
    }
    uint32_t keep = 0, tie = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t kk = float_key(fabsf(v[e]));
      if (j0 >= ff) continue;
      if (by_window) {
        const float sv = key_to_float(kk);
        if (sv > hi) {
          keep |= 1u << e;
        } else if (sv >= lo) {  // within the window: look the channel up in the decided list
          for (int q = 0; q < n_cand; ++q)
            if (sm.cand_idx[q] == j0 + e && sm.cand_keep[q]) keep |= 1u << e;
        }
      } else {
        if (kk > key_thr) keep |= 1u << e;
        if (kk == key_thr) tie |= 1u << e;
      }
    }
    int incl = __popc(tie);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    __syncthreads();  // earlier readers of sm.scan are done
    if (lane == 31) sm.scan[0][warp] = incl;
    __syncthreads();
    int before = ties_taken + incl - __popc(tie);
    for (int w = 0; w < WARPS; ++w) {
      const int x = sm.scan[0][w];
      if (w < warp) before += x;
      ties_taken += x;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if ((tie >> e) & 1u) {
        if (before < tie_need) keep |= 1u << e;
        ++before;
      }
    if (j0 < ff) {
      uint32_t hw[4] = {0, 0, 0, 0}, lw[4] = {0, 0, 0, 0}, kw[2] = {0, 0};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if ((keep >> e) & 1u) {
          const uint16_t hv = f2bf(v[e]), lv = f2bf(v[e] - bf2f(hv));
          hw[e >> 1] |= (uint32_t)hv << (16 * (e & 1));
          lw[e >> 1] |= (uint32_t)lv << (16 * (e & 1));
          kw[e >> 2] |= 1u << (8 * (e & 3));
        }
      unsigned char* dst = p.t_op + act_piece_offset(2 * p.Mpad, b, j0 >> 3);
      *reinterpret_cast<uint4*>(dst) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
      *reinterpret_cast<uint4*>(dst + (size_t)p.Mpad * 128) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
      *reinterpret_cast<uint2*>(p.keep + (size_t)b * ff + j0) = make_uint2(kw[0], kw[1]);
      if (keep) p.live[j0 >> 5] = 1;
    }
    total += __popc(keep);
  }
  total = block_count<CR_THREADS>(total, 1, sm);
  if (tid == 0) p.kept_cnt[b] = total;
}

// Grid (CTAs per token, tokens).  Nearly always most CTAs leave at once, so the kernel is kept small enough to be resident
// beside any other (as a kernel of 124 registers and 100 KB of unrolled code it took 1.7 us of a single sequence's layer,
// this 0.7).  Where open candidates may be handed over, a CTA of a token with a selection to make rehearses settle_open
// while the kernels before are still running, so that its code is in the instruction caches.
__global__ void __launch_bounds__(CR_THREADS, 2) channel_select_rest_kernel(const ChanDev p) {
  __shared__ SelectSmem sm;
  const int b = blockIdx.y;
  pdl_trigger();
  const int m = (int)(((long long)(1000 - p.p_permille[b]) * p.ff + 999) / 1000);
  if (m <= 0 || m >= p.ff) {  // all or nothing: never left to this kernel
    pdl_wait();
    return;
  }
  int live = 0, n_open = p.hand_over > 0 ? 1 : 0, need = 1;
#pragma unroll 1
  for (;;) {
    asm volatile("" : "+r"(live));  // one code for both
    if (n_open > 0) settle_open(p, sm, b, n_open, need, live);
    if (live) return;
    pdl_wait();
    const uint32_t* sel = p.sel + (size_t)b * CH_SEL_WORDS;
    if (__ldcg(sel + CH_FALLBACK) != 0u) {
      if (blockIdx.x == 0) redo_token(p, sm, b);
      return;
    }
    const uint32_t open = __ldcg(sel + CH_OPEN);
    n_open = (int)(open >> 16);
    need = (int)(open & 0xffffu);
    live = 1;
    __syncthreads();  // the rehearsal's candidate is not read any more
  }
}

// ============================================================================
// channel_select_multi
// ============================================================================
constexpr int CM_THREADS = 256;

constexpr int CM_EXACT = 32;  // candidates recomputed at a time
struct ChanMultiSmem {
  int scan[CM_THREADS / 32];
  int pick;
  int n_open, n_sure;
  int flag;
  float thr_hi, thr_lo;
  int idx[CH_CAND_CAP];
  float2 av[CH_CAND_CAP];          // a candidate's float32 |t| and the bound of its error
  int open[CH_CAND_CAP];           // the channels to recompute
  double val[CH_CAND_CAP];         // their exact |t|
  size_t row_off[CM_EXACT];        // of up to CM_EXACT of them: where their weight rows start, the rows' swizzle,
  int row_swz[CM_EXACT];
  double2 part[CM_EXACT][CM_THREADS / 32];  // the warps' sums of g and u
};

// Exact |t| of up to CM_EXACT open candidates, by the whole CTA: g_j = scale * sum_e x_e w_je with x the quantizer codes (or
// the bf16 row), in float64.  A thread owns elements 8 tid .. + 7 of every 2048; the rows are on their way to L2 before the
// first is read, and the next candidate's pieces travel while one is worked on.  One short rolled loop, because this
// code runs cold: four candidates side by side, in float64 or in float pairs, gained at d_model 4096 what their code cost
// at the other sizes (24 us here, 26 and 23 for 16 candidates of a Llama-8B layer; 2.0, 3.2 and 3.8 for one at d_model 256).
__device__ __forceinline__ void exact_candidates(const ChanDev& p, ChanMultiSmem& sm, int b, int i0, int n) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, d = p.d;
  const uint32_t chunk_bytes = (uint32_t)p.R * 128;
  if (tid < n) {  // where the candidate's gate row starts (its up row follows 128 bytes later)
    const int row = 2 * sm.open[i0 + tid], tile = row / p.R, r = row - tile * p.R;
    sm.row_off[tid] = ((size_t)tile * p.chunks * p.R + r) * 128;
    sm.row_swz[tid] = r & 7;
  }
  for (int i = tid; i < n * (CM_THREADS / 32); i += CM_THREADS) (&sm.part[0][0])[i] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int q = tid; q < n * (d / 64); q += CM_THREADS) {  // 256 bytes of both rows per 64 elements
    const int i = q / (d / 64), chunk = q - i * (d / 64);
    const unsigned char* src = p.w_gu + sm.row_off[i] + (size_t)chunk * chunk_bytes;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(src + 128));
  }
#pragma unroll 1
  for (int base = 0; base < d; base += CM_THREADS * 8) {
    const int e0 = base + tid * 8, piece = (e0 >> 3) & 7;
    const bool in = e0 < d;
    double x[8];
    {
      uint4 xv = make_uint4(0u, 0u, 0u, 0u);
      if (in) xv = *reinterpret_cast<const uint4*>(p.a_op + act_piece_offset(p.Mpad, b, e0 >> 3));
      const uint32_t xa[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        x[2 * q] = operand_to_f64(xa[q] << 16);
        x[2 * q + 1] = operand_to_f64(xa[q]);
      }
    }
    const unsigned char* chunk_src = p.w_gu + (size_t)(e0 >> 6) * chunk_bytes;
    uint4 g_next = make_uint4(0u, 0u, 0u, 0u), u_next = g_next;
    auto load = [&](int i) {
      if (in && i < n) {
        const int swz = sm.row_swz[i];  // even: a gate row is an even row
        g_next = *reinterpret_cast<const uint4*>(chunk_src + sm.row_off[i] + ((piece ^ swz) * 16));
        u_next = *reinterpret_cast<const uint4*>(chunk_src + sm.row_off[i] + 128 + ((piece ^ (swz + 1)) * 16));
      }
    };
    load(0);
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const uint32_t ga[4] = {g_next.x, g_next.y, g_next.z, g_next.w}, ua[4] = {u_next.x, u_next.y, u_next.z, u_next.w};
      load(i + 1);
      double g = 0.0, u = 0.0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        g = fma(x[2 * q], weight_to_f64(ga[q] << 16), g);
        u = fma(x[2 * q], weight_to_f64(ua[q] << 16), u);
        g = fma(x[2 * q + 1], weight_to_f64(ga[q]), g);
        u = fma(x[2 * q + 1], weight_to_f64(ua[q]), u);
      }
      g = warp_sum_d(g);
      u = warp_sum_d(u);
      if (lane == 0) {
        sm.part[i][warp].x += g;
        sm.part[i][warp].y += u;
      }
    }
  }
  __syncthreads();
  if (tid < n) {
    double g = 0.0, u = 0.0;
#pragma unroll
    for (int w = 0; w < CM_THREADS / 32; ++w) {
      g += sm.part[tid][w].x;
      u += sm.part[tid][w].y;
    }
    sm.val[i0 + tid] = exact_score(g, u, (double)p.scale[b]);
  }
  __syncthreads();
}

// CM_GROUPS: groups of four channels per thread, so CM_THREADS * 4 * CM_GROUPS channels per CTA: the launch takes
// two groups when one group per thread would need more CTAs than are resident at once (a second, partly filled
// wave of these latency-bound CTAs cost 15 % at batch 128; four groups were slower again: 37 against 34 us).
template <int CM_GROUPS>
__global__ void __launch_bounds__(CM_THREADS, 3) channel_select_multi_kernel(const ChanDev p) {
  constexpr int CM_SLICE = CM_THREADS * 4 * CM_GROUPS;
  __shared__ ChanMultiSmem sm;
  const int slice = blockIdx.x, b = blockIdx.y, S = gridDim.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ff = p.ff, d = p.d;
  pdl_trigger();
  pdl_wait();
  uint32_t* sel = p.sel + (size_t)b * CH_SEL_WORDS;
  const int m = (int)(((long long)(1000 - p.p_permille[b]) * ff + 999) / 1000);
  // What the later steps read is requested now, so that it arrives while the histogram is scanned: this CTA's
  // channels of t (and of g, u when there is a selection to make).
  const bool selecting = m > 0 && m < ff;
  float4 v[CM_GROUPS], gq[CM_GROUPS], uq[CM_GROUPS];
#pragma unroll
  for (int gi = 0; gi < CM_GROUPS; ++gi) {
    const int j0 = slice * CM_SLICE + (gi * CM_THREADS + tid) * 4;
    v[gi] = gq[gi] = uq[gi] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j0 < ff) {  // ff is a multiple of 4: a thread's group is present or absent as a whole
      v[gi] = *reinterpret_cast<const float4*>(p.t + (size_t)b * ff + j0);
      if (selecting) {
        gq[gi] = *reinterpret_cast<const float4*>(p.g + (size_t)b * ff + j0);
        uq[gi] = *reinterpret_cast<const float4*>(p.u + (size_t)b * ff + j0);
      }
    }
  }

  // ---- the histogram bin of the m-th largest |t| (every CTA of the token finds the same one) ----
  // keep at or above hi_edge + e_j, drop below lo_edge - e_j, listed in between; e_j = eps * (1.1 |u_j| + |g_j|)
  // bounds the error of this channel's own float32 |t|
  float hi_edge = 0.f, lo_edge = 0.f, eps = 0.f;
  if (m >= ff) {
    hi_edge = 0.f;  // everything is kept
    lo_edge = 0.f;
  } else if (m <= 0) {
    hi_edge = INFINITY;
    lo_edge = INFINITY;
  } else {
    constexpr int BPT = CH_BINS / CM_THREADS;  // bins per thread, descending
    static_assert(BPT == 16, "four 16-byte reads per thread");
    const uint4* own = reinterpret_cast<const uint4*>(sel + CH_BINS - (tid + 1) * BPT);
    const uint4 h0 = own[0], h1 = own[1], h2 = own[2], h3 = own[3];
    const float gmax = __uint_as_float(sel[CH_GMAX]), umax = __uint_as_float(sel[CH_UMAX]);
    const uint32_t hh[BPT] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w, h2.x, h2.y, h2.z, h2.w, h3.x, h3.y, h3.z, h3.w};
    int mine = 0;
#pragma unroll
    for (int q = 0; q < BPT; ++q) mine += (int)hh[q];
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    if (lane == 31) sm.scan[warp] = incl;
    __syncthreads();
    int before = incl - mine;
    for (int w = 0; w < warp; ++w) before += sm.scan[w];
    if (before < m && m <= before + mine) {
      int a = before;
      bool found = false;
#pragma unroll
      for (int q = BPT - 1; q >= 0; --q) {
        a += (int)hh[q];
        if (!found && m <= a) {
          sm.pick = CH_BINS - (tid + 1) * BPT + q;
          found = true;
        }
      }
    }
    __syncthreads();
    const int tb = sm.pick;
    const float bin_lo = chan_bin_lo(tb), bin_hi = tb >= CH_BINS - 1 ? INFINITY : chan_bin_lo(tb + 1);
    // error taken for g_j, u_j: the tensor cores add each 16-long slice of the dot product to the running
    // float32 sum with truncation, so the error grows with the d/16 steps: (d/16) * 2^-24 of the largest
    // magnitude, and never less than 2^-18 of it; carried into t through |silu'| <= 1.1, |silu(g)| <= |g|
    // (a multiple of the error that was measured, no proven bound; the product of both errors is left out)
    eps = fmaxf(3.814697265625e-06f, (float)(d / 16) * 5.9604644775390625e-08f) * fmaxf(gmax, umax);
    // the m-th largest exact |t| lies within the largest error any channel can carry of the bin; a channel is
    // settled when its own error cannot carry it across that
    const float delta = eps * (1.1f * umax + gmax) + 1e-6f * (tb >= CH_BINS - 1 ? bin_lo : bin_hi);
    lo_edge = bin_lo - delta;
    hi_edge = bin_hi + delta;
  }

  // ---- classify this CTA's channels: CM_GROUPS groups of four per thread ----
  int n_above = 0;
  uint32_t between = 0;  // bit 4 gi + e
#pragma unroll
  for (int gi = 0; gi < CM_GROUPS; ++gi) {
    const int j0 = slice * CM_SLICE + (gi * CM_THREADS + tid) * 4;
    const bool in = j0 < ff;
    const float vv[4] = {v[gi].x, v[gi].y, v[gi].z, v[gi].w}, gg[4] = {gq[gi].x, gq[gi].y, gq[gi].z, gq[gi].w},
                uu[4] = {uq[gi].x, uq[gi].y, uq[gi].z, uq[gi].w};
    uint32_t hw[2] = {0, 0}, lw[2] = {0, 0}, kw = 0;
    bool any = false;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float a = fabsf(vv[e]);
      if (!in) continue;
      const float ej = eps * (1.1f * fabsf(uu[e]) + fabsf(gg[e]));
      if (a >= hi_edge + ej) {
        const uint16_t hv = f2bf(vv[e]);
        const uint16_t lv = f2bf(vv[e] - bf2f(hv));
        hw[e >> 1] |= (uint32_t)hv << (16 * (e & 1));
        lw[e >> 1] |= (uint32_t)lv << (16 * (e & 1));
        kw |= 1u << (8 * e);
        ++n_above;
        any = true;
      } else if (a >= lo_edge - ej) {
        between |= 1u << (4 * gi + e);
      }
    }
    if (in) {  // four channels: half a piece of the packed operand
      unsigned char* dst = p.t_op + act_piece_offset(2 * p.Mpad, b, j0 >> 3) + (j0 & 7) * 2;
      *reinterpret_cast<uint2*>(dst) = make_uint2(hw[0], hw[1]);
      *reinterpret_cast<uint2*>(dst + (size_t)p.Mpad * 128) = make_uint2(lw[0], lw[1]);
      *reinterpret_cast<uint32_t*>(p.keep + (size_t)b * ff + j0) = kw;
      if (any) p.live[j0 >> 5] = 1;
    }
  }
  if (!selecting) {  // all or nothing: there is no candidate to wait for
    if (slice == 0 && tid == 0) p.kept_cnt[b] = m >= ff ? ff : 0;
    return;
  }
  // the candidates' places: one request per warp
  n_above = __reduce_add_sync(0xffffffffu, n_above);
  if (lane == 0 && n_above) atomicAdd(sel + CH_N_ABOVE, (uint32_t)n_above);
  {
    const int mine = __popc(between);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    uint32_t slot = 0;
    if (lane == 31 && incl) slot = atomicAdd(sel + CH_N_CAND, (uint32_t)incl);
    slot = __shfl_sync(0xffffffffu, slot, 31) + (uint32_t)(incl - mine);
#pragma unroll
    for (int gi = 0; gi < CM_GROUPS; ++gi) {
      const float vv[4] = {v[gi].x, v[gi].y, v[gi].z, v[gi].w}, gg[4] = {gq[gi].x, gq[gi].y, gq[gi].z, gq[gi].w},
                  uu[4] = {uq[gi].x, uq[gi].y, uq[gi].z, uq[gi].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (!((between >> (4 * gi + e)) & 1u)) continue;
        if (slot < (uint32_t)CH_CAND_CAP) {
          const float a = fabsf(vv[e]), ej = eps * (1.1f * fabsf(uu[e]) + fabsf(gg[e]));
          // and what the fast exponential and division add
          reinterpret_cast<float2*>(p.cand_val)[(size_t)b * CH_CAND_CAP + slot] = make_float2(a, ej + 2e-6f * a);
          p.cand_idx[(size_t)b * CH_CAND_CAP + slot] = slice * CM_SLICE + (gi * CM_THREADS + tid) * 4 + e;
        }
        ++slot;
      }
    }
  }

  // ---- the last CTA of the token settles the candidates ----
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    sm.flag = atomicAdd(sel + CH_DONE, 1u) == (uint32_t)(S - 1) ? 1 : 0;
    sm.n_open = sm.n_sure = 0;
  }
  __syncthreads();
  if (!sm.flag) return;
  __threadfence();
  const int n_cand = (int)__ldcg(sel + CH_N_CAND);
  const int need = m - (int)__ldcg(sel + CH_N_ABOVE);
  if (n_cand > CH_CAND_CAP || need < 0 || need > n_cand) {  // more candidates than the list holds: redo the token
    if (tid == 0) {
      sel[CH_FALLBACK] = 1u;
      atomicAdd(p.status + ST_CH_OVERFLOW, 1);
    }
    return;
  }
  for (int c = tid; c < n_cand; c += CM_THREADS) {
    sm.av[c] = __ldcg(reinterpret_cast<const float2*>(p.cand_val) + (size_t)b * CH_CAND_CAP + c);
    sm.idx[c] = __ldcg(p.cand_idx + (size_t)b * CH_CAND_CAP + c);
  }
  if (tid == 0) {
    sm.thr_hi = -INFINITY;  // need == 0: every candidate lies above "the" threshold's bounds nowhere
    sm.thr_lo = INFINITY;
  }
  __syncthreads();
  // the need-th largest exact |t| of the list lies between the need-th largest of |t| - e and the need-th largest of
  // |t| + e (four threads per candidate; equal values rank by position, any of them gives the same number)
  if (need > 0) {
    for (int c0 = 0; c0 < n_cand; c0 += CM_THREADS / 4) {
      const int c = c0 + (tid >> 2);
      const float2 a = c < n_cand ? sm.av[c] : make_float2(0.f, 0.f);
      const float lo = a.x - a.y, hi = a.x + a.y;
      int rank_lo = 0, rank_hi = 0;
      for (int o = tid & 3; o < n_cand; o += 4) {
        const float2 x = sm.av[o];
        rank_lo += (x.x - x.y > lo) || (x.x - x.y == lo && o < c);
        rank_hi += (x.x + x.y > hi) || (x.x + x.y == hi && o < c);
      }
      rank_lo += __shfl_xor_sync(0xffffffffu, rank_lo, 1);
      rank_hi += __shfl_xor_sync(0xffffffffu, rank_hi, 1);
      rank_lo += __shfl_xor_sync(0xffffffffu, rank_lo, 2);
      rank_hi += __shfl_xor_sync(0xffffffffu, rank_hi, 2);
      if (c < n_cand && rank_lo == need - 1) sm.thr_lo = lo;
      if (c < n_cand && rank_hi == need - 1) sm.thr_hi = hi;
    }
  } else if (tid == 0) {
    sm.thr_hi = INFINITY;  // nothing is kept: every candidate lies below
  }
  __syncthreads();
  for (int c = tid; c < n_cand; c += CM_THREADS) {
    const float2 a = sm.av[c];
    if (a.x + a.y < sm.thr_lo) continue;  // surely dropped
    if (a.x - a.y > sm.thr_hi) {          // surely kept: fewer than `need` candidates can be
      atomicAdd(&sm.n_sure, 1);
      keep_channel(p, b, sm.idx[c]);
    } else {
      sm.open[atomicAdd(&sm.n_open, 1)] = sm.idx[c];
    }
  }
  __syncthreads();
  const int n_open = sm.n_open, need_open = min(max(need - sm.n_sure, 0), n_open);
  if (tid == 0) p.kept_cnt[b] = m;
  if (p.hand_over > 0 && n_open * d > p.hand_over) {
    for (int i = tid; i < n_open; i += CM_THREADS) p.cand_idx[(size_t)b * CH_CAND_CAP + i] = sm.open[i];
    if (tid == 0) sel[CH_OPEN] = ((uint32_t)n_open << 16) | (uint32_t)need_open;
    return;
  }
  if (n_open == 0) return;
#pragma unroll 1
  for (int i0 = 0; i0 < n_open; i0 += CM_EXACT) exact_candidates(p, sm, b, i0, min(CM_EXACT, n_open - i0));
  for (int c0 = 0; c0 < n_open; c0 += CM_THREADS / 4) {  // four threads per channel
    const int c = c0 + (tid >> 2);
    const double mine = c < n_open ? sm.val[c] : 0.0;
    const int j = c < n_open ? sm.open[c] : 0;
    int rank = 0;
    for (int o = tid & 3; o < n_open; o += 4) {
      const double vo = sm.val[o];
      rank += (vo > mine) || (vo == mine && sm.open[o] < j);
    }
    rank += __shfl_xor_sync(0xffffffffu, rank, 1);
    rank += __shfl_xor_sync(0xffffffffu, rank, 2);
    if (c < n_open && rank < need_open && (tid & 3) == 0) keep_channel(p, b, j);
  }
  if (tid == 0) atomicAdd(p.status + ST_CH_REFINED, n_open);
}

// ============================================================================
// channel_list: keep mask -> ascending index list (only when a caller asks for the list)
// ============================================================================
template <int THREADS, int KPT>
__global__ void __launch_bounds__(THREADS) channel_list_kernel(const unsigned char* __restrict__ keep, int ff,
                                                               int32_t* __restrict__ kept_ch) {
  __shared__ SelectSmem sm;
  pdl_trigger();
  pdl_wait();
  const int b = blockIdx.x, j0 = threadIdx.x * KPT;
  const unsigned char* k = keep + (size_t)b * ff;
  compact_indices<THREADS, KPT>([&](int i) { return j0 + i < ff && k[j0 + i] != 0; }, kept_ch + (size_t)b * ff, sm);
}

void launch_channel_select(const ChannelSelectArgs& a, cudaStream_t st) {
  ChanDev c;
  c.d = a.d; c.ff = a.ff; c.p_permille = a.p_permille; c.g = a.g; c.u = a.u; c.t = a.t;
  c.a_op = static_cast<const unsigned char*>(a.a_op); c.scale = a.scale;
  c.w_gu = static_cast<const unsigned char*>(a.w_gate_up);
  const NKGeom geo = nk_geom_gate_up(a.ff, a.d, sm_count());
  c.R = geo.R; c.chunks = geo.chunks; c.Mpad = pad_rows(a.B);
  c.sel = a.sel; c.cand_val = a.cand_val; c.cand_idx = a.cand_idx; c.keep = a.keep;
  c.kept_ch = a.kept_ch; c.kept_cnt = a.kept_cnt;
  c.t_op = static_cast<unsigned char*>(a.t_op);
  c.live = a.live; c.status = a.status;
  const long long resident = 3LL * sm_count();
  const int groups = (long long)((a.ff + CM_THREADS * 4 - 1) / (CM_THREADS * 4)) * a.B > resident ? 2 : 1;
  const dim3 mgrid((a.ff + CM_THREADS * 4 * groups - 1) / (CM_THREADS * 4 * groups), a.B);
  // Where a token can have eight CTAs of its own, more than CH_HAND_OVER elements of open candidates are recomputed by them
  // instead of by its last CTA of the first kernel: three tokens of a Llama-8B layer with 13 to 20 candidates of 4096 elements
  // each 38 us for both kernels, this 21; 16 tokens of a Llama-1B layer with 4 of 2048 16 and 18; 64 tokens of a Llama-8B layer,
  // two CTAs each, 44 both ways.
  constexpr int CH_HAND_OVER = 24576;
  const int per_token = sm_count() >= 8 * a.B ? 8 : 1;
  c.hand_over = per_token > 1 ? CH_HAND_OVER : 0;
  if (groups == 1) SOL_LAUNCH("channel_select", channel_select_multi_kernel<1>, mgrid, dim3(CM_THREADS), 0, st, c);
  else SOL_LAUNCH("channel_select", channel_select_multi_kernel<2>, mgrid, dim3(CM_THREADS), 0, st, c);
  const dim3 grid(a.B);
  if (!a.keeps_all)
    SOL_LAUNCH("channel_select_exact", channel_select_rest_kernel, dim3(per_token, a.B), dim3(CR_THREADS), 0, st, c);
  if (a.kept_ch != nullptr) {
    if (a.ff <= 4096) SOL_LAUNCH("channel_list", (channel_list_kernel<256, 16>), grid, dim3(256), 0, st, a.keep, a.ff, a.kept_ch);
    else if (a.ff <= 16384) SOL_LAUNCH("channel_list", (channel_list_kernel<1024, 16>), grid, dim3(1024), 0, st, a.keep, a.ff, a.kept_ch);
    else SOL_LAUNCH("channel_list", (channel_list_kernel<1024, 48>), grid, dim3(1024), 0, st, a.keep, a.ff, a.kept_ch);
  }
}

}  // namespace sol
