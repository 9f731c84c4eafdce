// RMSNorm + per-token symmetric activation quantizer.  One token per CTA; the
// token's row is a few KB, so the kernel is latency-bound: 128-bit loads, the
// row held in registers, two block reductions (sum of squares, absmax).
//
// Quantizer (appendix "Activation quantization", "Quantizer"):
//   q_max = 2^(b-1) - 1, a = max|x|, s = a / q_max, code = clip(rne(x / s)).
// Both divisions are IEEE float32 (__fdiv_rn) so the codes are reproducible
// bit for bit.
#include <type_traits>

#include "sol_common.cuh"
#include "sol_internal.h"
#include "sol_select.cuh"

namespace sol {

constexpr int NQ_THREADS = 256;
constexpr int NQ_VEC = 8;                       // elements per 128-bit bf16 load

__device__ __forceinline__ float block_reduce(float v, bool is_max, float* sh) {
  v = is_max ? warp_max(v) : warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();  // protect sh from the previous use
  if (l == 0) sh[w] = v;
  __syncthreads();
  float r = sh[0];
  for (int i = 1; i < NQ_THREADS / 32; ++i) r = is_max ? fmaxf(r, sh[i]) : r + sh[i];
  return r;
}

// What the input-channel gating of the MLP block needs beside the row (GATE variant only).
struct GateArgs {
  const int32_t* p_permille;  // [B] prune rate: ceil((1 - p) d) channels of largest |x| survive
  float* xm;                  // optional tap: [B][d] the masked normalised row
};
struct NoSmem {
  int unused;
};

// NV: vectors of eight elements per thread (d <= NV * 2048).  Latency-bound: what needs nothing of the kernels before (the
// gains, the width) is read while they run, unless it is the first kernel of a call, and the code is compiled for the row's
// length.  Where it is not the first kernel of a call, the row's code is run once on zeros ahead of the wait (a rehearsal, which
// reads nothing that an earlier kernel writes and writes nothing), so that it is in the instruction caches.
// In the chain, per launch: a single sequence 4.9 us, this 3.3; 24 to 32 sequences 7.3 and 5.5; with the input gating 16.5
// and 12.1.
// PART: the row comes with the partial sums of a projection.  Their loads in flight take 110 to 199 registers (219 to 255 with the
// gating), one CTA per SM, which a layer's 128 rows fit; on an SM that holds a row the projections around it find no room.  The
// stand-alone quantizer takes any number of rows and has none of that (26 to 64 registers; 4096 rows of 2048 elements 14 us, of
// 4096 elements 25.5; with the partial sums' registers a call of thousands of rows took three times as long).
template <bool IN_F32, bool GATE, int NV, bool PART>
__global__ void __launch_bounds__(NQ_THREADS)
norm_quant_kernel(const void* __restrict__ in, const float* __restrict__ part, int ksplit, size_t part_stride,
                  float* __restrict__ sum_out, const uint16_t* __restrict__ gamma, float eps,
                  const int32_t* __restrict__ bits, int d, uint16_t* __restrict__ a_op, int a_op_rows,
                  float* __restrict__ scale,
                  float* __restrict__ xn, int8_t* __restrict__ codes, int16_t* __restrict__ codes16, int* __restrict__ status,
                  uint32_t* __restrict__ clear, int clear_words, int32_t* __restrict__ zero_flags, int n_zero_flags,
                  bool first, const GateArgs gate) {
  __shared__ float sh[NQ_THREADS / 32];
  __shared__ typename std::conditional<GATE, SelectSmem, NoSmem>::type gsm;
  constexpr int NQ_MAX_PER_THREAD = NV;
  constexpr int ZB = NV == 1 ? 12 : 4;  // slices of the partial sums in flight
  const int row = blockIdx.x;
  pdl_trigger();
  if (first) pdl_wait();
  uint4 gains[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    const int v = threadIdx.x + i * NQ_THREADS;
    gains[i] = make_uint4(0u, 0u, 0u, 0u);
    if (gamma != nullptr && v < d / NQ_VEC) gains[i] = reinterpret_cast<const uint4*>(gamma)[v];
  }
  const int width = bits ? __ldcg(bits + row) : 16;
  // a bf16 row without partial sums is an input of the call: that kernel is the first one, or the stand-alone quantizer
  constexpr bool REHEARSE = PART || IN_F32;
  int live = !REHEARSE || first ? 1 : 0;
#pragma unroll 1
  for (;; live = 1) {
    if (REHEARSE) asm volatile("" : "+r"(live));  // one code for a rehearsal and the row
    if (live) pdl_wait();
    int b = width;
    if (zero_flags != nullptr && live)
      for (int i = blockIdx.x * NQ_THREADS + threadIdx.x; i < n_zero_flags; i += gridDim.x * NQ_THREADS) zero_flags[i] = 0;
    if (clear != nullptr && live)  // this token's scratch of the kernels that follow
      for (int i = threadIdx.x; i < clear_words; i += NQ_THREADS) clear[(size_t)row * clear_words + i] = 0u;
    const int nvec = d / NQ_VEC;
    float x[NQ_MAX_PER_THREAD][NQ_VEC];

    // load the row (zero-fill vectors beyond d)
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < NQ_MAX_PER_THREAD; ++i) {
      const int v = threadIdx.x + i * NQ_THREADS;
#pragma unroll
      for (int e = 0; e < NQ_VEC; ++e) x[i][e] = 0.f;
      if (v < nvec) {
        float4 a[PART ? ZB : 1], b4[PART ? ZB : 1];
        const float* src = part + (size_t)row * d + 8 * v;
        if (PART && part != nullptr) {  // partial sums of the projection that produced this row: ZB slices' loads in flight
#pragma unroll
          for (int q = 0; q < ZB; ++q) {
            a[q] = load4_if(src + (size_t)q * part_stride, live && q < ksplit);
            b4[q] = load4_if(src + (size_t)q * part_stride + 4, live && q < ksplit);
          }
        }
        if (IN_F32) {
          const float* p = static_cast<const float*>(in) + (size_t)row * d + 8 * v;
          const float4 a0 = load4_if(p, live), b0 = load4_if(p + 4, live);
          x[i][0] = a0.x; x[i][1] = a0.y; x[i][2] = a0.z; x[i][3] = a0.w;
          x[i][4] = b0.x; x[i][5] = b0.y; x[i][6] = b0.z; x[i][7] = b0.w;
        } else {
          uint4 w = make_uint4(0u, 0u, 0u, 0u);
          if (live) w = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(in) + (size_t)row * d)[v];
          x[i][0] = bf16_lo(w.x); x[i][1] = bf16_hi(w.x); x[i][2] = bf16_lo(w.y); x[i][3] = bf16_hi(w.y);
          x[i][4] = bf16_lo(w.z); x[i][5] = bf16_hi(w.z); x[i][6] = bf16_lo(w.w); x[i][7] = bf16_hi(w.w);
        }
        if (GATE && !live) {  // distinct values for the selection
#pragma unroll
          for (int e = 0; e < NQ_VEC; ++e) x[i][e] = (float)((8 * v + e) * 389 & 0x1fff);
        }
        if (PART && part != nullptr) {  // added in slice order
#pragma unroll 1
          for (int z0 = 0;;) {
#pragma unroll
            for (int q = 0; q < ZB; ++q) {
              x[i][0] += a[q].x; x[i][1] += a[q].y; x[i][2] += a[q].z; x[i][3] += a[q].w;
              x[i][4] += b4[q].x; x[i][5] += b4[q].y; x[i][6] += b4[q].z; x[i][7] += b4[q].w;
            }
            z0 += ZB;
            if (z0 >= ksplit) break;
#pragma unroll
            for (int q = 0; q < ZB; ++q) {
              a[q] = load4_if(src + (size_t)(z0 + q) * part_stride, live && z0 + q < ksplit);
              b4[q] = load4_if(src + (size_t)(z0 + q) * part_stride + 4, live && z0 + q < ksplit);
            }
          }
        }
        if (sum_out != nullptr && live) {
          float4* o = reinterpret_cast<float4*>(sum_out + (size_t)row * d) + 2 * v;
          o[0] = make_float4(x[i][0], x[i][1], x[i][2], x[i][3]);
          o[1] = make_float4(x[i][4], x[i][5], x[i][6], x[i][7]);
        }
#pragma unroll
        for (int e = 0; e < NQ_VEC; ++e) ss += x[i][e] * x[i][e];
      }
    }

    if (gamma != nullptr) {
      const float tot = block_reduce(ss, false, sh);
      const float inv = 1.0f / sqrtf(tot / (float)d + eps);
#pragma unroll
      for (int i = 0; i < NQ_MAX_PER_THREAD; ++i) {
        const int v = threadIdx.x + i * NQ_THREADS;
        if (v < nvec) {
          const uint4 w = gains[i];
          float gm[NQ_VEC] = {bf16_lo(w.x), bf16_hi(w.x), bf16_lo(w.y), bf16_hi(w.y),
                              bf16_lo(w.z), bf16_hi(w.z), bf16_lo(w.w), bf16_hi(w.w)};
#pragma unroll
          for (int e = 0; e < NQ_VEC; ++e) x[i][e] = (x[i][e] * gm[e]) * inv;
        }
      }
    }

    if (xn != nullptr && live) {
#pragma unroll
      for (int i = 0; i < NQ_MAX_PER_THREAD; ++i) {
        const int v = threadIdx.x + i * NQ_THREADS;
        if (v < nvec) {
          float4* p = reinterpret_cast<float4*>(xn + (size_t)row * d) + 2 * v;
          p[0] = make_float4(x[i][0], x[i][1], x[i][2], x[i][3]);
          p[1] = make_float4(x[i][4], x[i][5], x[i][6], x[i][7]);
        }
      }
    }

    if constexpr (GATE) {
      // The paper's structured MLP pruning (appendix "Structured MLP activation pruning"): keep the
      // m = ceil((1 - p) d) channels of largest |x|, ties to the lower index, zero the rest.  |x| orders like its
      // bit pattern; element j = 8 v + e of the row is slot i * 8 + e of thread v - 256 i.
      const int m = (int)(((long long)(1000 - gate.p_permille[row]) * d + 999) / 1000);
      if (m < d) {
        auto key = [&](int q) -> uint32_t {
          const int v = threadIdx.x + (q >> 3) * NQ_THREADS;
          return v < nvec ? __float_as_uint(fabsf(x[q >> 3][q & 7])) : 0u;
        };
        int tie_need = 0;
        uint32_t thr = 0xffffffffu;
        if (m > 0) thr = select_kth<NQ_THREADS, NQ_MAX_PER_THREAD * NQ_VEC>(key, m, tie_need, gsm, NQ_MAX_PER_THREAD * NQ_VEC);
        // ties at the threshold are kept in index order until tie_need runs out: index order is (i, thread, e)
        int taken = 0;  // ties granted to earlier rounds (block-uniform)
#pragma unroll
        for (int i = 0; i < NQ_MAX_PER_THREAD; ++i) {
          const int v = threadIdx.x + i * NQ_THREADS;
          uint32_t tie_mask = 0;
#pragma unroll
          for (int e = 0; e < NQ_VEC; ++e)
            if (m > 0 && v < nvec && __float_as_uint(fabsf(x[i][e])) == thr) tie_mask |= 1u << e;
          // exclusive prefix of the tie counts over the threads of this round
          const int mine = __popc(tie_mask);
          int incl = mine;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if ((threadIdx.x & 31) >= o) incl += y;
          }
          __syncthreads();
          if ((threadIdx.x & 31) == 31) gsm.scan[0][threadIdx.x >> 5] = incl;
          __syncthreads();
          int before = taken + incl - mine, total = 0;
          for (int wq = 0; wq < NQ_THREADS / 32; ++wq) {
            const int y = gsm.scan[0][wq];
            if (wq < (int)(threadIdx.x >> 5)) before += y;
            total += y;
          }
          taken += total;
#pragma unroll
          for (int e = 0; e < NQ_VEC; ++e) {
            const uint32_t kk = __float_as_uint(fabsf(x[i][e]));
            bool keep = m > 0 && kk > thr;
            if ((tie_mask >> e) & 1u) {
              keep = before < tie_need;
              ++before;
            }
            if (!keep) x[i][e] = 0.f;
          }
        }
      }
      if (gate.xm != nullptr && live) {
#pragma unroll
        for (int i = 0; i < NQ_MAX_PER_THREAD; ++i) {
          const int v = threadIdx.x + i * NQ_THREADS;
          if (v < nvec) {
            float4* p = reinterpret_cast<float4*>(gate.xm + (size_t)row * d) + 2 * v;
            p[0] = make_float4(x[i][0], x[i][1], x[i][2], x[i][3]);
            p[1] = make_float4(x[i][4], x[i][5], x[i][6], x[i][7]);
          }
        }
      }
    }

    // widths of 9..15 bits need int16 codes, and their codes are no exact bf16 numbers: they are served only where
    // no tensor-core operand is produced (the stand-alone wide quantizer call)
    const int b_max = (codes16 != nullptr && a_op == nullptr) ? 15 : 8;
    if (b != 16 && (b < 2 || b > b_max)) {  // no kernel for this width: pass through and flag it
      if (threadIdx.x == 0 && status != nullptr && live) atomicOr(status + ST_ERR, ERR_BAD_ACTION);
      b = 16;
    }
    float s = 1.0f;
    float q_max = 0.f;
    if (b != 16) {
      float a = 0.f;
#pragma unroll
      for (int i = 0; i < NQ_MAX_PER_THREAD; ++i)
#pragma unroll
        for (int e = 0; e < NQ_VEC; ++e) a = fmaxf(a, fabsf(x[i][e]));
      a = block_reduce(a, true, sh);
      q_max = (float)((1 << (b - 1)) - 1);
      s = __fdiv_rn(a, q_max);
    }
    if (threadIdx.x == 0 && scale != nullptr && live) scale[row] = s;

#pragma unroll
    for (int i = 0; i < NQ_MAX_PER_THREAD; ++i) {
      const int v = threadIdx.x + i * NQ_THREADS;
      if (v >= nvec) continue;
      float c[NQ_VEC];
      if (b == 16) {
#pragma unroll
        for (int e = 0; e < NQ_VEC; ++e) c[e] = x[i][e];
      } else {
#pragma unroll
        for (int e = 0; e < NQ_VEC; ++e) {
          float r = (s == 0.f) ? 0.f : rintf(__fdiv_rn(x[i][e], s));
          c[e] = fminf(fmaxf(r, -q_max), q_max) + 0.0f;  // +0.0f turns a rounded -0 into +0
        }
      }
      if (a_op != nullptr && live) {
        uint4 w;
        w.x = pack_bf16(c[0], c[1]); w.y = pack_bf16(c[2], c[3]);
        w.z = pack_bf16(c[4], c[5]); w.w = pack_bf16(c[6], c[7]);
        // vector v is the 16-byte piece of elements 8 v .. 8 v + 7: its place in the packed operand layout, or in the plain row
        if (a_op_rows > 0) *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(a_op) + act_piece_offset(a_op_rows, row, v)) = w;
        else reinterpret_cast<uint4*>(a_op + (size_t)row * d)[v] = w;
      }
      if (codes16 != nullptr && live) {
        int q[NQ_VEC];
#pragma unroll
        for (int e = 0; e < NQ_VEC; ++e) q[e] = (b == 16) ? 0 : (int)c[e];
        uint4 w;
        w.x = (q[0] & 0xffff) | ((uint32_t)(q[1] & 0xffff) << 16);
        w.y = (q[2] & 0xffff) | ((uint32_t)(q[3] & 0xffff) << 16);
        w.z = (q[4] & 0xffff) | ((uint32_t)(q[5] & 0xffff) << 16);
        w.w = (q[6] & 0xffff) | ((uint32_t)(q[7] & 0xffff) << 16);
        reinterpret_cast<uint4*>(codes16 + (size_t)row * d)[v] = w;
      }
      if (codes != nullptr && live) {
        int q[NQ_VEC];
#pragma unroll
        for (int e = 0; e < NQ_VEC; ++e) q[e] = (b == 16) ? 0 : (int)c[e];
        uint2 w;
        w.x = (q[0] & 0xff) | ((q[1] & 0xff) << 8) | ((q[2] & 0xff) << 16) | ((uint32_t)(q[3] & 0xff) << 24);
        w.y = (q[4] & 0xff) | ((q[5] & 0xff) << 8) | ((q[6] & 0xff) << 16) | ((uint32_t)(q[7] & 0xff) << 24);
        reinterpret_cast<uint2*>(codes + (size_t)row * d)[v] = w;
      }
    }
    if (live) return;
    if (GATE) __syncthreads();  // the rehearsal's selection is not read any more
  }
}

void launch_norm_quant(const NormQuantArgs& a, cudaStream_t st) {
  const size_t stride = a.part_stride ? a.part_stride : (size_t)a.B * a.d;
  GateArgs g;
  g.p_permille = a.gate_p_permille;
  g.xm = a.xm;
#define SOL_NQ_LAUNCH(F32, GATE, NV, PART)                                                                                   \
  SOL_LAUNCH("norm_quant", (norm_quant_kernel<F32, GATE, NV, PART>), dim3(a.B), dim3(NQ_THREADS), 0, st, a.in, a.part,         \
             a.ksplit, stride, a.sum_out, static_cast<const uint16_t*>(a.gamma_bf16), a.eps, a.bits, a.d,              \
             static_cast<uint16_t*>(a.a_op), a.a_op_rows, a.scale, a.xn, a.codes, a.codes16, a.status, a.clear,         \
             a.clear_words, a.zero_flags, a.n_zero_flags, a.first, g)
#define SOL_NQ_BY_SIZE(F32, GATE, PART)                    \
  do {                                                     \
    if (a.d <= 2048) SOL_NQ_LAUNCH(F32, GATE, 1, PART);      \
    else if (a.d <= 4096) SOL_NQ_LAUNCH(F32, GATE, 2, PART); \
    else SOL_NQ_LAUNCH(F32, GATE, 4, PART);                  \
  } while (0)
#define SOL_NQ_BY_PART(F32, GATE)                          \
  do {                                                     \
    if (a.part != nullptr) SOL_NQ_BY_SIZE(F32, GATE, true); \
    else SOL_NQ_BY_SIZE(F32, GATE, false);                  \
  } while (0)
  if (a.gate_p_permille != nullptr) {  // the second RMSNorm of a layer: always with the partial sums of the output projection
    if (a.in_f32) SOL_NQ_BY_SIZE(true, true, true);
    else SOL_NQ_BY_SIZE(false, true, true);
  } else {
    if (a.in_f32) SOL_NQ_BY_PART(true, false);
    else SOL_NQ_BY_PART(false, false);
  }
#undef SOL_NQ_BY_PART
#undef SOL_NQ_BY_SIZE
#undef SOL_NQ_LAUNCH
}

// ============================================================================
// fake-quantization of the MLP output (the paper's placement of the quantizer)
// ============================================================================
// One token per CTA: z = sum of the down projection's partial sums; per-token symmetric quantizer at
// bits[row] on z (appendix "Activation quantization": a = max|z|, s = a / q_max, code = clip(rne(z / s))),
// z_hat = code * s, from 16 bits on z_hat = z; out = resid + z_hat.
__global__ void __launch_bounds__(NQ_THREADS)
quant_out_kernel(const float* __restrict__ partial, int chunks, size_t chunk_stride, int d, const void* __restrict__ resid,
                 int resid_f32, const int32_t* __restrict__ bits, uint16_t* __restrict__ out_bf16, float* __restrict__ out_f32,
                 float* __restrict__ out_f32_b, float* __restrict__ z_tap, int16_t* __restrict__ z_codes,
                 float* __restrict__ z_scale, int32_t* __restrict__ live, int n_live, int* __restrict__ status) {
  __shared__ float sh[NQ_THREADS / 32];
  pdl_trigger();
  pdl_wait();
  const int row = blockIdx.x;
  // the down projection has read the "granule is live" flags; the next selection starts from zero
  for (int i = blockIdx.x * NQ_THREADS + threadIdx.x; i < n_live; i += gridDim.x * NQ_THREADS) live[i] = 0;
  const int nvec = d / 4;
  constexpr int VPT = 8;  // float4 vectors per thread: d <= 8192
  float4 z[VPT];
  float a = 0.f;
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int v = threadIdx.x + i * NQ_THREADS;
    z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (v < nvec) {
      for (int c0 = 0; c0 < chunks; c0 += 4) {  // four partials' loads in flight, added in order
        float4 t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          t[q] = c0 + q < chunks ? reinterpret_cast<const float4*>(partial + (size_t)(c0 + q) * chunk_stride + (size_t)row * d)[v]
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          z[i].x += t[q].x; z[i].y += t[q].y; z[i].z += t[q].z; z[i].w += t[q].w;
        }
      }
      if (z_tap) reinterpret_cast<float4*>(z_tap + (size_t)row * d)[v] = z[i];
      a = fmaxf(a, fmaxf(fmaxf(fabsf(z[i].x), fabsf(z[i].y)), fmaxf(fabsf(z[i].z), fabsf(z[i].w))));
    }
  }
  int b = bits[row];
  if (b < 2) {
    if (threadIdx.x == 0 && status != nullptr) atomicOr(status + ST_ERR, ERR_BAD_ACTION);
    b = 16;
  }
  float s = 1.0f, q_max = 0.f;
  if (b < 16) {
    a = block_reduce(a, true, sh);
    q_max = (float)((1 << (b - 1)) - 1);
    s = __fdiv_rn(a, q_max);
  }
  if (threadIdx.x == 0 && z_scale) z_scale[row] = s;
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int v = threadIdx.x + i * NQ_THREADS;
    if (v >= nvec) continue;
    float zz[4] = {z[i].x, z[i].y, z[i].z, z[i].w};
    int cc[4] = {0, 0, 0, 0};
    if (b < 16) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float r = (s == 0.f) ? 0.f : rintf(__fdiv_rn(zz[e], s));
        const float c = fminf(fmaxf(r, -q_max), q_max) + 0.0f;
        cc[e] = (int)c;
        zz[e] = __fmul_rn(c, s);
      }
    }
    if (z_codes) {
      uint2 w;
      w.x = (cc[0] & 0xffff) | ((uint32_t)(cc[1] & 0xffff) << 16);
      w.y = (cc[2] & 0xffff) | ((uint32_t)(cc[3] & 0xffff) << 16);
      reinterpret_cast<uint2*>(z_codes + (size_t)row * d)[v] = w;
    }
    float4 acc = make_float4(zz[0], zz[1], zz[2], zz[3]);
    if (resid != nullptr) {
      if (resid_f32) {
        const float4 r = reinterpret_cast<const float4*>(static_cast<const float*>(resid) + (size_t)row * d)[v];
        acc.x += r.x; acc.y += r.y; acc.z += r.z; acc.w += r.w;
      } else {
        const uint2 r = reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(resid) + (size_t)row * d)[v];
        acc.x += bf16_lo(r.x); acc.y += bf16_hi(r.x); acc.z += bf16_lo(r.y); acc.w += bf16_hi(r.y);
      }
    }
    if (out_bf16) {
      uint2 o;
      o.x = pack_bf16(acc.x, acc.y);
      o.y = pack_bf16(acc.z, acc.w);
      reinterpret_cast<uint2*>(out_bf16 + (size_t)row * d)[v] = o;
    }
    if (out_f32) reinterpret_cast<float4*>(out_f32 + (size_t)row * d)[v] = acc;
    if (out_f32_b) reinterpret_cast<float4*>(out_f32_b + (size_t)row * d)[v] = acc;
  }
}

void launch_quant_out(const QuantOutArgs& a, cudaStream_t st) {
  SOL_LAUNCH("mlp_out_quant_residual", quant_out_kernel, dim3(a.M), dim3(NQ_THREADS), 0, st, a.partial, a.chunks,
             (size_t)a.Mpad * a.d, a.d, a.resid, a.resid_f32, a.bits, static_cast<uint16_t*>(a.out_bf16), a.out_f32, a.out_f32_b,
             a.z_tap, a.z_codes, a.z_scale, a.live, a.n_live, a.status);
}

}  // namespace sol
