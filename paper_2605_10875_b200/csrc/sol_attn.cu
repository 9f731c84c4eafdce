// Decode attention with a per-sequence keep-rate, as four kernels:
//
//   attn_prep     rotary embedding of q and the new k, append k/v to the paged
//                 cache, split q into three bf16 parts (hi + mid + lo == q to
//                 2^-24) laid out as tensor-core operand rows
//   attn_score    pass 1: stream every K page once (cp.async.bulk into shared
//                 memory), logits of the G heads of the group with m16n8k16
//                 MMAs (tokens are the M side, the split query rows the N
//                 side), group-summed selection score sigma.  Rows that keep
//                 every token need no selection and are left to pass 2
//   token_select  exact top-k per (sequence, kv-head): the bin of the k-th
//                 float32 score from a histogram, then every score within a
//                 small window of the threshold is re-scored in float64 from
//                 the cache rows, so the kept set does not depend on float32
//                 rounding; the outcome is one edge per row: kept is score >
//                 edge (kept tokens of the window get an infinite score)
//   attn_gather   pass 2: walks the scores, reads the V rows of the kept tokens
//                 only (of a row that keeps every token: its K and V rows);
//                 online softmax over the kept logits; split over the row +
//                 combine
//
// Kept count: ceil(r*T) clamped to [0, T] (appendix "Token sparsity",
// "Budgeted token selection"), raised to the forced set (sinks, window; the
// newest token by default).  Softmax over kept tokens only equals the paper's
// additive -inf mask on dropped keys.
#include <math.h>

#include "sol_common.cuh"
#include "sol_internal.h"
#include "sol_select.cuh"

namespace sol {

constexpr int PLAN_STRIDE = 132;  // words of a cumulative work list: entry b is the count before sequence b (per kv-head), entry B the total
constexpr int PLAN_GROUP_TOKENS = 4 * PAGE;  // tokens of one pass-1 unit (a CTA of attn_score: one page per warp)
// Tokens per token_select CTA.  A row of several segments costs a flush of its histogram, a ticket and a second walk over its
// scores: with 8192 (and three CTAs per SM) the selection of 64 sequences of 16384 tokens took 42 us, this 33; 128 ragged
// sequences 39 and 34.
constexpr int TH_SEG = 16384;

// What every selection kernel derives from a row's length and keep-rate.
struct RowPlan {
  int T, n_sink, n_win, nf, k, mode;  // mode 0: keep all; 1: forced only; 2: selection
  __device__ __forceinline__ bool forced(int j) const { return j < n_sink || j >= T - n_win; }
  // every token is kept: no scores, no selection; pass 2 reads keys and values together
  __device__ __forceinline__ bool dense() const { return mode == 0 && T > 0; }
};
__device__ __forceinline__ RowPlan row_plan(const sol_shape_t& sh, const sol_kv_t& kv, const int32_t* r_permille, int b) {
  RowPlan r;
  r.T = min(kv.seq_lens[b], kv.max_pages_per_seq * PAGE);  // never index past the page table
  const int Tp = max(r.T, 0);
  r.n_sink = min(max(sh.n_sink, 0), Tp);
  r.n_win = min(max(sh.n_window, 0), Tp - r.n_sink);
  r.nf = r.n_sink + r.n_win;
  long long bud = ((long long)r_permille[b] * Tp + 999) / 1000;
  if (bud > Tp) bud = Tp;
  r.k = min(Tp, max((int)bud, r.nf));
  r.mode = r.k >= Tp ? 0 : (r.k <= r.nf ? 1 : 2);
  return r;
}

// Warps of a pass-2 CTA (one CTA per SM).
constexpr int gather_warps(int hd, int gmax) { return hd == 64 ? (gmax == 4 ? 16 : 12) : 8; }

// Tokens of a row per pass-2 item, for items of about c kept tokens each; min_len (the token count of a slot of the
// partial results) at least.  A multiple of 128, so that the scores of an item start on a full line.
__device__ __forceinline__ int gather_item_tokens(const RowPlan& rp, int c, int min_len) {
  const int items = max(1, (rp.k + c - 1) / c);
  const int len = ((rp.T + items - 1) / items + 127) & ~127;
  return max(len, min_len);
}

// The flat work lists of the selection and of pass 2 are made by every CTA for itself from the lengths and keep-rates,
// which are inputs of the step, while the kernels before are still running; a list made by one CTA of attn_prep stood in
// that kernel's way and cost the readers a round trip to memory.

// A barrier of the first 128 threads of a CTA.
__device__ __forceinline__ void plan_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// cum[b + 1] = cnt of sequences 0 .. b (cnt: this thread's sequence); cum[0] = 0.  By the first 128 threads of the CTA; wsum:
// four words of shared memory.
__device__ __forceinline__ void plan_scan(int cnt, int* cum, int* wsum) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) wsum[warp] = incl;
  plan_sync();
  for (int w = 0; w < warp; ++w) incl += wsum[w];
  cum[tid + 1] = incl;
  if (tid == 0) cum[0] = 0;
  plan_sync();
}

// The pass-2 items of every sequence into cum; returns the kept tokens c of an item, a power of two from 64 to 1024: the
// one with the least time by the rounds its items take on the resident warps, each round as long as the longest item and
// the ITEM_FILL tokens that filling a warp's ring of row copies is worth, and the ITEM_MERGE tokens that merging the
// partial results is worth where a row has several.  (Long items alone left the chip half empty in a second round: 134 MB
// of values of 32 sequences in 55 us.)
constexpr int ITEM_FILL = 256;  // measured: 64 to 192 cut long rows into too many items (290 -> 365 us where all of
                                // 128 ragged sequences' tokens are kept), 512 gave up balance (32 equal sequences 98 -> 122)
constexpr int ITEM_MERGE = 160;
constexpr int ITEM_C0 = 64, ITEM_NC = 5;
struct PlanSmem {
  int cum[PLAN_STRIDE];
  int n_items[ITEM_NC], longest[ITEM_NC];  // per option: items of a kv-head, kept tokens of the longest
  int sel_units;  // units of token_select of a kv-head
  int wsum[4], per_item;
};
// By the first 128 threads of the CTA.  The options are tried in a rolled loop: this runs once per CTA, at the pace at which
// its code is fetched.
__device__ __forceinline__ int plan_items(const sol_shape_t& sh, const sol_kv_t& kv, const int32_t* r_permille, int B, int min_len,
                                          int target_items, PlanSmem& ps) {
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < ITEM_NC) ps.n_items[tid] = ps.longest[tid] = 0;
  if (tid == 0) ps.sel_units = 0;
  plan_sync();
  RowPlan rp;
  rp.T = rp.k = rp.mode = 0;
  if (tid < B) rp = row_plan(sh, kv, r_permille, tid);
  const int units = __reduce_add_sync(0xffffffffu, rp.mode == 2 ? (rp.T + TH_SEG - 1) / TH_SEG : 0);
  if (lane == 0 && units) atomicAdd(&ps.sel_units, units);
  auto items_of = [&](int c) {  // one item at least, so that the output is always written
    const int len = gather_item_tokens(rp, c, min_len);
    return max(1, (rp.T + len - 1) / len);
  };
#pragma unroll 1
  for (int q = 0; q < ITEM_NC; ++q) {
    const int n = tid < B ? items_of(ITEM_C0 << q) : 0;
    const int sum = __reduce_add_sync(0xffffffffu, n);
    const int most = __reduce_max_sync(0xffffffffu, n > 0 ? max(rp.k, 0) / n : 0);
    if (lane == 0 && sum) {
      atomicAdd(&ps.n_items[q], sum);
      atomicMax(&ps.longest[q], most);
    }
  }
  plan_sync();
  uint32_t key = 0xffffffffu;  // a lane per option; the larger c where two cost the same
  if (lane < ITEM_NC) {
    const int rounds = (ps.n_items[lane] * sh.n_kv_heads + target_items - 1) / target_items;
    const int cost = rounds * (ps.longest[lane] + ITEM_FILL) + (ps.n_items[lane] > B ? ITEM_MERGE : 0);
    key = ((uint32_t)cost << 3) | (uint32_t)(ITEM_NC - 1 - lane);
  }
  const int c = ITEM_C0 << (ITEM_NC - 1 - (int)(__reduce_min_sync(0xffffffffu, key) & 7u));
  plan_scan(tid < B ? items_of(c) : 0, ps.cum, ps.wsum);
  return c;
}

// The sequence that holds flat unit `u` of a cumulative list (cum[b] <= u < cum[b + 1]); n entries + total.
__device__ __forceinline__ int plan_find(const int* cum, int n, int u) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (cum[mid] <= u) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// ============================================================================
// attn_prep
// ============================================================================
// Rotation of an element pair.  The multiply-adds are spelled out: left to the compiler, which of the two products is rounded
// by itself differed between the queries and the keys, and between builds.
__device__ __forceinline__ float2 rotate(float x0, float x1, float c, float s) {
  return make_float2(__fmaf_rn(x0, c, -__fmul_rn(x1, s)), __fmaf_rn(x1, c, __fmul_rn(x0, s)));
}

struct PrepDev {
  sol_shape_t sh;
  sol_kv_t kv;
  const float* qkv;  // [ksplit][B][ldq] partial sums of the QKV projection, or nullptr
  int ldq, ksplit, B;
  const float* qkv_scale;  // [B]
  const uint16_t* q_bf16;  // [B][Hq][hd] or nullptr
  float* q_rot;
  uint16_t* q_split;
  int32_t* work_ctr;  // zeroed here
  uint32_t* row_hist; // zeroed here: [B*Hkv][SEL_BINS] score histogram of rows that span several selection CTAs
  uint32_t* row_ctl;  // zeroed here: [B*Hkv][RC_WORDS]
  int32_t* kept_cnt;  // [B*Hkv], written here; token_select writes it again for the rows it settles
  const int32_t* r_permille;
  int* status;
  int rehearse;
};

constexpr int PREP_THREADS = 128;
// words of AttnArgs::row_ctl, per (sequence, kv-head): segments whose scores are in the histogram, largest |score|,
// keep edge (float bits), non-zero if a score is not a number
enum : int { RC_DONE = 0, RC_MAX, RC_EDGE, RC_NAN, RC_WORDS = 8 };

// One CTA per (kv-head, sequence): the G query heads of the group, the new k row and the new v row.
__global__ void __launch_bounds__(PREP_THREADS) attn_prep_kernel(const PrepDev p) {
  __shared__ float cs[64], sn[64];  // hd/2 <= 64
  const int kvh = blockIdx.x, b = blockIdx.y;
  const int Hq = p.sh.n_q_heads, Hkv = p.sh.n_kv_heads, hd = p.sh.head_dim, half = hd / 2;
  const int G = Hq / Hkv, HG = (G + 3) / 4;
  const int tid = threadIdx.x;
  const bool layer = p.qkv != nullptr;
  const bool rope = layer && p.sh.rope_theta > 0.f;
  if (!layer) pdl_wait();  // the stand-alone attention begins with this kernel
  pdl_trigger();
  const int T = min(p.kv.seq_lens[b], p.kv.max_pages_per_seq * PAGE);  // never index past the page table
  const int pos = T - 1;
  // the angles need only the lengths (an input of the step): float64 functions are slow here, and the projection is
  // still running
  if (tid < half) {
    float c = 1.f, s = 0.f;
    if (rope) {
      // angle = pos * theta^(-2i/hd) in float64, reduced to [-pi, pi] before the float32 sine and cosine
      const double inv = exp2(-2.0 * (double)tid / (double)hd * log2((double)p.sh.rope_theta));
      const double a = (double)pos * inv;
      const double k = rint(a * 0.15915494309189535);
      const float r = (float)fma(-k, 6.283185307179586, a);
      sincosf(r, &s, &c);
    }
    cs[tid] = c;
    sn[tid] = s;
  }
  // In a layer of at most one CTA per SM, the code below is run once ahead of the wait (a rehearsal, which reads nothing that
  // an earlier kernel writes and writes nothing), so that it is in the instruction caches: a single sequence 4.5 us in the
  // chain, this 3.7; 192 and 256 CTAs the same either way; 512 6.9 and 8.3, 1024 5.3 and 6.7, where later CTAs wait for it.
  __shared__ alignas(16) float rowbuf[(8 + 2) * 128];
  const size_t bk = (size_t)b * Hkv + kvh;
  uint16_t* qs = p.q_split + bk * HG * 16 * hd;
  int live = p.rehearse ? 0 : 1;
#pragma unroll 1
  for (;; live = 1) {
    asm volatile("" : "+r"(live));  // one code for both
    if (live) pdl_wait();

    // this (sequence, kv-head)'s part of the q/k/v row: G query heads, the k head, the v head.  The K
    // slices of the projection are summed in order (four columns per thread, eight slices in flight) and scaled.
    if (layer) {
      const float row_scale = p.qkv_scale && live ? p.qkv_scale[b] : 1.0f;
      const float* base = p.qkv + (size_t)b * p.ldq;
      const size_t zs = (size_t)p.B * p.ldq;
#pragma unroll 1
      for (int i = tid * 4; i < (G + 2) * hd; i += PREP_THREADS * 4) {  // hd is a multiple of 4: the four belong to one head
        const int col = i < G * hd ? kvh * G * hd + i
                                   : (i < (G + 1) * hd ? Hq * hd + kvh * hd + (i - G * hd)
                                                       : (Hq + Hkv) * hd + kvh * hd + (i - (G + 1) * hd));
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int z0 = 0; z0 < p.ksplit; z0 += 8) {
          float4 v[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) v[q] = load4_if(base + (size_t)(z0 + q) * zs + col, live && z0 + q < p.ksplit);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            a.x += v[q].x;
            a.y += v[q].y;
            a.z += v[q].z;
            a.w += v[q].w;
          }
        }
        *reinterpret_cast<float4*>(rowbuf + i) = make_float4(a.x * row_scale, a.y * row_scale, a.z * row_scale, a.w * row_scale);
      }
    }

    if (live) {
      if (tid == 0) {
        p.work_ctr[WC_DONE + bk] = 0;
        if (b == 0 && kvh == 0) p.work_ctr[WC_NEXT] = p.work_ctr[WC_SELECT] = 0;
        p.kept_cnt[bk] = row_plan(p.sh, p.kv, p.r_permille, b).k;
      }
      // scratch of the token selection of this (sequence, kv-head)
      if (tid < RC_WORDS) p.row_ctl[bk * RC_WORDS + tid] = 0u;
      if (T > TH_SEG) {  // rows of one segment keep their histogram in shared memory
        uint4* hz = reinterpret_cast<uint4*>(p.row_hist + bk * SEL_BINS);
        for (int i = tid; i < SEL_BINS / 4; i += PREP_THREADS) hz[i] = make_uint4(0u, 0u, 0u, 0u);
      }
      // zero the operand rows of this (sequence, kv-head): pad rows and the unused fourth slot stay zero
      for (int i = tid * 8; i < HG * 16 * hd; i += PREP_THREADS * 8) *reinterpret_cast<uint4*>(qs + i) = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();

    // queries of the group: element pair (f, f + half) of one head per iteration
    for (int i = tid; i < G * half; i += PREP_THREADS) {
      const int gi = i / half, f = i % half, h = kvh * G + gi;
      float q0, q1;
      if (layer) {
        const float2 v = rotate(rowbuf[gi * hd + f], rowbuf[gi * hd + f + half], cs[f], sn[f]);
        q0 = v.x;
        q1 = v.y;
      } else {
        const uint16_t* src = p.q_bf16 + ((size_t)b * Hq + h) * hd;
        q0 = bf2f(src[f]);
        q1 = bf2f(src[f + half]);
      }
      float* qr = p.q_rot + ((size_t)b * Hq + h) * hd;
      if (live) {
        qr[f] = q0;
        qr[f + half] = q1;
      }
      const int hg = gi >> 2, t = gi & 3;
      uint16_t* base = qs + (size_t)(hg * 16) * hd;
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const float q = w ? q1 : q0;
        const int e = w ? f + half : f;
        const uint16_t hi = f2bf(q);
        const float r1 = q - bf2f(hi);
        const uint16_t mid = f2bf(r1);
        const float r2 = r1 - bf2f(mid);
        if (live) {
          base[(2 * t) * hd + e] = hi;
          base[(2 * t + 1) * hd + e] = mid;
          base[(8 + 2 * t) * hd + e] = f2bf(r2);
        }
      }
    }

    if (layer && T > 0) {
      // new k (rotated) and v, rounded to bf16, written at position T-1
      const int lp = pos / PAGE, slot = pos % PAGE;
      const int page = lp < p.kv.max_pages_per_seq ? p.kv.page_table[(size_t)b * p.kv.max_pages_per_seq + lp] : -1;
      const bool good = page >= 0 && page < p.kv.num_pages;
      if (!good && live && tid == 0) atomicOr(p.status + ST_ERR, ERR_BAD_PAGE);
      uint16_t* kp = static_cast<uint16_t*>(p.kv.k_pool);
      uint16_t* vp = static_cast<uint16_t*>(p.kv.v_pool);
      const float* kr = rowbuf + G * hd;
      const float* vr = rowbuf + (G + 1) * hd;
      const size_t dst = (((size_t)page * Hkv + kvh) * PAGE + slot) * hd;
      for (int f = tid; f < half; f += PREP_THREADS) {
        const float2 k = rotate(kr[f], kr[f + half], cs[f], sn[f]);
        const uint16_t k0 = f2bf(k.x), k1 = f2bf(k.y);
        const uint16_t v0 = f2bf(vr[f]), v1 = f2bf(vr[f + half]);
        if (good && live) {
          kp[dst + f] = k0;
          kp[dst + f + half] = k1;
          vp[dst + f] = v0;
          vp[dst + f + half] = v1;
        }
      }
    }
    if (live) return;
    __syncthreads();  // the rehearsal's row is not read any more
  }
}

// ============================================================================
// outputs, and the merge of a row's partial results
// ============================================================================
struct AttnOut {  // each optional
  float* f32;          // [B][Hq][hd]
  uint16_t* bf16;      // [B][Hq][hd]
  unsigned char* hi;   // packed operand of the output projection (2 `rows` rows: high parts, then low parts)
  int rows, Hq, G;
};
// elements e, e + 1 (e even) of one query head
template <int HD>
__device__ __forceinline__ void attn_write(const AttnOut& o, int b, int head, int e, float o0, float o1) {
  const size_t idx = ((size_t)b * o.Hq + head) * HD + e;
  if (o.f32) *reinterpret_cast<float2*>(o.f32 + idx) = make_float2(o0, o1);
  if (o.bf16) *reinterpret_cast<uint32_t*>(o.bf16 + idx) = pack_bf16(o0, o1);
  if (o.hi) {
    const uint16_t h0 = f2bf(o0), h1 = f2bf(o1);
    const int k = head * HD + e;  // column of the projection's input; e is even, so k and k + 1 share a piece
    unsigned char* dst = o.hi + act_piece_offset(2 * o.rows, b, k >> 3) + (k & 7) * 2;
    *reinterpret_cast<uint32_t*>(dst) = (uint32_t)h0 | ((uint32_t)h1 << 16);
    *reinterpret_cast<uint32_t*>(dst + (size_t)o.rows * 128) = pack_bf16(o0 - bf2f(h0), o1 - bf2f(h1));
  }
}

// Merges the ns partial results of a (sequence, kv-head), [ns][G][HD + 2] floats each (weighted sums, maximum in the
// base-2 domain, sum of the weights), by one warp.  fac: 2 * ns * G floats of shared memory.  `live`: false for a rehearsal,
// which writes nothing.
template <int HD, int GMAX>
__device__ __forceinline__ void merge_partials(const AttnOut& o, const float* src0, int ns, int b, int kvh, float* fac, int lane,
                                               bool live) {
  const int G = o.G;
  const size_t stride = (size_t)G * (HD + 2);
  // a lane's columns 2 lane, 2 lane + 1 of every 64: four such pairs of MU partials in flight, the first of them requested
  // before the factors are made (four partials in flight, after the factors: 24 sequences of 2000 tokens 24.0 us, this 22.8;
  // one pair of eight partials: 7.6 us for the 16 partials of a 4096-token row alone)
  constexpr int MU = 8;
  float2 v[4][MU];
  auto request = [&](int p0, int q) {
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int e0 = lane * 2 + 64 * (p0 + x), h = e0 / HD, e = e0 % HD;
      const float* src = src0 + (size_t)q * stride + (size_t)h * (HD + 2) + e;
#pragma unroll
      for (int u = 0; u < MU; ++u)
        v[x][u] = p0 + x < G * HD / 64 && q + u < ns ? __ldcg(reinterpret_cast<const float2*>(src + u * stride)) : make_float2(0.f, 0.f);
    }
  };
  request(0, 0);
  // factors of the partials: f[q][h] = 2^(m_q - M_h) / sum_q l_q 2^(m_q - M_h).  A lane takes one head of GMAX of every 32
  // partials, all requested at once.  The order of a sum is fixed, as the last bits of the results depend on it: the partials
  // that are equal modulo 32 one after the other with the final maximum, then a tree over those 32 (16 apart, 8, 4, 2, 1).
  // (A partial per lane and one head after the other, in the same order: one sequence of 32000 tokens, 250 partials per row of
  // 128-wide heads, 75 us for the attention, this 69; of 2000 tokens 0.5 to 1 us more.)
  {
    constexpr int QL = 32 / GMAX;  // lanes of a head
    const int h = lane % GMAX, q0 = lane / GMAX;
    const float* src = src0 + (size_t)h * (HD + 2) + HD;
    float* const sum = fac + ns * G;
    float2 ml[GMAX];
    auto fetch = [&](int q) {
#pragma unroll
      for (int u = 0; u < GMAX; ++u)
        ml[u] = h < G && q + QL * u < ns ? __ldcg(reinterpret_cast<const float2*>(src + (q + QL * u) * stride)) : make_float2(-INFINITY, 0.f);
    };
    float mm = -INFINITY;
#pragma unroll 1
    for (int q = q0 + 32; q < ns; q += 32) {  // rows of more than 32 partials: the others by way of shared memory
      fetch(q);
#pragma unroll
      for (int u = 0; u < GMAX; ++u) {
        mm = fmaxf(mm, ml[u].x);
        if (h < G && q + QL * u < ns) {
          fac[(q + QL * u) * G + h] = ml[u].x;
          sum[(q + QL * u) * G + h] = ml[u].y;
        }
      }
    }
    fetch(q0);
#pragma unroll
    for (int u = 0; u < GMAX; ++u) mm = fmaxf(mm, ml[u].x);
#pragma unroll
    for (int o = GMAX; o < 32; o <<= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, o));
    float l[GMAX];
#pragma unroll
    for (int u = 0; u < GMAX; ++u) {
      ml[u].x = ml[u].x == -INFINITY ? 0.f : exp2f(ml[u].x - mm);
      l[u] = __fmul_rn(ml[u].y, ml[u].x);
    }
#pragma unroll 1
    for (int q = q0 + 32; q < ns; q += 32) {
#pragma unroll
      for (int u = 0; u < GMAX; ++u)
        if (h < G && q + QL * u < ns) {
          const int at = (q + QL * u) * G + h;
          const float m2 = fac[at], f = m2 == -INFINITY ? 0.f : exp2f(m2 - mm);
          l[u] = __fmaf_rn(sum[at], f, l[u]);
          fac[at] = f;
        }
    }
#pragma unroll
    for (int o = GMAX / 2; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < o; ++u) l[u] = __fadd_rn(l[u], l[u + o]);
#pragma unroll
    for (int o = 16; o >= GMAX; o >>= 1) l[0] = __fadd_rn(l[0], __shfl_xor_sync(0xffffffffu, l[0], o));
    const float inv = l[0] > 0.f ? 1.0f / l[0] : 0.f;
#pragma unroll
    for (int u = 0; u < GMAX; ++u)
      if (h < G && q0 + QL * u < ns) fac[(q0 + QL * u) * G + h] = ml[u].x * inv;
#pragma unroll 1
    for (int q = q0 + 32; q < ns; q += 32)
#pragma unroll
      for (int u = 0; u < GMAX; ++u)
        if (h < G && q + QL * u < ns) fac[(q + QL * u) * G + h] *= inv;
  }
  __syncwarp();
#pragma unroll 1
  for (int p0 = 0; p0 < G * HD / 64; p0 += 4) {
    float2 a[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) a[x] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int q = 0; q < ns; q += MU) {
      if (p0 + q > 0) request(p0, q);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int h = min((lane * 2 + 64 * (p0 + x)) / HD, G - 1);
#pragma unroll
        for (int u = 0; u < MU; ++u) {
          const float f = q + u < ns ? fac[(q + u) * G + h] : 0.f;
          a[x].x = fmaf(v[x][u].x, f, a[x].x);
          a[x].y = fmaf(v[x][u].y, f, a[x].y);
        }
      }
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int e0 = lane * 2 + 64 * (p0 + x);
      if (p0 + x < G * HD / 64 && live) attn_write<HD>(o, b, kvh * G + e0 / HD, e0 % HD, a[x].x, a[x].y);
    }
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src, bool valid) {
  const uint32_t n = valid ? 16u : 0u;  // 0: the 16 bytes are filled with zeros and the source is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst_smem), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// O^T[dim][head] += V^T[dim][token] P^T[token][head] for the 16 tokens tok0 .. of a tile of V rows in shared memory
// (row r: HD bf16, piece c at piece position c ^ (r & 7) of its group of eight).  The eight columns of the
// m16n8k16 tile are weights as bf16 numbers; acc[j] is the tile of dims 16 j .. 16 j + 15.
template <int HD>
__device__ __forceinline__ void pv_step(float (&acc)[HD / 16][4], uint32_t tile, int tok0, int lane, uint32_t b0, uint32_t b1) {
  const int tok = tok0 + (lane & 7) + ((lane >> 4) & 1) * 8;
  const uint32_t row = tile + tok * (HD * 2);
#pragma unroll
  for (int j = 0; j < HD / 16; ++j) {
    const int piece = 2 * j + ((lane >> 3) & 1);
    uint32_t a[4];
    ldsm_x4_trans(a, row + ((piece & ~7) | ((piece ^ tok) & 7)) * 16);
    mma_bf16(acc[j], a[0], a[1], a[2], a[3], b0, b1);
  }
}
// The weights of four tokens as a B fragment: their bf16 high parts, or what those leave (low).
__device__ __forceinline__ void weight_fragment(float w0, float w1, float w2, float w3, bool low, uint32_t& b0, uint32_t& b1) {
  if (low) {
    w0 -= bf2f(f2bf(w0));
    w1 -= bf2f(f2bf(w1));
    w2 -= bf2f(f2bf(w2));
    w3 -= bf2f(f2bf(w3));
  }
  b0 = pack_bf16(w0, w1);
  b1 = pack_bf16(w2, w3);
}

// ============================================================================
// attn_score (pass 1)
// ============================================================================
struct ScoreDev {
  sol_shape_t sh;
  sol_kv_t kv;
  const int32_t* r_permille;
  int Hkv, G, HG, Tmax;
  const uint16_t* q_split;
  float* logits;
  float* sigma;
  int B;
  int* status;
};

constexpr int SC_WARPS = 4;  // pages per CTA
static_assert(SC_WARPS * PAGE == PLAN_GROUP_TOKENS, "a unit of attn_score is one page per warp");
constexpr int SC_PER_SM = 12;  // CTAs per SM of the grid: twice what is resident at head_dim 64 (6), four times at 128 (3: a CTA
                               // holds 64 KB of keys); 6 and 24 measured the same within 1 %

template <int HD, int HG>
__global__ void __launch_bounds__(SC_WARPS * 32) attn_score_kernel(const ScoreDev p) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int PAGE_BYTES = PAGE * HD * 2;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SC_WARPS * PAGE_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  pdl_trigger();
  // The units (sequence, kv-head, group of four pages) that exist are numbered along the batch: every CTA adds up the
  // sequences' group counts itself from the lengths and keep-rates (inputs of the step, so before the wait for the
  // earlier kernels) and takes every gridDim.x-th unit.  A row that keeps every token has no units: pass 2 reads its
  // keys with its values.  (A 3-D grid over the longest row the page table allows spends ~0.5 ns of CTA issue on every
  // empty CTA, and a CTA per unit its set-up: 64 sequences of 16384 tokens 352 us, this 341; 128 ragged sequences 161
  // and 147.)
  __shared__ int s_cum[SC_WARPS * 32 + 1], s_len[SC_WARPS * 32], s_wsum[SC_WARPS];
  int Tt = 0;
  if (tid < p.B) {
    const RowPlan rp = row_plan(p.sh, p.kv, p.r_permille, tid);
    Tt = rp.dense() ? 0 : max(rp.T, 0);  // never indexes past the page table
  }
  int my_incl = (Tt + PLAN_GROUP_TOKENS - 1) / PLAN_GROUP_TOKENS;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, my_incl, o);
    if (lane >= o) my_incl += x;
  }
  if (lane == 31) s_wsum[warp] = my_incl;
  if (tid == 0) {
    s_cum[0] = 0;
    for (int i = 0; i < SC_WARPS; ++i) mbar_init(&bars[i], 1);
    fence_mbar_init();
  }
  __syncthreads();
  for (int w = 0; w < warp; ++w) my_incl += s_wsum[w];
  s_cum[tid + 1] = my_incl;
  s_len[tid] = Tt;
  __syncthreads();
  const int n_units = s_cum[p.B] * p.Hkv;
  // a launch may have no work at all; its first CTA still waits for the kernels before, on which the ones after rely
  if ((int)blockIdx.x >= max(n_units, 1)) return;
  pdl_wait();
  const int g = lane >> 2, t = lane & 3;
  constexpr int KS = HD / 32;  // pair steps (two MMAs of k=16 each)
  uint32_t phase = 0;
  bool dead = false;  // a wait ran out: no more work, but the block-wide counts below still need this warp
#pragma unroll 1
  for (int u = blockIdx.x; u < n_units; u += gridDim.x) {
    // sequence of unit u: how many cumulative counts lie at or below u / Hkv
    const int key = u / p.Hkv;
    const int b = __syncthreads_count(tid < p.B && my_incl <= key);
    const int first = s_cum[b], n_groups = s_cum[b + 1] - first;
    const int rem = u - first * p.Hkv;
    const int kvh = rem / n_groups, grp = rem - kvh * n_groups;
    const int T = s_len[b];
    const int lp = grp * SC_WARPS + warp;  // logical page
    if (dead || lp * PAGE >= T || lp >= p.kv.max_pages_per_seq) continue;
    const int page = p.kv.page_table[(size_t)b * p.kv.max_pages_per_seq + lp];
    if (page < 0 || page >= p.kv.num_pages) {
      if (lane == 0) atomicOr(p.status + ST_ERR, ERR_BAD_PAGE);
      continue;
    }
    unsigned char* tile = smem + warp * PAGE_BYTES;
    if (lane == 0) {
      mbar_expect_tx(&bars[warp], PAGE_BYTES);
      bulk_g2s(tile, static_cast<const uint16_t*>(p.kv.k_pool) + ((size_t)page * p.Hkv + kvh) * PAGE * HD, PAGE_BYTES,
               &bars[warp]);
    }

    // query operand fragments: B[k][n] = q_split[n][k]; this lane holds rows g and 8+g, 8 k-values per pair step
    uint4 qf[HG][KS][2];
#pragma unroll
    for (int hg = 0; hg < HG; ++hg) {
      const uint16_t* qb = p.q_split + ((size_t)((b * p.Hkv + kvh) * HG + hg) * 16) * HD;
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        qf[hg][s][0] = *reinterpret_cast<const uint4*>(qb + (size_t)g * HD + s * 32 + t * 8);
        qf[hg][s][1] = *reinterpret_cast<const uint4*>(qb + (size_t)(8 + g) * HD + s * 32 + t * 8);
      }
    }

    if (!mbar_wait(&bars[warp], phase, p.status)) {
      dead = true;
      continue;
    }
    phase ^= 1;

    const uint32_t tb = smem_u32(tile);
    const size_t row0 = ((size_t)b * p.Hkv + kvh) * p.Tmax;
#pragma unroll 1
    for (int mt = 0; mt < PAGE / 16; ++mt) {
      uint4 ka[KS][2];
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        ka[s][0] = lds128(tb + (mt * 16 + g) * (HD * 2) + (s * 32 + t * 8) * 2);
        ka[s][1] = lds128(tb + (mt * 16 + g + 8) * (HD * 2) + (s * 32 + t * 8) * 2);
      }
      float sig0 = 0.f, sig1 = 0.f;  // tokens g and g+8 of this m-tile
      const int tok0 = lp * PAGE + mt * 16 + g, tok1 = tok0 + 8;
#pragma unroll
      for (int hg = 0; hg < HG; ++hg) {
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int s = 0; s < KS; ++s) {
          mma_bf16(d0, ka[s][0].x, ka[s][1].x, ka[s][0].y, ka[s][1].y, qf[hg][s][0].x, qf[hg][s][0].y);
          mma_bf16(d0, ka[s][0].z, ka[s][1].z, ka[s][0].w, ka[s][1].w, qf[hg][s][0].z, qf[hg][s][0].w);
          mma_bf16(d1, ka[s][0].x, ka[s][1].x, ka[s][0].y, ka[s][1].y, qf[hg][s][1].x, qf[hg][s][1].y);
          mma_bf16(d1, ka[s][0].z, ka[s][1].z, ka[s][0].w, ka[s][1].w, qf[hg][s][1].z, qf[hg][s][1].w);
        }
        // columns 2t, 2t+1 of the first n-tile are head t's hi and mid parts; column 2t of the second its lo part
        const float s0 = d0[0] + (d0[1] + d1[0]);
        const float s1 = d0[2] + (d0[3] + d1[2]);
        const int head = hg * 4 + t;
        if (head < p.G) {
          if (tok0 < T) p.logits[(row0 + tok0) * p.G + head] = s0;
          if (tok1 < T) p.logits[(row0 + tok1) * p.G + head] = s1;
        }
        float q0 = s0, q1 = s1;  // rows of absent heads are zero, so they add nothing
        q0 += __shfl_xor_sync(0xffffffffu, q0, 1);
        q1 += __shfl_xor_sync(0xffffffffu, q1, 1);
        q0 += __shfl_xor_sync(0xffffffffu, q0, 2);
        q1 += __shfl_xor_sync(0xffffffffu, q1, 2);
        sig0 += q0;
        sig1 += q1;
      }
      if (t == 0) {
        if (tok0 < T) p.sigma[row0 + tok0] = sig0 + 0.0f;  // -0 becomes +0: the selection compares floats and keys
        if (tok1 < T) p.sigma[row0 + tok1] = sig1 + 0.0f;
      }
    }
    __syncwarp();  // the tile is rewritten by the next unit's copy
  }
}

// ============================================================================
// token selection: token_select (+ token_list)
// ============================================================================
// Exact top-k of a (sequence, kv-head) row of scores.
//
//   token_select one CTA per 16384 tokens: histogram of its scores over 4096 value bins in shared memory,
//                flushed (non-empty bins) to the row's histogram in global memory, and the largest |score|.
//                The CTA that finishes last (rows of one segment go straight on) finds the bin of the k-th
//                largest score and two values: everything above `edge` (the bin's upper end plus a small
//                window) is kept, everything below `lo` is dropped.  It walks the row's scores again (from
//                L2), counts what lies above the edge and lists the few tokens between lo and edge, ranks these
//                in float32, re-scores those within the window of the k-th value in float64 from the cache
//                rows, and gives the kept ones an infinite score: kept is now "score > edge, or forced", which is
//                all that pass 2 needs to know.
//   token_list   only when a caller asks for the kept indices: the ascending list.
//
// (A list of the kept tokens in memory, written by kernels of its own over 2048-token segments and read back by
// pass 2, cost 16 bytes of traffic per kept token and, with the settling, two more latency-bound launches: 24 + 35 +
// 21 us per layer on 128 ragged sequences.)
// Latency-bound: a chain of barriers and L2 round trips per row.  Hence one bulk copy for a segment's scores and short
// rolled loops over them in shared memory (unrolled over registers, the code of a unit was fetched cold for 14 us even
// where a launch has one unit of 2000 scores), and 512 threads.
constexpr int TS_THREADS = 512;
constexpr int TS_PER_SM = 2;  // CTAs per SM of the persistent grid: 85 KB of shared memory
constexpr float TS_FLT_MAX = 3.402823466e+38f;

struct SelectDev {
  sol_shape_t sh;
  sol_kv_t kv;
  const int32_t* r_permille;
  int Tmax, B;
  const float* q_rot;
  float* sigma;          // kept candidates are overwritten with +inf
  uint32_t* row_hist;    // [B*Hkv][SEL_BINS], zero on entry (rows of several segments)
  uint32_t* row_ctl;     // [B*Hkv][RC_WORDS], zero on entry
  int32_t* kept_cnt;
  int32_t* work_ctr;
  int few;               // the grid is a quarter of the SMs at most
  int* status;
};

// Exclusive prefix sum of v over the TS_THREADS threads (in thread order) and the block total.
__device__ __forceinline__ int ts_block_scan(int v, int& total, int* warp_tot) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  __syncthreads();  // earlier readers of warp_tot are done
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  int before = incl - v;
  total = 0;
#pragma unroll
  for (int w = 0; w < TS_THREADS / 32; ++w) {
    const int x = warp_tot[w];
    if (w < warp) before += x;
    total += x;
  }
  return before;
}

struct SelSmem {
  alignas(128) float score[TH_SEG];  // the segment's scores
  alignas(16) SelectSmemOverlay sm;  // the candidates are listed when the histogram is no longer read
  uint64_t bar;
  double qsum[128];
  float fmax_w[TS_THREADS / 32];
  int s_flag;
  int cum[PLAN_STRIDE], wsum[4];
  alignas(16) int len[128];      // tokens of a sequence that needs a selection, 0 of the others
  unsigned char order[128];      // the sequences, those with the most units first
  int unit_b, unit_kvh, unit_seg;  // the next unit (unit_b < 0: none)
};

// The end of a row's selection, by one CTA: n_list tokens lie above the edge or are forced; ns_all candidates lie
// between the edges (the first SEL_CAND_CAP of them in sm.cand_idx and sm.f32).  Ranks the candidates in
// float32, re-scores those within the window of the k-th value in float64 from the cache rows, and gives the
// kept ones an infinite score.
__device__ __forceinline__ void settle_row(const SelectDev& p, SelectSmemOverlay& sm, double* qsum, const RowPlan& rp, int b,
                                           int kvh, int n_list, float edge, float lo, float delta, int ns_all, bool live) {
  const int Hkv = p.sh.n_kv_heads, hd = p.sh.head_dim, G = p.sh.n_q_heads / Hkv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int WARPS = TS_THREADS / 32;
  const int bk = b * Hkv + kvh;
  const int T = rp.T;
  float* sig = p.sigma + (size_t)bk * p.Tmax;
  const int32_t* table = p.kv.page_table + (size_t)b * p.kv.max_pages_per_seq;
  const int need_s = rp.k - n_list;
  if (ns_all > SEL_CAND_CAP || need_s < 0 || need_s > ns_all) {
    // More scores between the edges than the list holds (long runs of equal scores): float32 order with
    // ties to the lower index, by a radix select over the row's keys that lie between the edges.
    if (tid == 0) atomicAdd(p.status + ST_TOK_OVERFLOW, 1);
    auto between = [&](int j, float& v) {
      if (j >= T || rp.forced(j)) return false;
      v = sig[j];
      return v <= edge && v >= lo;
    };
    const int per = (T + TS_THREADS - 1) / TS_THREADS;
    auto key = [&](int i) -> uint32_t {
      float v;
      return between(i * TS_THREADS + tid, v) ? float_key(v) : 0u;
    };
    int tie_need = 0;
    const int want = min(max(need_s, 1), max(ns_all, 1));
    __syncthreads();  // the histogram takes the candidates' space
    const uint32_t key_thr = select_kth<TS_THREADS, 0, true>(key, want, tie_need, sm, per);
    int ties_taken = 0, at = n_list;
#pragma unroll 1
    for (int base0 = 0; base0 < T && need_s > 0; base0 += TS_THREADS * 8) {  // in index order: ties are kept until tie_need runs out
      const int q0 = base0 + tid * 8;
      uint32_t above_mask = 0, tie_mask = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float v;
        if (between(q0 + e, v)) {
          const uint32_t kk = float_key(v);
          if (kk > key_thr) above_mask |= 1u << e;
          if (kk == key_thr) tie_mask |= 1u << e;
        }
      }
      int tot_ties;
      const int t_before = ties_taken + ts_block_scan(__popc(tie_mask), tot_ties, sm.scan[0]);
      uint32_t take = above_mask;
      int taken = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (((tie_mask >> e) & 1u) && t_before + taken < tie_need) {
          take |= 1u << e;
          ++taken;
        }
      }
      int tot_take;
      ts_block_scan(__popc(take), tot_take, sm.scan[1]);
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if ((take >> e) & 1u) sig[q0 + e] = INFINITY;
      at += tot_take;
      ties_taken += tot_ties;
    }
    n_list = at;
  } else if (need_s > 0) {
    const int ns = ns_all;
    const float* sup_val = sm.f32;
    // float32 rank inside the list: the element of rank need_s - 1 carries the k-th value.  A warp per candidate: a
    // thread per candidate walked the list alone, a chain of up to some hundred shared-memory reads.
    for (int c = warp; c < ns; c += WARPS) {
      const float v = sup_val[c];
      const int j = sm.cand_idx[c];
      int rank = 0;
      for (int o = lane; o < ns; o += 32) {
        const float vo = sup_val[o];
        rank += (vo > v) || (vo == v && sm.cand_idx[o] < j);
      }
      if (__reduce_add_sync(0xffffffffu, rank) == need_s - 1) sm.pick[1] = __float_as_int(v);
    }
    __syncthreads();
    const float thr32 = __int_as_float(sm.pick[1]);
    const float whi = thr32 + delta, wlo = thr32 - delta;
    // classes: above the window (kept, ranks first), inside it (re-scored), below it (dropped)
    int n_above = 0, n_in = 0;
    for (int c = tid; c < ns; c += TS_THREADS) {
      const float v = sup_val[c];
      unsigned char cls = 0;
      if (v > whi) {
        cls = 1;
        ++n_above;
        sm.cand_val[c] = 1.0e300;
      } else if (v >= wlo) {
        cls = 2;
        ++n_in;
        sm.cand_val[c] = (double)v;
      } else {
        sm.cand_val[c] = -1.0e300;
      }
      sm.cand_keep[c] = cls;
    }
    n_above = block_count<TS_THREADS>(n_above, 0, sm);
    n_in = block_count<TS_THREADS>(n_in, 1, sm);
    __syncthreads();
    if (n_above + n_in != need_s) {  // the window holds more than are needed: settle it in float64
      if (tid == 0) atomicAdd(p.status + ST_TOK_REFINED, n_in);
      for (int e = tid; e < hd; e += TS_THREADS) {
        double a = 0.0;
        for (int h = 0; h < G; ++h) a += (double)p.q_rot[((size_t)b * p.sh.n_q_heads + kvh * G + h) * hd + e];
        qsum[e] = a;
      }
      __syncthreads();
      const uint16_t* kp = static_cast<const uint16_t*>(p.kv.k_pool);
      for (int c = warp; c < ns; c += WARPS) {
        if (sm.cand_keep[c] != 2) continue;  // warp-uniform
        const int j = sm.cand_idx[c];
        const int page = table[j / PAGE];
        double a = 0.0;
        if (page >= 0 && page < p.kv.num_pages) {
          const uint16_t* kr = kp + (((size_t)page * Hkv + kvh) * PAGE + (j % PAGE)) * hd;
          for (int e = lane; e < hd; e += 32) a += qsum[e] * (double)bf2f(kr[e]);
        }
        a = warp_sum_d(a);
        if (lane == 0) sm.cand_val[c] = a;
      }
      __syncthreads();
    }
    for (int c = warp; c < ns; c += WARPS) {  // the need_s best of the list are kept
      const double v = sm.cand_val[c];
      const int j = sm.cand_idx[c];
      int rank = 0;
      for (int o = lane; o < ns; o += 32) {
        const double vo = sm.cand_val[o];
        rank += (vo > v) || (vo == v && sm.cand_idx[o] < j);
      }
      if (__reduce_add_sync(0xffffffffu, rank) < need_s && lane == 0 && live) sig[j] = INFINITY;
    }
    n_list += need_s;
  }
  if (tid == 0 && live) p.kept_cnt[bk] = n_list;
}

constexpr int TS_REHEARSAL = 1024;  // scores of a rehearsal

// One (sequence, kv-head, 16384-token segment) of a row that needs a selection; the phase of hs.bar is the caller's.
// live == false: a rehearsal on made-up scores, 1/64 apart, which reads and writes shared memory only.  scores_read: called
// by all threads when hs.score is no longer needed (the caller then lets the next unit's scores come).
template <typename ScoresRead>
__device__ __forceinline__ void token_select_item(const SelectDev& p, SelSmem& hs, int b, int kvh, int seg, uint32_t& phase, bool live,
                                                  ScoresRead scores_read) {
  SelectSmemOverlay& sm = hs.sm;
  uint32_t* hist = sm.hist;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  RowPlan rp = row_plan(p.sh, p.kv, p.r_permille, b);
  if (!live) {
    rp.T = TS_REHEARSAL;
    rp.k = TS_REHEARSAL / 4;
    rp.n_sink = 0;
    rp.nf = rp.n_win = 1;
    rp.mode = 2;
    seg = 0;
  }
  const int T = rp.T;
  const int bk = b * p.sh.n_kv_heads + kvh;
  const float* sig = p.sigma + (size_t)bk * p.Tmax;
  uint32_t* ctl = p.row_ctl + (size_t)bk * RC_WORDS;
  uint32_t* gh = p.row_hist + (size_t)bk * SEL_BINS;
  const int nseg = (T + TH_SEG - 1) / TH_SEG;
  const int j_first = seg * TH_SEG, n_here = min(T - j_first, TH_SEG);
  if (!live)
    for (int i = tid; i < TS_REHEARSAL; i += TS_THREADS) hs.score[i] = (float)((i * 389) & (TS_REHEARSAL - 1)) * 0.015625f;
  for (int i = tid; i < SEL_BINS / 4; i += TS_THREADS) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  if (live) {
    mbar_wait(&hs.bar, phase, p.status);  // a wait that gives up is reported; what follows stays in bounds
    phase ^= 1;
  }

  float mx = 0.f;
  bool nan_here = false;
#pragma unroll 1
  for (int i = tid * 4; i < n_here; i += TS_THREADS * 4) {
    const float4 v = *reinterpret_cast<const float4*>(hs.score + i);
    const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int j = j_first + i + e;
      if (j < T && !rp.forced(j)) {
        atomicAdd(&hist[key_value_bin(float_key(vv[e]))], 1u);
        mx = fmaxf(mx, fabsf(vv[e]));
        nan_here = nan_here || vv[e] != vv[e];
      }
    }
  }
  mx = warp_max(mx);
  if (lane == 0) hs.fmax_w[warp] = mx;
  int any_nan = __syncthreads_or(nan_here ? 1 : 0);
  mx = warp_max(lane < TS_THREADS / 32 ? hs.fmax_w[lane] : 0.f);
  if (nseg > 1) {  // only the CTA that arrives last goes on
    scores_read();
    for (int i = tid; i < SEL_BINS; i += TS_THREADS) {
      const uint32_t c = hist[i];
      if (c) atomicAdd(gh + i, c);
    }
    if (tid == 0) {
      atomicMax(ctl + RC_MAX, __float_as_uint(mx));
      if (any_nan) atomicOr(ctl + RC_NAN, 1u);
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) hs.s_flag = atomicAdd(ctl + RC_DONE, 1u) == (uint32_t)(nseg - 1) ? 1 : 0;
    __syncthreads();
    if (!hs.s_flag) return;
    __threadfence();
    for (int i = tid; i < SEL_BINS / 4; i += TS_THREADS)
      reinterpret_cast<uint4*>(hist)[i] = __ldcg(reinterpret_cast<const uint4*>(gh) + i);
    mx = __uint_as_float(__ldcg(ctl + RC_MAX));
    any_nan = (int)__ldcg(ctl + RC_NAN);
    __syncthreads();
  }

  // ---- the bin that holds the `want`-th largest of the histogrammed scores, how many lie above it, how many in it:
  //      thread t owns a run of bins, the first thread the highest
  auto rank_bin = [&](int want) {
    constexpr int BPT = SEL_BINS / TS_THREADS;
    const uint4* own = reinterpret_cast<const uint4*>(hist + SEL_BINS - BPT * (tid + 1));
    int mine = 0;
#pragma unroll
    for (int q = 0; q < BPT / 4; ++q) {
      const uint4 x = own[q];
      mine += (int)(x.x + x.y + x.z + x.w);
    }
    int total;
    const int before = ts_block_scan(mine, total, sm.scan[0]);
    if (before < want && want <= before + mine) {
      int a = before;
#pragma unroll 1
      for (int q = 0; q < BPT; ++q) {
        const int bin = SEL_BINS - 1 - tid * BPT - q;
        const int c = (int)hist[bin];
        if (want <= a + c) {
          sm.pick[0] = bin;
          sm.pick[1] = a;
          sm.pick[2] = c;
          break;
        }
        a += c;
      }
    }
    __syncthreads();
  };
  const int need_total = rp.k - rp.nf;
  rank_bin(need_total);
  const int vbin = sm.pick[0];
  int above = sm.pick[1];  // scores above the bin
  uint32_t klo, khi;
  value_bin_key_range(vbin, klo, khi);
  const bool prefix_bin = vbin != 0 && vbin != SEL_BINS / 2 - 1 && vbin != SEL_BINS / 2 && vbin != SEL_BINS - 1;
  if (sm.pick[2] > SEL_CAND_CAP / 2 && prefix_bin) {
    // A crowded bin (many nearly equal scores): histogram the next 12 key bits of the bin's keys (they share
    // their upper 15 bits) and take the sub-bin of the k-th score, so that the candidate list stays short.
    __syncthreads();
    for (int i = tid; i < SEL_BINS; i += TS_THREADS) hist[i] = 0;
    __syncthreads();
#pragma unroll 4
    for (int j = tid; j < T; j += TS_THREADS) {
      if (rp.forced(j)) continue;
      const uint32_t kk = float_key(sig[j]);
      if (kk >= klo && kk <= khi) atomicAdd(&hist[(kk >> 5) & 0xfffu], 1u);
    }
    __syncthreads();
    rank_bin(need_total - above);
    above += sm.pick[1];
    klo = (klo & 0xfffe0000u) | ((uint32_t)sm.pick[0] << 5);
    khi = klo | 31u;
  }
  // window: 2^-16 of the largest score, far above the float32 accumulation error of a head_dim-long dot product
  const float delta = mx * 1.52587890625e-05f;
  const float bin_hi = key_to_float(khi);
  const float lo = key_to_float(klo) - delta;
  const float edge = fminf(bin_hi + delta, TS_FLT_MAX);
  if (tid == 0) {
    if (live) ctl[RC_EDGE] = __float_as_uint(edge);  // for pass 2 and token_list
    sm.counts[0] = 0;
  }
  __syncthreads();  // the histogram is not read any more: the candidates take its space

  // ---- what lies between the edges is listed; `above` loses those of the list that lie above the bin ----
  int in_window = 0;
  auto list_candidates = [&](float4 v, int j0) {
    const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (vv[e] >= lo && vv[e] <= edge) {
        const int j = j0 + e;
        if (j < T && !rp.forced(j)) {
          if (vv[e] > bin_hi) ++in_window;
          const int slot = atomicAdd(&sm.counts[0], 1);
          if (slot < SEL_CAND_CAP) {
            sm.cand_idx[slot] = j;
            sm.f32[slot] = vv[e];
          }
        }
      }
    }
  };
  if (nseg == 1) {
#pragma unroll 1
    for (int i = tid * 4; i < n_here; i += TS_THREADS * 4) list_candidates(*reinterpret_cast<const float4*>(hs.score + i), i);
  } else {
#pragma unroll 1
    for (int j0 = tid * 4; j0 < T; j0 += TS_THREADS * 16) {  // four loads in flight
      float4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int j = j0 + q * TS_THREADS * 4;
        v[q] = *reinterpret_cast<const float4*>(sig + (j < T ? j : 0));
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (j0 + q * TS_THREADS * 4 < T) list_candidates(v[q], j0 + q * TS_THREADS * 4);
    }
  }
  in_window = block_count<TS_THREADS>(in_window, 0, sm);  // the barrier inside also publishes the candidates
  above -= in_window;
  if (nseg == 1) scores_read();
  // Counted again where the histogram's ranks say something else than "above the edge": it ranks what is not a number as
  // a large score, but that is never kept; and where the k-th score lies in the top bin, whose end is +inf, scores of
  // +inf are no higher than the bin but above the edge, and all of them are kept.
  if (any_nan || mx == INFINITY) {
    int n = 0;
    for (int j = tid; j < T; j += TS_THREADS) n += !rp.forced(j) && sig[j] > edge ? 1 : 0;
    above = block_count<TS_THREADS>(n, 1, sm);
  }
  settle_row(p, sm, hs.qsum, rp, b, kvh, above + rp.nf, edge, lo, delta, sm.counts[0], live);
}

// Persistent CTAs over the flat list of (sequence, kv-head, segment) units of the rows that need a selection, the longest
// rows first: their last CTA has the whole row to settle.  A CTA's first unit is its index, the later ones are claimed; the
// last warp claims a unit while the one before is worked on and requests its scores as soon as they may be overwritten
// (with the units in batch order, claimed in the way of the first warp and their scores requested when the unit began, 128
// ragged sequences took 48 us; this, with segments of 8192 tokens, 39).
// `rehearse`: the unit's code is run once on made-up scores ahead of the wait and is then in the instruction caches; its first
// pass through code that comes from L2 took as long again (a single sequence of 2000 tokens: 9.1 us in the chain, 6.8).
__global__ void __launch_bounds__(TS_THREADS, TS_PER_SM) token_select_kernel(const SelectDev p, int rehearse) {
  extern __shared__ __align__(128) unsigned char ts_smem[];
  SelSmem& hs = *reinterpret_cast<SelSmem*>(ts_smem);
  const int tid = threadIdx.x, Hkv = p.sh.n_kv_heads;
  const bool fetcher = tid == TS_THREADS - 32;
  pdl_trigger();
  if (fetcher) {
    mbar_init(&hs.bar, 1);
    fence_mbar_init();
  }
  int len = 0;
  if (tid < p.B) {
    const RowPlan rp = row_plan(p.sh, p.kv, p.r_permille, tid);
    if (rp.mode == 2) len = rp.T;
  }
  // Nothing to select: pass 2 is not kept waiting for the order of the units, and has the SMs at once.  The first CTA waits for
  // the kernels before, on which the ones after rely.
  if (p.few && __syncthreads_or(len) == 0) {
    if (blockIdx.x == 0) pdl_wait();
    return;
  }
  if (tid < 128) {
    hs.len[tid] = len;
    plan_sync();
    int rank = 0;
#pragma unroll 1
    for (int j = 0; j < 128; j += 4) {
      const int4 x = *reinterpret_cast<const int4*>(hs.len + j);
      rank += (x.x > len || (x.x == len && j < tid)) + (x.y > len || (x.y == len && j + 1 < tid)) +
              (x.z > len || (x.z == len && j + 2 < tid)) + (x.w > len || (x.w == len && j + 3 < tid));
    }
    hs.order[rank] = (unsigned char)tid;
    plan_sync();
    plan_scan((hs.len[hs.order[tid]] + TH_SEG - 1) / TH_SEG, hs.cum, hs.wsum);
  }
  __syncthreads();
  const int n_units = hs.cum[128] * Hkv;
  if (p.few && (int)blockIdx.x >= n_units) return;  // makes room for pass 2
  uint32_t phase = 0;
  int live = rehearse && (int)blockIdx.x < n_units ? 0 : 1;
  int unit = blockIdx.x, next = blockIdx.x;
  // by the fetcher: looks unit u up and requests its scores
  auto fetch = [&](int u) {
    hs.unit_b = -1;
    if (u < n_units) {
      const int at = plan_find(hs.cum, 128, u / Hkv), b = hs.order[at];
      const int n = hs.cum[at + 1] - hs.cum[at], rem = u - hs.cum[at] * Hkv, kvh = rem / n, seg = rem - kvh * n;
      hs.unit_b = b;
      hs.unit_kvh = kvh;
      hs.unit_seg = seg;
      // a row's space ends on a full page, so whole groups of four may be read
      const uint32_t bytes = (uint32_t)((min(hs.len[b] - seg * TH_SEG, TH_SEG) + 3) & ~3) * 4;
      mbar_expect_tx(&hs.bar, bytes);
      bulk_g2s(hs.score, p.sigma + (size_t)(b * Hkv + kvh) * p.Tmax + seg * TH_SEG, bytes, &hs.bar);
    }
  };
  if (live) {
    pdl_wait();
    if (fetcher) fetch(unit);
  } else if (tid == 0) {
    hs.unit_b = hs.unit_kvh = hs.unit_seg = 0;
  }
  __syncthreads();
#pragma unroll 1
  for (;;) {
    asm volatile("" : "+r"(live));  // one code for a rehearsal and a unit
    const int b = hs.unit_b, kvh = hs.unit_kvh, seg = hs.unit_seg;
    if (b < 0) break;
    if (live && fetcher) next = n_units > (int)gridDim.x ? (int)gridDim.x + atomicAdd(p.work_ctr + WC_SELECT, 1) : n_units;
    token_select_item(p, hs, b, kvh, seg, phase, live != 0, [&] {
      if (live && fetcher) fetch(next);
    });
    if (!live) {
      pdl_wait();
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the made-up scores are overwritten by a bulk copy
      __syncthreads();
      live = 1;
      if (fetcher) fetch(unit);
    }
    __syncthreads();
  }
}

struct ListDev {
  sol_shape_t sh;
  sol_kv_t kv;
  const int32_t* r_permille;
  int Tmax;
  const float* sigma;
  const uint32_t* row_ctl;
  int32_t* kept_idx;  // [B*Hkv][Tmax] ascending
};

// One CTA per (sequence, kv-head): the kept token indices in ascending order, for a caller that asks for them.
__global__ void __launch_bounds__(TS_THREADS) token_list_kernel(const ListDev p) {
  __shared__ int warp_tot[TS_THREADS / 32];
  const int kvh = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
  pdl_trigger();
  const RowPlan rp = row_plan(p.sh, p.kv, p.r_permille, b);
  pdl_wait();
  const int bk = b * p.sh.n_kv_heads + kvh;
  const size_t row = (size_t)bk * p.Tmax;
  const float edge = rp.mode == 2 ? __uint_as_float(p.row_ctl[(size_t)bk * RC_WORDS + RC_EDGE]) : TS_FLT_MAX;
  int at = 0;
#pragma unroll 1
  for (int base0 = 0; base0 < rp.T; base0 += TS_THREADS * 8) {
    const int j0 = base0 + tid * 8;
    uint32_t keep = 0;
    if (j0 < rp.T) {
      float vv[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (rp.mode == 2) {
        const float4 v0 = *reinterpret_cast<const float4*>(p.sigma + row + j0);
        const float4 v1 = *reinterpret_cast<const float4*>(p.sigma + row + j0 + 4);
        vv[0] = v0.x; vv[1] = v0.y; vv[2] = v0.z; vv[3] = v0.w; vv[4] = v1.x; vv[5] = v1.y; vv[6] = v1.z; vv[7] = v1.w;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (j0 + e < rp.T && (rp.mode == 0 || rp.forced(j0 + e) || (rp.mode == 2 && vv[e] > edge))) keep |= 1u << e;
    }
    int total;
    int pos = at + ts_block_scan(__popc(keep), total, warp_tot);
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if ((keep >> e) & 1u) p.kept_idx[row + pos++] = j0 + e;
    at += total;
  }
}

// ============================================================================
// attn_gather (pass 2) with the combine step folded in
// ============================================================================
struct GatherDev {
  sol_shape_t sh;
  sol_kv_t kv;
  const int32_t* r_permille;
  int B, Hkv, G, Tmax, S, min_len, sms;
  const uint16_t* q_split;
  const float* logits;
  const float* sigma;
  const uint32_t* row_ctl;
  int32_t* work_ctr;
  float* part;  // [B][Hkv][S][G][HD + 2]
  float scale_log2;
  AttnOut out;
  int* status;
  int sure_ctas;  // CTAs that are there before the selection ends, whatever it has to do; 0: no rule on that
};

constexpr int GA_BATCH = 32;   // kept tokens per warp step: one per lane in the softmax part
constexpr int GA_CHUNK = 256;  // tokens whose scores a warp looks at together: eight per lane
constexpr int GA_QUEUE = GA_CHUNK + GA_BATCH;
constexpr int GA_DENSE = 16;   // tokens per warp step of a row that keeps every token: keys and values share a stage

// Pass 2 is a gather of 128- or 256-byte V rows with G multiply-adds per element: bound by how many row
// fetches are in flight, so the rows travel by asynchronous 16-byte copies into per-warp rings of shared
// memory (about 190 KB per SM; of a ring's three batches one is worked on and two are in flight) and the registers only
// hold accumulators.
//
// The warps of one persistent CTA per SM work through the list of items, each warp on its own: an item is
// (sequence, kv-head, run of tokens of which about 64 to 1024 are kept); a warp's first item is dealt by its index
// (neighbouring items to different SMs), the later ones are claimed from a counter one item ahead.
//
// A run of a selected row: the warp takes the scores 256 at a time (the next 512 are on their way meanwhile), queues
// the kept tokens' offsets, and works on the kept tokens in batches of 32, NST batches deep: lane l pops token l
// of a batch (and looks its cache row up) one step before the batch's rows and logits are requested; when they have
// landed the warp updates its running maximum per head, every lane computes its token's softmax weights, and the
// weights (as bf16 high and low parts: the eight columns of the m16n8k16 tile, see pv_step) multiply the rows on
// the tensor cores.  The logits travel with the rows: when the memory system is busy every load takes microseconds,
// and a load into registers one step ahead of its use set the pace of the whole warp.
//
// A run of a row that keeps every token: sixteen tokens' keys and values per stage, whole pages in order; the logits
// come from the keys on the tensor cores (the query in three bf16 parts, as in pass 1) and stay on the SM.  (Through
// pass 1, the selection and the lists such a row cost 52 bytes of scratch traffic per token.)
//
// A row of one item goes straight to the output; otherwise one partial per item (accumulators, maximum,
// sum) is written and the warp that finishes the last item of a (sequence, kv-head) merges the partials.
// The pipeline's fill, steady state and drain are one rolled loop: a launch that gives every warp one item of a few
// batches runs its code cold.
// Sixteen warps with rings of three batches, where shared memory allows it: a warp's steps are chains of dependent
// instructions, so more warps beat deeper rings (12 warps with four batches: 118 against 79 us at r = 0.25 on 128 ragged
// sequences, 139 against 129 at r = 0.5, the same where every token is kept).
template <int HD, int GMAX>
struct GatherCfg {
  static constexpr int WARPS = gather_warps(HD, GMAX);
  static constexpr int NST = 3;                              // batches of rows per warp ring
  static constexpr int STAGE_BYTES = GA_BATCH * HD * 2;      // 4 KB / 8 KB
  static constexpr int REHEARSE = WARPS - WARPS / 4;         // the first of the warps that rehearse
  static constexpr int THREADS = WARPS * 32;
  static constexpr int RING_BYTES = WARPS * NST * STAGE_BYTES;  // 192 KB (hd 64, G > 4: 144 KB)
  static constexpr int LOG_BYTES = GA_BATCH * GMAX * 4;         // logits of a batch, then its weights
  static constexpr int W_BYTES = WARPS * NST * LOG_BYTES;
  static constexpr int Q_BYTES = WARPS * GA_QUEUE * 2;
  static constexpr int SMEM = RING_BYTES + W_BYTES + Q_BYTES;
  // a warp's ring holds two floats per head and partial of the longest row (see merge_partials)
  static_assert(NST * STAGE_BYTES >= 2 * 4 * GMAX * (MAX_PAGES_PER_SEQ * PAGE / (HD == 64 ? 256 : 128)), "");
};

template <int HD, int GMAX>
__global__ void __launch_bounds__(GatherCfg<HD, GMAX>::THREADS, 1) attn_gather_kernel(const GatherDev p) {
  using C = GatherCfg<HD, GMAX>;
  constexpr int WARPS = C::WARPS, NST = C::NST, HG = GMAX / 4;
  constexpr int CPR = HD / 8;  // 16-byte pieces per row
  extern __shared__ __align__(128) unsigned char gsm[];
  __shared__ PlanSmem ps;
  const int* const cum = ps.cum;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = p.G, Hkv = p.Hkv;
  const uint16_t* kp = static_cast<const uint16_t*>(p.kv.k_pool);
  const uint16_t* vp = static_cast<const uint16_t*>(p.kv.v_pool);
  const int g = lane >> 2, t = lane & 3;  // row group and column pair of the MMA fragments
  unsigned char* my_ring = gsm + (size_t)warp * NST * C::STAGE_BYTES;
  float* my_w = reinterpret_cast<float*>(gsm + C::RING_BYTES + (size_t)warp * NST * C::LOG_BYTES);  // [NST][32][GMAX]
  uint16_t* my_q = reinterpret_cast<uint16_t*>(gsm + C::RING_BYTES + C::W_BYTES) + warp * GA_QUEUE;
  float* ml = reinterpret_cast<float*>(my_q);  // at the end of an item: [GMAX] maxima, [GMAX] sums
  pdl_trigger();
  // The first four warps make the list of items; the others wait for it at a barrier that the first four only arrive at.
  // Where CTAs are there early (the first `sure_ctas`), the last quarter of the warps rehearse meanwhile: they run the code of
  // an item on absent tokens (even warps that of a selected row, odd ones that of a row that keeps every token; the merge
  // loads whatever the first slot of the partial results holds and drops it), write nothing and leave the code in the
  // instruction caches.  The first pass through code that comes from L2 was half of the time of a launch with one item per
  // warp (a single sequence of 2000 tokens: 19.5 us in the chain, 11.8 with the rehearsal).
  // The selection's CTAs hold SMs until it ends, and the CTAs of this kernel that wait for those are there late: where the
  // others have a warp for every item, they take all of them (attention of four sequences of 8000 tokens, a quarter kept, 64-wide
  // heads: 38.4 us, dealt to every CTA 40.6); else every CTA has its share (128-wide heads, more items than the others have
  // warps: 52.7 us, with the rest left to whoever is free first 62.8).  Up to three items per CTA go to the CTAs that are
  // there whatever the selection does (2000 tokens, all kept: 20.2, dealt to every CTA 21.6).
  int live = 1, per_item = 0, n_items = 0, item = 0;
  bool planned = false, waited = false;
  const int total_warps = gridDim.x * WARPS;
  auto read_plan = [&] {
    per_item = ps.per_item;
    n_items = cum[p.B] * Hkv;
    const int grid = gridDim.x, early = min(grid, max(p.sure_ctas, p.sms - ps.sel_units * Hkv));
    const int deal = p.sure_ctas == 0 ? grid : n_items <= 3 * p.sure_ctas ? min(grid, p.sure_ctas) : n_items <= early * WARPS ? early : grid;
    item = (int)blockIdx.x < deal ? warp * deal + blockIdx.x : n_items;
    planned = true;
  };
  if (warp < 4) {
    const int c = plan_items(p.sh, p.kv, p.r_permille, p.B, p.min_len, p.sms * WARPS, ps);
    if (threadIdx.x == 0) ps.per_item = c;
    plan_sync();
    read_plan();
    asm volatile("bar.arrive 2, %0;" ::"n"(C::THREADS) : "memory");  // the list is there
  } else if ((int)blockIdx.x < p.sure_ctas && warp >= C::REHEARSE) {
    live = 0;
  }
#pragma unroll 1
  for (;;) {
    asm volatile("" : "+r"(live));  // one code for both
    if (live) {
      if (!planned) {
        asm volatile("bar.sync 2, %0;" ::"n"(C::THREADS) : "memory");
        read_plan();
      }
      if (item >= n_items) break;
    }
    int b = 0, ns = 1, kvh = 0, slot = 0;
    if (live) {
      b = plan_find(cum, p.B, item / Hkv);
      ns = cum[b + 1] - cum[b];  // items of every (sequence, kv-head) of this sequence
      const int rem = item - cum[b] * Hkv;
      kvh = rem / ns;
      slot = rem - kvh * ns;
    }
    const bool split = !live || ns > 1;
    const int bk = b * Hkv + kvh;
    const RowPlan rp = row_plan(p.sh, p.kv, p.r_permille, b);
    const int len = gather_item_tokens(rp, live ? per_item : ITEM_C0, p.min_len);
    const int n0 = slot * len, n1 = min(rp.T, n0 + len);  // this item's tokens; n0 is a multiple of 128
    const int32_t* table = p.kv.page_table + (size_t)b * p.kv.max_pages_per_seq;
    if (live && !waited) {
      pdl_wait();
      waited = true;
    }
    // the next item is claimed now, while this one is worked on
    int claimed = n_items;
    if (live && n_items > total_warps && lane == 0) claimed = total_warps + atomicAdd(p.work_ctr + WC_NEXT, 1);

    float acc[HD / 16][4];
#pragma unroll
    for (int j = 0; j < HD / 16; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[j][c] = 0.f;

    if (live ? rp.dense() : (warp & 1) != 0) {
      // ================= a run of a row that keeps every token =================
      // a lane's page of the run (1024 tokens at most)
      int pg = -1;
      if (live && n0 + lane * PAGE < n1) {
        pg = table[n0 / PAGE + lane];
        if (pg < 0 || pg >= p.kv.num_pages) {
          atomicOr(p.status + ST_ERR, ERR_BAD_PAGE);
          pg = -1;
        }
      }
      // queries: columns of the two n-tiles are rows 0..7 and 8..15 of q_split (see attn_prep)
      uint32_t qb[HG][HD / 16][2][2];
#pragma unroll
      for (int hg = 0; hg < HG; ++hg) {
        const uint16_t* q = p.q_split + ((size_t)(bk * ((G + 3) / 4) + hg) * 16) * HD;
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks)
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int x = 0; x < 2; ++x)
              qb[hg][ks][n][x] =
                  hg * 4 < G && live ? *reinterpret_cast<const uint32_t*>(q + (size_t)(8 * n + g) * HD + ks * 16 + x * 8 + 2 * t) : 0u;
      }
      float mt[HG], lt[HG];  // head 4 hg + t: running maximum, this lane's share of the sum
#pragma unroll
      for (int hg = 0; hg < HG; ++hg) {
        mt[hg] = -INFINITY;
        lt[hg] = 0.f;
      }
      const int nstep = live ? (n1 - n0 + GA_DENSE - 1) / GA_DENSE : 1;
      int slot_w = 0;
#pragma unroll 1
      for (int s = 0; s - (NST - 1) < nstep; ++s) {
        const int page = __shfl_sync(0xffffffffu, pg, (s >> 2) & 31);
        if (s < nstep) {  // 16 tokens' keys, then their values, into slot s mod NST
          const uint32_t dst0 = smem_u32(my_ring + slot_w * C::STAGE_BYTES);
          const size_t src = ((size_t)((page < 0 ? 0 : page) * Hkv + kvh) * PAGE + (s & 3) * GA_DENSE) * HD;
#pragma unroll
          for (int i = 0; i < GA_DENSE * CPR / 32; ++i) {
            const int c = i * 32 + lane, r = c / CPR, part = c % CPR;
            const uint32_t off = r * (HD * 2) + ((part & ~7) | ((part ^ r) & 7)) * 16;
            const bool valid = page >= 0 && n0 + s * GA_DENSE + r < n1;
            cp_async16(dst0 + off, kp + src + (size_t)c * 8, valid);
            cp_async16(dst0 + GA_DENSE * HD * 2 + off, vp + src + (size_t)c * 8, valid);
          }
        }
        cp_async_commit();  // an empty group keeps the count of groups per step fixed
        slot_w = slot_w + 1 == NST ? 0 : slot_w + 1;
        const int m = s - (NST - 1);  // the step worked on now: it is in the slot that is written next
        if (m < 0) continue;
        cp_async_wait<NST - 1>();
        const int page_m = __shfl_sync(0xffffffffu, pg, (m >> 2) & 31);
        __syncwarp();  // every lane's pieces have landed
        const uint32_t st = smem_u32(my_ring + slot_w * C::STAGE_BYTES);
        float* wt = my_w;  // [16][GMAX] weights of the step
        float sc[HG], d[HG][2][4];
#pragma unroll
        for (int hg = 0; hg < HG; ++hg)
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int c = 0; c < 4; ++c) d[hg][n][c] = 0.f;
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
          const int r = (lane & 7) + ((lane >> 3) & 1) * 8, piece = 2 * ks + (lane >> 4);
          uint32_t a[4];
          ldsm_x4(a, st + r * (HD * 2) + ((piece & ~7) | ((piece ^ r) & 7)) * 16);
#pragma unroll
          for (int hg = 0; hg < HG; ++hg)
#pragma unroll
            for (int n = 0; n < 2; ++n) mma_bf16(d[hg][n], a[0], a[1], a[2], a[3], qb[hg][ks][n][0], qb[hg][ks][n][1]);
        }
        const int tok = n0 + m * GA_DENSE + g;
#pragma unroll
        for (int hg = 0; hg < HG; ++hg) {
          // columns 2t, 2t+1 of the first n-tile are head t's hi and mid parts; column 2t of the second its lo part
          float x0 = (d[hg][0][0] + (d[hg][0][1] + d[hg][1][0])) * p.scale_log2;
          float x1 = (d[hg][0][2] + (d[hg][0][3] + d[hg][1][2])) * p.scale_log2;
          if (page_m < 0 || tok >= n1) x0 = -INFINITY;
          if (page_m < 0 || tok + 8 >= n1) x1 = -INFINITY;
          float mx = fmaxf(x0, x1);
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
          const float nm = fmaxf(mt[hg], mx);
          sc[hg] = mt[hg] == -INFINITY ? 0.f : exp2f(mt[hg] - nm);
          const float w0 = x0 == -INFINITY ? 0.f : exp2f(x0 - nm), w1 = x1 == -INFINITY ? 0.f : exp2f(x1 - nm);
          mt[hg] = nm;
          lt[hg] = lt[hg] * sc[hg] + (w0 + w1);
          wt[g * GMAX + hg * 4 + t] = w0;
          wt[(g + 8) * GMAX + hg * 4 + t] = w1;
        }
        // this lane's accumulator columns: heads 2t, 2t + 1 (modulo 4 where the columns are high and low parts)
        float sc0 = 1.f, sc1 = 1.f;
#pragma unroll
        for (int hg = 0; hg < HG; ++hg) {
          const float y0 = __shfl_sync(0xffffffffu, sc[hg], (2 * t) & 3), y1 = __shfl_sync(0xffffffffu, sc[hg], (2 * t + 1) & 3);
          if (HG == 1 || (t >> 1) == hg) {
            sc0 = y0;
            sc1 = y1;
          }
        }
#pragma unroll
        for (int j = 0; j < HD / 16; ++j) {
          acc[j][0] *= sc0;
          acc[j][1] *= sc1;
          acc[j][2] *= sc0;
          acc[j][3] *= sc1;
        }
        __syncwarp();
        {
          const float* w = wt + 2 * t * GMAX + (g & (GMAX - 1));
          const float w0 = w[0], w1 = w[GMAX], w2 = w[8 * GMAX], w3 = w[9 * GMAX];
          uint32_t b0, b1;
          weight_fragment(w0, w1, w2, w3, GMAX == 4 && g >= 4, b0, b1);
          pv_step<HD>(acc, st + GA_DENSE * HD * 2, 0, lane, b0, b1);
          if (GMAX == 8) {
            weight_fragment(w0, w1, w2, w3, true, b0, b1);
            pv_step<HD>(acc, st + GA_DENSE * HD * 2, 0, lane, b0, b1);
          }
        }
        __syncwarp();  // the weights and the ring slot are rewritten by the next steps
      }
#pragma unroll
      for (int hg = 0; hg < HG; ++hg) {
        float l = lt[hg];
        l += __shfl_xor_sync(0xffffffffu, l, 4);
        l += __shfl_xor_sync(0xffffffffu, l, 8);
        l += __shfl_xor_sync(0xffffffffu, l, 16);
        if (g == 0) {
          ml[hg * 4 + t] = mt[hg];
          ml[GMAX + hg * 4 + t] = l;
        }
      }
    } else {
      // ======================== a run of a selected row ========================
      const size_t row = (size_t)bk * p.Tmax;
      const float* sig = p.sigma + row;
      const float* lgrow = p.logits + row * G;
      const bool scored = rp.mode == 2 && live;
      const float edge = scored ? __uint_as_float(p.row_ctl[(size_t)bk * RC_WORDS + RC_EDGE]) : INFINITY;

      // ---- the queue of kept tokens' offsets from n0; the scores of the next two chunks wait in registers: lane l holds
      //      tokens 4 l .. 4 l + 3 of both halves of a chunk ----
      int q_head = 0, q_tail = 0, c_at = n0;
      float4 sv[2], sw[2];
      auto fetch_scores = [&](int base, float4 (&v)[2]) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int j = base + x * (GA_CHUNK / 2) + lane * 4;
          v[x] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
          if (j < n1 && scored) v[x] = *reinterpret_cast<const float4*>(sig + j);  // a row's space ends on a full page
        }
      };
      fetch_scores(c_at, sv);
      fetch_scores(c_at + GA_CHUNK, sw);
      const uint32_t below = (1u << lane) - 1u;
      // the next (up to) 32 kept tokens, one per lane: (cache row or -1, token)
      auto pop = [&]() {
#pragma unroll 1
        while (q_tail - q_head < GA_BATCH && c_at < n1) {  // warp-uniform
          const int left = q_tail - q_head;
          const uint16_t moved = lane < left ? my_q[q_head + lane] : (uint16_t)0;
          uint32_t keep = 0;
          {
            const float vv[8] = {sv[0].x, sv[0].y, sv[0].z, sv[0].w, sv[1].x, sv[1].y, sv[1].z, sv[1].w};
#pragma unroll
            for (int e = 0; e < 8; ++e)
              if (vv[e] > edge) keep |= 1u << e;
          }
          sv[0] = sw[0];
          sv[1] = sw[1];
          fetch_scores(c_at + 2 * GA_CHUNK, sw);
          if (c_at < rp.n_sink || c_at + GA_CHUNK > min(n1, rp.T - rp.n_win)) {  // warp-uniform: forced tokens, the run's end
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int j = c_at + (e >> 2) * (GA_CHUNK / 2) + lane * 4 + (e & 3);
              if (rp.forced(j)) keep |= 1u << e;
              if (j >= n1) keep &= ~(1u << e);
            }
          }
          if (!live) {
            keep = 0;
            c_at = n1;
          }
          __syncwarp();
          if (lane < left) my_q[lane] = moved;
          q_tail = left;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const bool k = (keep >> e) & 1u;
            const uint32_t all = __ballot_sync(0xffffffffu, k);
            if (k) my_q[q_tail + __popc(all & below)] = (uint16_t)(c_at - n0 + (e >> 2) * (GA_CHUNK / 2) + lane * 4 + (e & 3));
            q_tail += __popc(all);
          }
          q_head = 0;
          c_at += GA_CHUNK;
          __syncwarp();
        }
        int2 e = make_int2(-1, 0);
        if (q_head + lane < q_tail) {
          const int j = n0 + my_q[q_head + lane], page = table[j / PAGE];
          if (page >= 0 && page < p.kv.num_pages) e = make_int2((page * Hkv + kvh) * PAGE + (j % PAGE), j);
          else atomicOr(p.status + ST_ERR, ERR_BAD_PAGE);
        }
        return e;
      };

      float mt[HG], lt[HG];  // head 4 hg + t: running maximum, this lane's share of the sum
#pragma unroll
      for (int hg = 0; hg < HG; ++hg) {
        mt[hg] = -INFINITY;
        lt[hg] = 0.f;
      }
      int2 e_cur = make_int2(-1, 0);
      int nb = 0x7fffffff;   // batches of the item: known once a pop comes back empty
      int slot_w = NST - 1;  // ring slot of batch s
#pragma unroll 1
      for (int s = -1; s - (NST - 1) < nb; ++s) {
        if (s >= 0 && s < nb) {  // the rows and the logits of batch s
          const uint32_t dst0 = smem_u32(my_ring + slot_w * C::STAGE_BYTES);
#pragma unroll
          for (int i = 0; i < CPR; ++i) {
            const int c = i * 32 + lane, r = c / CPR, part = c % CPR;
            const int ridx = __shfl_sync(0xffffffffu, e_cur.x, r);
            // piece `part` of row r sits at piece position part ^ (r & 7): the transposing matrix loads then touch
            // every bank once
            cp_async16(dst0 + r * (HD * 2) + ((part & ~7) | ((part ^ r) & 7)) * 16, vp + (size_t)(ridx < 0 ? 0 : ridx) * HD + part * 8,
                       ridx >= 0);
          }
          float* lg = my_w + (slot_w * GA_BATCH + lane) * GMAX;
          if (e_cur.x < 0) {  // an absent token weighs nothing
#pragma unroll
            for (int h = 0; h < GMAX; ++h) lg[h] = -INFINITY;
          } else if (GMAX == 4 && G == 4) {
            cp_async16(smem_u32(lg), lgrow + (size_t)e_cur.y * 4, true);
          } else {
#pragma unroll
            for (int h = 0; h < GMAX; ++h)
              if (h < G) cp_async4(smem_u32(lg + h), lgrow + (size_t)e_cur.y * G + h);
          }
        }
        cp_async_commit();  // an empty group keeps the count of groups per step fixed
        e_cur = make_int2(-1, 0);
        if (s + 1 < nb) {
          e_cur = pop();
          if (q_tail == q_head && (live || s >= 0)) nb = s + 1;  // (a rehearsal takes one batch of absent tokens)
          q_head = min(q_tail, q_head + GA_BATCH);
        }
        slot_w = slot_w + 1 == NST ? 0 : slot_w + 1;
        if (s - (NST - 1) < 0) continue;
        // ---- the batch that was requested NST - 1 steps ago, in the slot that is written next ----
        cp_async_wait<NST - 1>();
        __syncwarp();  // every lane's pieces of the batch have landed
        // softmax weights relative to the running maximum, in the logits' place: lane (g, t) takes head t of tokens g,
        // g + 8, g + 16, g + 24, so that a maximum over the batch is three exchanges
        float* wt = my_w + slot_w * GA_BATCH * GMAX;  // [32][GMAX]
        float sc0 = 0.f, sc1 = 0.f;                   // rescaling of this lane's accumulator columns
#pragma unroll
        for (int hg = 0; hg < HG; ++hg) {
          float x[4], mx = -INFINITY;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            x[q] = hg * 4 + t < G ? wt[(g + 8 * q) * GMAX + hg * 4 + t] * p.scale_log2 : -INFINITY;
            mx = fmaxf(mx, x[q]);
          }
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
          mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
          const float nm = fmaxf(mt[hg], mx);
          const float sc = mt[hg] == -INFINITY ? 0.f : exp2f(mt[hg] - nm);
          mt[hg] = nm;
          float l = 0.f;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float w = x[q] == -INFINITY ? 0.f : exp2f(x[q] - nm);
            l += w;
            wt[(g + 8 * q) * GMAX + hg * 4 + t] = w;
          }
          lt[hg] = lt[hg] * sc + l;
          // this lane's accumulator columns: heads 2t, 2t + 1 (modulo 4 where the columns are high and low parts)
          const float y0 = __shfl_sync(0xffffffffu, sc, (2 * t) & 3), y1 = __shfl_sync(0xffffffffu, sc, (2 * t + 1) & 3);
          if (HG == 1 || (t >> 1) == hg) {
            sc0 = y0;
            sc1 = y1;
          }
        }
#pragma unroll
        for (int j = 0; j < HD / 16; ++j) {
          acc[j][0] *= sc0;
          acc[j][1] *= sc1;
          acc[j][2] *= sc0;
          acc[j][3] *= sc1;
        }
        __syncwarp();  // the weights are in place
        const uint32_t st = smem_u32(my_ring + slot_w * C::STAGE_BYTES);
#pragma unroll
        for (int ks = 0; ks < GA_BATCH / 16; ++ks) {
          // B fragment: column g is head g % 4's high (g < 4) or low part, or (GMAX 8) head g; tokens 2t, 2t+1, 2t+8, 2t+9
          const float* w = wt + (ks * 16 + 2 * t) * GMAX + (g & (GMAX - 1));
          const float w0 = w[0], w1 = w[GMAX], w2 = w[8 * GMAX], w3 = w[9 * GMAX];
          uint32_t b0, b1;
          weight_fragment(w0, w1, w2, w3, GMAX == 4 && g >= 4, b0, b1);
          pv_step<HD>(acc, st, ks * 16, lane, b0, b1);
          if (GMAX == 8) {
            weight_fragment(w0, w1, w2, w3, true, b0, b1);
            pv_step<HD>(acc, st, ks * 16, lane, b0, b1);
          }
        }
        __syncwarp();  // the weights and the ring slot are rewritten by the next steps
      }
      __syncwarp();  // the queue is not read any more
#pragma unroll
      for (int hg = 0; hg < HG; ++hg) {
        float l = lt[hg];
        l += __shfl_xor_sync(0xffffffffu, l, 4);
        l += __shfl_xor_sync(0xffffffffu, l, 8);
        l += __shfl_xor_sync(0xffffffffu, l, 16);
        if (g == 0) {
          ml[hg * 4 + t] = mt[hg];
          ml[GMAX + hg * 4 + t] = l;
        }
      }
    }
    cp_async_wait<0>();
    __syncwarp();

    // ---- the item's sums, through the (idle) ring: [G][HD] ----
    float* ob = reinterpret_cast<float*>(my_ring);
#pragma unroll
    for (int j = 0; j < HD / 16; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float v = acc[j][c];
        if (GMAX == 4) v += __shfl_xor_sync(0xffffffffu, v, 2);  // high and low parts
        const int h = 2 * t + (c & 1);
        if (h < GMAX) ob[h * HD + 16 * j + g + (c >> 1) * 8] = v;
      }
    __syncwarp();
    float* dst = p.part + ((size_t)bk * p.S + slot) * G * (HD + 2);
#pragma unroll 1
    for (int e0 = lane * 2; e0 < G * HD; e0 += 64) {
      const int h = e0 / HD, e = e0 % HD;
      const float2 v = *reinterpret_cast<const float2*>(ob + e0);
      if (!split) {  // the row is this one item: its output goes out directly
        const float l = ml[GMAX + h], inv = l > 0.f ? 1.0f / l : 0.f;
        attn_write<HD>(p.out, b, kvh * G + h, e, v.x * inv, v.y * inv);
      } else if (live) {
        *reinterpret_cast<float2*>(dst + h * (HD + 2) + e) = v;
        if (e == 0) *reinterpret_cast<float2*>(dst + h * (HD + 2) + HD) = make_float2(ml[h], ml[GMAX + h]);
      }
    }
    if (split) {  // the last item of this (sequence, kv-head) merges the partials
      int last = 1;
      if (live) {
        __threadfence();
        __syncwarp();
        if (lane == 0) last = atomicAdd(p.work_ctr + WC_DONE + bk, 1) == ns - 1 ? 1 : 0;
        last = __shfl_sync(0xffffffffu, last, 0);
      }
      if (last) {
        if (live) __threadfence();
        merge_partials<HD, GMAX>(p.out, p.part + (size_t)bk * p.S * G * (HD + 2), ns, b, kvh, ob, lane, live);
      }
    }
    __syncwarp();  // the ring and the tables are rewritten by the next item
    if (live) item = __shfl_sync(0xffffffffu, claimed, 0);
    else live = 1;
  }
  if (!waited) pdl_wait();
}

// ============================================================================
// host side
// ============================================================================
template <int HD, int HG>
static void launch_score(const ScoreDev& d, int groups_per_row, cudaStream_t st) {
  const int smem = SC_WARPS * PAGE * HD * 2 + SC_WARPS * 8 + 32;
  ensure_dynamic_smem(reinterpret_cast<const void*>(&attn_score_kernel<HD, HG>), smem);
  const long long units = (long long)groups_per_row * d.Hkv * d.B, ctas = (long long)SC_PER_SM * sm_count();
  SOL_LAUNCH("attn_score", (attn_score_kernel<HD, HG>), dim3((unsigned)(units < ctas ? units : ctas)), dim3(SC_WARPS * 32), smem, st, d);
}

// Persistent: at most one CTA per SM.
template <int HD, int GMAX>
static void launch_gather(const GatherDev& d, long long items, cudaStream_t st) {
  using C = GatherCfg<HD, GMAX>;
  ensure_dynamic_smem(reinterpret_cast<const void*>(&attn_gather_kernel<HD, GMAX>), C::SMEM);
  const int grid = (int)(items < d.sms ? items : d.sms);
  SOL_LAUNCH("attn_gather_v", (attn_gather_kernel<HD, GMAX>), dim3(grid), dim3(C::THREADS), C::SMEM, st, d);
}

void launch_attention(const AttnArgs& a, cudaStream_t st) {
  const sol_shape_t& sh = a.shape;
  const int Hq = sh.n_q_heads, Hkv = sh.n_kv_heads, hd = sh.head_dim, G = Hq / Hkv, HG = (G + 3) / 4;
  const int Tmax = a.kv.max_pages_per_seq * PAGE;

  PrepDev pd;
  pd.sh = sh; pd.kv = a.kv; pd.qkv = a.qkv_f32; pd.ldq = a.ldq; pd.ksplit = a.qkv_ksplit; pd.B = a.B;
  pd.qkv_scale = a.qkv_scale;
  pd.q_bf16 = static_cast<const uint16_t*>(a.q_bf16);
  pd.q_rot = a.q_rot; pd.q_split = static_cast<uint16_t*>(a.q_split); pd.work_ctr = a.work_ctr; pd.status = a.status;
  pd.row_hist = a.row_hist; pd.row_ctl = a.row_ctl; pd.kept_cnt = a.kept_cnt;
  pd.r_permille = a.r_permille;
  pd.rehearse = a.qkv_f32 != nullptr && Hkv * a.B <= sm_count();
  SOL_LAUNCH("attn_prep_rope_append", attn_prep_kernel, dim3(Hkv, a.B), dim3(PREP_THREADS), 0, st, pd);

  if (a.span_tokens > 0) {  // KV refresh: the rows are spans of one sequence's tokens, every token before a row's own is kept
    launch_span_attention(a, a.span_tokens, st);
    return;
  }
  if (sh.token_select == SOL_SELECT_QUEST_PAGES) {
    // the paper's page selection per query head (sol_quest.cu) instead of pass 1 and the token selection; a
    // layer step has just appended a key, so the extrema of its block are taken again first
    launch_quest_selection(a, a.qkv_f32 != nullptr, st);
    launch_quest_attend(a, st);
    return;
  }
  AttnOut out;
  out.f32 = a.out_f32;
  out.bf16 = static_cast<uint16_t*>(a.out_bf16);
  out.hi = static_cast<unsigned char*>(a.out_hi);
  out.rows = a.out_rows; out.Hq = Hq; out.G = G;

  ScoreDev sd;
  sd.sh = sh; sd.kv = a.kv; sd.r_permille = a.r_permille; sd.Hkv = Hkv; sd.G = G; sd.HG = HG; sd.Tmax = Tmax;
  sd.q_split = static_cast<const uint16_t*>(a.q_split);
  sd.logits = a.logits; sd.sigma = a.sigma; sd.status = a.status; sd.B = a.B;
  const int groups_per_row = (a.kv.max_pages_per_seq + SC_WARPS - 1) / SC_WARPS;
  if (hd == 64) {
    if (HG == 1) launch_score<64, 1>(sd, groups_per_row, st);
    else launch_score<64, 2>(sd, groups_per_row, st);
  } else {
    if (HG == 1) launch_score<128, 1>(sd, groups_per_row, st);
    else launch_score<128, 2>(sd, groups_per_row, st);
  }

  SelectDev se;
  se.sh = sh; se.kv = a.kv; se.r_permille = a.r_permille; se.Tmax = Tmax; se.q_rot = a.q_rot; se.B = a.B;
  se.sigma = a.sigma; se.row_hist = a.row_hist; se.row_ctl = a.row_ctl; se.kept_cnt = a.kept_cnt;
  se.status = a.status; se.work_ctr = a.work_ctr;
  // persistent grid: a few CTAs per SM, never more than there can be units
  const long long sel_units = (long long)a.B * Hkv * ((Tmax + TH_SEG - 1) / TH_SEG), sel_res = (long long)sm_count() * TS_PER_SM;
  ensure_dynamic_smem(reinterpret_cast<const void*>(&token_select_kernel), (int)sizeof(SelSmem));
  const int sel_ctas = (int)(sel_units < sel_res ? sel_units : sel_res);
  // Few CTAs: those without a unit leave ahead of the kernels before, so that pass 2 has their SMs (four sequences of 8000 tokens,
  // every token kept: 30 us with it, 33 with those SMs left out).  Of many this does not pay throughout: steps of 48, 64 and 96
  // sequences of 500 tokens, every token kept, 3 to 5 % slower, of 24 and 128 as much faster.
  se.few = sel_ctas <= sm_count() / 4;
  const long long score_ctas = (long long)a.B * Hkv * groups_per_row;
  // A rehearsal (about 3 us) pays where a CTA is there well before pass 1 ends: where the CTAs of both leave room for each
  // other on every SM.  Elsewhere a CTA starts when one of pass 1 ends, and a rehearsal is in its way (16 sequences of 4096
  // tokens: 10.2 us without, 12.9 with it).
  const int rehearse_select = score_ctas + sel_ctas <= 3LL * sm_count();
  SOL_LAUNCH("token_select", token_select_kernel, dim3((unsigned)sel_ctas), dim3(TS_THREADS), sizeof(SelSmem), st, se, rehearse_select);
  if (a.kept_idx_out != nullptr) {
    ListDev ld;
    ld.sh = sh; ld.kv = a.kv; ld.r_permille = a.r_permille; ld.Tmax = Tmax; ld.sigma = a.sigma; ld.row_ctl = a.row_ctl;
    ld.kept_idx = a.kept_idx_out;
    SOL_LAUNCH("token_list", token_list_kernel, dim3(Hkv, a.B), dim3(TS_THREADS), 0, st, ld);
  }

  GatherDev gd;
  gd.sh = sh; gd.kv = a.kv; gd.r_permille = a.r_permille; gd.B = a.B; gd.Hkv = Hkv; gd.G = G; gd.Tmax = Tmax;
  gd.S = a.splits; gd.min_len = attn_split_len(hd);
  gd.q_split = static_cast<const uint16_t*>(a.q_split);
  gd.logits = a.logits; gd.sigma = a.sigma; gd.row_ctl = a.row_ctl; gd.work_ctr = a.work_ctr; gd.sms = sm_count();
  gd.part = a.part; gd.scale_log2 = (float)(1.4426950408889634 / sqrt((double)hd)); gd.out = out; gd.status = a.status;
  const long long items = (long long)a.B * Hkv * a.splits;
  // Where the selection's CTAs are few, the CTAs of pass 2 that are surely there before it ends have the time for a rehearsal.
  // Where they are many, a rehearsal delays the items (24 sequences of about 2000 tokens: 22.8 us without, 25.2 with it).
  gd.sure_ctas = se.few ? sm_count() - sel_ctas : 0;
  if (hd == 64) {
    if (G <= 4) launch_gather<64, 4>(gd, items, st);
    else launch_gather<64, 8>(gd, items, st);
  } else {
    if (G <= 4) launch_gather<128, 4>(gd, items, st);
    else launch_gather<128, 8>(gd, items, st);
  }
}

}  // namespace sol
