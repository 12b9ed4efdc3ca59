// Single-token decode (Table 1 "Decode time per token"): one query per head attends over the
// m readout rows of the state plus the window tokens [b, t].  ONE kernel per step: every CTA rotates
// the query heads it serves (and, where its rows end with the new token, that token's key), streams
// its share of the rows with 16-byte loads into an online softmax, and the row splits of a head - a
// thread-block cluster - merge their partial results through distributed shared memory; few heads over many rows take several
// clusters per head (plan_decode), of which the last to arrive merges.
// What bounds it: with many heads HBM (K_hat, V_hat and the window are read once); with few the
// latency of launch, first loads and merge, and on the host the launch itself, which is why the rotation of the
// token and the merge are not kernels of their own: 32 heads over 256 + window rows took 1.9 + 7.4 + 3.1 us
// in three kernels and 18.5 us per step on the host's side; now 7.0 us per step, 4.5 with the rows fetched ahead (decode_short_kernel).  64 x 32 heads over 4096 + window
// rows: 763 -> 695 us per step with its share of the block's fold, the set-up of a step under the tail of the one before.
#include <cooperative_groups.h>

#include <algorithm>

#include <utility>

#include "kvm_internal.h"
#include "ln_rows.cuh"
#include "tc_common.cuh"

namespace kvm {

// One rotary channel: `val` with its partner `oth` of the other rotary half.
__device__ __forceinline__ float rope_pair(float val, float oth, float cs, float sn, bool lower) {
  return lower ? val * cs - oth * sn : oth * sn + val * cs;
}

struct DecodeParams {
  const __nv_bfloat16 *q, *k, *v;   // [B*Hq, D], [U, D]
  const float* gate;                // [U] or NULL
  const double* inv_freq;
  const float *lnq_w, *lnq_b, *lnk_w, *lnk_b;
  const __half *Khat, *Vhat;
  __half *ringK, *ringV;
  float* ringG;
  const float *tau_s, *tau_b;
  __nv_bfloat16* out;
  int32_t* sat_counter;
  int64_t Mcap, ringCap, t;
  int m, n;              // state rows; all rows: m + window tokens, the new one last
  int ringLen, slot_b;   // ring slot of the window's first token
  int slot_t;            // ring slot of the new token
  int Hq, Hkv, G, nsplit, r;
  int nclus;             // clusters of nsplit CTAs per group of heads
  float* part;           // (nclus > 1) merged results of the clusters, [CTA group][rank][cluster][share + 2]
  int32_t* ticket;       // (nclus > 1) [CTA group][rank], zero between launches
  uint32_t *seen;        // (short steps) the step that has last met the end of the one before it, by its number
  uint32_t no, base;     // number of this step, and of the first one since a kernel other than a step wrote rows or window slots
  int rpw;               // (short steps) rows per warp
  int32_t* status;
  float qk_ln_eps;
};

__device__ __forceinline__ void unpack8(const uint4& w, float (&f)[8]) {
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
  const float2 c = __half22float2(*reinterpret_cast<const __half2*>(&w.z));
  const float2 e = __half22float2(*reinterpret_cast<const __half2*>(&w.w));
  f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y; f[4] = c.x; f[5] = c.y; f[6] = e.x; f[7] = e.y;
}

// A row that is read once.  Not the non-coherent path (.nc): a step is resident while the kernel before it still writes
// window slots or readout rows, and only ordinary loads are ordered by griddepcontrol.wait.
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 r;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

// The new token's share of a CTA's set-up: the query heads [bh0, bh0 + GQ) rotated into s_q, and, where `fresh`
// (the CTA's rows end with the new token), its rotated key and its value into s_new; the first query head's CTA of a
// kv group (`store`) also writes them to the window ring, and `count_q` says which CTA of a head counts the inputs that
// had to be clamped to the fp16 range.  Plain rows: one thread per channel.
template <int D, int GQ, typename F>
__device__ __forceinline__ void new_token(const DecodeParams& p, int bh0, int64_t u, bool fresh, bool store, bool count_q,
                                          __half (*s_q)[D], __half (*s_new)[D], F&& behind_wait) {
  const int x = threadIdx.x % D;
  const int half = p.r >> 1;
  float cs = 1.f, sn = 0.f;
  int partner = x;
  if (x < p.r) {
    const int pidx = x < half ? x : x - half;
    double s, c;
    sincos((double)p.t * p.inv_freq[pidx], &s, &c);
    cs = (float)c; sn = (float)s;
    partner = x < half ? x + half : x - half;
  }
  // (the step before this one, or whatever wrote the inputs and the rows, may still be running up to here)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  behind_wait();
  int nsat = 0;
  for (int i = threadIdx.x / D; i < GQ + (fresh ? 1 : 0); i += 256 / D) {
    const bool isq = i < GQ;
    const __nv_bfloat16* row = isq ? p.q + (int64_t)(bh0 + i) * D : p.k + u * D;
    const float val = __bfloat162float(row[x]), oth = __bfloat162float(row[partner]);
    const float o = (x < p.r) ? rope_pair(val, oth, cs, sn, x < half) : val;
    const __half h = __float2half_rn(fminf(fmaxf(o, -65504.f), 65504.f));
    const int sat = !(fabsf(o) <= 65504.f) ? 1 : 0;
    if (isq) {
      s_q[i][x] = h;
      if (count_q) nsat += sat;
    } else {
      const float vv = __bfloat162float(p.v[u * D + x]);
      const __half hv = __float2half_rn(fminf(fmaxf(vv, -65504.f), 65504.f));
      s_new[0][x] = h; s_new[1][x] = hv;
      if (store) {
        const int64_t at = (u * p.ringCap + p.slot_t) * D + x;
        p.ringK[at] = h; p.ringV[at] = hv;
        nsat += sat + (!(fabsf(vv) <= 65504.f) ? 1 : 0);
      }
    }
  }
  if (nsat) atomicAdd(p.sat_counter, nsat);
}

// The same with LN_q / LN_k applied first (fused front end): one warp per row, d / 8 lanes hold it as eight channels
// each (ln_chunk8: the arithmetic of kvm_head_layernorm), the other lane groups compute copies and store nothing.
// The partner channel of the rotation comes from the lane that holds it.
template <int D, int GQ, typename F>
__device__ __forceinline__ void new_token_ln(const DecodeParams& p, int bh0, int64_t u, bool fresh, bool store, bool count_q,
                                             __half (*s_q)[D], __half (*s_new)[D], F&& behind_wait) {
  constexpr int LPR = D / 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane % LPR;
  const int half = p.r >> 1, ch0 = sub * 8;
  const bool inr = ch0 < p.r, lower = ch0 < half;   // (r / 2 is a multiple of 8: a partner chunk is a whole lane's)
  float cs[8], sn[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) { cs[i] = 1.f; sn[i] = 0.f; }
  if (inr && warp < GQ + (fresh ? 1 : 0)) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      double s, c;
      sincos((double)p.t * p.inv_freq[(lower ? ch0 : ch0 - half) + i], &s, &c);
      cs[i] = (float)c; sn[i] = (float)s;
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  behind_wait();
  int nsat = 0;
  for (int row_i = warp; row_i < GQ + (fresh ? 1 : 0); row_i += 8) {   // (uniform over the warp)
    const bool isq = row_i < GQ;
    const int h = isq ? (bh0 + row_i) % p.Hq : (int)(u % p.Hkv);
    float x[8];
    {
      const uint4 raw = *reinterpret_cast<const uint4*>((isq ? p.q + (int64_t)(bh0 + row_i) * D : p.k + u * D) + ch0);
      const __nv_bfloat162* pv = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(pv[i]);
        x[2 * i] = f.x; x[2 * i + 1] = f.y;
      }
    }
    float w8[8], b8[8];
    ln_load_affine<D>(isq ? p.lnq_w : p.lnk_w, isq ? p.lnq_b : p.lnk_b, h, sub, w8, b8);
    ln_chunk8<D>(x, w8, b8, p.qk_ln_eps);
    const int src = (lane & ~(LPR - 1)) + (inr ? (lower ? sub + half / 8 : sub - half / 8) : sub);
    alignas(16) __half hv[8];
    int sat = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float oth = __shfl_sync(0xffffffffu, x[i], src);
      const float o = inr ? rope_pair(x[i], oth, cs[i], sn[i], lower) : x[i];
      sat += !(fabsf(o) <= 65504.f) ? 1 : 0;
      hv[i] = __float2half_rn(fminf(fmaxf(o, -65504.f), 65504.f));
    }
    if (lane >= LPR) continue;
    if (isq) {
      *reinterpret_cast<uint4*>(&s_q[row_i][ch0]) = *reinterpret_cast<const uint4*>(hv);
      if (count_q) nsat += sat;
    } else {
      alignas(16) __half vh[8];
      const uint4 raw = *reinterpret_cast<const uint4*>(p.v + u * D + ch0);
      const __nv_bfloat162* pv = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __bfloat1622float2(pv[i]);
        sat += (!(fabsf(f.x) <= 65504.f) ? 1 : 0) + (!(fabsf(f.y) <= 65504.f) ? 1 : 0);
        vh[2 * i] = __float2half_rn(fminf(fmaxf(f.x, -65504.f), 65504.f));
        vh[2 * i + 1] = __float2half_rn(fminf(fmaxf(f.y, -65504.f), 65504.f));
      }
      *reinterpret_cast<uint4*>(&s_new[0][ch0]) = *reinterpret_cast<const uint4*>(hv);
      *reinterpret_cast<uint4*>(&s_new[1][ch0]) = *reinterpret_cast<const uint4*>(vh);
      if (store) {
        const int64_t at = (u * p.ringCap + p.slot_t) * D + ch0;
        *reinterpret_cast<uint4*>(p.ringK + at) = *reinterpret_cast<const uint4*>(hv);
        *reinterpret_cast<uint4*>(p.ringV + at) = *reinterpret_cast<const uint4*>(vh);
        nsat += sat;
      }
    }
  }
  if (nsat) atomicAdd(p.sat_counter, nsat);
}

// Sums of LEFT values over 2 O lanes: a lane with bit O set goes on with the upper half of the values that are left, the
// other one with the lower half; a single value left is summed over the remaining lanes.
template <int LEFT, int O, int N>
__device__ __forceinline__ void lane_sums(float (&v)[N], int gl) {
  if constexpr (O > 0) {
    if constexpr (LEFT > 1) {
      const bool up = gl & O;
#pragma unroll
      for (int k = 0; k < LEFT / 2; ++k) {
        const float give = up ? v[k] : v[k + LEFT / 2], keep = up ? v[k + LEFT / 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, give, O);
      }
      lane_sums<LEFT / 2, O / 2>(v, gl);
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], O);
      lane_sums<1, O / 2>(v, gl);
    }
  }
}

// grid (nsplit * nclus, B*Hq / GQ), nsplit CTAs of a row a cluster; block 256 = 8 warps.  LPR = D/8 lanes cover one
// row with 16-byte loads, a warp covers RPW = 32/LPR rows per load instruction and UNR such instructions per
// step.  A CTA serves GQ query heads that share one kv head (grouped queries): every key / value row is loaded
// once and meets all GQ queries, so the bytes streamed per step do not grow with the group size.  MULTI: nclus > 1 (a build of
// its own: the steps of one cluster, 5 us each for few rows, took 1 to 3 % longer with the merge of several in the kernel).
template <int D, int GQ, bool LN, bool MULTI>
__global__ void __launch_bounds__(256) decode_step_kernel(DecodeParams p) {
  constexpr int LPR = D / 8;
  constexpr int RPW = 32 / LPR;
  constexpr int UNR = 4;
  constexpr int STEP = RPW * UNR;       // rows per warp per iteration
  __shared__ float s_m[8][GQ], s_l[8][GQ];
  __shared__ __align__(16) float s_acc[8][GQ][D];
  __shared__ float s_part[GQ][D + 2];   // this split's merged result: channels, maximum, sum
  __shared__ __align__(16) __half s_q[GQ][D], s_new[2][D];
  __shared__ int s_last;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int split = blockIdx.x;
  const int bh0 = blockIdx.y * GQ;                 // first query head of this CTA (GQ divides the group size G)
  const int bb = bh0 / p.Hq, hq0 = bh0 % p.Hq, hk = hq0 / p.G;
  const int64_t u = (int64_t)bb * p.Hkv + hk;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = lane / LPR, gl = lane % LPR;   // row group inside the warp, lane inside the row

  const int m = p.m, n = p.n, ns_all = MULTI ? p.nsplit * p.nclus : p.nsplit;
  int per = (n + ns_all - 1) / ns_all;
  per = (per + 8 * STEP - 1) / (8 * STEP) * (8 * STEP);
  const int r0 = split * per;
  const int r1 = min(n, r0 + per);
  const bool fresh = r0 < n && r1 == n;          // this CTA's rows end with the new token

  if (LN) new_token_ln<D, GQ>(p, bh0, u, fresh, fresh && hq0 % p.G == 0, split == 0, s_q, s_new, [] {});
  else new_token<D, GQ>(p, bh0, u, fresh, fresh && hq0 % p.G == 0, split == 0, s_q, s_new, [] {});
  if (fresh && hq0 % p.G == 0 && tid == 0) p.ringG[u * p.ringCap + p.slot_t] = p.gate ? p.gate[u] : 1.0f;
  __syncthreads();

  // Which of a step's GQ * UNR logits of a row group a lane ends up with (index g * UNR + i: head g, row i of the
  // group): the reduction over the LPR lanes of a row halves the values together with the lanes, so every sum costs
  // about one exchange instead of log2(LPR) and every exponential is taken once.
  constexpr int NV = GQ * UNR;
  constexpr int NVL = NV > LPR ? NV / LPR : 1;        // logits per lane
  constexpr int LPV = NV > LPR ? 1 : LPR / NV;        // lanes that hold the same logit
  const int v0 = gl / LPV * NVL;                      // this lane's first logit
  const int my_g = v0 / UNR;
  const float kLog2e = 1.4426950408889634f;
  const float scale_s = p.tau_s[hq0 + my_g] * rsqrtf((float)D) * kLog2e;
  const float scale_b = p.tau_b[hq0 + my_g] * rsqrtf((float)D) * kLog2e;
  float qf[GQ][8];
#pragma unroll
  for (int g = 0; g < GQ; ++g) unpack8(*reinterpret_cast<const uint4*>(&s_q[g][gl * 8]), qf[g]);
  float m_run = -INFINITY, l_run = 0.f;   // of head my_g: maximum over the warp's rows, sum over this lane's
  float acc[GQ][8];
#pragma unroll
  for (int g = 0; g < GQ; ++g)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[g][c] = 0.f;

  const __half* KhatU = p.Khat + u * p.Mcap * D + gl * 8;
  const __half* VhatU = p.Vhat + u * p.Mcap * D + gl * 8;
  const __half* ringKU = p.ringK + u * p.ringCap * D + gl * 8;
  const __half* ringVU = p.ringV + u * p.ringCap * D + gl * 8;

  for (int base = r0 + warp * STEP; base < r1; base += 8 * STEP) {
    uint4 kw[UNR], vw[UNR];
#pragma unroll
    for (int i = 0; i < UNR; ++i) {
      const int row = base + i * RPW + grp;
      if (row < r1 && row < n - 1) {
        const __half *kp, *vp;
        if (row < m) {
          kp = KhatU + (int64_t)row * D;
          vp = VhatU + (int64_t)row * D;
        } else {
          int slot = p.slot_b + (row - m);   // (the window is no longer than the ring)
          if (slot >= p.ringLen) slot -= p.ringLen;
          kp = ringKU + (int64_t)slot * D;
          vp = ringVU + (int64_t)slot * D;
        }
        kw[i] = ldg_stream(kp);
        vw[i] = ldg_stream(vp);
      } else if (row < r1) {   // the new token
        kw[i] = *reinterpret_cast<const uint4*>(&s_new[0][gl * 8]);
        vw[i] = *reinterpret_cast<const uint4*>(&s_new[1][gl * 8]);
      } else {
        kw[i] = make_uint4(0, 0, 0, 0);
        vw[i] = make_uint4(0, 0, 0, 0);
      }
    }
    float lg[NV];
#pragma unroll
    for (int i = 0; i < UNR; ++i) {
      float kf[8];
      unpack8(kw[i], kf);
#pragma unroll
      for (int g = 0; g < GQ; ++g) {
        float dot = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) dot = fmaf(qf[g][c], kf[c], dot);
        lg[g * UNR + i] = dot;
      }
    }
    lane_sums<NV, LPR / 2>(lg, gl);
    float tmax = -INFINITY;
#pragma unroll
    for (int k = 0; k < NVL; ++k) {
      const int row = base + (v0 + k) % UNR * RPW + grp;
      lg[k] = row < r1 ? lg[k] * (row < m ? scale_s : scale_b) : -INFINITY;
      tmax = fmaxf(tmax, lg[k]);
    }
    // maximum of the head over the rows of the step: the lanes of its other rows, the other row groups
#pragma unroll
    for (int o = LPV; o < LPV * UNR / NVL; o <<= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    // (a step has a valid row, so tmax is finite for every head)
    if (__any_sync(0xffffffffu, tmax > m_run)) {
      const float mnew = fmaxf(m_run, tmax);
      const float corr = exp2f(m_run - mnew);
      m_run = mnew;
      l_run *= corr;
#pragma unroll
      for (int g = 0; g < GQ; ++g) {
        const float cg = __shfl_sync(0xffffffffu, corr, g * UNR / NVL * LPV);
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[g][c] *= cg;
      }
    }
#pragma unroll
    for (int k = 0; k < NVL; ++k) {
      lg[k] = exp2f(lg[k] - m_run);   // 0 for invalid rows
      l_run += lg[k];
    }
#pragma unroll
    for (int i = 0; i < UNR; ++i) {
      float vf[8];
      unpack8(vw[i], vf);
#pragma unroll
      for (int g = 0; g < GQ; ++g) {
        const int idx = g * UNR + i;   // held by lane idx / NVL * LPV of the row group
        const float pr = __shfl_sync(0xffffffffu, lg[idx % NVL], grp * LPR + idx / NVL * LPV);
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[g][c] = fmaf(pr, vf[c], acc[g][c]);
      }
    }
  }
  // merge the row groups of the warp (all share m_run; l_run is per lane)
#pragma unroll
  for (int o = LPV; o < LPV * UNR / NVL; o <<= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, o);
#pragma unroll
  for (int o = 16; o >= LPR; o >>= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, o);
  if (grp == 0 && gl % (LPV * UNR / NVL) == 0) { s_m[warp][my_g] = m_run; s_l[warp][my_g] = l_run; }
#pragma unroll
  for (int g = 0; g < GQ; ++g) {
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[g][c] += __shfl_xor_sync(0xffffffffu, acc[g][c], o);
    if (grp == 0) {
#pragma unroll
      for (int c = 0; c < 8; ++c) s_acc[warp][g][gl * 8 + c] = acc[g][c];
    }
  }
  __syncthreads();
  for (int e = tid; e < GQ * D; e += 256) {
    const int g = e / D, x = e % D;
    float mx = -INFINITY;
#pragma unroll
    for (int w = 0; w < 8; ++w) mx = fmaxf(mx, s_m[w][g]);
    float l = 0.f, a = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const float f = (s_m[w][g] == -INFINITY) ? 0.f : exp2f(s_m[w][g] - mx);
      l += s_l[w][g] * f;
      a += s_acc[w][g][x] * f;
    }
    if (!MULTI && ns_all == 1) {
      p.out[(int64_t)(bh0 + g) * D + x] = __float2bfloat16_rn(a / l);
    } else {
      s_part[g][x] = a;
      if (x == 0) { s_part[g][D] = mx; s_part[g][D + 1] = l; }
    }
  }
  if (!MULTI && ns_all == 1) return;
  // the splits of these heads: every CTA of the cluster merges its share of the channels
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  cl.sync();
  const int rank = MULTI ? (int)cl.block_rank() : split, share = (GQ * D + p.nsplit - 1) / p.nsplit, e0 = rank * share;
  // several clusters: nsplit == 8, a share lies in one head
  float* part = p.part + ((int64_t)blockIdx.y * p.nsplit + rank) * p.nclus * (share + 2);
  for (int e = e0 + tid; e < min(GQ * D, e0 + share); e += 256) {
    const int g = e / D, x = e % D;
    const float* mine = &s_part[g][0];
    float mx = -INFINITY;
    for (int z = 0; z < p.nsplit; ++z) mx = fmaxf(mx, cl.map_shared_rank(mine, z)[D]);
    float l = 0.f, a = 0.f;
    for (int z = 0; z < p.nsplit; ++z) {
      const float* pz = cl.map_shared_rank(mine, z);
      const float ms = pz[D];
      const float f = (ms == -INFINITY) ? 0.f : exp2f(ms - mx);
      l += pz[D + 1] * f;
      a += pz[x] * f;
    }
    if (!MULTI) {
      p.out[(int64_t)(bh0 + g) * D + x] = __float2bfloat16_rn(a / l);
    } else {
      float* mine_out = part + split / p.nsplit * (share + 2);
      mine_out[e - e0] = a;
      if (e == e0) { mine_out[share] = mx; mine_out[share + 1] = l; }
    }
  }
  // (no CTA leaves while another still reads its shared memory)
  if constexpr (!MULTI) {
    cl.sync();
  } else {
    auto gone = cl.barrier_arrive();
    // the clusters of these heads: of the CTAs with the same share the one that arrives last merges it (nobody waits)
    __threadfence();
    __syncthreads();
    int32_t* ticket = p.ticket + (int64_t)blockIdx.y * p.nsplit + rank;
    if (tid == 0) s_last = atomicAdd(ticket, 1) == p.nclus - 1 ? 1 : 0;
    __syncthreads();
    if (s_last) {
      __threadfence();
      if (tid == 0) *ticket = 0;
      const float* all = part;
      // (s_acc is idle by now) weight of every cluster; then the partial sums of the thread groups
      float *s_w = &s_acc[0][0][0], *s_sum = s_w + 128;
      static_assert(8 * 64 >= 128 + 256, "scratch of the merge");
      if (warp == 0) {   // (at most 64 clusters: plan_decode)
        float ms[2], ls[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int z = lane + 32 * k;
          ms[k] = z < p.nclus ? __ldcg(all + z * (share + 2) + share) : -INFINITY;
          ls[k] = z < p.nclus ? __ldcg(all + z * (share + 2) + share + 1) : 0.f;
        }
        float mx = fmaxf(ms[0], ms[1]), l = 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float f = (ms[k] == -INFINITY) ? 0.f : exp2f(ms[k] - mx);
          s_w[lane + 32 * k] = f;
          l += ls[k] * f;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) s_w[64] = l;
      }
      __syncthreads();
      // a group of `share` threads takes every (256 / share)-th cluster, four loads in flight
      const int ng = 256 / share, grp_z = tid / share, ch = tid % share;
      float a = 0.f;
      for (int z0 = grp_z; z0 < p.nclus; z0 += 4 * ng) {
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = z0 + k * ng < p.nclus ? __ldcg(all + (z0 + k * ng) * (share + 2) + ch) : 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) a += v[k] * (z0 + k * ng < p.nclus ? s_w[z0 + k * ng] : 0.f);
      }
      s_sum[tid] = a;
      __syncthreads();
      if (tid < share) {
        a = 0.f;
        for (int k = 0; k < ng; ++k) a += s_sum[k * share + tid];
        p.out[(int64_t)bh0 * D + e0 + tid] = __float2bfloat16_rn(a / s_w[64]);
      }
    }
    cl.barrier_wait(std::move(gone));
  }
}

// A step over few rows (a warp has at most 8 * RPW of them): bound by latencies, so what does not depend on the kernel before it is
// done under that one's tail.  The rows are fetched before griddepcontrol.wait as far as they are known to be complete: a step
// that has waited for everything before it stores its number with release, a later one that reads it with acquire may read what
// was complete then - the state's rows and all window slots but those of the `back` steps in between, which follow
// behind the wait, under the latency of the new token's own loads.  (Numbers from before `base`, or not below this step's own - a
// replayed graph -, say nothing: then every row is fetched behind the wait.)  The splits of a head, a cluster, send each other
// their shares of the channels (st.async, bytes counted by the receiver): one exchange instead of two cluster barriers and
// a round of remote loads.  us per step in a graph, with the loop above
// and with this: 32 heads, 630 rows 6.3, 4.5; 890 rows 6.6, 5.1; 16 heads, 850 rows 6.2, 3.8; 32 on 8, 700 rows 6.9, 4.9; 8 heads, 90 rows 3.9, 3.1.
// ONE: no warp has more than one pass over rows (with the loop's bookkeeping 0.3 us longer).
template <int D, int GQ, bool LN, bool ONE>
__global__ void __launch_bounds__(256, 2) decode_short_kernel(const __grid_constant__ DecodeParams p) {
  constexpr int LPR = D / 8, RPW = 32 / LPR, UNR = 8;
  __shared__ float s_m[8][GQ], s_l[8][GQ];
  __shared__ __align__(16) float s_acc[8][GQ][D];
  __shared__ __align__(16) __half s_q[GQ][D], s_new[2][D];
  __shared__ float s_in[GQ * D + kDecodeCluster], s_in_ml[kDecodeCluster][GQ][2];   // what the splits send: [split][share], [split]
  __shared__ uint64_t s_bar;
  __shared__ uint32_t s_seen;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int split = blockIdx.x, ns = p.nsplit;
  const int bh0 = blockIdx.y * GQ;
  const int bb = bh0 / p.Hq, hq0 = bh0 % p.Hq, hk = hq0 / p.G;
  const int64_t u = (int64_t)bb * p.Hkv + hk;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = lane / LPR, gl = lane % LPR;
  const int m = p.m, n = p.n;
  const int share = (GQ * D + ns - 1) / ns, e0 = split * share, nmine = min(share, GQ * D - e0);
  if (tid == 0) {
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(s_seen) : "l"(p.seen) : "memory");
    tc::mbar_init(&s_bar, 1);
    tc::fence_barrier_init();
    if (ns > 1) tc::mbar_expect_tx(&s_bar, (uint32_t)(ns * 4 * (nmine + 2 * GQ)));
  }
  __syncthreads();
  if (ns > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");   // (this CTA is there, with its barrier)

  const uint32_t back = p.no - s_seen;
  const int safe = back - 1u < p.no - p.base ? max(m, n - 1 - (int)back) : 0;
  const int rw = (split * 8 + warp) * p.rpw, rend = min(n, rw + p.rpw);   // this warp's rows
  const __half* KhatU = p.Khat + u * p.Mcap * D + gl * 8;
  const __half* VhatU = p.Vhat + u * p.Mcap * D + gl * 8;
  const __half* ringKU = p.ringK + u * p.ringCap * D + gl * 8;
  const __half* ringVU = p.ringV + u * p.ringCap * D + gl * 8;
  uint4 kw[UNR], vw[UNR];
  auto fetch = [&](int r, int lo, int hi) {   // of the rows [r, r + UNR RPW) those in [lo, hi)
#pragma unroll
    for (int i = 0; i < UNR; ++i) {
      const int row = r + i * RPW + grp;
      if (row >= lo && row < hi) {
        const __half *kp, *vp;
        if (row < m) {
          kp = KhatU + (int64_t)row * D;
          vp = VhatU + (int64_t)row * D;
        } else {
          int slot = p.slot_b + (row - m);
          if (slot >= p.ringLen) slot -= p.ringLen;
          kp = ringKU + (int64_t)slot * D;
          vp = ringVU + (int64_t)slot * D;
        }
        kw[i] = ldg_stream(kp);
        vw[i] = ldg_stream(vp);
      }
    }
  };
#pragma unroll
  for (int i = 0; i < UNR; ++i) kw[i] = vw[i] = make_uint4(0, 0, 0, 0);
  const int known = min(rend, n - 1);   // (the new token's row is not in memory)
  fetch(rw, 0, min(known, safe));
  constexpr int NV = GQ * UNR;
  constexpr int NVL = NV > LPR ? NV / LPR : 1;
  constexpr int LPV = NV > LPR ? 1 : LPR / NV;
  const int v0 = gl / LPV * NVL;
  const int my_g = v0 / UNR;
  const float kLog2e = 1.4426950408889634f;
  const float scale_s = p.tau_s[hq0 + my_g] * rsqrtf((float)D) * kLog2e;
  const float scale_b = p.tau_b[hq0 + my_g] * rsqrtf((float)D) * kLog2e;
  const bool fresh = (n - 1) / (8 * p.rpw) == split;   // this CTA's rows end with the new token
  const bool store = fresh && hq0 % p.G == 0;
  auto behind_wait = [&] {
    if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p.seen), "r"(p.no) : "memory");
    if (safe < known) fetch(rw, safe, known);
  };
  if (LN) new_token_ln<D, GQ>(p, bh0, u, fresh, store, split == 0, s_q, s_new, behind_wait);
  else new_token<D, GQ>(p, bh0, u, fresh, store, split == 0, s_q, s_new, behind_wait);
  if (store && tid == 0) p.ringG[u * p.ringCap + p.slot_t] = p.gate ? p.gate[u] : 1.0f;
  __syncthreads();

  float m_run = -INFINITY, l_run = 0.f;   // of head my_g: maximum over the warp's rows, sum over this lane's
  float acc[GQ][8];
#pragma unroll
  for (int g = 0; g < GQ; ++g)
#pragma unroll
    for (int c = 0; c < 8; ++c) acc[g][c] = 0.f;
  for (int r = rw; ONE ? r == rw : r < rend; r += UNR * RPW) {
    if (!ONE && r > rw) fetch(r, 0, known);
    float lg[NV];
#pragma unroll
    for (int i = 0; i < UNR; ++i) {
      if (r + i * RPW + grp == n - 1 && rend == n) {   // (the last rows of a warp may be the next one's)
        kw[i] = *reinterpret_cast<const uint4*>(&s_new[0][gl * 8]);
        vw[i] = *reinterpret_cast<const uint4*>(&s_new[1][gl * 8]);
      }
      float kf[8];
      unpack8(kw[i], kf);
#pragma unroll
      for (int g = 0; g < GQ; ++g) {
        float qf[8];
        unpack8(*reinterpret_cast<const uint4*>(&s_q[g][gl * 8]), qf);
        float dot = 0.f;
#pragma unroll
        for (int c = 0; c < 8; ++c) dot = fmaf(qf[c], kf[c], dot);
        lg[g * UNR + i] = dot;
      }
    }
    lane_sums<NV, LPR / 2>(lg, gl);
    float tmax = -INFINITY;
#pragma unroll
    for (int k = 0; k < NVL; ++k) {
      const int row = r + (v0 + k) % UNR * RPW + grp;
      lg[k] = row < rend ? lg[k] * (row < m ? scale_s : scale_b) : -INFINITY;
      tmax = fmaxf(tmax, lg[k]);
    }
#pragma unroll
    for (int o = LPV; o < LPV * UNR / NVL; o <<= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    const float mnew = fmaxf(m_run, tmax);   // (finite, but where a single pass meets no row)
    if (!ONE && r > rw) {
      const float corr = exp2f(m_run - mnew);
      l_run *= corr;
#pragma unroll
      for (int g = 0; g < GQ; ++g) {
        const float cg = __shfl_sync(0xffffffffu, corr, g * UNR / NVL * LPV);
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[g][c] *= cg;
      }
    }
    m_run = mnew;
#pragma unroll
    for (int k = 0; k < NVL; ++k) {
      lg[k] = ONE && lg[k] == -INFINITY ? 0.f : exp2f(lg[k] - m_run);   // 0 for invalid rows
      l_run += lg[k];
    }
#pragma unroll
    for (int i = 0; i < UNR; ++i) {
      float vf[8];
      unpack8(vw[i], vf);
#pragma unroll
      for (int g = 0; g < GQ; ++g) {
        const int idx = g * UNR + i;
        const float pr = __shfl_sync(0xffffffffu, lg[idx % NVL], grp * LPR + idx / NVL * LPV);
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[g][c] = fmaf(pr, vf[c], acc[g][c]);
      }
    }
  }
#pragma unroll
  for (int o = LPV; o < LPV * UNR / NVL; o <<= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, o);
#pragma unroll
  for (int o = 16; o >= LPR; o >>= 1) l_run += __shfl_xor_sync(0xffffffffu, l_run, o);
  if (grp == 0 && gl % (LPV * UNR / NVL) == 0) { s_m[warp][my_g] = m_run; s_l[warp][my_g] = l_run; }
#pragma unroll
  for (int g = 0; g < GQ; ++g) {
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[g][c] += __shfl_xor_sync(0xffffffffu, acc[g][c], o);
    if (grp == 0) {
#pragma unroll
      for (int c = 0; c < 8; c += 4)
        *reinterpret_cast<float4*>(&s_acc[warp][g][gl * 8 + c]) = make_float4(acc[g][c], acc[g][c + 1], acc[g][c + 2], acc[g][c + 3]);
    }
  }
  __syncthreads();
  if (ns > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // (every CTA of the cluster is there)
  for (int e = tid; e < GQ * D; e += 256) {
    const int g = e / D, x = e % D;
    float mx = -INFINITY;
#pragma unroll
    for (int w = 0; w < 8; ++w) mx = fmaxf(mx, s_m[w][g]);
    float l = 0.f, a = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      const float f = s_m[w][g] == -INFINITY ? 0.f : exp2f(s_m[w][g] - mx);
      l += s_l[w][g] * f;
      a += s_acc[w][g][x] * f;
    }
    if (ns == 1) {
      p.out[(int64_t)(bh0 + g) * D + x] = __float2bfloat16_rn(a / l);
      continue;
    }
    auto send = [&](float* at, int r, float v) {
      asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
                   ::"r"(tc::cluster_addr(at, r)), "r"(__float_as_uint(v)), "r"(tc::cluster_addr(&s_bar, r)) : "memory");
    };
    send(&s_in[split * share + e % share], e / share, a);
    if (x < ns) { send(&s_in_ml[split][g][0], x, mx); send(&s_in_ml[split][g][1], x, l); }
  }
  if (ns == 1) return;
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  if (tc::mbar_wait_cluster(&s_bar, 0)) {
    for (int e = tid; e < nmine; e += 256) {
      const int g = (e0 + e) / D;
      float mx = -INFINITY;
      for (int z = 0; z < ns; ++z) mx = fmaxf(mx, s_in_ml[z][g][0]);
      float l = 0.f, a = 0.f;
      for (int z = 0; z < ns; ++z) {
        const float ms = s_in_ml[z][g][0], f = ms == -INFINITY ? 0.f : exp2f(ms - mx);
        l += s_in_ml[z][g][1] * f;
        a += s_in[z * share + e] * f;
      }
      p.out[(int64_t)bh0 * D + e0 + e] = __float2bfloat16_rn(a / l);
    }
  } else {
    atomicExch(p.status, (int)KVM_ERR_TIMEOUT);
  }
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // (nobody leaves while another may still send to it)
}

template <int D, int GQ, bool LN, bool ONE>
static bool launch_decode_short(const DecodeParams& p, int ncta, bool early, cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(p.nsplit, ncta); lc.blockDim = dim3(256); lc.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = p.nsplit; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  lc.attrs = at; lc.numAttrs = p.nsplit > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&lc, decode_short_kernel<D, GQ, LN, ONE>, p) == cudaSuccess;
}

template <int D, int GQ, bool LN, bool MULTI>
static bool launch_decode_step(const DecodeParams& p, int ncta, bool early, cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(p.nsplit * p.nclus, ncta); lc.blockDim = dim3(256); lc.stream = s;
  cudaLaunchAttribute at[2];
  // the set-up of this step (launch, the rotation's angles) runs under the tail of the kernel before it on the stream
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = p.nsplit; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  lc.attrs = at; lc.numAttrs = p.nsplit > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&lc, decode_step_kernel<D, GQ, LN, MULTI>, p) == cudaSuccess;
}

// CTAs per cluster of decode_short_kernel for a step over n rows, 0 where decode_step_kernel is the better one.  Measured: us per step,
// the loop and this, steps of a block in a graph (launched one by one the host is the longer side up to 5.8 us).
// kFit: clusters of 1 to 8 CTAs up to which this is the faster one; the GPU holds 296, 148, 93, 71, 56, 45, 37, 33 at two CTAs per SM, and
// the last ones cost what the early loads save (single heads, 630 rows in 5 splits: 52 6.59, 5.77; 53 6.60, 6.08; 55 6.61, 6.88; 56
// 6.60, 7.35; 890 rows in 7: 36 6.68, 6.20; 37 6.67, 6.79; 1020 in 8: 32 6.84, 5.90; 33 6.85, 7.15; 296 in one 5.57, 4.62; 148 in two
// 6.82, 6.12; 71 in four 6.37, 5.76).  Two heads per CTA, where the loop has no more of 128 channels: 52 in 5 6.88, 7.06; 36 in 7 7.55,
// 8.12; 32 in 8 6.91, 7.23; 30 6.67, 6.07.
// The fewest splits whose warps have all their rows in flight at once, one pass; 8 for 8 to 16 groups of heads, where two steps
// fit beside each other, from the rows on that pay for the exchange (16 heads, 40 rows in one split and in 8: 2.90, 3.55; 90 rows 3.17,
// 3.55; 240 rows in two 3.88, 3.60; 700 rows in 6 3.97, 3.74; 12 pairs, 60 rows in one 3.3, 4.7; 200 in two 4.2, 4.7).
// Two passes of 8 splits (8 heads, 1300 rows 6.21, 5.00; 32 heads 8.04, 7.33; three: 8 heads, 2400 rows 8.2, 8.8) up to 32 single heads
// (1800 rows 9.14, 8.48; 33 9.11, 9.13; 1950 rows, where the loop's last pass is nearly full, 16 heads 7.21, 7.44, 32 9.06, 9.33) and 20
// pairs (1600 rows 8.93, 8.11; 24 at 1500 7.53, 8.06), but for pairs over 10.5 to 12 passes, the end of the loop's third (20 pairs, 1300
// rows 8.07, 7.67; 1400 7.37, 7.66; 1500 7.56, 7.99).  Where the loop takes four or eight heads per CTA two are better all along: 32 on 8, 900 rows 6.2,
// 5.4; 64 on 8, 2000 rows 10.97, 9.31.
DecodeShortPlan plan_decode_short(int nQ, int G, int d, int64_t n) {
  static const int kFit[2][kDecodeCluster] = {{296, 148, 88, 71, 53, 45, 36, 32}, {296, 148, 88, 71, 51, 45, 35, 30}};
  const int heads = G % 2 == 0 ? 2 : 1, groups = nQ / heads;
  const bool same = G % 4 != 0;             // the loop has as many heads per CTA
  const int rows1 = 256 / d;                // rows that a warp loads at once
  const int64_t pass = 8 * 8 * rows1;       // rows of a CTA in one pass
  int64_t ns = (n + pass - 1) / pass;
  if (ns > 2 * kDecodeCluster) return {0, 0, 0};
  if (ns > kDecodeCluster) {
    if (same && (heads == 1 ? groups > 32 : groups > 20 || (2 * n > 21 * pass && ns <= 12))) return {0, 0, 0};
    ns = kDecodeCluster;
  } else if (groups >= 8 && groups <= 16 && ns >= 2 * heads) {
    ns = kDecodeCluster;
  }
  if (groups > kFit[heads == 2 && same && d == 128][ns - 1]) return {0, 0, 0};
  return {heads, (int)ns, (int)(((n + 8 * ns - 1) / (8 * ns) + rows1 - 1) / rows1 * rows1)};
}

// How a step over n rows is cut.  Query heads per CTA (they share a kv head): the largest of 8, 4, 2, 1 that divides the group
// size, but four of eight while all splits of four fit at once, two CTAs per SM: the rows are fetched twice, mostly from L2, by
// twice the warps (us per step of 8 and 4: 64 heads on 8, 900 rows 10.0, 8.7; 16600 rows 69, 41 in two clusters; 96 on 12, 2400
// rows 15.6, 14.2; 50000 rows 197, 179; 128 on 16 - 16 clusters of eight CTAs do not fit at one per SM - 900 rows 19, 10).
DecodePlan plan_decode(int nQ, int G, int d, int64_t n) {
  int heads = (G % 8 == 0) ? 8 : (G % 4 == 0) ? 4 : (G % 2 == 0) ? 2 : 1;
  if (heads == 8 && nQ / 4 <= 33) heads = 4;
  DecodePlan pl;
  pl.heads = heads;
  pl.splits = pl.clusters = 1;
  // Row splits, up to the portable cluster size (clusters of 16 took 13.5 us per step where 8 take 8.5): waves of clusters
  // times the length of a CTA, its set-up and merge counted as 300 rows.  kFit: clusters of 1 to 8 CTAs that the GPU holds at
  // once at 1, 2, 3 CTAs per SM (cudaOccupancyMaxActiveClusters; a cluster lies in one group of SMs, and one too many is another
  // wave: 136 heads on 17, 900 rows, clusters of 8: 18.6 us, of 6: 12).  By registers 3, 2, 2, 1 CTAs of 1, 2, 4, 8 heads fit an SM.
  // This picks the fastest of 1, 2, 3, 4, 6, 8 splits, or one within 2 % of it, in all of 15 measured shapes (64 to 768 heads,
  // 900 to 2400 rows; e.g. us per step of 256 heads over 2430 rows: 59, 68, 55, 61, 64, 70; of 512 heads: 123, 109, 106, 108,
  // 123, 131).  (The fewest of equal counts.)
  static const int kFit[3][kDecodeCluster] = {{148, 74, 45, 33, 26, 22, 15, 15}, {296, 148, 93, 71, 56, 45, 37, 33}, {444, 222, 142, 104, 82, 71, 56, 48}};
  const int* fit = kFit[heads == 1 ? 2 : heads == 8 ? 0 : 1];
  const int64_t ncta = nQ / heads, rows1 = 8 * 4 * (256 / d);
  auto rows_of = [&](int64_t ns) { return ((n + ns - 1) / ns + rows1 - 1) / rows1 * rows1; };
  int64_t t = INT64_MAX;
  for (int ns = 1; ns <= kDecodeCluster; ++ns) {
    const int64_t tn = (ncta + fit[ns - 1] - 1) / fit[ns - 1] * (rows_of(ns) + 300);
    if (tn < t) { t = tn; pl.splits = ns; }
  }
  // Few heads over many rows: several clusters of eight per group of heads, while all of them fit at once (another wave costs
  // what the shorter CTAs save), merged through global memory by the CTAs that arrive last.  That takes 1.5 us and 5 to 9 ns per CTA longer, where a CTA takes 80 (1, 2 heads)
  // or 45 rows of 128 channels per us.  Measured, us per step, one cluster and as chosen: 1 head of 128 channels over 2300
  // rows 7.5, 6.7; 6400 rows 13.3, 7.9; 131072 rows 281, 19; 8 heads on one, 50000 rows 171, 21; 8 on 8,
  // 16600 rows 41, 19; 32 on 8, 50000 rows 158, 61; 16 on 16, 50000 rows 127, 67.  Left in one cluster: 32 on 8, 1300 rows 8.8
  // (10.2 with three); 2 x 8 heads of 64 channels, 4400 rows 9.4 (10.2).  A twentieth has to be gained: 32 on 8 over 1870
  // rows 10.6, 11.9 with four.
  t -= t / 20;
  for (int64_t nc = 2; ncta * nc <= fit[kDecodeCluster - 1]; ++nc) {
    const int64_t merge = ((heads <= 2 ? 120 : 70) + 2 * kDecodeCluster * ncta * nc / 5) * 128 / d;
    const int64_t tn = rows_of(kDecodeCluster * nc) + 300 + merge;
    if (tn < t) { t = tn; pl.splits = kDecodeCluster; pl.clusters = (int)nc; }
  }
  return pl;
}

#define KVM_DEC_EACH(F, L) \
  F(128, 8, L, false) F(128, 4, L, false) F(128, 2, L, false) F(128, 1, L, false) F(64, 8, L, false) F(64, 4, L, false) F(64, 2, L, false) F(64, 1, L, false) \
  F(128, 4, L, true) F(128, 2, L, true) F(128, 1, L, true) F(64, 4, L, true) F(64, 2, L, true) F(64, 1, L, true)

int launch_decode(State* st, const DecodeArgs& a, cudaStream_t s) {
  const int nQ = st->B * st->Hq;
  DecodeParams p;
  p.q = a.q; p.k = a.k; p.v = a.v; p.gate = a.gate; p.inv_freq = st->inv_freq;
  p.lnq_w = st->lnq_w; p.lnq_b = st->lnq_b; p.lnk_w = st->lnk_w; p.lnk_b = st->lnk_b; p.qk_ln_eps = st->qk_ln_eps;
  p.Khat = st->KhatBuf[st->nfolds & 1]; p.Vhat = st->VhatBuf[st->nfolds & 1];
  p.ringK = st->ringK; p.ringV = st->ringV; p.ringG = st->ringG;
  p.tau_s = st->tau_s; p.tau_b = st->tau_b; p.out = a.out; p.sat_counter = st->status + 4;
  p.Mcap = st->Mcap; p.ringCap = (int64_t)st->w * st->Cmax; p.t = a.t;
  p.m = (int)a.m; p.n = (int)(a.m + (a.t - a.b + 1));
  p.ringLen = (int)st->ringLen; p.slot_b = (int)(a.b % st->ringLen); p.slot_t = (int)(a.t % st->ringLen);
  p.Hq = st->Hq; p.Hkv = st->Hkv; p.G = st->G; p.r = st->r;
  p.part = st->decPart; p.ticket = st->decTicket;
  const bool early = st->prof_hook == nullptr;
  p.seen = st->decSeen; p.no = st->decNo++; p.base = early ? st->decBase : p.no; p.status = st->status;   // (with the timing hook on nothing overlaps)
  const DecodeShortPlan sp = plan_decode_short(nQ, st->G, st->d, p.n);
  if (sp.splits > 0) {
    p.nsplit = sp.splits; p.nclus = 1; p.rpw = sp.rows_per_warp;
#define KVM_DEC_SHORT(DD, GG, LL)                                                                \
  if (st->d == DD && sp.heads == GG && st->fusedLn == LL) {                                       \
    if (p.rpw <= 8 * (256 / DD)) launch_decode_short<DD, GG, LL, true>(p, nQ / GG, early, s);     \
    else launch_decode_short<DD, GG, LL, false>(p, nQ / GG, early, s);                            \
  }
    KVM_DEC_SHORT(128, 1, false) KVM_DEC_SHORT(128, 2, false) KVM_DEC_SHORT(64, 1, false) KVM_DEC_SHORT(64, 2, false)
    KVM_DEC_SHORT(128, 1, true) KVM_DEC_SHORT(128, 2, true) KVM_DEC_SHORT(64, 1, true) KVM_DEC_SHORT(64, 2, true)
#undef KVM_DEC_SHORT
    return 1;
  }
  const DecodePlan pl = plan_decode(nQ, st->G, st->d, p.n);
  const int GQ = pl.heads;
  p.nsplit = pl.splits; p.nclus = pl.clusters;
#define KVM_DEC_GO(DD, GG, LL, MM) \
  if (st->d == DD && GQ == GG && st->fusedLn == LL && (pl.clusters > 1) == MM) launch_decode_step<DD, GG, LL, MM>(p, nQ / GQ, early, s);
  KVM_DEC_EACH(KVM_DEC_GO, true)
  KVM_DEC_EACH(KVM_DEC_GO, false)
#undef KVM_DEC_GO
  return 1;
}

}  // namespace kvm
