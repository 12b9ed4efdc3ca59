// Single-token decode (Table 1 "Decode time per token"): one query per head attends over the
// m readout rows of the state plus the window tokens [b, t].  ONE kernel per step: every CTA rotates
// the query heads it serves (and, where its rows end with the new token, that token's key), streams
// its share of the rows with 16-byte loads into an online softmax, and the row splits of a head - a
// thread-block cluster - merge their partial results through distributed shared memory.
// What bounds it: with many heads HBM (K_hat, V_hat and the window are read once); with few the
// latency of launch, first loads and merge, and on the host the launch itself, which is why the rotation of the
// token and the merge are not kernels of their own: 32 heads over 256 + window rows took 1.9 + 7.4 + 3.1 us
// in three kernels and 18.5 us per step on the host's side; now 9.5 us per step.  64 x 32 heads over 4096 + window
// rows: 763 -> 716 us per step (6.57 TB/s), the set-up of a step under the tail of the one before.
#include <cooperative_groups.h>

#include "kvm_internal.h"
#include "ln_rows.cuh"

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
template <int D, int GQ>
__device__ __forceinline__ void new_token(const DecodeParams& p, int bh0, int64_t u, bool fresh, bool store, bool count_q,
                                          __half (*s_q)[D], __half (*s_new)[D]) {
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
template <int D, int GQ>
__device__ __forceinline__ void new_token_ln(const DecodeParams& p, int bh0, int64_t u, bool fresh, bool store, bool count_q,
                                             __half (*s_q)[D], __half (*s_new)[D]) {
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

// grid (nsplit, B*Hq / GQ), the nsplit CTAs of a row a cluster; block 256 = 8 warps.  LPR = D/8 lanes cover one
// row with 16-byte loads, a warp covers RPW = 32/LPR rows per load instruction and UNR such instructions per
// step.  A CTA serves GQ query heads that share one kv head (grouped queries): every key / value row is loaded
// once and meets all GQ queries, so the bytes streamed per step do not grow with the group size.
template <int D, int GQ, bool LN>
__global__ void __launch_bounds__(256) decode_step_kernel(DecodeParams p) {
  constexpr int LPR = D / 8;
  constexpr int RPW = 32 / LPR;
  constexpr int UNR = 4;
  constexpr int STEP = RPW * UNR;       // rows per warp per iteration
  __shared__ float s_m[8][GQ], s_l[8][GQ];
  __shared__ __align__(16) float s_acc[8][GQ][D];
  __shared__ float s_part[GQ][D + 2];   // this split's merged result: channels, maximum, sum
  __shared__ __align__(16) __half s_q[GQ][D], s_new[2][D];

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int split = blockIdx.x;
  const int bh0 = blockIdx.y * GQ;                 // first query head of this CTA (GQ divides the group size G)
  const int bb = bh0 / p.Hq, hq0 = bh0 % p.Hq, hk = hq0 / p.G;
  const int64_t u = (int64_t)bb * p.Hkv + hk;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = lane / LPR, gl = lane % LPR;   // row group inside the warp, lane inside the row

  const int m = p.m, n = p.n;
  int per = (n + p.nsplit - 1) / p.nsplit;
  per = (per + 8 * STEP - 1) / (8 * STEP) * (8 * STEP);
  const int r0 = split * per;
  const int r1 = min(n, r0 + per);
  const bool fresh = r0 < n && r1 == n;          // this CTA's rows end with the new token

  if (LN) new_token_ln<D, GQ>(p, bh0, u, fresh, fresh && hq0 % p.G == 0, split == 0, s_q, s_new);
  else new_token<D, GQ>(p, bh0, u, fresh, fresh && hq0 % p.G == 0, split == 0, s_q, s_new);
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
    if (p.nsplit == 1) {
      p.out[(int64_t)(bh0 + g) * D + x] = __float2bfloat16_rn(a / l);
    } else {
      s_part[g][x] = a;
      if (x == 0) { s_part[g][D] = mx; s_part[g][D + 1] = l; }
    }
  }
  if (p.nsplit == 1) return;
  // the splits of these heads: every CTA of the cluster merges its share of the channels
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  cl.sync();
  const int share = (GQ * D + p.nsplit - 1) / p.nsplit;
  for (int e = split * share + tid; e < min(GQ * D, (split + 1) * share); e += 256) {
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
    p.out[(int64_t)(bh0 + g) * D + x] = __float2bfloat16_rn(a / l);
  }
  cl.sync();   // (no CTA leaves while another still reads its shared memory)
}

template <int D, int GQ, bool LN>
static bool launch_decode_step(const DecodeParams& p, int ncta, bool early, cudaStream_t s) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(p.nsplit, ncta); lc.blockDim = dim3(256); lc.stream = s;
  cudaLaunchAttribute at[2];
  // the set-up of this step (launch, the rotation's angles) runs under the tail of the kernel before it on the stream
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = p.nsplit; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  lc.attrs = at; lc.numAttrs = p.nsplit > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&lc, decode_step_kernel<D, GQ, LN>, p) == cudaSuccess;
}

// query heads of one kv group share a CTA: the largest of 8, 4, 2, 1 that divides the group size
static int decode_heads_per_cta(const State* st) { return (st->G % 8 == 0) ? 8 : (st->G % 4 == 0) ? 4 : (st->G % 2 == 0) ? 2 : 1; }

#define KVM_DEC_EACH(F)                                                                                                 \
  F(128, 8, true) F(128, 4, true) F(128, 2, true) F(128, 1, true) F(64, 8, true) F(64, 4, true) F(64, 2, true) F(64, 1, true) \
  F(128, 8, false) F(128, 4, false) F(128, 2, false) F(128, 1, false) F(64, 8, false) F(64, 4, false) F(64, 2, false) F(64, 1, false)

int launch_decode(State* st, const DecodeArgs& a, cudaStream_t s) {
  const int nQ = st->B * st->Hq, GQ = decode_heads_per_cta(st);
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
  // Row splits, up to the portable cluster size (clusters of 16 took 13.5 us per step where 8 take 8.5): waves of CTAs
  // times the length of a CTA, its set-up and merge counted as 300 rows.  `slots` = CTAs that fit the GPU at once (3, 2,
  // 2, 1 per SM by registers for 1, 2, 4, 8 heads).  This picks the fastest of 1, 2, 3, 4, 6, 8 splits, or one within 2 %
  // of it, in all of 15 measured shapes (64 to 768 heads, 900 to 2400 rows; e.g. us per step of 256 heads over 2430
  // rows: 59, 68, 55, 61, 64, 70; of 512 heads: 123, 109, 106, 108, 123, 131).
  const int nCta = nQ / GQ, rows1 = 8 * 4 * (256 / st->d), slots = 148 * (GQ == 1 ? 3 : GQ == 8 ? 1 : 2);
  int nsplit = 1;
  int64_t least = INT64_MAX;
  for (int ns = 1; ns <= 8; ++ns) {
    const int64_t rows = ((p.n + ns - 1) / ns + rows1 - 1) / rows1 * rows1;
    const int64_t t = ((int64_t)nCta * ns + slots - 1) / slots * (rows + 300);
    if (t < least) { least = t; nsplit = ns; }
  }
  p.nsplit = nsplit;
  const bool early = st->prof_hook == nullptr;
#define KVM_DEC_GO(DD, GG, LL) \
  if (st->d == DD && GQ == GG && st->fusedLn == LL) launch_decode_step<DD, GG, LL>(p, nCta, early, s);
  KVM_DEC_EACH(KVM_DEC_GO)
#undef KVM_DEC_GO
  return 1;
}

}  // namespace kvm
