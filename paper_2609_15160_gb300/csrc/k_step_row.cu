// The shared block of a decode step for small float32 models, one CTA per row (Eq. 6-11).
//
// The rows of a step are independent between the router and the LM head, and the block of a small model is a few
// hundred kilobytes: as launches of their own its stages (norm, QKV, rotary and append, attention, O, norm, gate/up,
// SwiGLU, down per loop and layer) were all launch latency, 112 us a step for four loops of one layer of width 64; as one
// launch the step is 62 us (host, router, plan and LM head included). Here a CTA takes its row through every loop the row
// runs, with the residual and every activation in shared memory and only block barriers between stages, so an exited row
// costs nothing and no stage of another row is waited for. Weights that fit are staged in shared memory by bulk copies
// while the router and the plan run; larger ones, and K and V, are read through L2, which pays as long as they cross one
// SM's port in less time than the launches take (step_path in tlf_api.cu).
//
// A projection gives each output to a group of lanes (16 for a reduction of up to 64, else a warp), float4 loads and a
// shuffle reduction; the pre-norm's factor is applied to the sum. Attention: a thread per (head, key) for the scores, a
// warp per head for the softmax, and a thread per (key split, head, element) for the values.
#include "tlf_internal.cuh"

namespace tlf {

constexpr int SR_THREADS = 512;
constexpr int SR_SMEM = 232448 - 2560;  // less the static shared memory
constexpr int SR_VAHEAD = 8;            // values a thread loads ahead of the softmax

// Shared memory: activations, then (if they fit) the weights of all layers.
struct SrLayout {
  int scores, total_act, weights;  // floats
};
static __host__ __device__ int sr_outputs(const ModelDims& md) {
  const int n = md.qkv_dim > 2 * md.ff ? md.qkv_dim : 2 * md.ff;
  return n > md.d ? n : md.d;
}
static __host__ __device__ SrLayout sr_layout(const ModelDims& md) {
  SrLayout l;
  // h, a projection's outputs, o, u; partial value sums; score rows
  const int part = SR_THREADS > md.q_dim ? SR_THREADS : md.q_dim;
  l.scores = (md.d + sr_outputs(md) + md.q_dim + md.ff + part + md.Hq + 3) / 4 * 4;
  l.total_act = l.scores + md.Hq * RowStep::MAX_KEYS;
  l.weights = md.J * (md.qkv_dim * md.d + md.d * md.q_dim + 3 * md.ff * md.d + 2 * md.d);  // matrices, norm gains
  return l;
}

// y[o] = dot(W[o], x) for o < N, W row-major with K columns (a multiple of 4), x and y in shared memory; ends with the
// block's barrier. One copy of the code serves every projection: a launch runs it a few times only, so its size is its
// time (inlined per projection, gate/up alone waited 4 us for its instructions).
__device__ __noinline__ void sr_gemv(const float* W, int N, int K, const float* x, float* y) {
  const int lg = K <= 64 ? 16 : 32;  // lanes per output
  const int grp = threadIdx.x / lg, l = threadIdx.x % lg, ngrp = SR_THREADS / lg, gw = grp % (32 / lg), k4 = K / 4;
  for (int ob = grp - gw; ob < N; ob += 4 * ngrp) {  // (the groups of a warp run the same trips: warp-wide shuffles)
    const int o0 = ob + gw;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int c = l; c < k4; c += lg) {
      const float4 v = reinterpret_cast<const float4*>(x)[c];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (o0 + q * ngrp < N) {
          const float4 w = reinterpret_cast<const float4*>(W + (size_t)(o0 + q * ngrp) * K)[c];
          acc[q] = fmaf(w.x, v.x, fmaf(w.y, v.y, fmaf(w.z, v.z, fmaf(w.w, v.w, acc[q]))));
        }
    }
#pragma unroll 1
    for (int o = lg / 2; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    // lane q of the group keeps output q
    float v = acc[0];
    v = l == 1 ? acc[1] : v;
    v = l == 2 ? acc[2] : v;
    v = l == 3 ? acc[3] : v;
    if (l < 4 && o0 + l * ngrp < N) y[o0 + l * ngrp] = v;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(SR_THREADS, 1) k_step_row(RowStep a) {
  extern __shared__ __align__(16) float smf[];
  __shared__ __align__(8) uint64_t wbar;
  // of every loop the row runs, read in one go: pages of its cache, page / slot / position of the new entry, keys
  __shared__ int pages_s[16][RowStep::MAX_KEYS / 64];
  __shared__ int4 info_s[16];
  __shared__ int keys_s[16];
  __shared__ float2 cs_s[64];  // rotary factors of the row's position
  const ModelDims& md = a.md;
  const StepDev& s = a.s;
  const int d = md.d, hd = md.hd, q_dim = md.q_dim, qkv_dim = md.qkv_dim, ff = md.ff, M = md.M, J = md.J, Hq = md.Hq;
  const int G = Hq / md.Hkv, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SrLayout lay = sr_layout(md);
  float* h = smf;                 // [d] residual stream of the row
  float* y = h + d;               // a projection's outputs; QKV's become the rotated q (scaled)
  float* o = y + sr_outputs(md);  // [q_dim] attention output
  float* u = o + q_dim;           // [ff]
  float* part = u + ff;           // partial value sums
  float* lsum = part + (SR_THREADS > q_dim ? SR_THREADS : q_dim);  // [Hq] softmax sums
  float* sc = smf + lay.scores;   // [Hq][MAX_KEYS]
  float* wsm = smf + lay.total_act;
  const size_t per_layer = (size_t)lay.weights / J;
  const size_t nq = (size_t)qkv_dim * d, no = (size_t)d * q_dim, ng = (size_t)2 * ff * d, nd = (size_t)d * ff;
  if (a.weights_in_smem) {
    if (tid == 0) {
      mbar_init(smem_u32(&wbar), 1);
      fence_barrier_init();
      mbar_arrive_expect_tx(smem_u32(&wbar), (uint32_t)(lay.weights * 4));
      for (int j = 0; j < J; ++j) {
        float* w = wsm + per_layer * j;
        bulk_g2s(smem_u32(w), a.layer[j].wqkv, (uint32_t)(nq * 4), smem_u32(&wbar));
        bulk_g2s(smem_u32(w + nq), a.layer[j].wo, (uint32_t)(no * 4), smem_u32(&wbar));
        bulk_g2s(smem_u32(w + nq + no), a.layer[j].wgu, (uint32_t)(ng * 4), smem_u32(&wbar));
        bulk_g2s(smem_u32(w + nq + no + ng), a.layer[j].wd, (uint32_t)(nd * 4), smem_u32(&wbar));
        bulk_g2s(smem_u32(w + nq + no + ng + nd), a.layer[j].attn_norm, (uint32_t)(d * 4), smem_u32(&wbar));
        bulk_g2s(smem_u32(w + nq + no + ng + nd + d), a.layer[j].mlp_norm, (uint32_t)(d * 4), smem_u32(&wbar));
      }
    }
  }
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x;
  const int m = min(s.m[b], M), slot = s.slots[b];
  if (tid < d) h[tid] = s.H[(size_t)b * d + tid];
  const float fgain = tid < d ? a.final_norm[tid] : 0.f;
  if (tid < m) {
    const int k = s.col[tid * md.max_batch + b];  // the row's place in A_r
    info_s[tid] = s.rowinfo[tid * md.max_batch + k];
    keys_s[tid] = min(s.nch[tid * md.max_batch + k], RowStep::MAX_KEYS);
  }
  for (int i = tid; i < m * (RowStep::MAX_KEYS / 64); i += SR_THREADS) {
    const int r = i / (RowStep::MAX_KEYS / 64), p = i % (RowStep::MAX_KEYS / 64);
    pages_s[r][p] = p < md.max_pages ? s.page_table[((size_t)slot * M + r) * md.max_pages + p] : -1;
  }
  __syncthreads();
  if (tid < hd / 2) cs_s[tid] = a.rope[(size_t)info_s[0].z * (hd / 2) + tid];  // one position in every loop
  for (int i = tid; i < m * (RowStep::MAX_KEYS / 64); i += SR_THREADS) {
    const int r = i / (RowStep::MAX_KEYS / 64), p = i % (RowStep::MAX_KEYS / 64);
    if (p * 64 < keys_s[r] && (pages_s[r][p] < 0 || pages_s[r][p] >= md.n_pages)) {
      atomicOr(s.err, DEVERR_INDEX);
      pages_s[r][p] = 0;
    }
  }
  __syncthreads();
  if (a.weights_in_smem && !mbar_wait(smem_u32(&wbar), 0, s.err)) drain_copies();

  // every warp takes the row's RMSNorm factor for itself
  auto norm_factor = [&]() {
    float t = 0.f;
    for (int i = lane; i < d; i += 32) t = fmaf(h[i], h[i], t);
    return rsqrtf(warp_sum(t) / (float)d + md.eps);
  };
  const float qscale = 1.4426950408889634f * rsqrtf((float)hd);
  const int combos = M * (M + 1) / 2, half = hd / 2;

  for (int r = 0; r < m; ++r) {
    const int4 ri = info_s[r];
    const int L = keys_s[r];
    const int* pages = pages_s[r];
    // conditioning vector `p` of layer j for the row's (depth, loop)
    auto cvec = [&](int j, int p) { return a.cond + ((size_t)(j * combos + m * (m - 1) / 2 + r) * 4 + p) * d; };
    for (int j = 0; j < J; ++j) {
      const float* wq = a.weights_in_smem ? wsm + per_layer * j : a.layer[j].wqkv;
      const float* wo = a.weights_in_smem ? wsm + per_layer * j + nq : a.layer[j].wo;
      const float* wg = a.weights_in_smem ? wsm + per_layer * j + nq + no : a.layer[j].wgu;
      const float* wd = a.weights_in_smem ? wsm + per_layer * j + nq + no + ng : a.layer[j].wd;
      const float* ga = a.weights_in_smem ? wsm + per_layer * j + nq + no + ng + nd : a.layer[j].attn_norm;
      const float* gm = a.weights_in_smem ? wsm + per_layer * j + nq + no + ng + nd + d : a.layer[j].mlp_norm;
      // a pre-norm operand: h * gain (* (1 + gamma)) into `part`, the factor applied to the sums
      auto operand = [&](const float* gain, int p) {
        for (int i = tid; i < d; i += SR_THREADS) part[i] = h[i] * gain[i] * (a.cond ? 1.f + cvec(j, p)[i] : 1.f);
        __syncthreads();
      };
      // ---- QKV, rotary, append ----
      operand(ga, 2);
      float inv = norm_factor();
      sr_gemv(wq, qkv_dim, d, part, y);
      float* pool = reinterpret_cast<float*>(s.pool);
      for (int t = tid; t < (Hq + md.Hkv) * half + md.Hkv * hd; t += SR_THREADS) {
        if (t < (Hq + md.Hkv) * half) {
          const int hh = t / half, i = t - hh * half;
          const float x0 = y[hh * hd + i] * inv, x1 = y[hh * hd + i + half] * inv;
          const float2 cs = cs_s[i];
          const float r0 = x0 * cs.x - x1 * cs.y, r1 = x0 * cs.y + x1 * cs.x;
          if (hh < Hq) {
            y[hh * hd + i] = r0 * qscale;
            y[hh * hd + i + half] = r1 * qscale;
          } else if (ri.x >= 0) {
            float* kp = pool + (size_t)ri.x * md.page_elems + ((size_t)(j * 2 + 0) * md.Hkv + (hh - Hq)) * 64 * hd +
                        (size_t)ri.y * hd;
            kp[i] = r0;
            kp[i + half] = r1;
          }
        } else if (ri.x >= 0) {
          const int e = t - (Hq + md.Hkv) * half, hh = e / hd, i = e - hh * hd;
          pool[(size_t)ri.x * md.page_elems + ((size_t)(j * 2 + 1) * md.Hkv + hh) * 64 * hd + (size_t)ri.y * hd + i] =
              y[q_dim + md.kv_dim + e] * inv;
        }
      }
      __syncthreads();
      // ---- attention over the row's loop-r cache ----
      // a thread's values: keys sp, sp + splits, ... of element f; the first of them are loaded ahead of the scores
      const int splits = q_dim >= SR_THREADS ? 1 : SR_THREADS / q_dim;
      const int vsp = tid / q_dim, vf = tid - vsp * q_dim;
      const float* vbase = pool + ((size_t)(j * 2 + 1) * md.Hkv + (vf / hd) / G) * 64 * hd + vf % hd;
      auto value = [&](const float* vb, int key) {
        return vb[(size_t)pages[key >> 6] * md.page_elems + (size_t)(key & 63) * hd];
      };
      float va[SR_VAHEAD];
#pragma unroll
      for (int i = 0; i < SR_VAHEAD; ++i) {
        const int key = vsp + i * splits;
        va[i] = vsp < splits && key < L ? value(vbase, key) : 0.f;
      }
      for (int t = tid; t < Hq * L; t += SR_THREADS) {
        const int hh = t / L, key = t - hh * L;
        const float4* kp = reinterpret_cast<const float4*>(pool + (size_t)pages[key >> 6] * md.page_elems +
                                                           ((size_t)(j * 2 + 0) * md.Hkv + hh / G) * 64 * hd +
                                                           (size_t)(key & 63) * hd);
        const float4* qp = reinterpret_cast<const float4*>(y + hh * hd);
        float acc = 0.f;
        for (int c = 0; c < hd / 4; ++c) {
          const float4 x = kp[c], y = qp[c];
          acc = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, acc))));
        }
        sc[hh * RowStep::MAX_KEYS + key] = acc;
      }
      __syncthreads();
      for (int hh = warp; hh < Hq; hh += SR_THREADS / 32) {
        float* row = sc + hh * RowStep::MAX_KEYS;
        float mx = -INFINITY;
        for (int i = lane; i < L; i += 32) mx = fmaxf(mx, row[i]);
        mx = warp_max(mx);
        float t = 0.f;
        for (int i = lane; i < L; i += 32) {
          const float e = exp2f(row[i] - mx);
          row[i] = e;
          t += e;
        }
        t = warp_sum(t);
        if (lane == 0) lsum[hh] = t;
      }
      __syncthreads();
      for (int t = tid; t < splits * q_dim; t += SR_THREADS) {
        const int sp = t / q_dim, f = t - sp * q_dim, hh = f / hd;
        const float* row = sc + hh * RowStep::MAX_KEYS;
        const float* vb = pool + ((size_t)(j * 2 + 1) * md.Hkv + hh / G) * 64 * hd + f % hd;
        float acc = 0.f;
        int key = sp;
        if (t == tid) {
#pragma unroll
          for (int i = 0; i < SR_VAHEAD; ++i) {
            if (key < L) acc = fmaf(row[key], va[i], acc);
            key += splits;
          }
        }
#pragma unroll 4
        for (; key < L; key += splits) acc = fmaf(row[key], value(vb, key), acc);
        part[t] = acc;
      }
      __syncthreads();
      for (int f = tid; f < q_dim; f += SR_THREADS) {
        float t = 0.f;
        for (int sp = 0; sp < splits; ++sp) t += part[sp * q_dim + f];
        o[f] = t / lsum[f / hd];
      }
      __syncthreads();
      // ---- O projection and residual ----
      const float* al = a.cond ? cvec(j, 0) : nullptr;
      sr_gemv(wo, d, q_dim, o, y);
      if (tid < d) h[tid] += al ? al[tid] * y[tid] : y[tid];
      __syncthreads();
      // ---- SwiGLU and down projection ----
      operand(gm, 3);
      inv = norm_factor();
      sr_gemv(wg, 2 * ff, d, part, y);
      for (int f = tid; f < ff; f += SR_THREADS) {
        const float g = y[f] * inv;
        u[f] = g / (1.f + expf(-g)) * (y[ff + f] * inv);
      }
      __syncthreads();
      const float* am = a.cond ? cvec(j, 1) : nullptr;
      sr_gemv(wd, d, ff, u, y);
      if (tid < d) h[tid] += am ? am[tid] * y[tid] : y[tid];
      __syncthreads();
    }
  }
  // final norm for the LM head, and the cache lengths
  const float inv = norm_factor();
  if (tid < d) a.Xf[(size_t)b * d + tid] = h[tid] * inv * fgain;
  if (tid < m) s.len[slot * M + tid] += 1;
}

// Whether a step of this model may run row by row: the widths its shared memory takes, and layers of up to 1 MB (which
// steps do depends on their caches too).
bool step_row_fits(const ModelDims& md) {
  if (md.dtype != 0 || md.J > SS_LAYERS || md.d % 4 || md.ff % 4) return false;
  const SrLayout l = sr_layout(md);
  return (long long)l.weights / md.J * 4 <= (1 << 20) && (long long)l.total_act * 4 <= SR_SMEM && md.d <= SR_THREADS;
}

long long step_row_weight_bytes(const ModelDims& md) {
  const SrLayout l = sr_layout(md);
  return (long long)(l.total_act + l.weights) * 4 <= SR_SMEM ? 0 : (long long)l.weights / md.J * 4;
}

cudaError_t launch_step_row(RowStep a, int B, cudaStream_t st) {
  const SrLayout l = sr_layout(a.md);
  a.weights_in_smem = (long long)(l.total_act + l.weights) * 4 <= SR_SMEM;
  const int smem = (l.total_act + (a.weights_in_smem ? l.weights : 0)) * 4;
  (void)ensure_kernel_attrs((const void*)k_step_row, SR_SMEM);  // a failure shows at launch
  return launch_k(k_step_row, dim3(B), dim3(SR_THREADS), smem, st, a);
}

}  // namespace tlf
