// The shared block of a decode step for up to 16 rows in one persistent kernel (Eq. 6-11).
//
// With few rows a decode step is a chain of small dependent stages: five per (loop, layer), each a few
// megabytes of weights and kilobytes of activations. As launches of their own every stage paid for the
// release of its predecessor, its operand's first load, a split-K exchange over a cluster and the
// drain of its own stores, about 7 us a launch; here the stages are phases of one cooperative kernel (one
// CTA per SM), separated by grid barriers, and loops that no token reaches cost nothing.
//
// Projections. The unit is a tile of 8 weight rows over the whole reduction length, so no partial sum
// leaves the CTA. A CTA owns a contiguous range of tiles; their rows are fetched into shared memory by
// bulk copies two phases ahead of their use (weights depend on nothing), so at the barrier only the
// activations are waited for. The 16 consumer warps split K; each lane reads 16 contiguous bytes of a
// token row (hi and lo planes) and of a weight row, which feed two mma.sync m16n8k16 (tokens are the
// 16 MMA rows, the 8 weight rows its columns; K's order inside a 32-wide step is permuted alike on both
// sides). With 16 tokens a tcgen05 tile would leave the 128-row operand to the weights and need the
// cluster exchange again; the arithmetic here is far from bounding the phase either way. The warps' sums
// meet in shared memory in a fixed order, and the epilogue finishes the tile: RoPE and K/V append, SwiGLU,
// or the residual update with the next pre-norm's operand and its partial sums of squares.
//
// Attention. Two groups of eight warps and a producer warp per CTA each run the stream-K scheme of
// k_attn_decode on half of the CTA's share of the pages.
#include <type_traits>

#include "tlf_internal.cuh"

namespace tlf {

namespace {

constexpr int SS_THREADS = 2 * 288;  // two groups of 8 consumer warps and a producer warp
constexpr int SS_TILES = 5;          // most tiles of 8 weight rows a CTA may own in a phase
constexpr int SS_PAD = 64;           // bytes added to a staged weight row: 2 rows of a quarter warp on different banks
constexpr int SS_PS = 64;            // keys per page

constexpr __host__ __device__ int ss_tile_bytes(int K) { return 8 * (2 * K + SS_PAD); }

template <int HD, int G>
struct SsShape {
  static constexpr int VEC = 8, LPK = HD / VEC, KPW = 32 / LPK, KEYS_PER_WARP = SS_PS / 8;
  static constexpr int STEPS = KEYS_PER_WARP / KPW > 0 ? KEYS_PER_WARP / KPW : 1;
  static constexpr int SEG = SS_PS * HD * 2, STAGE = 2 * SEG;
  static constexpr int PSZ = G * (HD + 2);        // floats of one partial
  static constexpr int RED = 8 * PSZ * 4;         // a group's merge buffer
};

__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                          uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint4 ldcg16(const void* p) { return __ldcg(reinterpret_cast<const uint4*>(p)); }

// Tiles [u0, u1) of a phase with U tiles owned by CTA c of n.
__device__ __forceinline__ void ss_range(int U, int c, int n, int& u0, int& u1) {
  u0 = (int)((long long)c * U / n);
  u1 = (int)((long long)(c + 1) * U / n);
}

// Weight row of local row l (0..7) of tile u.
// QKV: four rotary pairs (i, i + hd/2) of a q or k head, or 8 features of a v head.
__device__ __forceinline__ int ss_row_qkv(const ModelDims& md, int u, int l) {
  const int f0 = 8 * u;
  if (f0 >= md.q_dim + md.kv_dim) return f0 + l;
  const int hb = f0 / md.hd * md.hd, i0 = (f0 % md.hd) / 2;
  return hb + i0 + (l & 3) + (l >> 2) * (md.hd / 2);
}
// gate/up: four gate features, then the matching up features (packed 64 gate, 64 up per 128 rows)
__device__ __forceinline__ int ss_row_gu(int u, int l) {
  const int f = 4 * u + (l & 3);
  return (f >> 6) * 128 + (f & 63) + (l >> 2) * 64;
}

}  // namespace

// What of a phase's weights a CTA stages: tile count, row source.
template <int KIND>  // 0 QKV, 1 gate/up, 2 plain rows
__device__ __forceinline__ void ss_prefetch(const ModelDims& md, const bf16* W, int K, int U, uint8_t* dst, uint32_t bar,
                                            int lane) {
  int u0, u1;
  ss_range(U, blockIdx.x, gridDim.x, u0, u1);
  const int rows = 8 * (u1 - u0), rs = 2 * K + SS_PAD;
  if (rows == 0) return;
  if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)(rows * 2 * K));
  __syncwarp();
  for (int i = lane; i < rows; i += 32) {
    const int u = u0 + (i >> 3), l = i & 7;
    const int row = KIND == 0 ? ss_row_qkv(md, u, l) : KIND == 1 ? ss_row_gu(u, l) : 8 * u + l;
    bulk_g2s(smem_u32(dst + (size_t)i * rs), W + (size_t)row * K, (uint32_t)(2 * K), bar);
  }
}

template <int HD, int G>
__global__ void __launch_bounds__(SS_THREADS, 1) k_step_small(SmallStep a) {
  using Sh = SsShape<HD, G>;
  extern __shared__ __align__(128) uint8_t sm[];
  const ModelDims& md = a.md;
  const StepDev& s = a.s;
  uint8_t* w1 = sm;                      // QKV and gate/up weights
  uint8_t* w2 = w1 + a.w1_bytes;         // O and down weights
  uint8_t* kv = w2 + a.w2_bytes;         // two K/V rings; the projections' partial sums between attentions
  float* att_red = reinterpret_cast<float*>(kv + 2 * a.nst * Sh::STAGE);
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(att_red) + 2 * Sh::RED);
  __shared__ int4 rowmeta[16];           // per compact row of the loop: page, slot in page, position, batch row
  // its compact row in the next loop plus 1 (0: none), and conditioning table rows of (depth, loop) and (depth, next loop)
  __shared__ uchar4 rowaux[16];
  __shared__ float scale[16];
  __shared__ int pbase[17], nkeys[16], slots[16];  // attention plan of the loop: first flat pages, keys, sequence slots
  __shared__ int flags[4];               // ticket outcome of the two groups; abort
  volatile int* abort_flag = &flags[2];
  auto kvfull = [&](int grp, int st) { return smem_u32(&bars[grp * 2 * a.nst + st]); };
  auto kvempty = [&](int grp, int st) { return smem_u32(&bars[grp * 2 * a.nst + a.nst + st]); };
  const uint32_t wbar1 = smem_u32(&bars[4 * a.nst]), wbar2 = smem_u32(&bars[4 * a.nst + 1]);  // weights in
  const uint32_t wfree1 = smem_u32(&bars[4 * a.nst + 2]), wfree2 = smem_u32(&bars[4 * a.nst + 3]);  // ... read

  const int tid = threadIdx.x, lane = tid & 31;
  const int grp = tid >= 288, w9 = (tid - 288 * grp) >> 5;  // group, warp of the group (8: producer)
  const bool producer = w9 == 8;
  const int wi = grp * 8 + w9;                             // consumer warp 0..15
  const int ct = grp * 256 + (tid - 288 * grp);            // consumer thread 0..511
  if (tid == 0) {
    for (int i = 0; i < 2 * a.nst; ++i) {
      mbar_init(smem_u32(&bars[(i / a.nst) * 2 * a.nst + i % a.nst]), 1);
      mbar_init(smem_u32(&bars[(i / a.nst) * 2 * a.nst + a.nst + i % a.nst]), 8);
    }
    mbar_init(wbar1, 1);
    mbar_init(wbar2, 1);
    mbar_init(wfree1, 16);
    mbar_init(wfree2, 16);
    flags[2] = 0;
    fence_barrier_init();
  }
  __syncthreads();
  const int d = md.d, q_dim = md.q_dim, ff = md.ff, M = md.M, J = md.J, maxB = md.max_batch;
  const int Uq = md.qkv_dim / 8, Uo = d / 8, Ug = ff / 4, Ud = d / 8;
  // group 0's producer warp keeps the QKV and gate/up weights coming, group 1's the O and down weights
  if (producer) {
    if (grp == 0) ss_prefetch<0>(md, a.layer[0].wqkv, d, Uq, w1, wbar1, lane);
    else ss_prefetch<2>(md, a.layer[0].wo, q_dim, Uo, w2, wbar2, lane);
  }
  pdl_wait();

  int epoch = 0;        // grid barriers passed
  uint32_t ph1 = 0, ph2 = 0;  // phases of the weight barriers
  uint32_t phf = 0;           // ... of the producer's "weights read" barrier
  int tq, tg, to, td;         // tiles of this CTA in each projection
  {
    int x0, x1;
    ss_range(Uq, blockIdx.x, gridDim.x, x0, x1); tq = x1 - x0;
    ss_range(Ug, blockIdx.x, gridDim.x, x0, x1); tg = x1 - x0;
    ss_range(Uo, blockIdx.x, gridDim.x, x0, x1); to = x1 - x0;
    ss_range(Ud, blockIdx.x, gridDim.x, x0, x1); td = x1 - x0;
  }
  int ring = 0;         // pages that went through this group's ring
  auto give_up = [&]() {
    atomicOr(s.err, DEVERR_WAIT);
    *abort_flag = 1;
  };
  // All CTAs' writes before it are visible to reads past L1 after it (consumer threads).
  auto grid_sync = [&](bool to_copies = false) {
    ++epoch;
    if (to_copies) fence_proxy_async_all();  // new K/V entries, and the partial sums' space, go to bulk copies
    named_sync(1, 512);
    if (ct < 32) {
      // arrivals spread over eight counters, one of which each of eight lanes watches
      if (ct == 0)
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.gbar + 32 * (blockIdx.x & 7)) : "memory");
      const unsigned want = (unsigned)epoch * ((gridDim.x + 7 - (ct & 7)) / 8);
      uint64_t t0 = 0;
      while (!*abort_flag) {
        unsigned got = want;
        if (ct < 8) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(a.gbar + 32 * ct) : "memory");
        if (__all_sync(0xffffffffu, got >= want)) break;
        const uint64_t t = globaltimer_ns();
        if (t0 == 0) t0 = t;
        if (t - t0 > kWaitLimitNs) give_up();
      }
      __syncwarp();
    }
    named_sync(1, 512);
  };
  auto wait_w = [&](uint32_t bar, uint32_t& ph) {
    if (!*abort_flag && !mbar_wait(bar, ph & 1u, s.err)) *abort_flag = 1;
    ++ph;
  };

  // A projection over this CTA's T tiles: the warps' partial sums [16][T][16 rows][8] to `red`; ends with the consumers'
  // barrier, after which sum(T, tile, m, l) may be taken. The token operand's loads are issued ahead of the wait for
  // the weights and of their use. Up to 8 rows the two terms of a row are the MMA's rows g and g + 8.
  float* red = reinterpret_cast<float*>(kv);
  auto project = [&](const uint8_t* ws, uint32_t wbar, uint32_t& ph, int K, int T, int n, const bf16* X, size_t lo_off,
                     bool free_next, uint32_t wfree, auto tm) {
    constexpr int TM = decltype(tm)::value;
    const int g = lane >> 2, t4 = lane & 3, rs = 2 * K + SS_PAD;
    float acc[TM][4];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
    const int steps = T > 0 ? (K + 31) / 32 : 0;
    const uint4 z = make_uint4(0, 0, 0, 0);
    const bf16* xg = X + (size_t)g * K + t4 * 8;
    bool waited = T == 0;
    if (n <= 8) {
      constexpr int SB = 3;  // steps whose operands are in flight at once
      for (int s0 = wi; s0 < steps; s0 += 16 * SB) {
        uint4 h[SB], l[SB];
#pragma unroll
        for (int q = 0; q < SB; ++q) {
          const int k = (s0 + 16 * q) * 32;
          const bool in = s0 + 16 * q < steps && k + t4 * 8 < K && g < n;
          h[q] = in ? ldcg16(xg + k) : z;
          l[q] = in ? ldcg16(xg + k + lo_off) : z;
        }
        if (!waited) wait_w(wbar, ph);
        waited = true;
#pragma unroll
        for (int q = 0; q < SB; ++q) {
          const int k = (s0 + 16 * q) * 32 + t4 * 8;
          if (s0 + 16 * q < steps)
#pragma unroll
            for (int i = 0; i < TM; ++i)
              if (i < T) {
                const uint4 w = k < K ? *reinterpret_cast<const uint4*>(ws + (size_t)(i * 8 + g) * rs + 2 * k) : z;
                mma_16816(acc[i], h[q].x, l[q].x, h[q].y, l[q].y, w.x, w.y);
                mma_16816(acc[i], h[q].z, l[q].z, h[q].w, l[q].w, w.z, w.w);
              }
        }
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        acc[i][0] += acc[i][2];
        acc[i][1] += acc[i][3];
      }
    } else {
      constexpr int SB = 2;
      for (int s0 = wi; s0 < steps; s0 += 16 * SB) {
        uint4 h0[SB], h1[SB], l0[SB], l1[SB];
#pragma unroll
        for (int q = 0; q < SB; ++q) {
          const int k = (s0 + 16 * q) * 32;
          const bool in = s0 + 16 * q < steps && k + t4 * 8 < K;  // (n > 8: row g exists)
          h0[q] = in ? ldcg16(xg + k) : z;
          l0[q] = in ? ldcg16(xg + k + lo_off) : z;
          h1[q] = in && g + 8 < n ? ldcg16(xg + (size_t)8 * K + k) : z;
          l1[q] = in && g + 8 < n ? ldcg16(xg + (size_t)8 * K + k + lo_off) : z;
        }
        if (!waited) wait_w(wbar, ph);
        waited = true;
#pragma unroll
        for (int q = 0; q < SB; ++q) {
          const int k = (s0 + 16 * q) * 32 + t4 * 8;
          if (s0 + 16 * q < steps)
#pragma unroll
            for (int i = 0; i < TM; ++i)
              if (i < T) {
                const uint4 w = k < K ? *reinterpret_cast<const uint4*>(ws + (size_t)(i * 8 + g) * rs + 2 * k) : z;
                mma_16816(acc[i], h0[q].x, h1[q].x, h0[q].y, h1[q].y, w.x, w.y);
                mma_16816(acc[i], h0[q].z, h1[q].z, h0[q].w, h1[q].w, w.z, w.w);
                mma_16816(acc[i], l0[q].x, l1[q].x, l0[q].y, l1[q].y, w.x, w.y);
                mma_16816(acc[i], l0[q].z, l1[q].z, l0[q].w, l1[q].w, w.z, w.w);
              }
        }
      }
    }
    if (!waited) wait_w(wbar, ph);  // (a warp without a step keeps the phase)
    __syncwarp();
    if (free_next && lane == 0) mbar_arrive(wfree);  // the producer may fetch the next weights of this region
#pragma unroll
    for (int i = 0; i < TM; ++i)
      if (i < T) {
        float* o = red + ((size_t)(wi * T + i) * 16 + g) * 8 + 2 * t4;
        *reinterpret_cast<float2*>(o) = make_float2(acc[i][0], acc[i][1]);
        if (n > 8) *reinterpret_cast<float2*>(o + 64) = make_float2(acc[i][2], acc[i][3]);
      }
    named_sync(1, 512);
  };
  auto sum = [&](int T, int i, int m, int l) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < 16; ++w) t += red[((size_t)(w * T + i) * 16 + m) * 8 + l];
    return t;
  };
  // RMSNorm factors of the loop's rows from the producer's partial sums of squares: warp wi takes row wi
  auto row_scale = [&](const float* ss, int ld, int n) {
    float t = 0.f;
    if (wi < n)
      for (int i = lane; i < ld / 4; i += 32) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(ss + (size_t)wi * ld) + i);
        t += (v.x + v.y) + (v.z + v.w);
      }
    t = warp_sum(t);
    if (lane == 0) scale[wi] = rsqrtf(t / (float)d + md.eps);
  };
  const size_t xlo = (size_t)maxB * d, olo = (size_t)maxB * q_dim, ulo = (size_t)maxB * ff;
  const int ld8 = d / 8;

  for (int r = 0; r < M; ++r) {
    const int n = min(16, __ldcg(s.n + r));
    if (n <= 0) break;  // active sets nest
    const bool more_loops = r + 1 < M && __ldcg(s.n + (r + 1 < M ? r + 1 : r)) > 0;
    if (!producer && ct < 17) {
      if (ct < n) {
        const int4 ri = __ldcg(s.rowinfo + r * maxB + ct);
        rowmeta[ct] = ri;
        const int nc = r + 1 < M ? __ldcg(s.col + (r + 1) * maxB + ri.w) + 1 : 0;
        const int m = min(max(__ldcg(s.m + ri.w), r + 1), M), mo = m * (m - 1) / 2 + r;
        rowaux[ct] = make_uchar4((unsigned char)nc, (unsigned char)mo, (unsigned char)min(mo + 1, m * (m + 1) / 2 - 1), 0);
        nkeys[ct] = __ldcg(s.nch + r * maxB + ct);
        slots[ct] = __ldcg(s.slots + ri.w);
      }
      if (ct <= n) pbase[ct] = __ldcg(s.item_base + r * (maxB + 1) + ct);
    }
    __syncthreads();
    // conditioning vector `part` of layer j for the rows' (depth, loop)
    const int combos = M * (M + 1) / 2;
    auto cvec = [&](int j, int off, int part) { return a.cond + ((size_t)(j * combos + off) * 4 + part) * d; };
    // What the epilogue of a residual projection needs besides its sums, for this thread's element (at most two tiles,
    // so one element a thread), loaded before the grid barrier: the CTA's own residual values, gains, modulation.
    struct Pre {
      float h, gain, alpha, gamma;
    };
    auto resid_pre = [&](int T, int u0, int j, int part, const float* gain, bool next_loop, int jn, int gpart) {
      Pre q = {0.f, 0.f, 1.f, 1.f};
      const int i = ct >> 7, m = (ct >> 3) & 15, f = 8 * (u0 + i) + (ct & 7);
      if (i < T && m < n) {
        q.h = __ldcg(s.H + (size_t)rowmeta[m].w * d + f);
        q.gain = gain[f];
        if (a.cond) {
          q.alpha = cvec(j, rowaux[m].y, part)[f];
          q.gamma = 1.f + cvec(jn, next_loop ? rowaux[m].z : rowaux[m].y, gpart)[f];
        }
      }
      return q;
    };
    // residual update of the CTA's tiles and the next pre-norm's operand
    auto resid_epilogue = [&](int T, int u0, const Pre& pre, bool has_next, bool next_loop) {
      if (ct < T * 128) {
        const int i = ct >> 7, m = (ct >> 3) & 15, l = ct & 7, f = 8 * (u0 + i) + l;
        float h = pre.h;
        int dst = -1;
        if (m < n) {
          h += pre.alpha * sum(T, i, m, l);
          s.H[(size_t)rowmeta[m].w * d + f] = h;
          if (has_next) dst = next_loop ? (int)rowaux[m].x - 1 : m;
          if (dst >= 0) {
            const float y = h * pre.gain * pre.gamma;
            const bf16 yh = __float2bfloat16_rn(y);
            a.X[(size_t)dst * d + f] = yh;
            a.X[xlo + (size_t)dst * d + f] = __float2bfloat16_rn(y - __bfloat162float(yh));
          }
        }
        float q = h * h;
        q += __shfl_xor_sync(0xffffffffu, q, 1);
        q += __shfl_xor_sync(0xffffffffu, q, 2);
        q += __shfl_xor_sync(0xffffffffu, q, 4);
        if (dst >= 0 && l == 0) a.ss8[(size_t)dst * ld8 + u0 + i] = q;
      }
    };

    for (int j = 0; j < J; ++j) {
      const SmallLayer L = a.layer[j];
      const bool last_layer = j + 1 == J, has_next = !last_layer || more_loops;
      const int jn = last_layer ? 0 : j + 1;
      int u0, u1;
      Pre pre;
      if (!producer) {
        // ---- QKV + RoPE + append ----
        ss_range(Uq, blockIdx.x, gridDim.x, u0, u1);
        {
          const int T = tq, i = ct >> 6, m = (ct >> 2) & 15, p = ct & 3, f = 8 * (u0 + i);  // (T <= 8: one item a thread)
          const bool mine = i < T && m < n;
          int4 ri = make_int4(-1, 0, 0, 0);
          float2 cs = make_float2(1.f, 0.f);
          if (mine) {
            ri = rowmeta[m];
            if (f < q_dim + md.kv_dim) cs = a.rope[(size_t)ri.z * (HD / 2) + (f % HD) / 2 + p];
          }
          const bool first = r == 0 && j == 0;
          row_scale(first ? a.ss : a.ss8, first ? a.ldss : ld8, n);
          project(w1, wbar1, ph1, d, T, n, a.X, xlo, tg > 0, wfree1, std::integral_constant<int, SS_TILES>{});
          if (mine) {
            const float x0 = sum(T, i, m, p) * scale[m], x1 = sum(T, i, m, p + 4) * scale[m];
            if (f < q_dim + md.kv_dim) {
              const int h = f / HD, e = (f % HD) / 2 + p;  // pair (e, e + HD/2) of head h
              const float r0 = x0 * cs.x - x1 * cs.y, r1 = x0 * cs.y + x1 * cs.x;
              if (h < md.Hq) {
                float* q = a.Q + ((size_t)m * md.Hq + h) * HD;
                q[e] = r0;
                q[e + HD / 2] = r1;
              } else if (ri.x >= 0) {
                bf16* kp = reinterpret_cast<bf16*>(s.pool) + (size_t)ri.x * md.page_elems +
                           ((size_t)(j * 2 + 0) * md.Hkv + (h - md.Hq)) * SS_PS * HD + (size_t)ri.y * HD;
                kp[e] = __float2bfloat16_rn(r0);
                kp[e + HD / 2] = __float2bfloat16_rn(r1);
              }
            } else if (ri.x >= 0) {
              const int fv = f - q_dim - md.kv_dim, h = fv / HD, e = fv % HD + p;
              bf16* vp = reinterpret_cast<bf16*>(s.pool) + (size_t)ri.x * md.page_elems +
                         ((size_t)(j * 2 + 1) * md.Hkv + h) * SS_PS * HD + (size_t)ri.y * HD;
              vp[e] = __float2bfloat16_rn(x0);
              vp[e + 4] = __float2bfloat16_rn(x1);
            }
          }
        }
        grid_sync(true);
      } else if (grp == 0 && tg > 0) {
        if (!*abort_flag && !mbar_wait(wfree1, phf & 1u, s.err)) *abort_flag = 1;
        ++phf;
        ss_prefetch<1>(md, L.wgu, d, Ug, w1, wbar1, lane);
      }
      // ---- attention: the group's share of the pages ----
      __syncthreads();  // the producers start here too
      {
        auto pages_of = [&](int kk) { return (nkeys[kk] + SS_PS - 1) / SS_PS; };
        const int total = pbase[n];
        const int nv = 2 * gridDim.x, v = 2 * blockIdx.x + grp;
        const int per = (total + nv - 1) / nv;
        const int p0 = v * per, p1 = min(total, p0 + per);
        if (p0 < total) {
          // (row, kv head, page) of flat page p0: the largest k with pbase[k] <= p0 (n <= 16 entries, one ballot)
          int k, h, g;
          {
            const unsigned le = __ballot_sync(0xffffffffu, lane < n && pbase[lane] <= p0);
            k = 31 - __clz((int)le);
            const int off = p0 - pbase[k], np = pages_of(k);
            h = off / np;
            g = off % np;
          }
          uint8_t* my_ring = kv + (size_t)grp * a.nst * Sh::STAGE;
          if (producer) {
            fence_proxy_async_all();  // behind the barrier: this step's K/V entries
            int page_l = -1;          // lane q: page of the q-th of the next 32 flat pages
            for (int p = p0; p < p1; ++p) {
              if (((p - p0) & 31) == 0) {
                const int pq = p + lane;
                page_l = -1;
                if (pq < p1) {
                  int kq = k;  // the row of a later page: rows ascend
                  while (kq + 1 < n && pbase[kq + 1] <= pq) ++kq;
                  page_l = s.page_table[((size_t)slots[kq] * M + r) * md.max_pages + (pq - pbase[kq]) % pages_of(kq)];
                }
                __syncwarp();
              }
              const int page = __shfl_sync(0xffffffffu, page_l, (p - p0) & 31);
              if (lane == 0) {
                const int i = ring + p - p0, st = i % a.nst;
                if (i >= a.nst && !*abort_flag && !mbar_wait(kvempty(grp, st), (uint32_t)(i / a.nst - 1) & 1u, s.err))
                  *abort_flag = 1;
                const uint32_t bar = kvfull(grp, st);
                const int valid = min(SS_PS, nkeys[k] - g * SS_PS);
                if (!*abort_flag) {
                if (page < 0 || page >= md.n_pages || valid <= 0) {
                  atomicOr(s.err, DEVERR_INDEX);
                  mbar_arrive(bar);  // complete the phase without data
                } else {
                  const bf16* pg = reinterpret_cast<const bf16*>(s.pool) + (size_t)page * md.page_elems;
                  const uint32_t bytes = (uint32_t)(valid * HD * 2);
                  uint8_t* dst = my_ring + st * Sh::STAGE;
                  const uint64_t pol = l2_policy_evict_first();  // pages are read once per step
                  mbar_arrive_expect_tx(bar, 2 * bytes);
                  bulk_g2s_hint(smem_u32(dst), pg + ((size_t)(j * 2 + 0) * md.Hkv + h) * SS_PS * HD, bytes, bar, pol);
                  bulk_g2s_hint(smem_u32(dst + Sh::SEG), pg + ((size_t)(j * 2 + 1) * md.Hkv + h) * SS_PS * HD, bytes, bar,
                                pol);
                }
                }
              }
              __syncwarp();
              if (++g == pages_of(k)) {
                g = 0;
                if (++h == md.Hkv) {
                  h = 0;
                  ++k;
                }
              }
            }
          } else {
            const int sub = lane / Sh::LPK, pl = lane % Sh::LPK;
            const float qscale = 1.4426950408889634f * rsqrtf((float)HD);
            float* mred = att_red + (size_t)grp * (Sh::RED / 4);
            const int gtid = tid - 288 * grp;
            int Lk = 0;
            float q[G][Sh::VEC], run_m[G], run_l[G], acc[G][Sh::VEC];
            auto begin_item = [&]() {
              Lk = nkeys[k];
              const float* qrow = a.Q + (size_t)k * md.Hq * HD;
#pragma unroll
              for (int gg = 0; gg < G; ++gg) {
                const float4* q4 = reinterpret_cast<const float4*>(qrow + (h * G + gg) * HD + pl * Sh::VEC);
                const float4 x = __ldcg(q4), y = __ldcg(q4 + 1);
                q[gg][0] = x.x * qscale; q[gg][1] = x.y * qscale; q[gg][2] = x.z * qscale; q[gg][3] = x.w * qscale;
                q[gg][4] = y.x * qscale; q[gg][5] = y.y * qscale; q[gg][6] = y.z * qscale; q[gg][7] = y.w * qscale;
                run_m[gg] = -INFINITY;
                run_l[gg] = 0.f;
#pragma unroll
                for (int e = 0; e < Sh::VEC; ++e) acc[gg][e] = 0.f;
              }
            };
            begin_item();
            for (int p = p0; p < p1; ++p) {
              const int i = ring + p - p0, st = i % a.nst;
              if (!*abort_flag && !mbar_wait(kvfull(grp, st), (uint32_t)(i / a.nst) & 1u, s.err)) *abort_flag = 1;
              const int valid = min(SS_PS, Lk - g * SS_PS);
              const bf16* sk = reinterpret_cast<const bf16*>(my_ring + st * Sh::STAGE);
              const bf16* sv = reinterpret_cast<const bf16*>(my_ring + st * Sh::STAGE + Sh::SEG);
              float sc[Sh::STEPS][G];
#pragma unroll
              for (int t = 0; t < Sh::STEPS; ++t) {
                const int key = w9 * Sh::KEYS_PER_WARP + t * Sh::KPW + sub;
                float x[Sh::VEC];
                const bool use = key < valid;
                if (use) {
                  Vec16<bf16>::load(sk + key * HD + pl * Sh::VEC, x);
                } else {
#pragma unroll
                  for (int e = 0; e < Sh::VEC; ++e) x[e] = 0.f;
                }
#pragma unroll
                for (int gg = 0; gg < G; ++gg) {
                  float dt = 0.f;
#pragma unroll
                  for (int e = 0; e < Sh::VEC; ++e) dt = fmaf(q[gg][e], x[e], dt);
#pragma unroll
                  for (int o = Sh::LPK / 2; o > 0; o >>= 1) dt += __shfl_xor_sync(0xffffffffu, dt, o);
                  sc[t][gg] = use ? dt : -INFINITY;
                }
              }
#pragma unroll
              for (int gg = 0; gg < G; ++gg) {
                float pm = sc[0][gg];
#pragma unroll
                for (int t = 1; t < Sh::STEPS; ++t) pm = fmaxf(pm, sc[t][gg]);
#pragma unroll
                for (int o = Sh::LPK; o < 32; o <<= 1) pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
                if (pm > run_m[gg]) {
                  const float cr = exp2f(run_m[gg] - pm);  // 0 when run_m was -inf
                  run_l[gg] *= cr;
#pragma unroll
                  for (int e = 0; e < Sh::VEC; ++e) acc[gg][e] *= cr;
                  run_m[gg] = pm;
                }
              }
#pragma unroll
              for (int t = 0; t < Sh::STEPS; ++t) {
                const int key = w9 * Sh::KEYS_PER_WARP + t * Sh::KPW + sub;
                if (key < valid) {
                  float x[Sh::VEC];
                  Vec16<bf16>::load(sv + key * HD + pl * Sh::VEC, x);
#pragma unroll
                  for (int gg = 0; gg < G; ++gg) {
                    const float pr = exp2f(sc[t][gg] - run_m[gg]);
                    run_l[gg] += pr;
#pragma unroll
                    for (int e = 0; e < Sh::VEC; ++e) acc[gg][e] = fmaf(pr, x[e], acc[gg][e]);
                  }
                }
              }
              __syncwarp();
              if (lane == 0) mbar_arrive(kvempty(grp, st));
              const int np = pages_of(k);
              if (g + 1 < np && p + 1 < p1) {
                ++g;
                continue;
              }
              // ---- the group's part of item (k, h) is done: merge the lane groups, then the warps ----
#pragma unroll
              for (int gg = 0; gg < G; ++gg)
#pragma unroll
                for (int o = Sh::LPK; o < 32; o <<= 1) {
                  run_l[gg] += __shfl_xor_sync(0xffffffffu, run_l[gg], o);
#pragma unroll
                  for (int e = 0; e < Sh::VEC; ++e) acc[gg][e] += __shfl_xor_sync(0xffffffffu, acc[gg][e], o);
                }
              if (sub == 0) {
#pragma unroll
                for (int gg = 0; gg < G; ++gg) {
                  float* rw = mred + (w9 * G + gg) * (HD + 2);
#pragma unroll
                  for (int e = 0; e < Sh::VEC; ++e) rw[pl * Sh::VEC + e] = acc[gg][e];
                  if (pl == 0) {
                    rw[HD] = run_m[gg];
                    rw[HD + 1] = run_l[gg];
                  }
                }
              }
              named_sync(2 + grp, 256);
              const int item = k * md.Hkv + h, first = pbase[k] + h * np;
              const int c_first = first / per, c_last = (first + np - 1) / per, nparts = c_last - c_first + 1;
              float* my = a.part + (size_t)(item + v) * Sh::PSZ;
              auto store_o = [&](int t, float val) {
                const size_t at = (size_t)k * q_dim + (size_t)h * G * HD + t;  // t = head of the group * HD + dim
                const bf16 hi = __float2bfloat16_rn(val);
                a.O[at] = hi;
                a.O[olo + at] = __float2bfloat16_rn(val - __bfloat162float(hi));
              };
              for (int t = gtid; t < G * HD; t += 256) {
                const int gg = t / HD, e = t % HD;
                float mx = -INFINITY;
#pragma unroll
                for (int w = 0; w < 8; ++w) mx = fmaxf(mx, mred[(w * G + gg) * (HD + 2) + HD]);
                float o = 0.f, l = 0.f;
#pragma unroll
                for (int w = 0; w < 8; ++w) {
                  const float* rw = mred + (w * G + gg) * (HD + 2);
                  const float fw = (rw[HD] == -INFINITY) ? 0.f : exp2f(rw[HD] - mx);
                  o = fmaf(fw, rw[e], o);
                  l = fmaf(fw, rw[HD + 1], l);
                }
                if (nparts == 1) {
                  store_o(t, o / l);
                } else {
                  my[gg * (HD + 2) + e] = o;
                  if (e == 0) {
                    my[gg * (HD + 2) + HD] = mx;
                    my[gg * (HD + 2) + HD + 1] = l;
                  }
                }
              }
              if (nparts > 1) {
                __threadfence();
                named_sync(2 + grp, 256);
                if (gtid == 0) flags[grp] = atomicAdd(s.cnt + item, 1) == nparts - 1;
                named_sync(2 + grp, 256);
                if (flags[grp]) {
                  // last contributor: merge the partials of shares c_first..c_last
                  __threadfence();
                  for (int t = gtid; t < G * HD; t += 256) {
                    const int gg = t / HD, e = t % HD;
                    float mx = -INFINITY;
                    // eight partials' loads in flight at a time
                    float o = 0.f, l = 0.f;
                    for (int c0 = c_first; c0 <= c_last; c0 += 8) {
                      float pm[8], po[8], pl8[8];
#pragma unroll
                      for (int q = 0; q < 8; ++q) {
                        const float* pp = a.part + (size_t)(item + min(c0 + q, c_last)) * Sh::PSZ + gg * (HD + 2);
                        pm[q] = c0 + q <= c_last ? __ldcg(pp + HD) : -INFINITY;
                        po[q] = __ldcg(pp + e);
                        pl8[q] = __ldcg(pp + HD + 1);
                      }
                      float nm = mx;
#pragma unroll
                      for (int q = 0; q < 8; ++q) nm = fmaxf(nm, pm[q]);
                      const float cr = exp2f(mx - nm);  // 0 for the first eight
                      o *= cr;
                      l *= cr;
                      mx = nm;
#pragma unroll
                      for (int q = 0; q < 8; ++q) {
                        const float fw = exp2f(pm[q] - mx);  // 0 past the last partial
                        o = fmaf(fw, po[q], o);
                        l = fmaf(fw, pl8[q], l);
                      }
                    }
                    store_o(t, o / l);
                  }
                  if (gtid == 0) s.cnt[item] = 0;  // ready for the next layer
                }
              }
              named_sync(2 + grp, 256);  // the merge buffer and flag are reused by the next item
              if (p + 1 < p1) {
                g = 0;
                if (++h == md.Hkv) {
                  h = 0;
                  ++k;
                }
                begin_item();
              }
            }
          }
          ring += p1 - p0;
        }
      }
      if (!producer) {
        ss_range(Uo, blockIdx.x, gridDim.x, u0, u1);
        pre = resid_pre(to, u0, j, 0, L.mlp_norm, false, j, 3);
        grid_sync();
        // ---- O projection + residual, MLP pre-norm operand ----
        project(w2, wbar2, ph2, q_dim, to, n, a.O, olo, td > 0, wfree2, std::integral_constant<int, 2>{});
        resid_epilogue(to, u0, pre, true, false);
        grid_sync();
        // ---- gate/up + SwiGLU ----
        ss_range(Ug, blockIdx.x, gridDim.x, u0, u1);
        row_scale(a.ss8, ld8, n);
        project(w1, wbar1, ph1, d, tg, n, a.X, xlo, has_next && tq > 0, wfree1, std::integral_constant<int, SS_TILES>{});
        {
          const int i = ct >> 6, m = (ct >> 2) & 15, p = ct & 3;  // (at most 8 tiles: one item a thread)
          if (i < tg && m < n) {
            const float gv = sum(tg, i, m, p) * scale[m], uv = sum(tg, i, m, p + 4) * scale[m];
            const float y = gv / (1.f + expf(-gv)) * uv;
            const bf16 yh = __float2bfloat16_rn(y);
            const size_t at = (size_t)m * ff + 4 * (u0 + i) + p;
            a.U[at] = yh;
            a.U[ulo + at] = __float2bfloat16_rn(y - __bfloat162float(yh));
          }
        }
        ss_range(Ud, blockIdx.x, gridDim.x, u0, u1);
        pre = resid_pre(td, u0, j, 1, a.layer[jn].attn_norm, last_layer, jn, 2);
        grid_sync();
        // ---- down projection + residual, next attention pre-norm operand ----
        project(w2, wbar2, ph2, ff, td, n, a.U, ulo, has_next && to > 0, wfree2, std::integral_constant<int, 2>{});
        resid_epilogue(td, u0, pre, has_next, last_layer);
        if (has_next) grid_sync();
      } else if (grp == 0) {
        if (has_next && tq > 0) {  // gate/up weights read: the next QKV weights
          if (!*abort_flag && !mbar_wait(wfree1, phf & 1u, s.err)) *abort_flag = 1;
          ++phf;
          ss_prefetch<0>(md, a.layer[jn].wqkv, d, Uq, w1, wbar1, lane);
        }
      } else {
        if (td > 0) {  // O weights read: the down weights
          if (!*abort_flag && !mbar_wait(wfree2, phf & 1u, s.err)) *abort_flag = 1;
          ++phf;
          ss_prefetch<2>(md, L.wd, ff, Ud, w2, wbar2, lane);
        }
        if (has_next && to > 0) {  // down weights read: the next O weights
          if (!*abort_flag && !mbar_wait(wfree2, phf & 1u, s.err)) *abort_flag = 1;
          ++phf;
          ss_prefetch<2>(md, a.layer[jn].wo, q_dim, Uo, w2, wbar2, lane);
        }
      }
    }
    __syncthreads();  // rowmeta is rewritten for the next loop
  }
}

// Shared memory of the kernel's parts for a model on a grid of `ctas` CTAs: fills the byte counts and ring depth of
// `a`, returns the dynamic shared memory (0: the model does not fit).
static int ss_layout(const ModelDims& md, int ctas, SmallStep* a) {
  auto tiles = [&](int U) { return (U + ctas - 1) / ctas; };
  const int tq = tiles(md.qkv_dim / 8), to = tiles(md.d / 8), tg = tiles(md.ff / 4), td = tiles(md.d / 8);
  if (tq > SS_TILES || tg > SS_TILES || to > 2 || td > 2) return 0;
  a->w1_bytes = ((tq > tg ? tq : tg) * ss_tile_bytes(md.d) + 127) / 128 * 128;
  const int wo = to * ss_tile_bytes(md.q_dim), wd = td * ss_tile_bytes(md.ff);
  a->w2_bytes = ((wo > wd ? wo : wd) + 127) / 128 * 128;
  const int G = md.Hq / md.Hkv, stage = 2 * SS_PS * md.hd * 2, red = 2 * 8 * G * (md.hd + 2) * 4;
  const int fixed = a->w1_bytes + a->w2_bytes + red;
  const int limit = 232448 - 640;  // less the static shared memory
  // the projections' partial sums (16 warps x tiles x 16 rows x 8) share the rings' space
  const int tm = tq > tg ? tq : tg;
  const int psum = 16 * (tm > td ? tm : td) * 16 * 8 * 4;
  for (int nst = 8; nst >= 2; --nst) {
    const int bytes = fixed + 2 * nst * stage + (4 * nst + 4) * 8;
    if (bytes <= limit && 2 * nst * stage >= psum) {
      a->nst = nst;
      return bytes;
    }
  }
  return 0;
}

template <typename F>
static cudaError_t ss_dispatch(const ModelDims& md, F&& f) {
  const int G = md.Hq / md.Hkv;
  if (md.hd == 128 && G == 1) return f(k_step_small<128, 1>);
  if (md.hd == 128 && G == 2) return f(k_step_small<128, 2>);
  if (md.hd == 128) return f(k_step_small<128, 4>);
  if (md.hd == 64 && G == 1) return f(k_step_small<64, 1>);
  if (md.hd == 64 && G == 2) return f(k_step_small<64, 2>);
  if (md.hd == 64) return f(k_step_small<64, 4>);
  if (G == 1) return f(k_step_small<32, 1>);
  return f(k_step_small<32, 2>);
}

bool step_small_fits(const ModelDims& md, int num_sms) {
  SmallStep a{};
  const int smem = ss_layout(md, num_sms, &a);
  if (smem == 0) return false;
  int blocks = 0;
  const cudaError_t e = ss_dispatch(md, [&](auto kernel) {
    const cudaError_t r = ensure_kernel_attrs((const void*)kernel, smem);
    return r != cudaSuccess ? r : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, SS_THREADS, smem);
  });
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return blocks >= 1;
}

cudaError_t launch_step_small(SmallStep a, int num_sms, cudaStream_t st) {
  const int smem = ss_layout(a.md, num_sms, &a);
  if (smem == 0) return cudaErrorInvalidValue;
  return ss_dispatch(a.md, [&](auto kernel) {
    (void)ensure_kernel_attrs((const void*)kernel, smem);  // a failure shows at launch
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(num_sms);
    cfg.blockDim = dim3(SS_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;  // the grid barriers need every CTA resident
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, a);
  });
}

}  // namespace tlf
