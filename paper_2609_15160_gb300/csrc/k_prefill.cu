// Batched prefill of a chunk of prompt tokens (T-LoopFormer Sec. 3.3 and App. B).
//
// A chunk holds up to C prompt tokens of one or more sequences, ordered by
// sequence and position. All its tokens are routed at once; loop r gathers the
// chunk tokens with m >= r (Eq. 6), runs the shared block on them, and writes
// their k, v into the loop-r caches of their sequences at the slots after the
// entries of earlier chunks, in position order (the original positions rho^(r)
// of App. B). Attention at loop r is causal over the loop-r cache of each
// sequence: the token with cache slot s sees slots 0..s, i.e. exactly the
// tokens before it (this or earlier chunks) that also ran loop r (Eq. 10 with
// the block-causal mask among gathered tokens).
//
// k_pf_plan       per loop r: compact rows A_r, each row's sequence slot, cache
//                 slot and position, per-sequence counts, first rows and query
//                 blocks of the attention.
// k_pf_attn_pair  causal attention of one block of queries of one sequence against
//                 that sequence's loop-r cache on the tensor cores (head_dim 64, 128).
// k_pf_attn       the same for head_dim 32, one block of QB queries
//                 against that sequence's loop-r cache, for the G query heads of
//                 one kv head; K is staged transposed in shared memory so each
//                 lane scores whole keys, online softmax in float32 (base 2).
// k_pf_len        cache lengths += tokens of the chunk that ran each loop.
#include "tlf_internal.cuh"

namespace tlf {

constexpr int PF_QB = 32;       // queries per attention block
constexpr int PF_WARPS = 8;     // 4 queries per warp

// Exclusive scan over a block of up to 1024 threads (one value per thread).
__device__ int pf_block_scan(int v, int* total, int* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int t = (lane < nw) ? warp_tot[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    if (lane < nw) warp_tot[lane] = t;
    if (lane == 31) warp_tot[32] = t;
  }
  __syncthreads();
  const int excl = x - v + (warp > 0 ? warp_tot[warp - 1] : 0);
  *total = warp_tot[32];
  __syncthreads();
  return excl;
}

// One CTA per loop (the loops' lists are independent). A thread owns eight consecutive tokens, whose depths
// stay in registers, so a chunk of up to 8192 tokens is counted and compacted in one pass (one CTA over all loops
// took 61 us for 8192 tokens and six loops, most of it in the scans' barriers).
__global__ void __launch_bounds__(1024) k_pf_plan(ModelDims md, PrefillDev p) {
  __shared__ int warp_tot[33];
  __shared__ int cnt_s[1024];
  __shared__ int first_s[1024];
  __shared__ int s0_s[1024];
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, T = p.T, S = p.S, C = p.C, M = md.M, r = blockIdx.x;
  constexpr int PER = 8;
  if (tid < S) cnt_s[tid] = 0;
  __syncthreads();
  for (int base = 0; base < T; base += PER * 1024) {
    const int t0 = base + tid * PER;
    int run = 0, sq = -1;  // tokens are ordered by sequence: one addition per run of a sequence
    for (int e = 0; e < PER && t0 + e < T; ++e) {
      const int q = p.seqidx[t0 + e];
      if (q != sq) {
        if (run) atomicAdd(&cnt_s[sq], run);
        run = 0;
        sq = q;
      }
      run += p.m[t0 + e] > r;
    }
    if (run) atomicAdd(&cnt_s[sq], run);
  }
  __syncthreads();
  const int v = tid < S ? cnt_s[tid] : 0;
  int n_r;
  const int first = pf_block_scan(v, &n_r, warp_tot);
  const int qb = (v + p.qblock - 1) / p.qblock;
  int tiles;
  const int tb = pf_block_scan(qb, &tiles, warp_tot);
  if (tid < S) {
    first_s[tid] = first;
    s0_s[tid] = p.len[p.seq_slot[tid] * M + r];
    p.first[r * p.Smax + tid] = first;
    p.cnt[r * p.Smax + tid] = v;
    p.s0[r * p.Smax + tid] = s0_s[tid];
    p.tile_base[r * (p.Smax + 1) + tid] = tb;
  }
  if (tid == 0) {
    p.n[r] = n_r;
    p.tile_base[r * (p.Smax + 1) + S] = tiles;
  }
  __syncthreads();
  int running = 0;
  for (int base = 0; base < T; base += PER * 1024) {
    const int t0 = base + tid * PER;
    unsigned act = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e)
      if (t0 + e < T && p.m[t0 + e] > r) act |= 1u << e;
    int btot;
    int k = running + pf_block_scan(__popc(act), &btot, warp_tot);
#pragma unroll
    for (int e = 0; e < PER; ++e)
      if (act >> e & 1u) {
        const int t = t0 + e, sq = p.seqidx[t];
        p.idx[r * C + k] = t;
        p.row_slot[r * C + k] = p.seq_slot[sq];
        p.row_cslot[r * C + k] = s0_s[sq] + (k - first_s[sq]);
        p.row_pos[r * C + k] = p.pos[t];
        ++k;
      }
    running += btot;
  }
}

template <typename T, int HD, int G>
__global__ void __launch_bounds__(32 * PF_WARPS) k_pf_attn(ModelDims md, PrefillDev p, StepDev s, int r, int j,
                                                           const float* __restrict__ Q, T* __restrict__ O) {
  constexpr int QH = (PF_QB / PF_WARPS) * G;  // query-heads per warp
  constexpr int DPL = HD / 32;                 // output dims per lane
  extern __shared__ float sm[];
  float* Qs = sm;                              // [QB][G][HD]
  float* Kt = Qs + PF_QB * G * HD;             // [HD][65]
  float* Vs = Kt + HD * 65;                    // [64][HD]
  float* Ps = Vs + 64 * HD;                    // [warps][QH][64]

  pdl_wait();
  pdl_trigger();
  const int S = p.S;
  const int* tbase = p.tile_base + r * (p.Smax + 1);
  const int tile = blockIdx.x, kvh = blockIdx.y;
  if (tile >= tbase[S]) return;
  int lo = 0, hi = S;  // sequence: largest sq with tbase[sq] <= tile
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tbase[mid] <= tile) lo = mid; else hi = mid;
  }
  const int sq = lo, qb = tile - tbase[sq];
  const int cnt = p.cnt[r * p.Smax + sq], first = p.first[r * p.Smax + sq], s0 = p.s0[r * p.Smax + sq];
  const int slot = p.seq_slot[sq];
  const int q0 = qb * PF_QB, nq = min(PF_QB, cnt - q0);
  const int last = s0 + q0 + nq - 1;  // cache slot of the block's last query
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float scale = 1.4426950408889634f * rsqrtf((float)HD);

  for (int e = tid; e < PF_QB * G * HD; e += blockDim.x) {
    const int qi = e / (G * HD), rem = e % (G * HD), g = rem / HD, d = rem % HD;
    Qs[e] = (qi < nq) ? Q[((size_t)(first + q0 + qi) * md.Hq + kvh * G + g) * HD + d] * scale : 0.f;
  }

  float m_run[QH], l_run[QH], acc[QH][DPL];
#pragma unroll
  for (int qh = 0; qh < QH; ++qh) {
    m_run[qh] = -INFINITY;
    l_run[qh] = 0.f;
#pragma unroll
    for (int t = 0; t < DPL; ++t) acc[qh][t] = 0.f;
  }
  const int* ptab = s.page_table + ((size_t)slot * md.M + r) * md.max_pages;
  const int npages = last / 64 + 1;
  for (int pg = 0; pg < npages; ++pg) {
    __syncthreads();  // previous page fully consumed
    const int page = ptab[pg];
    if (page < 0 || page >= md.n_pages) {
      if (tid == 0) atomicOr(s.err, DEVERR_INDEX);
      return;
    }
    const T* kseg = reinterpret_cast<const T*>(s.pool) + (size_t)page * md.page_elems +
                    ((size_t)(j * 2 + 0) * md.Hkv + kvh) * 64 * HD;
    const T* vseg = kseg + (size_t)md.Hkv * 64 * HD;
    const int valid = min(64, last + 1 - pg * 64);
    for (int e = tid; e < 64 * HD; e += blockDim.x) {
      const int key = e / HD, d = e % HD;
      const float kv = key < valid ? to_f32(kseg[e]) : 0.f;
      const float vv = key < valid ? to_f32(vseg[e]) : 0.f;
      Kt[d * 65 + key] = kv;
      Vs[e] = vv;
    }
    __syncthreads();
    // scores of keys lane and lane + 32 for this warp's query-heads
    float sc[QH][2];
#pragma unroll
    for (int qh = 0; qh < QH; ++qh) sc[qh][0] = sc[qh][1] = 0.f;
    const float* qw = Qs + (warp * (PF_QB / PF_WARPS)) * G * HD;  // QH consecutive [G][HD] rows
    for (int d = 0; d < HD; d += 4) {
      float k0[4], k1[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        k0[u] = Kt[(d + u) * 65 + lane];
        k1[u] = Kt[(d + u) * 65 + lane + 32];
      }
#pragma unroll
      for (int qh = 0; qh < QH; ++qh) {
        const float4 q4 = *reinterpret_cast<const float4*>(qw + qh * HD + d);
        sc[qh][0] = fmaf(q4.x, k0[0], fmaf(q4.y, k0[1], fmaf(q4.z, k0[2], fmaf(q4.w, k0[3], sc[qh][0]))));
        sc[qh][1] = fmaf(q4.x, k1[0], fmaf(q4.y, k1[1], fmaf(q4.z, k1[2], fmaf(q4.w, k1[3], sc[qh][1]))));
      }
    }
    float* pw = Ps + warp * QH * 64;
#pragma unroll
    for (int qh = 0; qh < QH; ++qh) {
      const int qi = warp * (PF_QB / PF_WARPS) + qh / G;
      const int qslot = s0 + q0 + qi;
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        const int ks = pg * 64 + lane + 32 * h2;
        if (qi >= nq || ks > qslot) sc[qh][h2] = -INFINITY;  // causal within the cache
      }
      const float pm = warp_max(fmaxf(sc[qh][0], sc[qh][1]));
      if (pm > m_run[qh]) {
        const float cr = exp2f(m_run[qh] - pm);
        l_run[qh] *= cr;
#pragma unroll
        for (int t = 0; t < DPL; ++t) acc[qh][t] *= cr;
        m_run[qh] = pm;
      }
      const float p0 = (sc[qh][0] == -INFINITY) ? 0.f : exp2f(sc[qh][0] - m_run[qh]);
      const float p1 = (sc[qh][1] == -INFINITY) ? 0.f : exp2f(sc[qh][1] - m_run[qh]);
      l_run[qh] += p0 + p1;
      pw[qh * 64 + lane] = p0;
      pw[qh * 64 + lane + 32] = p1;
    }
    __syncwarp();
    for (int key = 0; key < valid; key += 4) {
      float4 pk[QH];
#pragma unroll
      for (int qh = 0; qh < QH; ++qh) pk[qh] = *reinterpret_cast<const float4*>(pw + qh * 64 + key);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float vv[DPL];
#pragma unroll
        for (int t = 0; t < DPL; ++t) vv[t] = Vs[(key + u) * HD + lane + 32 * t];
#pragma unroll
        for (int qh = 0; qh < QH; ++qh) {
          const float pr = u == 0 ? pk[qh].x : (u == 1 ? pk[qh].y : (u == 2 ? pk[qh].z : pk[qh].w));
#pragma unroll
          for (int t = 0; t < DPL; ++t) acc[qh][t] = fmaf(pr, vv[t], acc[qh][t]);
        }
      }
    }
  }
#pragma unroll
  for (int qh = 0; qh < QH; ++qh) {
    const int qi = warp * (PF_QB / PF_WARPS) + qh / G, g = qh % G;
    const float l = warp_sum(l_run[qh]);
    if (qi < nq) {
      T* orow = O + (size_t)(first + q0 + qi) * md.q_dim + (kvh * G + g) * HD;
#pragma unroll
      for (int t = 0; t < DPL; ++t) orow[lane + 32 * t] = from_f32<T>(acc[qh][t] / l);
    }
  }
}

// ----------------------------------------------------------------------------
// Tensor-core causal attention of a chunk (bf16 models, head_dim 64 or 128)
// ----------------------------------------------------------------------------
// One CTA of 256 threads per (sequence, block of QT = 128/G queries, kv head): the 128 MMA rows
// are the G query heads of QT queries (row = query * G + head). For every page of 64 cache slots:
//   S = Q K^T   tcgen05.mma M=128, N=64, K=hd into TMEM; q enters as two bf16 terms (q = hi + lo),
//               so the scores keep q's float32 precision;
//   softmax     two threads share a row (warps w and w+4 reach the same TMEM lanes), each owning
//               32 of its 64 columns: they read S (tcgen05.ld), mask causally by cache slot (only
//               pages on the query's diagonal need the per-key test), exchange the row maximum
//               through shared memory and keep an online softmax in float32 (base 2); P goes to
//               shared memory in bf16;
//   O += P V    tcgen05.mma M=128, N=hd, K=64 accumulating in TMEM.
// The loop is software-pipelined: S has two TMEM buffers and the K / V^T operand tiles two
// shared-memory buffers, so the S product of page p+1 runs on the tensor cores while the threads
// do the softmax of page p, and the re-layout of page p+1 overlaps the P V product of page p.
// The running maximum is refreshed lazily: O (TMEM load, scale, store) and the row sum are
// rescaled only when a row's maximum grows by more than 8 (a factor of 256), so exponentials stay
// below 256 and rescaling is rare. The K and V segments of each page arrive by 1-D bulk copies in
// a two-deep staging ring; threads rewrite them into the swizzled K-major operand tiles (V
// transposed so that keys run along K), with zeros past the last valid slot.
constexpr int PFT_THREADS = 256;

template <int HD>
struct PfTcShape {
  static constexpr int A_BYTES = 128 * HD * 2;   // one of the hi / lo Q tiles [128][HD]
  static constexpr int BK_BYTES = 64 * HD * 2;   // K tile [64 keys][HD]
  static constexpr int BV_BYTES = HD * 64 * 2;   // V^T tile [HD][64 keys]
  static constexpr int P_BYTES = 128 * 64 * 2;   // P tile [128][64 keys]
  static constexpr int SEG = 64 * HD * 2;        // raw K (or V) segment of a page
  static constexpr int RAW_BYTES = 2 * SEG;
  static constexpr int OFF_AHI = 0;
  static constexpr int OFF_ALO = OFF_AHI + A_BYTES;
  static constexpr int OFF_BK = OFF_ALO + A_BYTES;   // two K tiles
  static constexpr int OFF_BV = OFF_BK + 2 * BK_BYTES;  // two V^T tiles
  static constexpr int OFF_P = OFF_BV + 2 * BV_BYTES;
  static constexpr int OFF_RAW = OFF_P + P_BYTES;
  static constexpr int OFF_BAR = OFF_RAW + 2 * RAW_BYTES;
  static constexpr int OFF_XCH = OFF_BAR + 64;         // [2][128] floats: row maxima, then row sums
  static constexpr int BYTES = OFF_XCH + 1024 + 1024;  // exchange, alignment slack
  static constexpr uint32_t TMEM_COLS = 256;          // S buffers in columns 0..127, O in 128..128+HD
  static constexpr int ACOL = 128 * 128;              // bytes of one 128-byte atom column of a Q tile
  static constexpr int BCOL = 64 * 128;               // ... of a K tile
};

// 2^x with the hardware approximation (relative error ~2^-22; the probabilities are then rounded
// to bf16)
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}


template <int HD, int G>
__global__ void __launch_bounds__(PFT_THREADS) k_pf_attn_tc(ModelDims md, PrefillDev p, StepDev s, int r, int j,
                                                             const float* __restrict__ Q, bf16* __restrict__ O) {
  using Sh = PfTcShape<HD>;
  constexpr int QT = 128 / G;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // staging 0, staging 1, S buffer 0 done, S buffer 1 done, P V done
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + Sh::OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 5);

  pdl_wait();
  const int S = p.S;
  const int* tbase = p.tile_base + r * (p.Smax + 1);
  const int tile = blockIdx.x, kvh = blockIdx.y;
  if (tile >= tbase[S]) return;
  int lo = 0, hi = S;  // sequence: largest sq with tbase[sq] <= tile
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tbase[mid] <= tile) lo = mid; else hi = mid;
  }
  const int sq = lo, qb = tile - tbase[sq];
  const int cnt = p.cnt[r * p.Smax + sq], first = p.first[r * p.Smax + sq], s0 = p.s0[r * p.Smax + sq];
  const int slot = p.seq_slot[sq];
  const int q0 = qb * QT, nq = min(QT, cnt - q0);
  const int last = s0 + q0 + nq - 1;  // cache slot of the block's last query
  const int npages = last / 64 + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quad = warp & 3, half = warp >> 2;  // TMEM lane quadrant and column half of this warp
  const int row = quad * 32 + lane;             // the MMA row (query * G + head) this thread serves
  float* xch = reinterpret_cast<float*>(sm + Sh::OFF_XCH);
  const int* ptab = s.page_table + ((size_t)slot * md.M + r) * md.max_pages;
  const uint32_t stg0 = smem_u32(&bars[0]), stg1 = smem_u32(&bars[1]);
  const uint32_t bar_s0 = smem_u32(&bars[2]), bar_s1 = smem_u32(&bars[3]), bar_o = smem_u32(&bars[4]);

  if (tid == 0) {
    for (int i = 0; i < 5; ++i) mbar_init(smem_u32(&bars[i]), 1);
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(tmem_slot), Sh::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();  // a dependent CTA on this SM could otherwise take the columns that this one still waits for
  const uint32_t tmem = *tmem_slot;
  const uint32_t t_row = tmem + ((uint32_t)(quad * 32) << 16);  // this warp's 32 TMEM lanes
  constexpr uint32_t OCOL = 128;                                 // first TMEM column of O

  bool dead = false;  // a wait of this thread ran out: it waits for nothing more
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (dead || mbar_wait(bar, parity, s.err)) return;
    dead = true;
    drain_copies();
  };
  auto stage_page = [&](int pg) {  // thread 0: K and V segments of page pg into staging buffer pg & 1
    if (dead) return;
    const uint32_t bar = (pg & 1) ? stg1 : stg0;
    const int page = ptab[pg];
    if (page < 0 || page >= md.n_pages) {
      atomicOr(s.err, DEVERR_INDEX);
      mbar_arrive(bar);  // complete the phase without data
      return;
    }
    const bf16* kseg = reinterpret_cast<const bf16*>(s.pool) + (size_t)page * md.page_elems +
                       ((size_t)(j * 2 + 0) * md.Hkv + kvh) * 64 * HD;
    const bf16* vseg = kseg + (size_t)md.Hkv * 64 * HD;
    uint8_t* dst = sm + Sh::OFF_RAW + (pg & 1) * Sh::RAW_BYTES;
    mbar_arrive_expect_tx(bar, Sh::RAW_BYTES);
    bulk_g2s(smem_u32(dst), kseg, Sh::SEG, bar);
    bulk_g2s(smem_u32(dst + Sh::SEG), vseg, Sh::SEG, bar);
  };
  // K tile of page pg (from its staging buffer) into K buffer pg & 1; rows = keys
  auto relayout_k = [&](int pg) {
    wait((pg & 1) ? stg1 : stg0, (pg >> 1) & 1);
    const uint8_t* raw = sm + Sh::OFF_RAW + (pg & 1) * Sh::RAW_BYTES;
    uint8_t* bk = sm + Sh::OFF_BK + (pg & 1) * Sh::BK_BYTES;
    const int valid = min(64, last + 1 - pg * 64);
    for (int e = tid; e < 64 * (HD / 8); e += PFT_THREADS) {
      const int key = e / (HD / 8), c = e % (HD / 8);
      const uint4 v = key < valid ? *reinterpret_cast<const uint4*>(raw + key * HD * 2 + c * 16) : make_uint4(0, 0, 0, 0);
      *reinterpret_cast<uint4*>(bk + (c / 8) * Sh::BCOL + sw128_off(key, c % 8)) = v;
    }
  };
  // V^T tile of page pg into V buffer pg & 1: row = hd index n, chunk c = keys 8c..8c+7
  auto relayout_v = [&](int pg) {
    const uint8_t* raw = sm + Sh::OFF_RAW + (pg & 1) * Sh::RAW_BYTES;
    uint8_t* bv = sm + Sh::OFF_BV + (pg & 1) * Sh::BV_BYTES;
    const int valid = min(64, last + 1 - pg * 64);
    const uint32_t* rv = reinterpret_cast<const uint32_t*>(raw + Sh::SEG);  // [64 keys][HD / 2] pairs
    for (int e = tid; e < (HD / 2) * 8; e += PFT_THREADS) {
      const int n2 = e % (HD / 2), c = e / (HD / 2);  // hd indices 2 n2, 2 n2 + 1; keys 8c..8c+7
      uint32_t x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = 8 * c + u < valid ? rv[(8 * c + u) * (HD / 2) + n2] : 0u;
      uint32_t we[4], wo[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        we[u] = __byte_perm(x[2 * u], x[2 * u + 1], 0x5410);  // low halves: hd index 2 n2
        wo[u] = __byte_perm(x[2 * u], x[2 * u + 1], 0x7632);  // high halves: hd index 2 n2 + 1
      }
      *reinterpret_cast<uint4*>(bv + sw128_off(2 * n2, c)) = make_uint4(we[0], we[1], we[2], we[3]);
      *reinterpret_cast<uint4*>(bv + sw128_off(2 * n2 + 1, c)) = make_uint4(wo[0], wo[1], wo[2], wo[3]);
    }
  };
  constexpr uint32_t IDS = idesc_bf16_f32(128, 64), IDO = idesc_bf16_f32(128, HD);
  auto issue_s = [&](int pg) {  // thread 0: S of page pg into TMEM columns 64 * (pg & 1)
    tc_fence_after();
    const uint32_t bk = smem_u32(sm + Sh::OFF_BK + (pg & 1) * Sh::BK_BYTES);
#pragma unroll
    for (int kc = 0; kc < HD / 64; ++kc)
#pragma unroll
      for (int k = 0; k < 4; ++k) {  // K = 16 per MMA: +32 bytes (encoded +2) inside the atom column
        const uint64_t db = smem_desc_sw128(bk + kc * Sh::BCOL) + 2 * k;
        const uint32_t d = tmem + 64u * (uint32_t)(pg & 1);
        tc_mma_f16(d, smem_desc_sw128(smem_u32(sm + Sh::OFF_AHI + kc * Sh::ACOL)) + 2 * k, db, IDS, (kc | k) ? 1u : 0u);
        tc_mma_f16(d, smem_desc_sw128(smem_u32(sm + Sh::OFF_ALO + kc * Sh::ACOL)) + 2 * k, db, IDS, 1u);
      }
    tc_commit((pg & 1) ? bar_s1 : bar_s0);
  };

  if (tid == 0) {
    stage_page(0);
    if (npages > 1) stage_page(1);
  }

  // Q tile: row = query * G + head, as hi and lo bf16 parts (zeros past the block's queries)
  for (int e = tid; e < 128 * (HD / 8); e += PFT_THREADS) {
    const int qr = e / (HD / 8), c = e % (HD / 8);
    const int qq = qr / G, gg = qr % G;
    float x[8];
    if (qq < nq) {
      const float4* q4 = reinterpret_cast<const float4*>(Q + ((size_t)(first + q0 + qq) * md.Hq + kvh * G + gg) * HD);
      const float4 a = q4[2 * c], b = q4[2 * c + 1];
      x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = 0.f;
    }
    uint32_t h[4], l[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float a0 = __bfloat162float(__float2bfloat16_rn(x[2 * u]));
      const float a1 = __bfloat162float(__float2bfloat16_rn(x[2 * u + 1]));
      h[u] = pack_bf16(a0, a1);
      l[u] = pack_bf16(x[2 * u] - a0, x[2 * u + 1] - a1);
    }
    const uint32_t off = (c / 8) * Sh::ACOL + sw128_off(qr, c % 8);
    *reinterpret_cast<uint4*>(sm + Sh::OFF_AHI + off) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(sm + Sh::OFF_ALO + off) = make_uint4(l[0], l[1], l[2], l[3]);
  }
  const int qi = row / G, g = row % G;
  const bool row_ok = qi < nq;
  // prologue: page 0's operand tiles and its S product
  relayout_k(0);
  relayout_v(0);
  fence_proxy_async_smem();
  __syncthreads();
  if (tid == 0) {
    if (npages > 2) stage_page(2);  // staging buffer 0 has been read
    issue_s(0);
  }
  __syncwarp();

  const int qslot = s0 + q0 + qi;  // cache slot of this row's query
  const float scale = 1.4426950408889634f * rsqrtf((float)HD);
  float m_run = -INFINITY, l_run = 0.f;

  for (int pg = 0; pg < npages; ++pg) {
    const bool more = pg + 1 < npages;
    // operand tiles of page pg+1: its K buffer was last read by S of page pg-1 (complete), its V^T
    // buffer by P V of page pg-1, which also frees P and lets O be rescaled
    if (more) relayout_k(pg + 1);
    if (pg > 0) wait(bar_o, (pg - 1) & 1);
    if (more) relayout_v(pg + 1);
    fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0 && more) {
      if (pg + 3 < npages) stage_page(pg + 3);  // staging buffer (pg+1) & 1 has been read
      issue_s(pg + 1);
    }
    __syncwarp();
    wait((pg & 1) ? bar_s1 : bar_s0, (pg >> 1) & 1);
    tc_fence_after();

    // this thread's 32 columns of the row
    float sc[32];
    tmem_ld_16(t_row + 64u * (uint32_t)(pg & 1) + 32u * half, sc);
    tmem_ld_16(t_row + 64u * (uint32_t)(pg & 1) + 32u * half + 16u, sc + 16);
    const int valid = min(64, last + 1 - pg * 64);
    const int kb = pg * 64 + 32 * half;  // cache slot of this thread's first column
    float pm = -INFINITY;
    if (row_ok && kb + 31 <= qslot && 32 * half + 31 < valid) {  // every key visible
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        sc[c] *= scale;
        pm = fmaxf(pm, sc[c]);
      }
    } else if (!row_ok || kb > qslot || 32 * half >= valid) {  // none visible
#pragma unroll
      for (int c = 0; c < 32; ++c) sc[c] = -INFINITY;
    } else {  // the diagonal: causal by cache slot
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const bool use = 32 * half + c < valid && kb + c <= qslot;
        sc[c] = use ? sc[c] * scale : -INFINITY;
        pm = fmaxf(pm, sc[c]);
      }
    }
    xch[half * 128 + row] = pm;
    __syncthreads();
    pm = fmaxf(pm, xch[(half ^ 1) * 128 + row]);
    // lazy maximum: rescale only when it grows by more than 8 (warp-uniform TMEM access); both
    // threads of a row take the same decision, each for its half of O and of the row sum
    const bool grow = pm > m_run + 8.f;
    const float cr = grow ? exp2f(m_run - pm) : 1.f;  // 0 when m_run was -inf
    if (__any_sync(0xffffffffu, grow) && pg > 0) {
#pragma unroll
      for (int c0 = 0; c0 < HD / 2; c0 += 16) {
        float o[16];
        tmem_ld_16(t_row + OCOL + (uint32_t)(half * (HD / 2) + c0), o);
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] *= cr;
        tmem_st_16(t_row + OCOL + (uint32_t)(half * (HD / 2) + c0), o);
      }
    }
    if (grow) {
      l_run *= cr;
      m_run = pm;
    }
    uint32_t pk[16];
    float psum = 0.f;
#pragma unroll
    for (int c = 0; c < 32; c += 2) {
      const float p0 = sc[c] == -INFINITY ? 0.f : ex2_approx(sc[c] - m_run);
      const float p1 = sc[c + 1] == -INFINITY ? 0.f : ex2_approx(sc[c + 1] - m_run);
      psum += p0 + p1;
      pk[c / 2] = pack_bf16(p0, p1);
    }
    l_run += psum;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<uint4*>(sm + Sh::OFF_P + sw128_off(row, 4 * half + q)) =
          make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      const uint32_t bv = smem_u32(sm + Sh::OFF_BV + (pg & 1) * Sh::BV_BYTES);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        tc_mma_f16(tmem + OCOL, smem_desc_sw128(smem_u32(sm + Sh::OFF_P)) + 2 * k, smem_desc_sw128(bv) + 2 * k, IDO,
                   (pg > 0 || k > 0) ? 1u : 0u);
      tc_commit(bar_o);
    }
    __syncwarp();
  }
  wait(bar_o, (npages - 1) & 1);
  tc_fence_after();
  xch[half * 128 + row] = l_run;  // the two halves of each row sum
  __syncthreads();
  const float l_tot = l_run + xch[(half ^ 1) * 128 + row];
  const float inv_l = l_tot > 0.f ? 1.f / l_tot : 0.f;
  bf16* orow = O + (size_t)(first + q0 + qi) * md.q_dim + (kvh * G + g) * HD + half * (HD / 2);
#pragma unroll
  for (int c0 = 0; c0 < HD / 2; c0 += 16) {
    float o[16];
    tmem_ld_16(t_row + OCOL + (uint32_t)(half * (HD / 2) + c0), o);
    if (row_ok) {
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = pack_bf16(o[2 * i] * inv_l, o[2 * i + 1] * inv_l);
      *reinterpret_cast<uint4*>(orow + c0) = make_uint4(w[0], w[1], w[2], w[3]);
      *reinterpret_cast<uint4*>(orow + c0 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, Sh::TMEM_COLS);
}

// ----------------------------------------------------------------------------
// Tensor-core causal attention of a chunk, two query tiles a CTA (bf16, head_dim 64 or 128)
// ----------------------------------------------------------------------------
// One CTA per (sequence, block of 2 x 128/G queries, kv head). The block is two tiles of 128 MMA rows
// (row = query * G + head) that share every K/V block of 128 cache slots (two pages), so that the tensor
// cores work on one tile while the other tile's softmax runs:
//   warps 0-3, 4-7  softmax of tile 0 and 1, one thread per row: read the row of S from TMEM, mask causally by
//                   cache slot, keep the running maximum (refreshed lazily: O is rescaled in TMEM only when a
//                   row's maximum grows by more than 8 in base 2) and sum in float32, write P in bf16 back to
//                   TMEM, where it is the A operand of the P V product; at the end normalise O and store it;
//   warp 8          TMA producer: the tiles' q rows as bf16 hi and lo planes (the scores keep q's float32
//                   precision), then K and V of every block through 3-D tensor maps into one ring;
//   warp 9          MMA issuer: S = Qhi K^T + Qlo K^T, O += P V with V taken as an MN-major operand.
// mbarriers connect the roles; every wait is bounded. A block past a sequence's last page loads its last
// page twice. Slots past the last query may hold anything (a released page keeps its entries), and P = 0 does not
// cancel an infinity, so warp 8 zeroes them in the last block's V while the softmax runs. (Products that end with a
// tile's last query instead cost the issuing thread 2 % of a prompt of 8192 tokens.)
//
// What bounds it: at head_dim 128 a block of a tile is 1536 cycles of MMAs (two S products for q's two terms, one P
// V) against about 1024 of exponentials, so the tiles' softmaxes hide behind each other's MMAs; at head_dim 64 the
// exponentials lead. Measured at 8192 causal rows: 310 us for 16 / 8 heads x 128 (890 useful TFLOP/s, 1330 counted
// with both q terms, 0.70 of the measured bf16 rate; one tile of 128 rows and 64-key pages a CTA took 549 us), and 67
// us for eight prompts of about 1000 rows, 16 heads x 64 (104 us). Scalar bf16 conversions instead of packed ones cost
// 8 %.
//
// Layouts: TMEM holds S of both tiles (128 columns each) and O of both (head_dim columns each). With
// head_dim 128 that is all 512 columns, so P overwrites its S; tcgen05 executes one thread's MMAs in
// order, so the next S of a tile may be issued right behind the P V product that reads P. With head_dim 64
// P has columns of its own and the next S is issued as soon as the softmax has read the one before.
constexpr int PFA_THREADS = 320;

template <int HD>
struct PfaShape {
  static constexpr int ATOMS = HD / 64;               // 128-byte atom columns of a row
  static constexpr int COL = 128 * 128;               // bytes of one atom column of 128 rows
  static constexpr int T_BYTES = ATOMS * COL;         // a tile of 128 rows: Q hi, Q lo, K or V
  static constexpr int NST = HD == 128 ? 3 : 8;       // K/V ring
  static constexpr int OFF_Q = 0;                     // tile 0 hi, lo, tile 1 hi, lo
  static constexpr int OFF_KV = 4 * T_BYTES;
  static constexpr int OFF_BAR = OFF_KV + NST * T_BYTES;
  static constexpr int NBAR = 2 * NST + 2 + 9;
  static constexpr int BYTES = OFF_BAR + NBAR * 8 + 16 + 1024;  // barriers, TMEM slot, alignment slack
  static constexpr bool SEP_P = HD == 64;
  static constexpr uint32_t SCOL = 0, OCOL = 256, PCOL = SEP_P ? 384 : 0;
  static constexpr uint32_t P_STEP = SEP_P ? 64 : 128;  // columns from tile 0's P to tile 1's
  static_assert(BYTES <= 232448, "shared memory of one CTA");
};

// D(tmem) (+)= A(tmem) * B(smem desc)
__device__ __forceinline__ void tc_mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// 32 lanes x 32-bit, 16 consecutive columns per thread, register -> TMEM; completes at tmem_st_wait().
__device__ __forceinline__ void tmem_st_16_issue(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

template <int HD, int G>
__global__ void __launch_bounds__(PFA_THREADS, 1) k_pf_attn_pair(ModelDims md, PrefillDev p, StepDev s, int r, int j,
                                                                 bf16* __restrict__ O,
                                                                 const __grid_constant__ CUtensorMap q_map,
                                                                 const __grid_constant__ CUtensorMap pool_map) {
  using Sh = PfaShape<HD>;
  constexpr int QT = 128 / G, NST = Sh::NST;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + Sh::OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + Sh::NBAR);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto bar = [&](int i) { return smem_u32(&bars[i]); };
  auto kv_full = [&](int st) { return bar(st); };
  auto kv_empty = [&](int st) { return bar(NST + st); };
  const uint32_t q_full0 = bar(2 * NST);                          // one per tile
  auto s_full = [&](int x) { return bar(2 * NST + 2 + x); };  // S of tile x written
  auto s_read = [&](int x) { return bar(2 * NST + 4 + x); };  // ... read by its softmax (SEP_P)
  auto p_full = [&](int x) { return bar(2 * NST + 6 + x); };  // P of tile x written
  auto o_done = [&](int x) { return bar(2 * NST + 8 + x); };  // its P V product done
  const uint32_t v_tail = bar(2 * NST + 10);                  // the last block's V zeroed behind the last query

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < NST; ++i) {
      mbar_init(kv_full(i), 1);
      mbar_init(kv_empty(i), 1);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(q_full0 + 8 * x, 1);
      mbar_init(s_full(x), 1);
      mbar_init(s_read(x), 4);
      mbar_init(p_full(x), 4);
      mbar_init(o_done(x), 1);
    }
    mbar_init(v_tail, 32);
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tensormap(&q_map);
    prefetch_tensormap(&pool_map);
  }
  if (warp == 9) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  pdl_wait();
  const int S = p.S;
  const int* tbase = p.tile_base + r * (p.Smax + 1);
  // 1-D grid, kv head fastest and query blocks in reverse order: the blocks with the most pages
  // (the last queries of a sequence) are dispatched first, so the last wave holds short ones
  const int ntiles = tbase[S];
  const int kvh = blockIdx.x % md.Hkv, tile = ntiles - 1 - (int)(blockIdx.x / md.Hkv);
  int lo = 0, hi = S;  // sequence: largest sq with tbase[sq] <= tile
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tbase[mid] <= tile) lo = mid; else hi = mid;
  }
  const int sq = lo, qb = tile < 0 ? 0 : tile - tbase[sq];
  const int cnt = p.cnt[r * p.Smax + sq], first = p.first[r * p.Smax + sq], s0 = p.s0[r * p.Smax + sq];
  const int slot = p.seq_slot[sq];
  const int q0 = qb * 2 * QT;
  // queries and key blocks of the two tiles (tile 1 may have none)
  const int nq0 = tile < 0 ? 0 : min(QT, cnt - q0), nq1 = tile < 0 ? 0 : max(0, min(QT, cnt - q0 - QT));
  const int nb0 = nq0 > 0 ? (s0 + q0 + nq0 - 1) / 128 + 1 : 0;
  const int nb1 = nq1 > 0 ? (s0 + q0 + QT + nq1 - 1) / 128 + 1 : 0;
  const int nb = max(nb0, nb1);
  const int last_page = (s0 + q0 + nq0 + nq1 - 1) / 64;
  tc_fence_before();
  __syncthreads();  // barriers initialised, TMEM allocated
  tc_fence_after();
  pdl_trigger();  // not before: a dependent CTA on this SM could take the columns that warp 9 still waits for
  const uint32_t tmem = *tmem_slot;
  // a bounded wait; once any role has given up, the others skip their waits and wind down
  auto wait = [&](uint32_t b, uint32_t parity) {
    if (*abort_flag) return false;
    if (!mbar_wait(b, parity, s.err)) {
      *abort_flag = 1;
      return false;
    }
    return true;
  };

  if (warp == 8) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      for (int x = 0; x < 2; ++x) {
        if (x == 1 && nq1 == 0) break;
        if (nq0 == 0) break;
        mbar_arrive_expect_tx(q_full0 + 8 * x, 2 * Sh::T_BYTES);
#pragma unroll
        for (int pl = 0; pl < 2; ++pl)
#pragma unroll
          for (int a = 0; a < Sh::ATOMS; ++a)
            tma_load_3d(smem_u32(sm + Sh::OFF_Q + (2 * x + pl) * Sh::T_BYTES + a * Sh::COL), &q_map, a * 64, kvh * G,
                        first + q0 + x * QT + pl * p.C, q_full0 + 8 * x);
      }
      const int* ptab = s.page_table + ((size_t)slot * md.M + r) * md.max_pages;
      const int rowK = ((j * 2 + 0) * md.Hkv + kvh) * 64, rowV = ((j * 2 + 1) * md.Hkv + kvh) * 64;
      bool ok = true;
      for (int i = 0; i < 2 * nb && ok; ++i) {  // K(0), V(0), K(1), V(1), ...
        const int st = i % NST, kb = i >> 1;
        if (i >= NST && !wait(kv_empty(st), (uint32_t)(i / NST - 1) & 1u)) break;
        int pg[2] = {ptab[2 * kb], ptab[min(2 * kb + 1, last_page)]};
        const bool okp = pg[0] >= 0 && pg[0] < md.n_pages && pg[1] >= 0 && pg[1] < md.n_pages;
        if (!okp) {
          atomicOr(s.err, DEVERR_INDEX);
          mbar_arrive(kv_full(st));  // complete the phase without data
          continue;
        }
        mbar_arrive_expect_tx(kv_full(st), Sh::T_BYTES);
        uint8_t* dst = sm + Sh::OFF_KV + st * Sh::T_BYTES;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int a = 0; a < Sh::ATOMS; ++a)
            tma_load_3d(smem_u32(dst + a * Sh::COL + h * (Sh::COL / 2)), &pool_map, a * 64, (i & 1) ? rowV : rowK, pg[h],
                        kv_full(st));
      }
    }
    __syncwarp();
    if (nb > 0) {
      // the last block's V behind the last query (a row of 128 bytes keeps its place in the swizzle)
      const int st = (2 * nb - 1) % NST, valid = s0 + q0 + nq0 + nq1 - (nb - 1) * 128;
      if (valid < 128) wait(kv_full(st), (uint32_t)((2 * nb - 1) / NST) & 1u);
      uint8_t* v = sm + Sh::OFF_KV + st * Sh::T_BYTES;
#pragma unroll 1
      for (int i = valid * 8 + lane; i < 1024; i += 32)
#pragma unroll
        for (int a = 0; a < Sh::ATOMS; ++a) *reinterpret_cast<uint4*>(v + a * Sh::COL + i * 16) = make_uint4(0, 0, 0, 0);
      fence_proxy_async_smem();
      mbar_arrive(v_tail);
    }
    __syncwarp();
  } else if (warp == 9) {
    // ---------------- MMA issuer ----------------
    if (lane == 0 && nb > 0) {
      constexpr uint32_t IDS = idesc_bf16_f32(128, 128), IDO = idesc_bf16_f32_bmn(128, HD);
      constexpr uint64_t T_E = Sh::T_BYTES >> 4, COL_E = Sh::COL >> 4, V16_E = 2048 >> 4;
      const uint64_t dq = smem_desc_sw128(smem_u32(sm + Sh::OFF_Q));
      const uint64_t dk = smem_desc_sw128(smem_u32(sm + Sh::OFF_KV));
      const uint64_t dv = smem_desc_sw128_mn(smem_u32(sm + Sh::OFF_KV), Sh::COL);
      auto issue_s = [&](int x, int kb) {
        const uint64_t kd = dk + (uint64_t)((2 * kb) % NST) * T_E, qd = dq + (uint64_t)(2 * x) * T_E;
        const uint32_t d = tmem + Sh::SCOL + 128u * (uint32_t)x;
#pragma unroll
        for (int pl = 0; pl < 2; ++pl)
#pragma unroll
          for (int kc = 0; kc < Sh::ATOMS; ++kc)
#pragma unroll
            for (int k = 0; k < 4; ++k)  // K = 16 per MMA: +32 bytes (encoded +2) inside the atom column
              tc_mma_f16(d, qd + pl * T_E + kc * COL_E + 2 * k, kd + kc * COL_E + 2 * k, IDS, (pl | kc | k) ? 1u : 0u);
        tc_commit(s_full(x));
      };
      auto issue_pv = [&](int x, int kb) {
        const uint64_t vd = dv + (uint64_t)((2 * kb + 1) % NST) * T_E;
        const uint32_t d = tmem + Sh::OCOL + (uint32_t)(HD * x), pa = tmem + Sh::PCOL + Sh::P_STEP * (uint32_t)x;
#pragma unroll
        for (int k = 0; k < 8; ++k)  // K = 16 keys per MMA: 8 TMEM columns of P, +2048 B (16 rows) of V
          tc_mma_f16_ts(d, pa + 8u * k, vd + V16_E * k, IDO, (kb > 0 || k > 0) ? 1u : 0u);
        tc_commit(o_done(x));
      };
      auto kfull = [&](int kb) { return wait(kv_full((2 * kb) % NST), (uint32_t)(2 * kb / NST) & 1u); };
      auto vfull = [&](int kb) { return wait(kv_full((2 * kb + 1) % NST), (uint32_t)((2 * kb + 1) / NST) & 1u); };
      bool ok = wait(q_full0, 0) && kfull(0);
      if (ok) {
        tc_fence_after();
        issue_s(0, 0);
        if (nb1 > 0) {
          ok = wait(q_full0 + 8, 0);
          tc_fence_after();
          if (ok) issue_s(1, 0);
        }
        tc_commit(kv_empty(0));
      }
      for (int kb = 0; kb < nb && ok; ++kb) {
        const bool next = kb + 1 < nb;
        if (Sh::SEP_P && next) {
          // both next S products first: each waits only for the softmax to have read the S before
          ok = kfull(kb + 1);
          for (int x = 0; x < 2 && ok; ++x)
            if (kb + 1 < (x ? nb1 : nb0)) {
              ok = wait(s_read(x), (uint32_t)kb & 1u);
              if (!ok) break;
              tc_fence_after();
              issue_s(x, kb + 1);
            }
          if (!ok) break;
          tc_commit(kv_empty((2 * kb + 2) % NST));
        }
        if (!vfull(kb) || (!next && !wait(v_tail, 0))) break;
        for (int x = 0; x < 2 && ok; ++x) {
          if (kb < (x ? nb1 : nb0)) {
            ok = wait(p_full(x), (uint32_t)kb & 1u);
            if (!ok) break;
            tc_fence_after();
            issue_pv(x, kb);
            if (x == 1 || nb1 <= kb) tc_commit(kv_empty((2 * kb + 1) % NST));
          }
          if (!Sh::SEP_P && kb + 1 < (x ? nb1 : nb0)) {
            ok = kfull(kb + 1);
            if (!ok) break;
            tc_fence_after();
            issue_s(x, kb + 1);
          }
        }
        if (!Sh::SEP_P && ok && next) tc_commit(kv_empty((2 * kb + 2) % NST));
      }
    }
    __syncwarp();
  } else {
    // ---------------- softmax: thread = MMA row = TMEM lane ----------------
    const int x = warp >> 2, quad = warp & 3, row = quad * 32 + lane;
    const uint32_t lane_off = (uint32_t)(quad * 32) << 16;
    const uint32_t t_s = tmem + lane_off + Sh::SCOL + 128u * (uint32_t)x;
    const uint32_t t_p = tmem + lane_off + Sh::PCOL + Sh::P_STEP * (uint32_t)x;
    const uint32_t t_o = tmem + lane_off + Sh::OCOL + (uint32_t)(HD * x);
    const int nbx = x ? nb1 : nb0, nqx = x ? nq1 : nq0;
    const int qi = row / G, g = row % G;
    const bool row_ok = qi < nqx;
    // cache slot of this row's query (-1: a row past the tile's queries, which sees no key)
    const int qslot = row_ok ? s0 + q0 + x * QT + qi : -1;
    const float scale = 1.4426950408889634f * rsqrtf((float)HD);
    float m_run = -INFINITY, l_run = 0.f;  // in units of the raw scores
    const float grow_by = 8.f / scale;
    bool ok = true;
    // waits taken by the whole warp: the TMEM accesses after them are warp-collective
    auto wait_w = [&](uint32_t b, uint32_t parity) { return __all_sync(0xffffffffu, wait(b, parity)); };
    for (int kb = 0; kb < nbx; ++kb) {
      if (!wait_w(s_full(x), (uint32_t)kb & 1u)) { ok = false; break; }
      tc_fence_after();
      uint32_t su[128];
#pragma unroll
      for (int c = 0; c < 128; c += 32) tmem_ld_32_issue(t_s + (uint32_t)c, su + c);
      tmem_ld_wait();
      if (Sh::SEP_P) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(s_read(x));
      }
      const int vis = qslot - kb * 128;  // columns 0..vis are visible
      float pm4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      if (__any_sync(0xffffffffu, vis < 127)) {
#pragma unroll
        for (int c = 0; c < 128; ++c)
          if (c > vis) su[c] = 0xff800000u;  // -inf
      }
#pragma unroll
      for (int c = 0; c < 128; ++c) pm4[c & 3] = fmaxf(pm4[c & 3], __uint_as_float(su[c]));
      const float pm = fmaxf(fmaxf(pm4[0], pm4[1]), fmaxf(pm4[2], pm4[3]));
      // lazy maximum: O is rescaled only when a row's maximum grows by more than 8 in base 2, after the
      // P V product before has landed (warp-uniform TMEM access)
      const bool grow = pm > m_run + grow_by;
      const float cr = grow ? exp2f((m_run - pm) * scale) : 1.f;  // 0 when m_run was -inf
      if (kb > 0 && (Sh::SEP_P || __any_sync(0xffffffffu, grow))) {
        if (!wait_w(o_done(x), (uint32_t)(kb - 1) & 1u)) { ok = false; break; }  // (with its own columns, P is free too)
        tc_fence_after();
        if (__any_sync(0xffffffffu, grow)) {
#pragma unroll
          for (int c0 = 0; c0 < HD; c0 += 16) {
            float o[16];
            tmem_ld_16(t_o + (uint32_t)c0, o);
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] *= cr;
            tmem_st_16(t_o + (uint32_t)c0, o);
          }
        }
      }
      if (grow) {
        l_run *= cr;
        m_run = pm;
      }
      const float mref = m_run == -INFINITY ? 0.f : m_run * scale;  // rows with no visible key so far: any finite value
      float ps4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c0 = 0; c0 < 128; c0 += 32) {
        uint32_t pk[16];
#pragma unroll
        for (int c = 0; c < 32; c += 2) {
          const float p0 = ex2_approx(fmaf(__uint_as_float(su[c0 + c]), scale, -mref));
          const float p1 = ex2_approx(fmaf(__uint_as_float(su[c0 + c + 1]), scale, -mref));
          ps4[(c >> 1) & 3] += p0 + p1;
          pk[c / 2] = pack_bf16(p0, p1);
        }
        tmem_st_16_issue(t_p + (uint32_t)(c0 / 2), pk);
      }
      l_run += (ps4[0] + ps4[1]) + (ps4[2] + ps4[3]);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full(x));
    }
    // the last P V product, then O / l out
    if (ok && nbx > 0 && wait_w(o_done(x), (uint32_t)(nbx - 1) & 1u)) {
      tc_fence_after();
      const float inv_l = l_run > 0.f ? 1.f / l_run : 0.f;
      bf16* orow = O + (size_t)(first + q0 + x * QT + qi) * md.q_dim + (kvh * G + g) * HD;
#pragma unroll
      for (int c0 = 0; c0 < HD; c0 += 32) {
        float o[32];
        tmem_ld_32(t_o + (uint32_t)c0, o);
        if (row_ok) {
#pragma unroll
          for (int i = 0; i < 32; i += 8)
            *reinterpret_cast<uint4*>(orow + c0 + i) =
                make_uint4(pack_bf16(o[i] * inv_l, o[i + 1] * inv_l), pack_bf16(o[i + 2] * inv_l, o[i + 3] * inv_l),
                           pack_bf16(o[i + 4] * inv_l, o[i + 5] * inv_l), pack_bf16(o[i + 6] * inv_l, o[i + 7] * inv_l));
        }
      }
    }
  }
  if (*abort_flag) drain_copies();
  tc_fence_before();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem, 512);
}

__global__ void k_pf_len(ModelDims md, PrefillDev p) {
  pdl_wait();
  pdl_trigger();
  for (int e = threadIdx.x; e < p.S * md.M; e += blockDim.x) {
    const int sq = e / md.M, r = e % md.M;
    p.len[p.seq_slot[sq] * md.M + r] += p.cnt[r * p.Smax + sq];
  }
}

template <typename T, int HD, int G>
static void pf_attn_launch(const ModelDims& md, const PrefillDev& p, const StepDev& s, int r, int j, const float* Q,
                           void* O, int tiles_bound, cudaStream_t st) {
  constexpr int smem = (PF_QB * G * HD + HD * 65 + 64 * HD + PF_WARPS * (PF_QB / PF_WARPS) * G * 64) * 4;
  (void)ensure_kernel_attrs((const void*)k_pf_attn<T, HD, G>, smem);  // a failure shows at launch
  launch_k(k_pf_attn<T, HD, G>, dim3(tiles_bound, md.Hkv), 32 * PF_WARPS, smem, st, md, p, s, r, j, Q, (T*)O);
}

void launch_pf_plan(const ModelDims& md, const PrefillDev& p, cudaStream_t st) {
  launch_k(k_pf_plan, md.M, 1024, 0, st, md, p);
}

template <int HD, int G>
static void pf_attn_tc_launch(const ModelDims& md, const PrefillDev& p, const StepDev& s, int r, int j,
                              const float* Q, void* O, int tiles_bound, cudaStream_t st) {
  constexpr int smem = PfTcShape<HD>::BYTES;
  (void)ensure_kernel_attrs((const void*)k_pf_attn_tc<HD, G>, smem);  // a failure shows at launch
  launch_k(k_pf_attn_tc<HD, G>, dim3(tiles_bound, md.Hkv), PFT_THREADS, smem, st, md, p, s, r, j, Q, (bf16*)O);
}

template <int HD, int G>
static void pf_attn_pair_launch(const ModelDims& md, const PrefillDev& p, const StepDev& s, int r, int j, void* O,
                                int tiles_bound, cudaStream_t st, const CUtensorMap* q_map, const CUtensorMap* pool_map) {
  constexpr int smem = PfaShape<HD>::BYTES;
  (void)ensure_kernel_attrs((const void*)k_pf_attn_pair<HD, G>, smem);  // a failure shows at launch
  launch_k(k_pf_attn_pair<HD, G>, dim3(tiles_bound * md.Hkv), PFA_THREADS, smem, st, md, p, s, r, j, (bf16*)O, *q_map,
           *pool_map);
}

// Tensor-core kernel for head_dim 64 and 128 (128-byte rows for the swizzled operand tiles); the
// CUDA-core kernel for head_dim 32.
static bool pf_attn_uses_tc(const ModelDims& md) { return md.hd == 64 || md.hd == 128; }

int pf_attn_qblock(const ModelDims& md, bool pair) {
  return pf_attn_uses_tc(md) ? (pair ? 256 : 128) / (md.Hq / md.Hkv) : PF_QB;
}

void launch_pf_attn_pair(const ModelDims& md, const PrefillDev& p, const StepDev& s, int r, int j, void* O,
                         int tiles_bound, cudaStream_t st, const CUtensorMap* q_map, const CUtensorMap* pool_map) {
  const int G = md.Hq / md.Hkv;
  if (md.hd == 128 && G == 1) pf_attn_pair_launch<128, 1>(md, p, s, r, j, O, tiles_bound, st, q_map, pool_map);
  else if (md.hd == 128 && G == 2) pf_attn_pair_launch<128, 2>(md, p, s, r, j, O, tiles_bound, st, q_map, pool_map);
  else if (md.hd == 128) pf_attn_pair_launch<128, 4>(md, p, s, r, j, O, tiles_bound, st, q_map, pool_map);
  else if (G == 1) pf_attn_pair_launch<64, 1>(md, p, s, r, j, O, tiles_bound, st, q_map, pool_map);
  else if (G == 2) pf_attn_pair_launch<64, 2>(md, p, s, r, j, O, tiles_bound, st, q_map, pool_map);
  else pf_attn_pair_launch<64, 4>(md, p, s, r, j, O, tiles_bound, st, q_map, pool_map);
}

void launch_pf_attn(const ModelDims& md, const PrefillDev& p, const StepDev& s, int r, int j, const float* Q,
                    void* O, int tiles_bound, cudaStream_t st) {
  const int G = md.Hq / md.Hkv;
  if (md.hd == 128 && G == 1) pf_attn_tc_launch<128, 1>(md, p, s, r, j, Q, O, tiles_bound, st);
  else if (md.hd == 128 && G == 2) pf_attn_tc_launch<128, 2>(md, p, s, r, j, Q, O, tiles_bound, st);
  else if (md.hd == 128 && G == 4) pf_attn_tc_launch<128, 4>(md, p, s, r, j, Q, O, tiles_bound, st);
  else if (md.hd == 64 && G == 1) pf_attn_tc_launch<64, 1>(md, p, s, r, j, Q, O, tiles_bound, st);
  else if (md.hd == 64 && G == 2) pf_attn_tc_launch<64, 2>(md, p, s, r, j, Q, O, tiles_bound, st);
  else if (md.hd == 64 && G == 4) pf_attn_tc_launch<64, 4>(md, p, s, r, j, Q, O, tiles_bound, st);
  else if (md.hd == 32 && G == 1) pf_attn_launch<bf16, 32, 1>(md, p, s, r, j, Q, O, tiles_bound, st);
  else pf_attn_launch<bf16, 32, 2>(md, p, s, r, j, Q, O, tiles_bound, st);
}

void launch_pf_len(const ModelDims& md, const PrefillDev& p, cudaStream_t st) {
  launch_k(k_pf_len, 1, 256, 0, st, md, p);
}

}  // namespace tlf
