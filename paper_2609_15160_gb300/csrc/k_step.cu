// The shared block of a decode step for up to 16 rows in one persistent kernel (Eq. 6-11).
//
// With few rows a decode step is a chain of small dependent stages: five per (loop, layer), each a few
// megabytes of weights and kilobytes of activations. As launches of their own every stage paid for the
// release of its predecessor, its operand's first load, a split-K exchange over a cluster and the
// drain of its own stores, about 7 us a launch; here the stages are phases of one cooperative kernel (one
// CTA per SM), separated by grid barriers, and loops that no token reaches cost nothing. Measured (device clock): about
// 21 us per (loop, layer) at one row of the mid-size model against 45 as launches, of which the five barriers take 1.3
// us each (the writes' release, the counter's round trip), a first load of what other SMs wrote 1.2 us each, and the
// attention of 47 pages a head 5 us. Steps, launches against this kernel: one row of 3000 keys of the mid-size model 770
// and 470 us, 8 rows of 1000 keys of the small model 324 and 250 us. Which steps take it: step_path in tlf_api.cu.
//
// Projections. The unit is a tile of 8 weight rows over the whole reduction length, so no partial sum
// leaves the CTA. A CTA owns a contiguous range of tiles; their rows are fetched into shared memory by
// bulk copies two phases ahead of their use (weights depend on nothing), so at the barrier only the
// activations are waited for. The 16 warps split K; each lane reads 16 contiguous bytes of a
// token row (hi and lo planes) and of a weight row, which feed two mma.sync m16n8k16 (tokens are the
// 16 MMA rows, the 8 weight rows its columns; K's order inside a 32-wide step is permuted alike on both
// sides). With 16 tokens a tcgen05 tile would leave the 128-row operand to the weights and need the
// cluster exchange again; the arithmetic here is far from bounding the phase either way. The warps' sums
// meet in shared memory in a fixed order, and the epilogue finishes the tile: RoPE and K/V append, SwiGLU,
// or the residual update with the next pre-norm's operand and its partial sums of squares.
//
// Attention. Two groups of eight warps a CTA each run the stream-K scheme of k_attn_decode on half of the
// CTA's share of the pages; the group's first warp also keeps its ring full, and fetches a layer's first pages while
// its QKV projection runs. The partials are merged by the O projection as it loads its operand: the grid barrier is
// there anyway, and a ticket would add an atomic's round trip and another set of loads. (Producer warps of their own left
// 96 registers a thread, and what spilled came back from L2: the barriers' acquires empty L1.)
#include <type_traits>

#include "tlf_internal.cuh"

namespace tlf {

namespace {

constexpr int SS_THREADS = 512;      // 16 warps: two attention groups of 8
constexpr int SS_TILES = 8;          // most tiles of 8 weight rows a CTA may own in a phase: one epilogue item a thread
constexpr int SS_PAD = 64;           // bytes added to a staged weight row: 2 rows of a quarter warp on different banks
constexpr int SS_PS = 64;            // keys per page

constexpr __host__ __device__ int ss_tile_bytes(int K) { return 8 * (2 * K + SS_PAD); }

template <int HD, int G>
struct SsShape {
  static constexpr int VEC = 8, LPK = HD / VEC, KPW = 32 / LPK, KEYS_PER_WARP = SS_PS / 8;
  static constexpr int STEPS = KEYS_PER_WARP / KPW > 0 ? KEYS_PER_WARP / KPW : 1;
  static constexpr int SEG = SS_PS * HD * 2, STAGE = 2 * SEG;
  static constexpr int PSZ = G * (HD + 4);        // floats of one partial: per head HD outputs, max, sum, padding
  static constexpr int RED = 8 * G * (HD + 2) * 4;  // a group's merge buffer
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

// Share of one warp (`wi` of 16) in fetching the weight rows of a CTA's tiles of a projection: KIND 0 QKV, 1 gate/up, 2
// plain rows. The caller has armed `bar` with all their bytes.
__device__ __forceinline__ void ss_fetch(int kind, const ModelDims& md, const bf16* W, int K, int u0, int T, uint8_t* dst,
                                         uint32_t bar, int wi, int lane) {
  const int i = wi + 16 * lane, rs = 2 * K + SS_PAD;  // rows spread over the warps: a copy is issued by one lane at a time
  if (i < 8 * T) {
    const int u = u0 + (i >> 3), l = i & 7;
    const int row = kind == 0 ? ss_row_qkv(md, u, l) : kind == 1 ? ss_row_gu(u, l) : 8 * u + l;
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
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  auto kvfull = [&](int grp, int st) { return smem_u32(&bars[grp * 2 * a.nst + st]); };
  auto kvempty = [&](int grp, int st) { return smem_u32(&bars[grp * 2 * a.nst + a.nst + st]); };
  const uint32_t wbar1 = smem_u32(&bars[4 * a.nst]), wbar2 = smem_u32(&bars[4 * a.nst + 1]);  // weights in

  const int tid = threadIdx.x, lane = tid & 31, wi = tid >> 5;
  const int grp = wi >> 3, w8 = wi & 7, gtid = tid & 255;  // attention group, warp and thread of the group
  if (tid == 0) {
    for (int g = 0; g < 2; ++g)
      for (int i = 0; i < a.nst; ++i) {
        mbar_init(kvfull(g, i), 1);
        mbar_init(kvempty(g, i), 8);
      }
    mbar_init(wbar1, 1);
    mbar_init(wbar2, 1);
    abort_word = 0;
    fence_barrier_init();
  }
  __syncthreads();
  const int d = md.d, q_dim = md.q_dim, ff = md.ff, M = md.M, J = md.J, maxB = md.max_batch;
  // this CTA's tiles of the projections
  int uq, tq, ug, tg, uo, to;
  ss_range(md.qkv_dim / 8, blockIdx.x, gridDim.x, uq, tq); tq -= uq;
  ss_range(ff / 4, blockIdx.x, gridDim.x, ug, tg); tg -= ug;
  ss_range(d / 8, blockIdx.x, gridDim.x, uo, to); to -= uo;  // O and down alike
  if (tid == 0) {
    if (tq > 0) mbar_arrive_expect_tx(wbar1, (uint32_t)(tq * 16 * d));
    if (to > 0) mbar_arrive_expect_tx(wbar2, (uint32_t)(to * 16 * q_dim));
  }
  __syncthreads();
  ss_fetch(0, md, a.layer[0].wqkv, d, uq, tq, w1, wbar1, wi, lane);
  ss_fetch(2, md, a.layer[0].wo, q_dim, uo, to, w2, wbar2, wi, lane);
  pdl_wait();

  int epoch = 0;              // grid barriers passed
  uint32_t ph1 = 0, ph2 = 0;  // phases of the weight barriers
  int ring_st = 0;            // this group's ring: the next page's stage,
  uint32_t ring_par = 0;      // and the parity of that stage's "full" phase
  auto give_up = [&]() {
    atomicOr(s.err, DEVERR_WAIT);
    *abort_flag = 1;
  };
  // All CTAs' writes before it are visible to reads past L1 after it.
  auto grid_sync = [&](bool to_copies) {
    ++epoch;
    if (to_copies) fence_proxy_async_all();  // new K/V entries, and the partial sums' space, go to bulk copies
    __syncthreads();
    if (tid == 0) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.gbar) : "memory");
      const unsigned want = (unsigned)epoch * gridDim.x;
      uint64_t t0 = 0;
      while (!*abort_flag) {
        unsigned got;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(a.gbar) : "memory");
        if (got >= want) break;
        const uint64_t t = globaltimer_ns();
        if (t0 == 0) t0 = t;
        if (t - t0 > kWaitLimitNs) give_up();
      }
    }
    __syncthreads();
  };
  auto wait_bar = [&](uint32_t bar, uint32_t parity) {
    if (!*abort_flag && !mbar_wait(bar, parity, s.err)) *abort_flag = 1;
  };

  // After a projection: the sum over the warps' partial sums `red` of row m, weight row l of tile i.
  auto sum = [&](const float* red, int T, int i, int m, int l) {
    const float* q = red + ((size_t)i * 16 + m) * 8 + l;
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < 16; ++w) t += q[w * T * 128];
    return t;
  };
  const size_t xlo = (size_t)maxB * d, ulo = (size_t)maxB * ff;
  // the merged attention output: hi plane, then lo plane, rows of q_dim + 8 elements, behind two tiles' partial sums
  bf16* om = reinterpret_cast<bf16*>(kv + 16 * 2 * 16 * 8 * 4);
  const int om_row = q_dim + 8;
  const int ld8 = d / 8;

  for (int r = 0; r < M; ++r) {
    const int n = min(16, __ldcg(s.n + r));
    if (n <= 0) break;  // active sets nest
    const bool more_loops = r + 1 < M && __ldcg(s.n + (r + 1 < M ? r + 1 : r)) > 0;
    if (tid < 17) {
      if (tid < n) {
        const int4 ri = __ldcg(s.rowinfo + r * maxB + tid);
        rowmeta[tid] = ri;
        const int nc = r + 1 < M ? __ldcg(s.col + (r + 1) * maxB + ri.w) + 1 : 0;
        const int m = min(max(__ldcg(s.m + ri.w), r + 1), M), mo = m * (m - 1) / 2 + r;
        rowaux[tid] = make_uchar4((unsigned char)nc, (unsigned char)mo, (unsigned char)min(mo + 1, m * (m + 1) / 2 - 1), 0);
        nkeys[tid] = __ldcg(s.nch + r * maxB + tid);
        slots[tid] = __ldcg(s.slots + ri.w);
      }
      if (tid <= n) pbase[tid] = __ldcg(s.item_base + r * (maxB + 1) + tid);
    }
    __syncthreads();
    // the attention's page shares: group v of nv takes flat pages [p0, p1)
    auto pages_of = [&](int kk) { return (nkeys[kk] + SS_PS - 1) / SS_PS; };
    const int total = pbase[n], nv = 2 * gridDim.x, v = 2 * blockIdx.x + grp;
    const int per = (total + nv - 1) / nv, p0 = v * per, p1 = min(total, p0 + per);
    // (row, kv head, page) of the group's first flat page: the largest k with pbase[k] <= p0 (n <= 16, one ballot)
    int k0 = 0, h0 = 0, g0 = 0;
    if (p0 < total) {
      const unsigned le = __ballot_sync(0xffffffffu, lane < n && pbase[min(lane, n)] <= p0);
      k0 = 31 - __clz((int)le);
      const int off = p0 - pbase[k0], np = pages_of(k0);
      h0 = off / np;
      g0 = off % np;
    }
    // Warp 0 of a group keeps its ring full. Lane q holds what it takes to fetch flat page p + q, the same in every layer
    // of the loop: element offset in the pool (-1: bad page), bytes of its K (or V) segment, whether it is its item's
    // last page.
    uint8_t* my_ring = kv + (size_t)grp * a.nst * Sh::STAGE;
    auto page_info = [&](int p, long long& off, int& bytes, bool& last) {
      const int pq = p + lane;
      off = -1;
      bytes = 0;
      last = false;
      if (pq < p1) {
        int kq = k0;  // the row of a later page: rows ascend
        while (kq + 1 < n && pbase[kq + 1] <= pq) ++kq;
        const int np = pages_of(kq), in_row = pq - pbase[kq], hq = in_row / np, gq = in_row - hq * np;
        const int page = s.page_table[((size_t)slots[kq] * M + r) * md.max_pages + gq];
        bytes = min(SS_PS, nkeys[kq] - gq * SS_PS) * HD * 2;
        last = gq + 1 == np;
        if (page >= 0 && page < md.n_pages && bytes > 0) off = (long long)page * md.page_elems + (long long)hq * SS_PS * HD;
        else atomicOr(s.err, DEVERR_INDEX);
      }
    };
    long long off_f = -1;
    int bytes_f = 0;
    bool last_f = false;
    if (w8 == 0) page_info(p0, off_f, bytes_f, last_f);
    // one lane's fetch of its page of layer j into stage st (whose readers are done)
    auto fetch = [&](int j, long long off, int bytes, int st) {
      const uint32_t bar = kvfull(grp, st);
      if (off < 0) {
        mbar_arrive(bar);  // complete the phase without data
      } else if (!*abort_flag) {
        const bf16* kp = reinterpret_cast<const bf16*>(s.pool) + off + (size_t)j * 2 * md.Hkv * SS_PS * HD;
        uint8_t* dst = my_ring + st * Sh::STAGE;
        const uint64_t pol = l2_policy_evict_first();  // pages are read once per step
        mbar_arrive_expect_tx(bar, 2 * bytes);
        bulk_g2s_hint(smem_u32(dst), kp, (uint32_t)bytes, bar, pol);
        bulk_g2s_hint(smem_u32(dst + Sh::SEG), kp + (size_t)md.Hkv * SS_PS * HD, (uint32_t)bytes, bar, pol);
      }
    };
    // The first pages of layer j, a lane each: those that can go while its QKV projection runs, or (late) the items' last
    // pages, which get the new entries. The ring is empty then.
    auto fill_ring = [&](int j, bool late) {
      if (lane < min(a.nst, p1 - p0) && last_f == late) {
        int st = ring_st + lane;
        if (st >= a.nst) st -= a.nst;
        fetch(j, off_f, bytes_f, st);
      }
      __syncwarp();
    };
    // The attention output of the loop's rows to `om`, from the partials of the groups that shared each item, eight of
    // them in flight at a time.
    auto merge_rows = [&]() {
      const int per_row = q_dim / 4;
#pragma unroll 1
      for (int i = tid; i < n * per_row; i += SS_THREADS) {
        const int k = i / per_row, kk = (i - k * per_row) * 4, hq = kk / HD, e = kk % HD;
        const int np = pages_of(k), item = k * md.Hkv + hq / G, first = pbase[k] + (hq / G) * np;
        const int c0 = first / per, c1 = (first + np - 1) / per;
        const float* base = a.part + (size_t)item * Sh::PSZ + (hq % G) * (HD + 4);
        float mx = -INFINITY, l = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int c = c0; c <= c1; c += 8) {
          float2 ml[8];
          float4 x[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float* src = base + (size_t)min(c + q, c1) * Sh::PSZ;
            ml[q] = __ldcg(reinterpret_cast<const float2*>(src + HD));
            x[q] = __ldcg(reinterpret_cast<const float4*>(src + e));
          }
          float nm = mx;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            if (c + q > c1) ml[q].x = -INFINITY;
            nm = fmaxf(nm, ml[q].x);
          }
          const float cr = exp2f(mx - nm);  // 0 for the first ones
          mx = nm;
          l *= cr;
#pragma unroll
          for (int w = 0; w < 4; ++w) o[w] *= cr;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float fw = exp2f(ml[q].x - mx);  // 0 past the last partial
            l = fmaf(fw, ml[q].y, l);
            o[0] = fmaf(fw, x[q].x, o[0]);
            o[1] = fmaf(fw, x[q].y, o[1]);
            o[2] = fmaf(fw, x[q].z, o[2]);
            o[3] = fmaf(fw, x[q].w, o[3]);
          }
        }
        uint32_t hb[2], lb[2];
#pragma unroll
        for (int w = 0; w < 2; ++w) {
          const float v0 = o[2 * w] / l, v1 = o[2 * w + 1] / l;
          const __nv_bfloat162 b = __floats2bfloat162_rn(v0, v1);
          const __nv_bfloat162 rest = __floats2bfloat162_rn(v0 - __low2float(b), v1 - __high2float(b));
          hb[w] = *reinterpret_cast<const uint32_t*>(&b);
          lb[w] = *reinterpret_cast<const uint32_t*>(&rest);
        }
        *reinterpret_cast<uint2*>(om + k * om_row + kk) = make_uint2(hb[0], hb[1]);
        *reinterpret_cast<uint2*>(om + (16 + k) * om_row + kk) = make_uint2(lb[0], lb[1]);
      }
      __syncthreads();
    };
    // conditioning vector `part` of layer j for rows at (depth, loop) `off`
    const int combos = M * (M + 1) / 2;
    auto cvec = [&](int j, int off, int part) { return a.cond + ((size_t)(j * combos + off) * 4 + part) * d; };

    for (int j = 0; j < J; ++j) {
      const bool last_layer = j + 1 == J, has_next = !last_layer || more_loops;
      const int jn = last_layer ? 0 : j + 1;
#pragma unroll 1
      for (int ph = 0; ph < 4; ++ph) {  // QKV, O, gate/up, down: one copy of the projection's code
        const bool wide = (ph & 1) == 0;  // QKV and gate/up: from the pre-norm operand, scaled by the rows' factors
        const int u0 = ph == 0 ? uq : ph == 2 ? ug : uo, T = ph == 0 ? tq : ph == 2 ? tg : to;
        const int K = ph == 1 ? q_dim : ph == 3 ? ff : d;
        // This thread's element of the epilogue (row m; wide: pair p of a tile's rows p, p + 4; else feature p), and
        // what it needs besides the sums, loaded ahead of the barrier: the CTA's own residual values, gains, rotary
        // factors.
        const int i = wide ? tid >> 6 : tid >> 7, m = wide ? (tid >> 2) & 15 : (tid >> 3) & 15, p = wide ? tid & 3 : tid & 7;
        const bool mine = i < T && m < n;
        float pre0 = 0.f, pre1 = 1.f, alpha = 1.f, gamma = 1.f;
        const int f = 8 * (u0 + i) + (wide ? 0 : p);
        if (mine) {
          if (ph == 0) {
            if (f < q_dim + md.kv_dim) {
              const float2 cs = a.rope[(size_t)rowmeta[m].z * (HD / 2) + (f % HD) / 2 + p];
              pre0 = cs.y;
              pre1 = cs.x;
            }
          } else if (!wide) {
            pre0 = __ldcg(s.H + (size_t)rowmeta[m].w * d + f);
            pre1 = ph == 1 ? a.layer[j].mlp_norm[f] : a.layer[jn].attn_norm[f];
            if (a.cond) {
              alpha = cvec(j, rowaux[m].y, ph == 1 ? 0 : 1)[f];
              gamma = 1.f + (ph == 1 ? cvec(j, rowaux[m].y, 3)[f] : cvec(jn, last_layer ? rowaux[m].z : rowaux[m].y, 2)[f]);
            }
          }
        }
        if (ph > 0 || j > 0 || r > 0) grid_sync(ph == 0);
        if (ph == 0 && w8 == 0) fill_ring(j, false);
        if (ph == 1 && T > 0) merge_rows();
        // partial sums: the rings' space between attentions; QKV's, which run beside the first pages' copies, behind its
        // weights
        float* red = reinterpret_cast<float*>(ph == 0 ? w1 + tq * ss_tile_bytes(d) : kv);

        // ---- the projection of this CTA's T tiles: warps split K, partial sums [16][T][16 rows][8] to `red`. The
        // token operand's loads come first, then the rows' norm factors, then the wait for the weights ----
        const uint8_t* ws = wide ? w1 : w2;
        {
          const bf16* X = wide ? a.X : ph == 1 ? om : a.U;  // (om in shared memory)
          const size_t lo_off = wide ? xlo : ph == 1 ? (size_t)16 * om_row : ulo;
          const int ldx = ph == 1 ? om_row : K;
          auto ldx16 = [&](const bf16* q) { return ph == 1 ? *reinterpret_cast<const uint4*>(q) : ldcg16(q); };
          const int g = lane >> 2, t4 = lane & 3, rs = 2 * K + SS_PAD;
          const int steps = T > 0 ? (K + 31) / 32 : 0;
          const uint4 z = make_uint4(0, 0, 0, 0);
          const bf16* xg = X + (size_t)g * ldx + t4 * 8;
          // partial sums of squares of row wi, for its RMSNorm factor
          float4 ssv[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
          const bool head = r == 0 && j == 0 && ph == 0;
          const int ldn = (head ? a.ldss : ld8) / 4;  // (at most 64: two a lane)
          if (wide && wi < n) {
            const float4* ss4 = reinterpret_cast<const float4*>(head ? a.ss + (size_t)wi * a.ldss : a.ss8 + (size_t)wi * ld8);
#pragma unroll
            for (int q = 0; q < 2; ++q)
              if (lane + 32 * q < ldn) ssv[q] = __ldcg(ss4 + lane + 32 * q);
          }
          bool first = true;
          auto between = [&]() {  // once, behind the first loads
            if (first && T > 0) wait_bar(wide ? wbar1 : wbar2, (wide ? ph1 : ph2) & 1u);
            first = false;
          };
          // This warp's K steps in batches whose token operands are in flight at once; each batch goes over the tiles in
          // a rolled loop (unrolled, the code of a phase ran once per phase and was bound by its fetch).
          float* po = red + ((size_t)wi * T * 16 + g) * 8 + 2 * t4;
          const uint8_t* wg = ws + (size_t)g * rs + t4 * 16;
          if (n <= 8) {
            // the two terms of a row are the MMA's rows g and g + 8
            constexpr int SB = 6;
            for (int s0 = wi; s0 < steps; s0 += 16 * SB) {
              uint4 h[SB], l[SB];
#pragma unroll
              for (int q = 0; q < SB; ++q) {
                const int k = (s0 + 16 * q) * 32;
                const bool in = k + t4 * 8 < K && g < n;
                h[q] = in ? ldx16(xg + k) : z;
                l[q] = in ? ldx16(xg + k + lo_off) : z;
              }
              between();
#pragma unroll 1
              for (int t = 0; t < T; ++t) {
                const uint8_t* wt = wg + (size_t)t * 8 * rs + s0 * 64;
                float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int q = 0; q < SB; ++q)
                  if ((s0 + 16 * q) * 32 < K) {
                    // (a lane past K holds zeros of the token operand; its weights must be finite too)
                    const uint4 w = (s0 + 16 * q) * 32 + t4 * 8 < K ? *reinterpret_cast<const uint4*>(wt + q * 1024) : z;
                    mma_16816(c, h[q].x, l[q].x, h[q].y, l[q].y, w.x, w.y);
                    mma_16816(c, h[q].z, l[q].z, h[q].w, l[q].w, w.z, w.w);
                  }
                float2* o = reinterpret_cast<float2*>(po + t * 128);
                float2 v = make_float2(c[0] + c[2], c[1] + c[3]);
                if (s0 != wi) {
                  v.x += o->x;
                  v.y += o->y;
                }
                *o = v;
              }
            }
          } else {
            constexpr int SB = 3;
            for (int s0 = wi; s0 < steps; s0 += 16 * SB) {
              uint4 h[SB], h8[SB], l[SB], l8[SB];
#pragma unroll
              for (int q = 0; q < SB; ++q) {
                const int k = (s0 + 16 * q) * 32;
                const bool in = k + t4 * 8 < K, in8 = in && g + 8 < n;  // (n > 8: row g exists)
                h[q] = in ? ldx16(xg + k) : z;
                l[q] = in ? ldx16(xg + k + lo_off) : z;
                h8[q] = in8 ? ldx16(xg + (size_t)8 * ldx + k) : z;
                l8[q] = in8 ? ldx16(xg + (size_t)8 * ldx + k + lo_off) : z;
              }
              between();
#pragma unroll 1
              for (int t = 0; t < T; ++t) {
                const uint8_t* wt = wg + (size_t)t * 8 * rs + s0 * 64;
                float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int q = 0; q < SB; ++q)
                  if ((s0 + 16 * q) * 32 < K) {
                    const uint4 w = (s0 + 16 * q) * 32 + t4 * 8 < K ? *reinterpret_cast<const uint4*>(wt + q * 1024) : z;
                    mma_16816(c, h[q].x, h8[q].x, h[q].y, h8[q].y, w.x, w.y);
                    mma_16816(c, h[q].z, h8[q].z, h[q].w, h8[q].w, w.z, w.w);
                    mma_16816(c, l[q].x, l8[q].x, l[q].y, l8[q].y, w.x, w.y);
                    mma_16816(c, l[q].z, l8[q].z, l[q].w, l8[q].w, w.z, w.w);
                  }
                float2* o = reinterpret_cast<float2*>(po + t * 128);
                float2 v0 = make_float2(c[0], c[1]), v1 = make_float2(c[2], c[3]);
                if (s0 != wi) {
                  v0.x += o->x; v0.y += o->y;
                  v1.x += o[32].x; v1.y += o[32].y;
                }
                o[0] = v0;
                o[32] = v1;
              }
            }
          }
          if (wi >= steps) {  // (a warp without a step)
            between();
            for (int t = 0; t < T; ++t) {
              *reinterpret_cast<float2*>(po + t * 128) = make_float2(0.f, 0.f);
              *reinterpret_cast<float2*>(po + t * 128 + 64) = make_float2(0.f, 0.f);
            }
          }
          if (T > 0) ++(wide ? ph1 : ph2);
          if (wide) {
            const float t = warp_sum((ssv[0].x + ssv[0].y) + (ssv[0].z + ssv[0].w) + (ssv[1].x + ssv[1].y) + (ssv[1].z + ssv[1].w));
            if (lane == 0) scale[wi] = rsqrtf(t / (float)d + md.eps);
          }
        }
        // the weights that follow these in their region: gate/up, down, the next QKV, the next O
        const int Tn = ph == 0 ? tg : ph == 1 ? to : has_next ? (ph == 2 ? tq : to) : 0;
        const int Kn = ph == 1 ? ff : ph == 3 ? q_dim : d;
        if (tid == 0 && Tn > 0) mbar_arrive_expect_tx(wide ? wbar1 : wbar2, (uint32_t)(Tn * 16 * Kn));
        __syncthreads();  // partial sums in, weights read
        if (Tn > 0 && ph > 0 && !*abort_flag) {
          const SmallLayer& Ln = a.layer[ph == 1 ? j : jn];
          ss_fetch(ph == 2 ? 0 : 2, md, ph == 1 ? Ln.wd : ph == 2 ? Ln.wqkv : Ln.wo, Kn, ph == 2 ? uq : uo, Tn,
                   wide ? w1 : w2, wide ? wbar1 : wbar2, wi, lane);
        }

        if (!wide) {
          // ---- residual update, and the next pre-norm's operand with its sums of squares ----
          if (tid < T * 128) {
            float h = pre0;
            int dst = -1;
            if (m < n) {
              h += alpha * sum(red, T, i, m, p);
              s.H[(size_t)rowmeta[m].w * d + f] = h;
              if (ph == 1 || has_next) dst = ph == 3 && last_layer ? (int)rowaux[m].x - 1 : m;
              if (dst >= 0) {
                const float y = h * pre1 * gamma;
                const bf16 yh = __float2bfloat16_rn(y);
                a.X[(size_t)dst * d + f] = yh;
                a.X[xlo + (size_t)dst * d + f] = __float2bfloat16_rn(y - __bfloat162float(yh));
              }
            }
            float q = h * h;
            q += __shfl_xor_sync(0xffffffffu, q, 1);
            q += __shfl_xor_sync(0xffffffffu, q, 2);
            q += __shfl_xor_sync(0xffffffffu, q, 4);
            if (dst >= 0 && p == 0) a.ss8[(size_t)dst * ld8 + u0 + i] = q;
          }
          continue;
        }
        if (mine) {
          const float x0 = sum(red, T, i, m, p) * scale[m], x1 = sum(red, T, i, m, p + 4) * scale[m];
          if (ph == 2) {
            // ---- SwiGLU ----
            const float y = x0 / (1.f + expf(-x0)) * x1;
            const bf16 yh = __float2bfloat16_rn(y);
            const size_t at = (size_t)m * ff + 4 * (u0 + i) + p;
            a.U[at] = yh;
            a.U[ulo + at] = __float2bfloat16_rn(y - __bfloat162float(yh));
          } else {
            // ---- RoPE on q and k, K/V append ----
            const int4 ri = rowmeta[m];
            if (f < q_dim + md.kv_dim) {
              const int h = f / HD, e = (f % HD) / 2 + p;  // pair (e, e + HD/2) of head h
              const float r0 = x0 * pre1 - x1 * pre0, r1 = x0 * pre0 + x1 * pre1;
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
        if (ph == 2) continue;

        // ---- attention: the group's share of the pages, after the QKV projection ----
        grid_sync(true);
        if (!*abort_flag) ss_fetch(1, md, a.layer[j].wgu, d, ug, tg, w1, wbar1, wi, lane);  // (its space held the partial sums till now)
        if (p0 >= total) continue;
        int k = k0, h = h0, g = g0;
        if (w8 == 0) {
          fence_proxy_async_all();  // behind the barrier: this step's K/V entries
          fill_ring(j, true);
        }
        const int sub = lane / Sh::LPK, pl = lane % Sh::LPK;
        const float qscale = 1.4426950408889634f * rsqrtf((float)HD);
        float* mred = att_red + (size_t)grp * (Sh::RED / 4);
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
        long long off_b = off_f;  // warp 0: the current 32 pages
        int bytes_b = bytes_f;
#pragma unroll 1
        for (int pp = p0; pp < p1; ++pp) {
          const int st = ring_st;
          const uint32_t par = ring_par;
          if (++ring_st == a.nst) {
            ring_st = 0;
            ring_par ^= 1u;
          }
          wait_bar(kvfull(grp, st), par);
          const int valid = min(SS_PS, Lk - g * SS_PS);
          const bf16* sk = reinterpret_cast<const bf16*>(my_ring + st * Sh::STAGE);
          const bf16* sv = reinterpret_cast<const bf16*>(my_ring + st * Sh::STAGE + Sh::SEG);
          float sc[Sh::STEPS][G];
#pragma unroll
          for (int t = 0; t < Sh::STEPS; ++t) {
            const int key = w8 * Sh::KEYS_PER_WARP + t * Sh::KPW + sub;
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
            const int key = w8 * Sh::KEYS_PER_WARP + t * Sh::KPW + sub;
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
          // the page before's stage is free by now, or soon: its next page
          const int pf = pp - 1 + a.nst;
          if (w8 == 0 && pp > p0 && pf < p1) {
            if (((pf - p0) & 31) == 0) {
              bool last_b;
              page_info(pf, off_b, bytes_b, last_b);
            }
            const int sp = st == 0 ? a.nst - 1 : st - 1;
            if (lane == ((pf - p0) & 31)) {
              wait_bar(kvempty(grp, sp), st == 0 ? par ^ 1u : par);
              fetch(j, off_b, bytes_b, sp);
            }
            __syncwarp();
          }
          const int np = pages_of(k);
          if (g + 1 < np && pp + 1 < p1) {
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
              float* rw = mred + (w8 * G + gg) * (HD + 2);
#pragma unroll
              for (int e = 0; e < Sh::VEC; ++e) rw[pl * Sh::VEC + e] = acc[gg][e];
              if (pl == 0) {
                rw[HD] = run_m[gg];
                rw[HD + 1] = run_l[gg];
              }
            }
          }
          named_sync(2 + grp, 256);
          float* my = a.part + (size_t)(k * md.Hkv + h + v) * Sh::PSZ;
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
            my[gg * (HD + 4) + e] = o;
            if (e == 0) *reinterpret_cast<float2*>(my + gg * (HD + 4) + HD) = make_float2(mx, l);
          }
          named_sync(2 + grp, 256);  // the merge buffer is reused by the next item
          if (pp + 1 < p1) {
            g = 0;
            if (++h == md.Hkv) {
              h = 0;
              ++k;
            }
            begin_item();
          }
        }
      }
    }
    __syncthreads();  // rowmeta is rewritten for the next loop
  }
  if (*abort_flag) drain_copies();
}

// Shared memory of the kernel's parts for a model on a grid of `ctas` CTAs: fills the byte counts and ring depth of
// `a`, returns the dynamic shared memory (0: the model does not fit).
static int ss_layout(const ModelDims& md, int ctas, SmallStep* a) {
  auto tiles = [&](int U) { return (U + ctas - 1) / ctas; };
  const int tq = tiles(md.qkv_dim / 8), to = tiles(md.d / 8), tg = tiles(md.ff / 4), td = tiles(md.d / 8);
  if (tq > SS_TILES || tg > SS_TILES || to > 2 || td > 2 || md.J > SS_LAYERS || md.d > 2048) return 0;
  // W1 holds QKV's tiles and, behind them, their partial sums (16 warps x tiles x 16 rows x 8), or gate/up's tiles
  const int w1q = tq * (ss_tile_bytes(md.d) + 16 * 16 * 8 * 4), w1g = tg * ss_tile_bytes(md.d);
  a->w1_bytes = ((w1q > w1g ? w1q : w1g) + 127) / 128 * 128;
  const int wo = to * ss_tile_bytes(md.q_dim), wd = td * ss_tile_bytes(md.ff);
  a->w2_bytes = ((wo > wd ? wo : wd) + 127) / 128 * 128;
  const int G = md.Hq / md.Hkv, stage = 2 * SS_PS * md.hd * 2, red = 2 * 8 * G * (md.hd + 2) * 4;
  const int fixed = a->w1_bytes + a->w2_bytes + red;
  const int limit = 232448 - 640;  // less the static shared memory
  // the other projections' partial sums share the rings' space, and so does the merged attention output
  int psum = 16 * (tg > td ? tg : td) * 16 * 8 * 4;
  const int merged = 16 * 2 * 16 * 8 * 4 + 2 * 16 * (md.q_dim + 8) * 2;
  if (merged > psum) psum = merged;
  for (int nst = 8; nst >= 2; --nst) {
    const int bytes = fixed + 2 * nst * stage + (4 * nst + 2) * 8;
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

// One partial per (item + group) index, for up to 16 rows.
size_t step_small_part_floats(const ModelDims& md, int num_sms) {
  return ((size_t)16 * md.Hkv + 2 * num_sms) * (md.Hq / md.Hkv) * (md.hd + 4);
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
