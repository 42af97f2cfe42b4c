// Dense projections of a prefill chunk (Eq. 6, 9): Y[row][o] = sum_k X[row][k] * W[o][k] for the
// hundreds to thousands of rows of a loop.
//
// k_gemm_pf: tcgen05 on a pair of SMs (cta_group::2). A cluster of two CTAs owns a tile of 256 rows
// (tokens, the MMA's M) x BN features (N); each CTA loads its 128 token rows and half of the weight
// rows by TMA and holds the accumulator of its 128 rows in TMEM. The grid is persistent (one pair per
// two SMs, tiles in a fixed stride) and warp-specialised:
//   warp 0      TMA producer: 64-wide K slabs of both operands into a ring; the bytes of both CTAs
//               complete on the leader's barrier;
//   warp 1      (leader CTA) MMA issuer, accumulating in one of two TMEM buffers, so the epilogue of a
//               tile runs under the MMAs of the next;
//   warps 2-9   epilogue: a thread holds one token row, so both halves of a rotary or gate/up pair and
//               the row's page and position are its own; 32 columns at a time go through a per-warp
//               staging tile and leave as whole 64- to 128-byte row segments.
// Epilogues: residual add + scatter (vector reductions, one writer per element), RoPE + q out + K/V
// append, SwiGLU.
//
// Tile and split: a pair on a 256 x 256 tile reads each operand byte from shared memory half as often as a
// single-CTA 128 x 256 tile, and with the tokens as M no partial tile is staged for another warp. Measured at 8192
// rows, K 2048, 11008 features with SwiGLU: 254 us, 1450 TFLOP/s, 0.74 of the measured bf16 rate (454 us with
// single-CTA tiles of k_gemm_tc, whose epilogue ran between the MMAs). Part of the rest is the last wave (1376 tiles
// over 76 pairs, 18.1 waves run as 19; 384 tiles, 5.05 waves run as 6, for the mid-size model's QKV) and the pipeline's
// ends; what holds the full waves is not measured (at the full MMA rate an SM would take 64 bytes a cycle from L2).
#include <type_traits>

#include "tlf_internal.cuh"

namespace tlf {

namespace {

constexpr int PG_THREADS = 320;
constexpr int PG_EPI_WARPS = 8;
constexpr int PG_BK = 64;
constexpr int PG_A_BYTES = 128 * PG_BK * 2;
constexpr int PG_SEG = 144;                     // bytes of a staged row: 32 floats, padded against bank conflicts
constexpr int PG_STAGE_TILE = 32 * PG_SEG;      // one epilogue warp's staging tile

template <int BN>
struct PgShape {
  static constexpr int B_BYTES = (BN / 2) * PG_BK * 2;
  static constexpr int ST_BYTES = PG_A_BYTES + B_BYTES;
  static constexpr int NS = BN == 256 ? 5 : 6;
  static constexpr int OFF_STG = NS * ST_BYTES;
  static constexpr int OFF_BAR = OFF_STG + PG_EPI_WARPS * PG_STAGE_TILE;
  static constexpr int NBAR = 2 * NS + 4;
  static constexpr uint32_t TMEM_COLS = 2 * BN;
  static constexpr int USED = OFF_BAR + NBAR * 8 + 16 + 1024;
  static constexpr int BYTES = USED > tmem_min_smem(TMEM_COLS) ? USED : tmem_min_smem(TMEM_COLS);
};

__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int32_t c0, int32_t c1,
                                                 uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_mma_f16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                                uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on the barrier at this offset in both CTAs of the pair once the MMAs issued so far are done.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}
// Arrive on a barrier of any CTA of the cluster (address from dsmem_map).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// The wait that pairs with a remote arrival.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, uint32_t* err) {
  uint64_t t0 = 0;
  while (true) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    const uint64_t t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    if (t - t0 > kWaitLimitNs) {
      atomicOr(err, DEVERR_WAIT);
      return false;
    }
  }
}



}  // namespace

template <int BN, int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PG_THREADS, 1)
    k_gemm_pf(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapW, GemmArgs a) {
  using Sh = PgShape<BN>;
  constexpr int NS = Sh::NS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + Sh::OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + Sh::NBAR);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto full = [&](int i) { return smem_u32(&bars[i]); };
  auto empty = [&](int i) { return smem_u32(&bars[NS + i]); };
  auto tfull = [&](int b) { return smem_u32(&bars[2 * NS + b]); };
  auto tempty = [&](int b) { return smem_u32(&bars[2 * NS + 2 + b]); };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  if (tid == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(full(i), 1);
      mbar_init(empty(i), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull(b), 1);
      mbar_init(tempty(b), 2 * PG_EPI_WARPS);
    }
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tensormap(&mapX);
    prefetch_tensormap(&mapW);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(tmem_slot), Sh::TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the pair's barriers are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // The row count comes from the plan kernel, which completed before this grid was launched (every
  // kernel triggers its successor only after its own wait), so it is read before pdl_wait().
  const int n = a.n_dev ? __ldcg(a.n_dev) : a.n_host;
  const int mt = (n + 255) / 256, ntl = (a.N + BN - 1) / BN, tiles = mt * ntl;
  const int nkb = (a.K + PG_BK - 1) / PG_BK;
  const int c_first = blockIdx.x >> 1, c_step = gridDim.x >> 1;
  auto wait = [&](uint32_t b, uint32_t parity) {
    if (*abort_flag) return false;
    if (!mbar_wait_cluster(b, parity, a.err)) {
      *abort_flag = 1;
      return false;
    }
    return true;
  };

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      int it = 0;  // k-slabs issued so far
      bool waited = false, ok = true;
      for (int t = c_first; t < tiles && ok; t += c_step) {
        const int m0 = (t / ntl) * 256 + (int)rank * 128, n0 = (t % ntl) * BN + (int)rank * (BN / 2);
        auto load = [&](int kb, int i, bool w, bool x) {
          const int st = i % NS;
          uint8_t* dst = sm + st * Sh::ST_BYTES;
          const uint32_t lead = dsmem_map(full(st), 0);
          if (w) {
            if (rank == 0) mbar_arrive_expect_tx(full(st), 2 * Sh::ST_BYTES);
            tma_load_2d_pair(smem_u32(dst + PG_A_BYTES), &mapW, kb * PG_BK, n0, lead);
          }
          if (x) tma_load_2d_pair(smem_u32(dst), &mapX, kb * PG_BK, m0, lead);
        };
        int kb = 0;
        if (!waited) {
          // the first slabs' weights go out before the wait on the preceding kernels
          const int pre = nkb < NS ? nkb : NS;
          for (int i = 0; i < pre; ++i) load(i, i, true, false);
          pdl_wait();
          pdl_trigger();
          waited = true;
          for (int i = 0; i < pre; ++i) load(i, i, false, true);
          kb = it = pre;
        }
        for (; kb < nkb; ++kb, ++it) {
          if (it >= NS && !wait(empty(it % NS), (uint32_t)(it / NS - 1) & 1u)) {
            ok = false;
            break;
          }
          load(kb, it, true, true);
        }
      }
      if (!waited) {
        pdl_wait();
        pdl_trigger();
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (leader CTA) ----------------
    pdl_wait();
    pdl_trigger();
    if (rank == 0 && lane == 0) {
      constexpr uint32_t IDESC = idesc_bf16_f32(256, BN);
      int it = 0, k = 0;  // slabs consumed, tiles started
      bool ok = true;
      for (int t = c_first; t < tiles && ok; t += c_step, ++k) {
        const int b = k & 1;
        if (k >= 2 && !wait(tempty(b), (uint32_t)(k / 2 - 1) & 1u)) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * BN);
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int st = it % NS;
          if (!wait(full(st), (uint32_t)(it / NS) & 1u)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t da = smem_desc_sw128(smem_u32(sm + st * Sh::ST_BYTES));
          const uint64_t db = smem_desc_sw128(smem_u32(sm + st * Sh::ST_BYTES + PG_A_BYTES));
#pragma unroll
          for (int q = 0; q < PG_BK / 16; ++q)
            tc_mma_f16_pair(d, da + 2 * q, db + 2 * q, IDESC, (kb > 0 || q > 0) ? 1u : 0u);
          tc_commit_pair(empty(st));
        }
        if (ok) tc_commit_pair(tfull(b));
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ----------------
    pdl_wait();
    pdl_trigger();
    const int quad = warp & 3, hf = (warp - 2) >> 2;  // TMEM lane quadrant, share of the columns
    uint8_t* stg = sm + Sh::OFF_STG + (warp - 2) * PG_STAGE_TILE;
    const ModelDims& md = a.md;
    int k = 0;
    for (int t = c_first; t < tiles; t += c_step, ++k) {
      const int b = k & 1;
      const int row = (t / ntl) * 256 + (int)rank * 128 + quad * 32 + lane, n0 = (t % ntl) * BN;
      const bool row_ok = row < n;
      // the row's destination, read while the tile's MMAs run
      int drow = -1;             // RESID: residual row; SWIGLU: row (-1: none)
      long long dkv = -1;        // QKV: element offset of the row's slot in its page (-1: no append)
      int pos = 0;
      const float* alpha = nullptr;
      if (EPI == EPI_CL_RESID) {
        if (row_ok) {
          drow = a.idx ? a.idx[row] : row;
          if (a.alpha.mod) alpha = cond_row(a.alpha, drow);
        }
      } else {
        if (row_ok) drow = row;
      }
      if (EPI == EPI_CL_QKV && row_ok) {
        const int slot = a.row_slot[row], L = a.row_cslot[row], ps = md.page_size;
        pos = a.row_pos[row];
        const int page = a.s.page_table[((size_t)slot * md.M + a.r) * md.max_pages + L / ps];
        if (page < 0 || page >= md.n_pages || pos < 0 || pos >= md.max_pos) {
          atomicOr(a.s.err, DEVERR_INDEX);
          pos = 0;
        } else {
          dkv = (long long)page * md.page_elems + (long long)(L % ps) * md.hd;
          if (a.j == 0 && n0 == 0 && hf == 0) a.s.pos_table[(size_t)page * ps + L % ps] = pos;
        }
      }
      if (!__all_sync(0xffffffffu, wait(tfull(b), (uint32_t)(k / 2) & 1u))) break;
      tc_fence_after();
      const uint32_t tr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * BN);
      float* srow = reinterpret_cast<float*>(stg + lane * PG_SEG);

      if constexpr (EPI == EPI_CL_RESID) {
        // units of 32 columns: a row segment of 128 bytes, 8 lanes each
        for (int u = hf; u < BN / 32; u += 2) {
          const int c0 = n0 + 32 * u;
          if (c0 >= a.N) break;
          float v[32];
          tmem_ld_32(tr + 32u * u, v);
          if (alpha) {
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              const float4 g = *reinterpret_cast<const float4*>(alpha + c0 + i);
              v[i] *= g.x; v[i + 1] *= g.y; v[i + 2] *= g.z; v[i + 3] *= g.w;
            }
          }
#pragma unroll
          for (int i = 0; i < 32; i += 4)
            *reinterpret_cast<float4*>(srow + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int rr = 4 * q + (lane >> 3);
            const int dst = __shfl_sync(0xffffffffu, drow, rr);
            const float4 x = *reinterpret_cast<const float4*>(stg + rr * PG_SEG + (lane & 7) * 16);
            if (dst >= 0)  // the only writer of these elements
              atomicAdd(reinterpret_cast<float4*>(a.resid + (size_t)dst * a.ldr + c0 + (lane & 7) * 4), x);
          }
          __syncwarp();
        }
      } else if constexpr (EPI == EPI_CL_SWIGLU) {
        // units of 32 outputs: 32 gate columns and the 32 up columns 64 further on
        for (int u = hf; u < BN / 64; u += 2) {
          const int cg = (u >> 1) * 128 + (u & 1) * 32;
          const int f0 = (n0 >> 1) + (u >> 1) * 64 + (u & 1) * 32;  // first output feature
          if (f0 >= md.ff) break;
          uint32_t g[32], w[32];
          tmem_ld_32_issue(tr + (uint32_t)cg, g);
          tmem_ld_32_issue(tr + (uint32_t)cg + 64u, w);
          tmem_ld_wait();
          uint32_t* sw = reinterpret_cast<uint32_t*>(srow);
#pragma unroll
          for (int i = 0; i < 32; i += 8) {
            uint32_t p[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float y[2];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const float gq = __uint_as_float(g[i + 2 * e + h]);
                y[h] = gq / (1.f + expf(-gq)) * __uint_as_float(w[i + 2 * e + h]);
              }
              p[e] = pack_bf16(y[0], y[1]);
            }
            *reinterpret_cast<uint4*>(sw + i / 2) = make_uint4(p[0], p[1], p[2], p[3]);
          }
          __syncwarp();
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int rr = 8 * q + (lane >> 2), c = (lane & 3) * 8;
            const int dst = __shfl_sync(0xffffffffu, drow, rr);
            const uint4 x = *reinterpret_cast<const uint4*>(stg + rr * PG_SEG + c * 2);
            if (dst >= 0 && f0 + c < md.ff)
              *reinterpret_cast<uint4*>(reinterpret_cast<bf16*>(a.U) + (size_t)dst * md.ff + f0 + c) = x;
          }
          __syncwarp();
        }
      } else {
        // EPI_CL_QKV, units of 32 columns: 16 rotary pairs (i, i + hd/2) of a q or k head, or 32 columns of
        // a v head. The two warps of a row quadrant split each head's units (or the heads, for hd 32), so
        // the rotary factors of 16 pairs are read once for all heads of the tile.
        const int hd = md.hd, half = hd / 2, upt = hd / 32;  // units per head
        const int heads = min(BN, md.qkv_dim - n0) / hd;
        const int h0 = upt > 1 ? 0 : hf, hstep = upt > 1 ? 1 : 2;
        for (int u = upt > 1 ? hf : 0; u < upt; u += 2) {
          float2 cs[16];
          {
            const float4* rp = reinterpret_cast<const float4*>(a.rope + (size_t)pos * half + 16 * u);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 x = rp[i];
              cs[2 * i] = make_float2(x.x, x.y);
              cs[2 * i + 1] = make_float2(x.z, x.w);
            }
          }
          for (int h = h0; h < heads; h += hstep) {
            const int f = n0 + h * hd;  // first feature of the head
            const bool is_q = f < md.q_dim, is_v = f >= md.q_dim + md.kv_dim;
            uint32_t x0[16], x1[16];
            const uint32_t ca = tr + (uint32_t)(h * hd) + (is_v ? 32u * u : 16u * u);
            tmem_ld_16_issue(ca, x0);
            tmem_ld_16_issue(ca + (is_v ? 16u : (uint32_t)half), x1);
            tmem_ld_wait();
            float r0[16], r1[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float p = __uint_as_float(x0[i]), q = __uint_as_float(x1[i]);
              r0[i] = is_v ? p : p * cs[i].x - q * cs[i].y;
              r1[i] = is_v ? q : p * cs[i].y + q * cs[i].x;
            }
            if (is_q && a.q_hi) {
              // 16 + 16 elements of the hi plane, then of the lo plane
              uint32_t* sw = reinterpret_cast<uint32_t*>(srow);
              auto split = [&](const float* v, int at) {
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                  const float a0 = __bfloat162float(__float2bfloat16_rn(v[i])), a1 = __bfloat162float(__float2bfloat16_rn(v[i + 1]));
                  sw[at + i / 2] = pack_bf16(a0, a1);
                  sw[16 + at + i / 2] = pack_bf16(v[i] - a0, v[i + 1] - a1);
                }
              };
              split(r0, 0);
              split(r1, 8);
              __syncwarp();
              const int c = (lane & 3) * 8;
              const int e = c < 16 ? 16 * u + c : half + 16 * u + c - 16;
              bf16* plane = (lane & 4) ? a.q_lo : a.q_hi;
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int rr = 4 * q + (lane >> 3);
                const int dst = __shfl_sync(0xffffffffu, drow, rr);
                const uint4 x = *reinterpret_cast<const uint4*>(stg + rr * PG_SEG + (lane & 7) * 16);
                if (dst >= 0) *reinterpret_cast<uint4*>(plane + (size_t)dst * md.q_dim + f + e) = x;
              }
            } else if (is_q) {
#pragma unroll
              for (int i = 0; i < 16; i += 4) {
                *reinterpret_cast<float4*>(srow + i) = make_float4(r0[i], r0[i + 1], r0[i + 2], r0[i + 3]);
                *reinterpret_cast<float4*>(srow + 16 + i) = make_float4(r1[i], r1[i + 1], r1[i + 2], r1[i + 3]);
              }
              __syncwarp();
              const int c = (lane & 7) * 4;  // staged column: pairs' lower elements, then their upper ones
              const int e = c < 16 ? 16 * u + c : half + 16 * u + c - 16;
#pragma unroll
              for (int q = 0; q < 8; ++q) {
                const int rr = 4 * q + (lane >> 3);
                const int dst = __shfl_sync(0xffffffffu, drow, rr);
                const float4 x = *reinterpret_cast<const float4*>(stg + rr * PG_SEG + c * 4);
                if (dst >= 0) *reinterpret_cast<float4*>(a.Q + (size_t)dst * md.q_dim + f + e) = x;
              }
            } else {
              uint32_t* sw = reinterpret_cast<uint32_t*>(srow);
#pragma unroll
              for (int i = 0; i < 16; i += 8) {
                *reinterpret_cast<uint4*>(sw + i / 2) = make_uint4(pack_bf16(r0[i], r0[i + 1]), pack_bf16(r0[i + 2], r0[i + 3]),
                                                                  pack_bf16(r0[i + 4], r0[i + 5]), pack_bf16(r0[i + 6], r0[i + 7]));
                *reinterpret_cast<uint4*>(sw + 8 + i / 2) =
                    make_uint4(pack_bf16(r1[i], r1[i + 1]), pack_bf16(r1[i + 2], r1[i + 3]), pack_bf16(r1[i + 4], r1[i + 5]),
                               pack_bf16(r1[i + 6], r1[i + 7]));
              }
              __syncwarp();
              const int c = (lane & 3) * 8;
              const int e = is_v ? 32 * u + c : (c < 16 ? 16 * u + c : half + 16 * u + c - 16);
              const int kh = (f - md.q_dim - (is_v ? md.kv_dim : 0)) / hd;
              bf16* base = reinterpret_cast<bf16*>(a.s.pool) +
                           ((size_t)(a.j * 2 + (is_v ? 1 : 0)) * md.Hkv + kh) * md.page_size * hd + e;
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int rr = 8 * q + (lane >> 2);
                const long long dst = __shfl_sync(0xffffffffu, dkv, rr);
                const uint4 x = *reinterpret_cast<const uint4*>(stg + rr * PG_SEG + c * 2);
                if (dst >= 0) *reinterpret_cast<uint4*>(base + dst) = x;
              }
            }
            __syncwarp();
          }
        }
      }
      // the accumulator buffer is read: the leader's MMAs may overwrite it
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(dsmem_map(tempty(b), 0));
    }
  }
  if (*abort_flag) drain_copies();
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // neither CTA leaves while the pair's MMAs, copies or arrivals may touch it
  if (warp == 1) tmem_dealloc_pair(tmem, Sh::TMEM_COLS);
}

template <int BN, int EPI>
static void launch_pf_t(const CUtensorMap* mapX, const CUtensorMap* mapW, const GemmArgs& a, int rows, int max_pairs,
                        cudaStream_t st) {
  constexpr int smem = PgShape<BN>::BYTES;
  (void)ensure_kernel_attrs((const void*)k_gemm_pf<BN, EPI>, smem);  // a failure shows at launch
  const int tiles = ((rows + 255) / 256) * ((a.N + BN - 1) / BN);
  const int pairs = tiles < max_pairs ? tiles : max_pairs;
  launch_k(k_gemm_pf<BN, EPI>, dim3(2 * pairs), PG_THREADS, smem, st, *mapX, *mapW, a);
}

int gemm_pf_max_pairs(int num_sms) {
  constexpr int smem = PgShape<256>::BYTES;
  const auto kernel = k_gemm_pf<256, EPI_CL_RESID>;
  if (ensure_kernel_attrs((const void*)kernel, smem) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(num_sms / 2 * 2);
  cfg.blockDim = dim3(PG_THREADS);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int pairs = 0;
  if (cudaOccupancyMaxActiveClusters(&pairs, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return pairs < num_sms / 2 ? pairs : num_sms / 2;
}

// Tile width by the time of the waves it needs: a tile costs its K steps (of 256 x BN x 16 MMAs, the
// narrower ones bound by operand reads) plus a fixed part for the pipeline's ends.
int gemm_pf_tile_n(int rows, int N, int K, int epi, int head_dim, int max_pairs) {
  const int widths[3] = {256, 128, 64};
  const int cycles[3] = {128, 72, 48};  // per K step of 16
  long long best = 0;
  int pick = 256;
  for (int i = 0; i < 3; ++i) {
    const int bn = widths[i];
    // a gate/up group (128 columns) and a head lie within one tile
    if (bn < 128 && (epi == EPI_CL_SWIGLU || (epi == EPI_CL_QKV && head_dim > 64))) continue;
    const long long tiles = (long long)((rows + 255) / 256) * ((N + bn - 1) / bn);
    const long long waves = (tiles + max_pairs - 1) / max_pairs;
    const long long cost = waves * ((long long)((K + 15) / 16) * cycles[i] + 1500);
    if (i == 0 || cost < best) {
      best = cost;
      pick = bn;
    }
  }
  return pick;
}

void launch_gemm_pf(const CUtensorMap* mapX, const CUtensorMap* mapW, int bn, const GemmArgs& a, int rows, int max_pairs,
                    cudaStream_t st) {
  if (a.epi == EPI_CL_RESID) {
    if (bn == 256) launch_pf_t<256, EPI_CL_RESID>(mapX, mapW, a, rows, max_pairs, st);
    else if (bn == 128) launch_pf_t<128, EPI_CL_RESID>(mapX, mapW, a, rows, max_pairs, st);
    else launch_pf_t<64, EPI_CL_RESID>(mapX, mapW, a, rows, max_pairs, st);
  } else if (a.epi == EPI_CL_SWIGLU) {
    if (bn == 256) launch_pf_t<256, EPI_CL_SWIGLU>(mapX, mapW, a, rows, max_pairs, st);
    else launch_pf_t<128, EPI_CL_SWIGLU>(mapX, mapW, a, rows, max_pairs, st);
  } else {
    if (bn == 256) launch_pf_t<256, EPI_CL_QKV>(mapX, mapW, a, rows, max_pairs, st);
    else if (bn == 128) launch_pf_t<128, EPI_CL_QKV>(mapX, mapW, a, rows, max_pairs, st);
    else launch_pf_t<64, EPI_CL_QKV>(mapX, mapW, a, rows, max_pairs, st);
  }
}

}  // namespace tlf
