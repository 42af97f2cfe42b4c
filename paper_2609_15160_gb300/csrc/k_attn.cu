// Recursion-wise decode attention (T-LoopFormer Sec. 3.3, Eq. 10).
//
// The query of a token at loop r, layer j attends only to cache (r, j) of its
// sequence. That cache holds exactly the tokens that ran loop r (Eq. 11), in
// position order, so the validity mask mu^(r) of Eq. 10 is realised by
// storage and the kernel reads no masked slots. The token's own entry was
// appended before this kernel runs, so the key count is len + 1.
//
// Without recursion-wise caches (the dense-cache ablation, MASKED) every loop
// cache holds a slot per position and slots of tokens that exited earlier are
// masked (position -1): the kernel then also copies each page's positions and
// skips masked keys, reading the masked slots' K/V as the ablation requires.
//
// Work split (stream-K over pages): an item is one (token, kv head); its keys
// live in ceil((len+1)/64) pages. The plan kernel lays all items' pages out in
// one flat order; CTA c of the persistent grid takes the contiguous page range
// [c*per, (c+1)*per), so every CTA streams the same number of pages whatever
// the lengths, and streams them without draining its pipeline at item
// boundaries. A producer warp copies the K and V segments of each page (64
// keys of one kv head, contiguous and 16-byte aligned) into an NST-deep
// shared-memory ring with 1-D bulk TMA copies that complete on mbarriers. The
// copies carry an L2 evict-first hint: each page is read once per launch, and the
// hint keeps the step's small reused buffers resident in L2. The
// eight consumer warps split every page (or four of them, taking pages in turn), release the stage on a per-stage
// mbarrier, and keep an online-softmax state (running max, sum, output slice)
// in float32 for the G query heads of the kv head (grouped-query attention),
// with LPK lanes sharing a key (16 bytes each) and xor-shuffle reductions.
// Scores are in base 2 (q pre-scaled by log2(e)/sqrt(hd)).
//
// When a CTA finishes its part of an item it merges its warps (with one query head
// a kv head, a merging warp does while the consumers go on). An item that
// lies inside one CTA's range is written out directly. Otherwise each
// contributing CTA stores a partial (max, sum, output) and takes a ticket with
// an atomic counter, and the CTA that takes the last ticket merges the
// partials and writes the output (no CTA ever waits for another). On the
// tcgen05 decode path the output also gets its lo plane, bf16(o - bf16(o)): the
// output projection then takes a two-term operand.
#include <type_traits>

#include "tlf_internal.cuh"

namespace tlf {

constexpr int ATT_PS = 64;     // keys per page (the only page size the library accepts)
constexpr int ATT_WARPS = 8;   // consumer warps

template <typename T, int HD, int G>
struct AttnShape {
  static constexpr int VEC = 16 / (int)sizeof(T);   // elements per lane per key
  static constexpr int LPK = HD / VEC;              // lanes per key
  static constexpr int KPW = 32 / LPK;              // keys per warp step
  static constexpr int SEG_BYTES = ATT_PS * HD * (int)sizeof(T);       // one page of K (or V) of one head
  static constexpr int STAGE_BYTES = 2 * SEG_BYTES;
  static constexpr int NST = (98304 / STAGE_BYTES) < 2 ? 2 : ((98304 / STAGE_BYTES) > 8 ? 8 : (98304 / STAGE_BYTES));
  // Page teams: with one query head a kv head the warps' chain per page, not its instructions, is what a page costs, so
  // two teams of four warps take the pages in turn (a ring stage then always belongs to one team, so its depth is even).
  // With the registers of two CTAs an SM: 200 rows of 64-700 keys, 16 heads x 64, 80 -> 69 us; 32 rows of 128-8192 keys
  // 98.5 -> 95 us. A ring of two stages is too short for two teams (float32 heads of 128: 32 rows of 128-8192 keys, 8
  // heads, 178 us, 173 with one).
  static constexpr int TEAMS = G == 1 && NST >= 4 && NST % 2 == 0 ? 2 : 1;
  // A warp of its own merges the parts of all items of a CTA but the last, out of REDS buffers, while the consumer warps
  // go on without a barrier: the 200 rows above 69 -> 62 us (5.1 TB/s), the 32 rows 95 -> 93 us (6.0 TB/s), 64 rows of
  // 500-1500 keys, 8 heads x 128, 50 us. The last item is the launch's tail, where all warps merge faster (one CTA an
  // item, 8 rows of 300-700 keys: 14.4 us, 15.5 with the one warp). With more query heads a kv head the tenth warp's
  // registers cost more than the barriers: 100 rows of 30-500 keys, 16 / 8 heads x 128, 40 -> 51 us. Float32 heads of 128
  // (one CTA an SM): 200 rows of 1-64 keys 31.4 us with the warp, 29.2 without.
  static constexpr bool MERGER = G == 1 && HD * sizeof(T) <= 256;
  static constexpr int THREADS = 32 * (ATT_WARPS + 1 + (MERGER ? 1 : 0));
  static constexpr int TEAM_WARPS = ATT_WARPS / TEAMS;
  static constexpr int KEYS_PER_WARP = ATT_PS / TEAM_WARPS;
  static constexpr int STEPS = KEYS_PER_WARP / KPW;
  static_assert(LPK >= 1 && LPK <= 32 && (32 % LPK) == 0, "head_dim / vector width mismatch");
  static_assert(STEPS >= 1, "page too small for the warp split");
};

// Merge buffers. MASKED (the dense-cache ablation): each stage also holds the page's 64 positions, -1 = masked slot, and
// heads of 128 give up a buffer for them, so that two CTAs still share an SM (16 rows of 2000 keys, 16 heads x 128: a
// step of 872 us; 1079 with four buffers and one CTA an SM; 898 before there were several).
template <typename T, int HD, int G, bool MASKED>
constexpr int attn_reds() { return !AttnShape<T, HD, G>::MERGER ? 1 : MASKED && HD == 128 ? 3 : 4; }
template <typename T, int HD, int G, bool MASKED>
constexpr int attn_smem_bytes() {
  using S = AttnShape<T, HD, G>;
  constexpr int REDS = attn_reds<T, HD, G, MASKED>();
  return 128 + S::NST * S::STAGE_BYTES + REDS * ATT_WARPS * G * (HD + 2) * 4 + (MASKED ? S::NST * ATT_PS * 4 : 0) +
         2 * (S::NST + REDS) * 8 + 16;
}
// Whether the shared memory of two CTAs fits an SM (228 KB, 1 KB of it reserved for each CTA).
template <typename T, int HD, int G, bool MASKED>
constexpr bool attn_two_per_sm() { return 2 * (attn_smem_bytes<T, HD, G, MASKED>() + 1024) <= 233472; }
static_assert(attn_two_per_sm<bf16, 128, 1, true>() && attn_two_per_sm<bf16, 64, 1, true>() &&
                  attn_two_per_sm<bf16, 32, 1, true>() && attn_two_per_sm<bf16, 128, 1, false>(),
              "the merge buffers cost the second CTA of an SM");

__device__ __forceinline__ void consumer_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * ATT_WARPS) : "memory");
}

// CTAs an SM that the registers are bounded for: two where the shared memory lets them, which gives one query head the
// registers it can use (96; 56 otherwise). Four heads then spill (96 registers, 180 to 224 bytes), which still pays at
// head_dim 64 (200 rows of 1-64 keys, 32 / 8 heads, 35.3 us, 38.6 with one CTA an SM; one row of 100 keys 13.0 and 12.8),
// but not at 128, where one CTA an SM takes 168: one row of 3000 keys, 16 / 4 heads, 28.7 us (33.3 with two CTAs), 36
// rows of about 2950 keys, 32 / 8 heads, 136 us (142), though 200 rows of 1-64 keys 47.7 us (45.5).
template <typename T, int HD, int G, bool MASKED>
constexpr int attn_ctas_per_sm() { return attn_two_per_sm<T, HD, G, MASKED>() && !(HD == 128 && G == 4) ? 2 : 1; }

template <typename T, int HD, int G, bool MASKED>
__global__ void __launch_bounds__(AttnShape<T, HD, G>::THREADS, attn_ctas_per_sm<T, HD, G, MASKED>())
    k_attn_decode(ModelDims md, StepDev s, int r, int j, const float* __restrict__ Q, float* __restrict__ part,
                  T* __restrict__ O, int* __restrict__ cnt, bool o_lo) {
  using S = AttnShape<T, HD, G>;
  constexpr int REDS = attn_reds<T, HD, G, MASKED>();
  // output element (token k, query head hq, dim e); with o_lo also the lo plane of the
  // projection's two-term operand (bf16 of the rounding remainder, max_batch rows down)
  auto store_o = [&](int k, int hq, int e, float val) {
    const size_t at = (size_t)k * md.q_dim + (size_t)hq * HD + e;
    const T hi = from_f32<T>(val);
    O[at] = hi;
    if (o_lo) O[(size_t)md.max_batch * md.q_dim + at] = from_f32<T>(val - to_f32(hi));
  };
  constexpr int PSZ = G * (HD + 2);  // floats of one partial: per head, HD outputs then max and sum
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  uint8_t* ring = smem;                                                   // [NST][K seg | V seg]
  float* red = reinterpret_cast<float*>(ring + S::NST * S::STAGE_BYTES);  // [warps][G][HD + 2]
  int* mring = reinterpret_cast<int*>(red + REDS * ATT_WARPS * PSZ);       // [NST][64] positions (MASKED)
  uint64_t* full = reinterpret_cast<uint64_t*>(mring + (MASKED ? S::NST * ATT_PS : 0));
  uint64_t* empty = full + S::NST;
  uint64_t* red_full = empty + S::NST;       // [REDS] an item's parts of all warps are in its buffer (MERGER)
  uint64_t* red_empty = red_full + REDS;     // [REDS] and merged
  int* flags = reinterpret_cast<int*>(red_empty + REDS);  // last contributor: consumers, merging warp
  volatile int* abort_flag = flags + 2;  // set when a bounded wait runs out: later waits are skipped

  pdl_wait();
  // bf16: the next projection's CTAs need more shared memory than two CTAs of this kernel leave, and start late enough.
  // Float32: those of the CUDA-core projection need registers only, and let start early they filled the first SMs that
  // this kernel's CTAs left instead of all SMs: a step of two layers of width 192 over 600 keys, 64 / 128 / 256 rows, 474 /
  // 716 / 1556 us against 411 / 617 / 1138 us when they start at the end; width 512, 1 / 256 rows, 317 / 2384 and 286 / 1875 us.
  if (sizeof(T) == 2) pdl_trigger();
  const int maxB = md.max_batch, M = md.M, Hkv = md.Hkv;
  const int n_r = s.n[r];
  const int* pbase = s.item_base + r * (maxB + 1);  // first flat page of each token's items
  const int* nkeys = s.nch + r * maxB;               // keys of each of the token's items (plan kernel)
  auto pages_of = [&](int kk) { return (nkeys[kk] + ATT_PS - 1) / ATT_PS; };
  const int total = (n_r > 0) ? pbase[n_r] : 0;
  const int per = (total + gridDim.x - 1) / gridDim.x;
  const int p0 = blockIdx.x * per;
  if (p0 >= total) return;
  const int p1 = min(total, p0 + per);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < S::NST; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), S::TEAM_WARPS);
    }
    for (int i = 0; i < REDS; ++i) {
      mbar_init(smem_u32(&red_full[i]), ATT_WARPS);
      mbar_init(smem_u32(&red_empty[i]), 1);
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  __syncthreads();

  // (token, kv head, page) of flat page p: the largest k with pbase[k] <= p, found by the warp
  // with independent loads (32 entries of pbase a round) and a ballot
  auto locate = [&](int p, int& k, int& h, int& g) {
    int kk = 0;
    for (int b = 0; b < n_r; b += 32) {
      const int i = b + lane;
      const unsigned le = __ballot_sync(0xffffffffu, i < n_r && pbase[i] <= p);
      if (le) kk = b + 31 - __clz((int)le);
      if (le != 0xffffffffu) break;  // pbase is non-decreasing: no later entry is <= p
    }
    k = kk;
    const int off = p - pbase[k], np = pages_of(k);
    h = off / np;
    g = off % np;
  };

  // Merge of the CTA's part of item (k, h), by NT threads (t0 is this one's index) that `sync` synchronises: written out,
  // or stored as a partial, which the last contributor merges with the others'.
  auto finish_item = [&](const float* mred, int* flag, int k, int h, int t0, auto nt, auto sync) {
    constexpr int NT = decltype(nt)::value;
    const int np = pages_of(k);
    const int item = k * Hkv + h;
    const int first = pbase[k] + h * np;
    const int c_first = first / per, c_last = (first + np - 1) / per;
    float* my = part + (size_t)(item + blockIdx.x) * PSZ;
    const int nparts = c_last - c_first + 1;
    // merged state of this CTA's warps: thread t owns (head gg, dim e)
    for (int t = t0; t < G * HD; t += NT) {
      const int gg = t / HD, e = t % HD;
      float mx = -INFINITY;
#pragma unroll
      for (int w = 0; w < ATT_WARPS; ++w) mx = fmaxf(mx, mred[(w * G + gg) * (HD + 2) + HD]);
      float o = 0.f, l = 0.f;
#pragma unroll
      for (int w = 0; w < ATT_WARPS; ++w) {
        const float* rw = mred + (w * G + gg) * (HD + 2);
        const float f = (rw[HD] == -INFINITY) ? 0.f : exp2f(rw[HD] - mx);
        o = fmaf(f, rw[e], o);
        l = fmaf(f, rw[HD + 1], l);
      }
      if (nparts == 1) {
        store_o(k, h * G + gg, e, o / l);
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
      sync();
      if (t0 == 0) {
        const int ticket = atomicAdd(cnt + item, 1);
        *flag = (ticket == nparts - 1);
      }
      sync();
      if (*flag) {
        // last contributor: merge the partials of CTAs c_first..c_last
        __threadfence();
        // a thread's elements of a head go together: their loads are in flight at once, and the head's maximum and
        // factors are read once. One at a time, the merging warp took four trips over the partials of a head of 128: one
        // row of 3000 keys, 8 heads x 128, 22.4 us, now 16.2 (17.0 before there was a merging warp); 8 rows of 300-700
        // keys 19.0, now 14.8 (16.0).
        constexpr int E = HD > NT ? HD / NT : 1;
        for (int t = t0; t < G * HD; t += NT * E) {
          const int gg = t / HD, e = t % HD;
          float mx = -INFINITY;
          for (int c = c_first; c <= c_last; ++c)
            mx = fmaxf(mx, __ldcg(part + (size_t)(item + c) * PSZ + gg * (HD + 2) + HD));
          float o[E] = {}, l = 0.f;
          for (int c = c_first; c <= c_last; ++c) {
            const float* pp = part + (size_t)(item + c) * PSZ + gg * (HD + 2);
            const float f = exp2f(__ldcg(pp + HD) - mx);
#pragma unroll
            for (int i = 0; i < E; ++i) o[i] = fmaf(f, __ldcg(pp + e + NT * i), o[i]);
            l = fmaf(f, __ldcg(pp + HD + 1), l);
          }
#pragma unroll
          for (int i = 0; i < E; ++i) store_o(k, h * G + gg, e + NT * i, o[i] / l);
        }
        if (t0 == 0) cnt[item] = 0;  // ready for the next launch
      }
    }
  };

  if (warp == ATT_WARPS) {
    // ---------------- producer warp ----------------
    int k, h, g;
    locate(p0, k, h, g);  // the whole warp (ballot)
    if (lane == 0) {
      const uint64_t kv_policy = l2_policy_evict_first();  // pages are read once per launch
      int slot = s.slots[s.idx[r * maxB + k]];
      int L = nkeys[k];
      for (int p = p0; p < p1; ++p) {
        const int i = p - p0, st = i % S::NST;
        if (i >= S::NST && (*abort_flag || !mbar_wait(smem_u32(&empty[st]), ((i / S::NST) - 1) & 1, s.err))) {
          *abort_flag = 1;
          break;
        }
        const uint32_t bar = smem_u32(&full[st]);
        const int page = s.page_table[((size_t)slot * M + r) * md.max_pages + g];
        const int valid = min(ATT_PS, L - g * ATT_PS);
        if (page < 0 || page >= md.n_pages || valid <= 0) {
          atomicOr(s.err, DEVERR_INDEX);
          mbar_arrive(bar);  // complete the phase without data
        } else {
          const T* pg = reinterpret_cast<const T*>(s.pool) + (size_t)page * md.page_elems;
          const uint32_t bytes = (uint32_t)(valid * HD * sizeof(T));
          uint8_t* dst = ring + st * S::STAGE_BYTES;
          mbar_arrive_expect_tx(bar, 2 * bytes + (MASKED ? ATT_PS * 4 : 0));
          if (MASKED) bulk_g2s(smem_u32(mring + st * ATT_PS), s.pos_table + (size_t)page * ATT_PS, ATT_PS * 4, bar);
          bulk_g2s_hint(smem_u32(dst), pg + ((size_t)(j * 2 + 0) * Hkv + h) * ATT_PS * HD, bytes, bar, kv_policy);
          bulk_g2s_hint(smem_u32(dst + S::SEG_BYTES), pg + ((size_t)(j * 2 + 1) * Hkv + h) * ATT_PS * HD, bytes, bar,
                        kv_policy);
        }
        if (++g == pages_of(k)) {
          g = 0;
          if (++h == Hkv) {
            h = 0;
            do {
              ++k;
            } while (k < n_r && nkeys[k] == 0);  // rows with no keys have no pages (no gather)
            if (k < n_r) {
              slot = s.slots[s.idx[r * maxB + k]];
              L = nkeys[k];
            }
          }
        }
      }
    }
    return;
  }

  if (S::MERGER && warp == ATT_WARPS + 1) {
    // ---------------- merging warp ----------------
    int k, h, g;
    locate(p0, k, h, g);
    for (int p = p0, it = 0; (p += pages_of(k) - g) < p1; ++it) {  // the items before the CTA's last
      const int b = it % REDS;
      if (!*abort_flag && !mbar_wait(smem_u32(&red_full[b]), (it / REDS) & 1, s.err)) *abort_flag = 1;
      finish_item(red + b * ATT_WARPS * PSZ, flags + 1, k, h, lane, std::integral_constant<int, 32>{}, [] { __syncwarp(); });
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&red_empty[b]));
      g = 0;
      if (++h == Hkv) {
        h = 0;
        do {
          ++k;
        } while (k < n_r && nkeys[k] == 0);
      }
    }
    return;
  }

  // ---------------- consumer warps ----------------
  const int grp = lane / S::LPK, part_lane = lane % S::LPK;
  const int team = warp / S::TEAM_WARPS, team_warp = warp % S::TEAM_WARPS;
  const float scale = 1.4426950408889634f * rsqrtf((float)HD);
  int k, h, g;
  locate(p0, k, h, g);
  int L = 0;
  float q[G][S::VEC];
  float run_m[G], run_l[G], acc[G][S::VEC];
  auto begin_item = [&]() {
    L = nkeys[k];
    const float* qrow = Q + (size_t)k * md.Hq * HD;
#pragma unroll
    for (int gg = 0; gg < G; ++gg) {
#pragma unroll
      for (int e = 0; e < S::VEC; ++e) q[gg][e] = qrow[(h * G + gg) * HD + part_lane * S::VEC + e] * scale;
      run_m[gg] = -INFINITY;
      run_l[gg] = 0.f;
#pragma unroll
      for (int e = 0; e < S::VEC; ++e) acc[gg][e] = 0.f;
    }
  };
  begin_item();
  int it = 0;  // items so far

  for (int p = p0; p < p1; ++p) {
    const int i = p - p0, st = i % S::NST;
    if (S::TEAMS == 1 || i % S::TEAMS == team) {  // this warp's team takes the page
      // a wait that runs out records the error word; the page is then computed on stale data
      if (!*abort_flag && !mbar_wait(smem_u32(&full[st]), (i / S::NST) & 1, s.err)) *abort_flag = 1;
      const int valid = min(ATT_PS, L - g * ATT_PS);
      const T* sk = reinterpret_cast<const T*>(ring + st * S::STAGE_BYTES);
      const T* sv = reinterpret_cast<const T*>(ring + st * S::STAGE_BYTES + S::SEG_BYTES);
      const int* smask = mring + st * ATT_PS;
      // key slot usable: inside the cache and, for a full-length cache, not masked (mu^(r) of Eq. 10)
      auto usable = [&](int key) { return key < valid && (!MASKED || smask[key] >= 0); };

      float sc[S::STEPS][G];
#pragma unroll
      for (int t = 0; t < S::STEPS; ++t) {
        const int key = team_warp * S::KEYS_PER_WARP + t * S::KPW + grp;
        float kv[S::VEC];
        const bool use = usable(key);
        if (use) {
          Vec16<T>::load(sk + key * HD + part_lane * S::VEC, kv);
        } else {
#pragma unroll
          for (int e = 0; e < S::VEC; ++e) kv[e] = 0.f;
        }
#pragma unroll
        for (int gg = 0; gg < G; ++gg) {
          float d = 0.f;
#pragma unroll
          for (int e = 0; e < S::VEC; ++e) d = fmaf(q[gg][e], kv[e], d);
#pragma unroll
          for (int o = S::LPK / 2; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
          sc[t][gg] = use ? d : -INFINITY;
        }
      }
#pragma unroll
      for (int gg = 0; gg < G; ++gg) {
        float pm = sc[0][gg];
#pragma unroll
        for (int t = 1; t < S::STEPS; ++t) pm = fmaxf(pm, sc[t][gg]);
#pragma unroll
        for (int o = S::LPK; o < 32; o <<= 1) pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
        if (pm > run_m[gg]) {
          const float cr = exp2f(run_m[gg] - pm);  // 0 when run_m was -inf
          run_l[gg] *= cr;
#pragma unroll
          for (int e = 0; e < S::VEC; ++e) acc[gg][e] *= cr;
          run_m[gg] = pm;
        }
      }
#pragma unroll
      for (int t = 0; t < S::STEPS; ++t) {
        const int key = team_warp * S::KEYS_PER_WARP + t * S::KPW + grp;
        if (usable(key)) {
          float vv[S::VEC];
          Vec16<T>::load(sv + key * HD + part_lane * S::VEC, vv);
#pragma unroll
          for (int gg = 0; gg < G; ++gg) {
            const float pr = exp2f(sc[t][gg] - run_m[gg]);
            run_l[gg] += pr;
#pragma unroll
            for (int e = 0; e < S::VEC; ++e) acc[gg][e] = fmaf(pr, vv[e], acc[gg][e]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&empty[st]));
    }

    const bool item_end = (g + 1 == pages_of(k));
    if (item_end || p + 1 == p1) {
      // ---- this CTA's part of item (k, h) is done: merge the lane groups, then the warps ----
      const int b = it % REDS;
      float* mred = red + b * ATT_WARPS * PSZ;
#pragma unroll
      for (int gg = 0; gg < G; ++gg) {
#pragma unroll
        for (int o = S::LPK; o < 32; o <<= 1) {
          run_l[gg] += __shfl_xor_sync(0xffffffffu, run_l[gg], o);
#pragma unroll
          for (int e = 0; e < S::VEC; ++e) acc[gg][e] += __shfl_xor_sync(0xffffffffu, acc[gg][e], o);
        }
      }
      if (S::MERGER && it >= REDS && !*abort_flag &&
          !mbar_wait(smem_u32(&red_empty[b]), ((it / REDS) - 1) & 1, s.err))
        *abort_flag = 1;
      ++it;
      if (grp == 0) {
#pragma unroll
        for (int gg = 0; gg < G; ++gg) {
          float* rw = mred + (warp * G + gg) * (HD + 2);
#pragma unroll
          for (int e = 0; e < S::VEC; ++e) rw[part_lane * S::VEC + e] = acc[gg][e];
          if (part_lane == 0) {
            rw[HD] = run_m[gg];
            rw[HD + 1] = run_l[gg];
          }
        }
      }
      if (S::MERGER && p + 1 < p1) {
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&red_full[b]));
      } else {
        consumer_sync();
        finish_item(mred, flags, k, h, tid, std::integral_constant<int, 32 * ATT_WARPS>{}, consumer_sync);
        if (!S::MERGER) consumer_sync();  // `red` and the flag are reused by the next item
      }
      if (p + 1 < p1) {
        g = 0;
        if (++h == Hkv) {
          h = 0;
          do {
            ++k;
          } while (k < n_r && nkeys[k] == 0);
        }
        begin_item();
      }
    } else {
      ++g;
    }
  }
  if (*abort_flag) drain_copies();
}

template <typename T, int HD, int G, bool MASKED>
static void attn_launch_v(const ModelDims& md, const StepDev& s, int r, int j, const float* Q, float* part, void* O,
                          int* cnt, int grid, cudaStream_t st, bool o_lo) {
  constexpr int smem = attn_smem_bytes<T, HD, G, MASKED>();
  (void)ensure_kernel_attrs((const void*)k_attn_decode<T, HD, G, MASKED>, smem);  // a failure shows at launch
  launch_k(k_attn_decode<T, HD, G, MASKED>, grid, AttnShape<T, HD, G>::THREADS, smem, st, md, s, r, j, Q, part, (T*)O, cnt, o_lo);
}

template <typename T, int HD, int G>
static void attn_launch(const ModelDims& md, const StepDev& s, int r, int j, const float* Q, float* part, void* O,
                        int* cnt, int grid, cudaStream_t st, bool o_lo) {
  o_lo = o_lo && std::is_same<T, bf16>::value;
  if constexpr (std::is_same<T, bf16>::value) {
    if (md.ablation == TLF_ABLATION_DENSE_CACHE) {
      attn_launch_v<T, HD, G, true>(md, s, r, j, Q, part, O, cnt, grid, st, o_lo);
      return;
    }
  }
  attn_launch_v<T, HD, G, false>(md, s, r, j, Q, part, O, cnt, grid, st, o_lo);
}

#define TLF_ATTN_DISPATCH(FN, ...)                                                              \
  do {                                                                                          \
    const int G_ = md.Hq / md.Hkv;                                                              \
    if (md.dtype == 1) {                                                                        \
      if (md.hd == 128 && G_ == 1) FN<bf16, 128, 1>(__VA_ARGS__);                               \
      else if (md.hd == 128 && G_ == 2) FN<bf16, 128, 2>(__VA_ARGS__);                          \
      else if (md.hd == 128 && G_ == 4) FN<bf16, 128, 4>(__VA_ARGS__);                          \
      else if (md.hd == 64 && G_ == 1) FN<bf16, 64, 1>(__VA_ARGS__);                            \
      else if (md.hd == 64 && G_ == 2) FN<bf16, 64, 2>(__VA_ARGS__);                            \
      else if (md.hd == 64 && G_ == 4) FN<bf16, 64, 4>(__VA_ARGS__);                            \
      else if (md.hd == 32 && G_ == 1) FN<bf16, 32, 1>(__VA_ARGS__);                            \
      else FN<bf16, 32, 2>(__VA_ARGS__);                                                        \
    } else {                                                                                    \
      if (md.hd == 128 && G_ == 1) FN<float, 128, 1>(__VA_ARGS__);                              \
      else if (md.hd == 128 && G_ == 2) FN<float, 128, 2>(__VA_ARGS__);                         \
      else if (md.hd == 64 && G_ == 1) FN<float, 64, 1>(__VA_ARGS__);                           \
      else if (md.hd == 64 && G_ == 2) FN<float, 64, 2>(__VA_ARGS__);                           \
      else if (md.hd == 32 && G_ == 1) FN<float, 32, 1>(__VA_ARGS__);                           \
      else if (md.hd == 32 && G_ == 2) FN<float, 32, 2>(__VA_ARGS__);                           \
      else if (md.hd == 16 && G_ == 1) FN<float, 16, 1>(__VA_ARGS__);                           \
      else FN<float, 16, 2>(__VA_ARGS__);                                                       \
    }                                                                                           \
  } while (0)

void launch_attn_decode(const ModelDims& md, const StepDev& s, int r, int j, const float* Q, float* part, void* O,
                        int* cnt, int grid, cudaStream_t st, bool o_lo) {
  TLF_ATTN_DISPATCH(attn_launch, md, s, r, j, Q, part, O, cnt, grid, st, o_lo);
}

// Resident CTAs: two per SM fit the ~104 KB ring of the largest head size.
int attn_decode_grid(const ModelDims& md, int num_sms) { return 2 * num_sms; }

// Floats of partial results one launch may write: one partial slot per (item + CTA) index.
size_t attn_partial_floats(const ModelDims& md, int grid) {
  const int G = md.Hq / md.Hkv;
  return ((size_t)md.max_batch * md.Hkv + grid) * G * (md.hd + 2);
}

}  // namespace tlf
