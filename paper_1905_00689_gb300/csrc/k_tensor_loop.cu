// Tensor-core path where the one-launch kernel per stream tile (k_tensor_seq.cu)
// does not apply: all T timesteps of a layer in one launch over all stream
// tiles, the factors resident on chip (bf16 factors, fp32 accumulate,
// activations as bf16 pairs as in k_tensor.cu).
//
// The per-timestep kernels of k_tensor.cu pay two or three dependent launches
// a step (their set-up, the wait for the whole grid before, the first copies)
// and stream the factors through shared memory again every step: 23.5 us a
// step at H = 512, B = 256, K = 512 with two intermediate depths, for 2 us of
// tensor work.  Here every CTA holds its share of both factors for the whole
// sequence and the CTAs exchange h and tau' through L2, ordered by counters
// (11.4 us a step):
//
//   role A (tau'): CTA group (row tile r, stream tiles) of ga CTAs; CTA z
//     holds 128 packed rows of V_h (rpg rows of each of 128 / rpg gates) x its
//     part of H (up to 512 columns) in shared memory, 128 KB.  Per stream tile
//     of NT streams: wait until every CTA has published h_{t-1} of the tile,
//     stream its pair in by TMA, accumulate in tensor memory; with ga > 1 the
//     group's partial sums go to the CTA that finishes the row (st.async) and
//     are added in rank order; tau' = sigma (sum + P_t) is stored as its pair
//     and the tile's tau' counter raised.
//   role B (gates and cells): CTA group (128 hidden units, stream tiles) of
//     4 / GP CTAs; CTA z holds the U rows of its GP gates, all K terms, in
//     tensor memory as the A operand of the MMAs (GP K / 2 columns; terms past
//     its capacity in shared memory).  Per stream tile: wait for tau' of every
//     row tile, stream its pair in, accumulate; with GP = 1 the gates' sums go
//     to the CTA that owns the streams (split by gate, a CTA sends one sum per
//     unit and stream where a split of the terms would send four); the cells
//     of Sec. II; h_t is stored as its pair and the tile's h counter raised,
//     then the outputs are written.
//
// A CTA has both roles and runs them in turn each step; the copies and MMAs
// of one stream tile overlap the epilogue of another.  Intermediate depths
// start a new accumulator segment (a depth inside a 16-term slice splits the
// slice into pieces whose other terms are zero), so no term is multiplied
// twice: the full depth is the sum of all segments and is finished first; the
// depths' cells run while the next step's tau' is on its way.  Long sums
// (K > 512) are cut into segments as well; without depths these take two
// accumulators in turn and are added up as they come.
//
// What bounds a step is latency and the epilogue's instructions, not bytes or
// the tensor pipe.  At H = 512, B = 256, K = 512 (SM cycles, CTA 0; 19,500 a
// step with the marks): h counter to MMAs done 2600, tau' stored 1300, its
// counter seen 4000 later (the store's release about 1200, the slowest CTA and
// the poll the rest), MMAs done 4500 (behind the depths), gate exchange 3600,
// cells 600, h counter seen 2100.
//
// One buffer each of h and tau' is enough: h_t of a tile is written only after
// every row tile has published tau'_t, hence read h_{t-1}; tau'_{t+1} only
// after all units have published h_t, hence read tau'_t.  The two receive
// buffers of an exchange alternate: a CTA sends use u + 2 only after receiving
// its peers' use u + 1, which they sent after finishing use u.
//
// The grid is at most one wave (one CTA per SM, cooperative launch), so every
// CTA is resident and each wait ends; every wait is bounded in wall time all
// the same: one that runs out writes the status word, all CTAs leave their
// loops, and CTAs of a cluster meet before any of them exits.
#include <cuda.h>

#include <climits>

#include "internal.h"
#include "ptx.cuh"

namespace lstm_approx_impl {
namespace {

using namespace lstm_approx_dev;

// Epilogue warps per 32-lane quarter of tensor memory, each taking 8 or 16 of a tile's streams.
__host__ __device__ constexpr int loop_epw(int nt) { return nt >= 32 ? 4 : 2; }
__host__ __device__ constexpr int loop_threads(int nt) { return 64 + 128 * loop_epw(nt); }
constexpr uint32_t kChunkBytes = 128 * 128;  // 128 factor rows x 64 bf16
constexpr int kMaxStages = 16;
constexpr int kMaxRegions = 4;  // accumulator regions per role
constexpr uint32_t kBarBytes = 1024;

struct LoopLayout {  // offsets from the 1024-byte aligned base
  uint32_t ux, ring, rxa, rxb, bar, total;
};
__host__ __device__ inline LoopLayout loop_layout(int nt, int nka, int ux_chunks, int stages, uint32_t rxa_bytes,
                                                  uint32_t rxb_bytes, bool share_rx) {
  LoopLayout l;
  l.ux = kChunkBytes * nka;
  l.ring = l.ux + kChunkBytes * ux_chunks;
  l.rxa = l.ring + (uint32_t)stages * nt * 256u;
  l.rxb = share_rx ? l.rxa : l.rxa + 2 * rxa_bytes;
  l.bar = share_rx ? l.rxa + 2 * (rxa_bytes > rxb_bytes ? rxa_bytes : rxb_bytes) : l.rxb + 2 * rxb_bytes;
  l.total = l.bar + kBarBytes + 1024u;
  return l;
}

// Eight terms [k, k + 8) of a U row, those outside [lo, hi) zero.
__device__ __forceinline__ uint4 masked_terms(const __nv_bfloat16* row, int k, int lo, int hi) {
  uint4 v = __ldg(reinterpret_cast<const uint4*>(row + k));
  uint32_t* w = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int k0 = k + 2 * e;
    if (k0 < lo || k0 >= hi) w[e] &= 0xFFFF0000u;
    if (k0 + 1 < lo || k0 + 1 >= hi) w[e] &= 0x0000FFFFu;
  }
  return v;
}

// Orders this thread's generic-proxy memory accesses against async-proxy (TMA) ones, either way.
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

__device__ __forceinline__ void red_release_gpu_add(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Named barrier `id` of `count` threads; returns whether any of them passed `pred`.
__device__ __forceinline__ bool block_or_named(int id, int count, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(pred ? 1u : 0u), "r"(id), "r"(count)
      : "memory");
  return r != 0u;
}

// 3-D tiled load (plane, row, 64 inner elements): the box at inner element c0 (a multiple of 8), row c1
// and plane c2, completing its bytes on the mbarrier `mb`.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, uint32_t mb, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::
          "r"(dst),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(mb), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// umma_bf16 with the A operand (128 rows x 16 terms, two terms per 32-bit column) in tensor memory.
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Two loads of 32 lanes x 8 consecutive columns and the wait for both in one statement.
template <bool kTogether = false>
__device__ __forceinline__ void tmem_ld8x2_sync(uint32_t ta, uint32_t tb, float (&va)[8], float (&vb)[8]) {
  uint32_t r[16];
  if constexpr (!kTogether) __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(ta), "r"(tb)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    va[i] = __uint_as_float(r[i]);
    vb[i] = __uint_as_float(r[8 + i]);
  }
}

// Store 8 consecutive 32-bit columns per lane into tensor memory; complete with tmem_wait_st().
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float (&v)[8]) {
  __syncwarp();
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr),
               "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
               "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
               "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
               : "memory");
}

// Bounded wait until *c has reached `target` (acquire at GPU scope), then
// orders later TMA reads of this thread after what the counter released.
__device__ __forceinline__ bool wait_counter(const unsigned* c, unsigned target, uint64_t limit,
                                             const volatile int* err) {
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(c) : "memory");
    if ((int)(v - target) >= 0) break;
    if ((i & 31u) == 0u) {
      if (*err != 0) return false;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit) return false;
    }
  }
  fence_proxy_async_all();
  return true;
}

// One unit's cell of one stream at the intermediate depth kd from the factor and the stored tau' pair, in place
// of sums in which a tau' past the depth that is not finite met a zero of U (see run_sets).  `u`, `tau`: the unit's
// and the stream's first gate; gate g follows at u + g gate_u and tau + g Ks.
__device__ __noinline__ void depth_cell(const __nv_bfloat16* u, long long gate_u, const __nv_bfloat16* tau,
                                        long long tau_plane, int Ks, int kd, const float* bias, int H, float c_prev,
                                        float* h_out, float* c_out) {
  float y[4];
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    float acc = 0.f;
#pragma unroll 2
    for (int k = 0; k < kd; k += 8) {
      const uint4 wu = __ldg(reinterpret_cast<const uint4*>(u + g * gate_u + k));
      const uint4 wh = __ldcg(reinterpret_cast<const uint4*>(tau + g * Ks + k));
      const uint4 wl = __ldcg(reinterpret_cast<const uint4*>(tau + tau_plane + g * Ks + k));
      const uint32_t* pu = reinterpret_cast<const uint32_t*>(&wu);
      const uint32_t* ph = reinterpret_cast<const uint32_t*>(&wh);
      const uint32_t* pl = reinterpret_cast<const uint32_t*>(&wl);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        auto value = [&](const uint32_t* w) {
          return __uint_as_float((e & 1) != 0 ? w[e >> 1] & 0xFFFF0000u : w[e >> 1] << 16);
        };
        if (k + e < kd) acc = fmaf(value(pu), value(ph) + value(pl), acc);
      }
    }
    y[g] = acc + bias[g * H];
  }
  float hh, cc;
  lstm_cell_s(y[0], y[1], y[2], y[3], c_prev, hh, cc);
  if (h_out != nullptr) *h_out = hh;
  if (c_out != nullptr) *c_out = cc;
}

// Position in the stage ring: slot and phase parity, advanced without divisions (one thread issues
// everything, so its instructions are on the path of every step).
struct RingPos {
  int slot = 0;
  uint32_t parity = 0;
  __device__ __forceinline__ void next(int stages) {
    if (++slot == stages) {
      slot = 0;
      parity ^= 1u;
    }
  }
};

// SD: an intermediate depth lies inside a 16-term slice (what that takes in the epilogue is left out of the other
// shapes' kernels: with it H = 1024, B = 1024, K = 128 without depths took 1132 us a run instead of 943)
template <int NT, int GP, bool MB, bool SD>
__global__ void __launch_bounds__(loop_threads(NT), 1)
    tc_loop_kernel(const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmu,
                   const __grid_constant__ CUtensorMap tmh, const __grid_constant__ CUtensorMap tmt, TcLoopArgs a) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int EWQ = loop_epw(NT);    // epilogue warps per quarter
  constexpr int EW = 4 * EWQ;
  constexpr int EPI = 32 * EW;
  constexpr int CW = NT / EWQ;         // streams per epilogue warp: 8 or 16
  constexpr int GB = 4 / GP;           // CTAs that share a unit tile's gates
  constexpr int SO = NT / GB;          // streams of a tile a CTA runs the cells of
  constexpr int CPT = GP == 4 ? 8 : SO / EWQ;  // cells per thread and round
  constexpr uint32_t kStage = NT * 256u;       // 64 elements x NT streams x 2 planes
  const LoopLayout L = loop_layout(NT, a.nka, a.ux_chunks, a.stages, a.rxa_bytes, a.rxb_bytes, a.share_rx != 0);
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gb_ = smem_raw + (base - raw);  // generic pointer to the base
  const uint32_t bar = base + L.bar;
  const uint32_t full0 = bar, empty0 = bar + 8u * kMaxStages, acc_a = bar + 16u * kMaxStages,
                 acc_b = acc_a + 8u * kMaxRegions, drain_a = acc_b + 8u * kMaxRegions,
                 drain_b = drain_a + 8u * kMaxRegions, setup_bar = drain_b + 8u * kMaxRegions, u_ready = setup_bar + 8u, final_bar = setup_bar + 16u,
                 rx0 = setup_bar + 24u;  // rx0: [set][buffer]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gb_ + L.bar + kBarBytes - 16);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = (int)blockIdx.x;
  const int T = a.T, B = a.B, H = a.H, K = a.K;
  const volatile int* err = a.err;
  const uint64_t limit = static_cast<uint64_t>(a.limit_ns);
  // role A: part z of H, row tile r, stream tiles [ta0, ta0 + na)
  const int ga = a.ga, za = cta % ga, ra = (cta / ga) % a.RT, ta0 = cta < a.nA ? cta / (ga * a.RT) * a.sa : a.ST;
  const int na = max(0, min(a.sa, a.ST - ta0));
  // role B: gates [GP zb, GP zb + GP), units [128 ut, +128), stream tiles [tb0, tb0 + nb)
  const int zb = cta % GB, ut = (cta / GB) % a.UT, tb0 = cta < a.nB ? cta / (GB * a.UT) * a.sb : a.ST;
  const int nb = max(0, min(a.sb, a.ST - tb0));
  const int nkh = min(a.nka, (H + 63) / 64 - za * a.nka);  // this CTA's 64-column chunks of H
  const int nkb = (K + 63) / 64, nsl = (K + 15) / 16;
  const int ncut = a.ncut, ndep = a.ndep;
  const bool stream = GP == 1 && a.stream_segs != 0;
  const int reg_segs = stream ? 1 : ncut + 1;  // segments of an accumulator region of role B
  const int regs_a = a.ra_regions, regs_b = a.rb_regions;
  const unsigned h_step = (unsigned)(a.UT * GB), tau_step = (unsigned)(a.RT * ga);  // counts per step and tile

  if (threadIdx.x == 0) {
    for (int i = 0; i < a.stages; ++i) {
      mbar_init(full0 + 8u * i, 1);
      mbar_init(empty0 + 8u * i, 1);
    }
    for (int i = 0; i < kMaxRegions; ++i) {
      mbar_init(acc_a + 8u * i, 1);
      mbar_init(acc_b + 8u * i, 1);
      mbar_init(drain_a + 8u * i, EW);
      mbar_init(drain_b + 8u * i, EW);
    }
    mbar_init(setup_bar, 1);
    mbar_init(u_ready, EW);
    mbar_init(final_bar, 1);
    for (int i = 0; i < 4; ++i) mbar_init(rx0 + 8u * i, 1);
    fence_mbarrier_init_cluster();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // every CTA's barriers are initialised before any push reaches them
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (elect_one()) {  // ---- TMA producer: the resident factors, then h and tau' of every step ----
      tma_prefetch_map(&tmv);
      tma_prefetch_map(&tmu);
      tma_prefetch_map(&tmh);
      tma_prefetch_map(&tmt);
      {
        const int gpt = 128 / a.rpg;  // gates per row tile (rpg < 128: the first rpg rows of each)
        const int kt = a.rpg == 128 ? ra % a.ktiles : 0, g0 = a.rpg == 128 ? ra / a.ktiles : ra * gpt;
        const int gates = a.rpg == 128 ? 1 : min(gpt, 4);
        const uint32_t vbytes = na > 0 ? (uint32_t)(nkh * gates * a.rpg) * 128u : 0u;
        const uint32_t ubytes = nb > 0 ? (uint32_t)a.ux_chunks * kChunkBytes : 0u;
        mbar_arrive_expect_tx(setup_bar, vbytes + ubytes);
        if (na > 0)
          for (int c = 0; c < nkh; ++c)
            for (int g = 0; g < gates; ++g)
              for (int r = 0; r < a.rpg; r += a.vbox)
                tma_load_2d(base + c * kChunkBytes + (uint32_t)(g * a.rpg + r) * 128u, &tmv, setup_bar,
                            64 * (za * a.nka + c), (g0 + g) * a.Ks + kt * 128 + r);
        if (nb > 0)
          for (int g = 0; g < GP; ++g)
            for (int kb = a.ures; kb < nkb; ++kb)
              tma_load_2d(base + L.ux + (uint32_t)(g * (nkb - a.ures) + kb - a.ures) * kChunkBytes, &tmu, setup_bar,
                          64 * kb, (GP * zb + g) * H + 128 * ut);
      }
      bool ok = true;
      const int stages = a.stages;
      int it = 0;  // loads issued, up to `stages` (then: every slot has been used)
      RingPos pos;
      auto load = [&](const CUtensorMap* m, int c0, int row) {
        // the slot's previous load (one ring round ago) has been consumed
        if (it == stages && !(ok = mbar_wait_bounded<false>(empty0 + 8u * pos.slot, pos.parity ^ 1u, limit, err))) return;
        const uint32_t bar_s = full0 + 8u * pos.slot;
        mbar_arrive_expect_tx(bar_s, kStage);
        tma_load_3d(base + L.ring + pos.slot * kStage, m, bar_s, c0, row, 0);
        if (it < stages) ++it;
        pos.next(stages);
      };
      for (int t = 0; t < T && ok; ++t) {
#pragma unroll 1
        for (int s = 0; s < na && ok; ++s) {
          if (!(ok = wait_counter(a.h_count + 32 * (ta0 + s), (unsigned)(t + 1) * h_step, limit, err))) break;
#pragma unroll 1
          for (int c = 0; c < nkh && ok; ++c) load(&tmh, 64 * (za * a.nka + c), (ta0 + s) * NT);
        }
#pragma unroll 1
        for (int s = 0; s < nb && ok; ++s) {
          if (!(ok = wait_counter(a.tau_count + 32 * (tb0 + s), (unsigned)(t + 1) * tau_step, limit, err))) break;
#pragma unroll 1
          for (int kb = 0; kb < nkb && ok; ++kb)
#pragma unroll 1
            for (int g = 0; g < GP && ok; ++g) load(&tmt, (GP * zb + g) * a.Ks + 64 * kb, (tb0 + s) * NT);
        }
      }
      if (!ok) atomicCAS(a.err, 0, kErrTcTimeout);
      // every issued copy has landed before the CTA may leave
      mbar_wait_bounded<false>(setup_bar, 0, limit, err);
      for (int s = 0; s < it; ++s)  // slot s was last filled in this turn of the ring (before the position) or the one before
        mbar_wait_bounded<false>(full0 + 8u * s, s < pos.slot ? pos.parity : pos.parity ^ 1u, limit, err);
    }
  } else if (warp == 1) {
    if (elect_one()) {  // ---- MMA issuer ----
      constexpr uint32_t idesc2 = umma_idesc_bf16(128, 2 * NT);
      constexpr uint32_t idesc_b = umma_idesc_bf16(128, MB ? 2 * NT : NT);
      bool ok = mbar_wait_bounded<false>(setup_bar, 0, limit, err) && mbar_wait_bounded<false>(u_ready, 0, limit, err);
      tc_fence_after();
      const int stages = a.stages;
      RingPos pos;
      // accumulators: a role's items (stream tiles) take its regions in turn, as stages of a ring; before one
      // is overwritten the epilogue has read it
      RingPos pa, pb;
      int used_a = 0, used_b = 0;
      auto drained = [&](uint32_t bars, const RingPos& p, int& used, int regions) {
        if (used < regions) {
          ++used;
          return true;
        }
        return mbar_wait_bounded<false>(bars + 8u * p.slot, p.parity ^ 1u, limit, err);
      };
      // the other role's accumulators in the same columns: its last item so far has been read
      auto last_drained = [&](uint32_t bars, const RingPos& p, int regions) {
        const int slot = p.slot == 0 ? regions - 1 : p.slot - 1;
        return mbar_wait_bounded<false>(bars + 8u * slot, p.slot == 0 ? p.parity ^ 1u : p.parity, limit, err);
      };
      constexpr uint32_t dg = NT * (MB ? 2 : 1);  // columns of one gate's accumulator
      constexpr uint32_t seg = GP * dg;           // of one depth segment
      const uint64_t ring_desc = umma_desc_sw128(base + L.ring), vh_desc = umma_desc_sw128(base),
                     ux_desc = umma_desc_sw128(base + L.ux);
      // both planes of the activation against one factor slice
      auto both_ss = [&](uint32_t d, uint64_t da, uint64_t db, uint32_t acc) {
        umma_bf16(d, da, db, idesc_b, acc);
        if (!MB) umma_bf16(d, da, db + (NT * 128u >> 4), idesc_b, 1u);
      };
      auto both_ts = [&](uint32_t d, uint32_t ta, uint64_t db, uint32_t acc) {
        umma_bf16_ts(d, ta, db, idesc_b, acc);
        if (!MB) umma_bf16_ts(d, ta, db + (NT * 128u >> 4), idesc_b, 1u);
      };
#pragma unroll 1
      for (int t = 0; t < T && ok; ++t) {
        if (a.shared_acc && t > 0 && nb > 0) ok = last_drained(drain_b, pb, regs_b);
#pragma unroll 1
        for (int s = 0; s < na && ok; ++s) {
          if (!(ok = drained(drain_a, pa, used_a, regs_a))) break;
          tc_fence_after();
          const uint32_t d = tmem + a.acc_a + (uint32_t)pa.slot * 2 * NT;
          uint64_t da = vh_desc;
          uint32_t acc = 0;
#pragma unroll 1
          for (int c = 0; c < nkh; ++c) {
            if (!(ok = mbar_wait_bounded<false>(full0 + 8u * pos.slot, pos.parity, limit, err))) break;
            tc_fence_after();
            const uint64_t db = ring_desc + (uint64_t)((uint32_t)pos.slot * (kStage >> 4));
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {  // both planes of h in one MMA: N = 2 NT
              umma_bf16(d, da + 2ull * kk, db + 2ull * kk, idesc2, acc);
              acc = 1;
            }
            umma_commit(empty0 + 8u * pos.slot);
            pos.next(stages);
            da += kChunkBytes >> 4;
          }
          if (ok) umma_commit(acc_a + 8u * pa.slot);
          pa.next(regs_a);
        }
        if (a.shared_acc && na > 0 && ok) ok = last_drained(drain_a, pa, regs_a);
#pragma unroll 1
        for (int s = 0; s < nb && ok; ++s) {
          if (!(ok = drained(drain_b, pb, used_b, regs_b))) break;
          tc_fence_after();
          uint32_t d0 = tmem + a.acc_b + (uint32_t)pb.slot * reg_segs * seg;  // the current segment's accumulators
          int cut = 0;
          int next_cut = ncut > 0 ? a.cut_k[0] : INT_MAX;
          uint32_t u_col = tmem;  // the next resident slice (or piece of one), in the order of issue
          uint32_t acc = 0;
#pragma unroll 1
          for (int kb = 0; kb < nkb; ++kb) {
            uint64_t db[GP];
            uint32_t freed[GP];  // the empty barriers of this chunk's slots
#pragma unroll
            for (int g = 0; g < GP; ++g) {
              ok = ok && mbar_wait_bounded<false>(full0 + 8u * pos.slot, pos.parity, limit, err);
              db[g] = ring_desc + (uint64_t)((uint32_t)pos.slot * (kStage >> 4));
              freed[g] = empty0 + 8u * pos.slot;
              pos.next(stages);
            }
            if (!ok) break;
            tc_fence_after();
            auto issue_ts = [&](int kk) {
#pragma unroll
              for (int g = 0; g < GP; ++g) both_ts(d0 + g * dg, u_col + 8 * g, db[g] + 2ull * kk, acc);
              acc = 1;
              u_col += 8 * GP;
            };
            auto next_segment = [&]() {  // the sums up to depth k_j are complete
              if (stream) {
                umma_commit(acc_b + 8u * pb.slot);
                pb.next(regs_b);
                ok = drained(drain_b, pb, used_b, regs_b);
                tc_fence_after();
                d0 = tmem + a.acc_b + (uint32_t)pb.slot * seg;
              } else {
                d0 += seg;
              }
              acc = 0;
              ++cut;
              next_cut = cut < ncut ? a.cut_k[cut] : INT_MAX;
            };
            if (kb < a.ures && next_cut >= 64 * kb + 64 && nsl >= 4 * kb + 4) {  // a whole chunk in tensor memory
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) issue_ts(kk);
            } else {
#pragma unroll 1
              for (int kk = 0; kk < 4 && 4 * kb + kk < nsl; ++kk) {
                const int k0 = 64 * kb + 16 * kk;
                if (next_cut == k0) next_segment();
                if (kb < a.ures) {
                  issue_ts(kk);
#pragma unroll 1
                  while (next_cut < k0 + 16) {  // a depth inside the slice: its next piece, in the next segment
                    next_segment();
                    issue_ts(kk);
                  }
                } else {
#pragma unroll
                  for (int g = 0; g < GP; ++g)
                    both_ss(d0 + g * dg,
                            ux_desc + (uint64_t)((uint32_t)(g * (nkb - a.ures) + kb - a.ures) * (kChunkBytes >> 4)) +
                                2ull * kk,
                            db[g] + 2ull * kk, acc);
                  acc = 1;
                }
              }
            }
#pragma unroll
            for (int g = 0; g < GP; ++g) umma_commit(freed[g]);
          }
          if (ok) umma_commit(acc_b + 8u * pb.slot);
          pb.next(regs_b);
        }
      }
      if (!ok) atomicCAS(a.err, 0, kErrTcTimeout);
      umma_commit(final_bar);  // every MMA issued has completed before tensor memory is freed
      mbar_wait_bounded<false>(final_bar, 0, limit, err);
    }
  } else {  // ---- epilogue ----
    const int e = threadIdx.x - 64, q = warp & 3, part = (warp - 2) >> 2;
    const uint32_t trow = tmem + ((32u * q) << 16);
    const int lrow = 32 * q + lane;    // tensor-memory lane: row of role A, unit of role B
    const int j = 128 * ut + lrow;     // hidden unit
    const bool unit_ok = nb > 0 && j < H;
    auto warp_arrive = [&](uint32_t mb) {
      __syncwarp();
      if (lane == 0) mbar_arrive(mb);
    };
    // U of this CTA's gates into tensor memory in the order the MMAs take it: for each 16-term slice, or
    // piece of one between two intermediate depths (its other terms zero), eight columns (two terms each)
    // per gate
    if (nb > 0) {
      int piece = 0, lo = 0, c = 0;
#pragma unroll 1
      for (int k0 = 0; k0 < min(64 * a.ures, 16 * nsl);) {
        while (c < ncut && a.cut_k[c] <= k0 + lo) ++c;
        const int hi = c < ncut && a.cut_k[c] < k0 + 16 ? a.cut_k[c] - k0 : 16;
        if (piece % EWQ == part) {
#pragma unroll 1
          for (int g = 0; g < GP; ++g) {
            const __nv_bfloat16* row = a.U + ((long long)(GP * zb + g) * H + (unit_ok ? j : 0)) * a.Ks;
            float v[8];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const uint4 w = unit_ok ? masked_terms(row, k0 + 8 * i, k0 + lo, min(K, k0 + hi)) : make_uint4(0, 0, 0, 0);
              v[4 * i] = __uint_as_float(w.x);
              v[4 * i + 1] = __uint_as_float(w.y);
              v[4 * i + 2] = __uint_as_float(w.z);
              v[4 * i + 3] = __uint_as_float(w.w);
            }
            __syncwarp();
            tmem_st8(trow + (uint32_t)(piece * GP + g) * 8, v);
          }
        }
        ++piece;
        lo = hi & 15;
        if (hi == 16) k0 += 16;
      }
      tmem_wait_st();
    }
    tc_fence_before();
    warp_arrive(u_ready);

    // row of role A: storage row of (gate, term), sigma
    struct RowA {
      int srow;    // storage row g Ks + k, or -1
      bool valid;  // k < K
    };
    auto row_a = [&](int lr) {
      RowA r;
      int g, k;
      if (a.rpg == 128) {
        g = ra / a.ktiles;
        k = (ra % a.ktiles) * 128 + lr;
      } else {
        g = ra * (128 / a.rpg) + lr / a.rpg;
        k = lr % a.rpg;
      }
      r.valid = g < 4 && k < K;
      r.srow = g < 4 ? g * a.Ks + k : -1;
      return r;
    };
    // with ga > 1 this thread finishes columns [fc0, fc0 + FC) of row frow of the CTA's 128 / ga rows
    const int RS = 128 / ga, RB = RS / 32;
    const int w16 = warp - 2;
    const int frow = ga == 1 ? lrow : za * RS + 32 * (w16 % RB) + lane;
    const int fcn = ga == 1 ? CW : NT * RB / EW, fc0 = ga == 1 ? part * CW : (w16 / RB) * fcn;
    const RowA fr = row_a(frow);
    const float sig = (na > 0 && fr.valid) ? a.sigma[fr.srow] : 0.f;
    float bias[4] = {0.f, 0.f, 0.f, 0.f};
    if (unit_ok)
#pragma unroll
      for (int g = 0; g < 4; ++g) bias[g] = a.bias[g * H + j];
    // the pairs of v0 and v1 (streams n, n + 1) at element `col` of their rows of `pitch`: neighbouring lanes
    // hold neighbouring elements, so an even lane stores stream n's two elements of a lane pair and an odd
    // lane stream n + 1's, one word per plane
    const int odd = lane & 1;
    const uint32_t sel = odd ? 0x7632u : 0x5410u;
    auto store_pair2 = [&](__nv_bfloat16* own, long long plane, float v0, float v1, bool write) {
      const __nv_bfloat162 hi = __floats2bfloat162_rn(v0, v1);
      const uint32_t h = *reinterpret_cast<const uint32_t*>(&hi);
      const __nv_bfloat162 lo =
          __floats2bfloat162_rn(v0 - __uint_as_float(h << 16), v1 - __uint_as_float(h & 0xFFFF0000u));
      const uint32_t l = *reinterpret_cast<const uint32_t*>(&lo);
      const uint32_t h2 = __shfl_xor_sync(0xffffffffu, h, 1), l2 = __shfl_xor_sync(0xffffffffu, l, 1);
      if (write) {
        *reinterpret_cast<uint32_t*>(own) = odd ? __byte_perm(h2, h, sel) : __byte_perm(h, h2, sel);
        *reinterpret_cast<uint32_t*>(own + plane) = odd ? __byte_perm(l2, l, sel) : __byte_perm(l, l2, sel);
      }
    };
    // rows and units come in pairs: a pair is stored when its first element exists (tau' rows past K and
    // the padding column of an odd H get zeros)
    const bool pair_a = fr.srow >= 0, pair_b = nb > 0 && (j & ~1) < H;
    // streams n, n + 1 of this thread's row of tau' / unit of h (n even, so both are of the same tile)
    auto store_tau2 = [&](int n, float v0, float v1) {
      store_pair2(a.tau + ((n + odd) * a.ldt + (fr.srow & ~1)), a.tau_plane, fr.valid ? v0 : 0.f, fr.valid ? v1 : 0.f,
                  pair_a && n + odd < B);
    };
    auto store_h2 = [&](__nv_bfloat16* base_, int ld, long long plane, int n, float v0, float v1) {
      store_pair2(base_ + ((n + odd) * ld + (j & ~1)), plane, unit_ok ? v0 : 0.f, unit_ok ? v1 : 0.f,
                  pair_b && n + odd < B);
    };
    // all of the epilogue's threads have written: raise the tile's counter (or, if a wait of any of
    // them ran out, leave together).  The consumer's proxy fence after its acquire orders its TMA
    // reads after these writes.
    auto publish = [&](bool failed, unsigned* count, bool withhold) -> bool {
      if (block_or_named(1, EPI, failed)) return false;
      if (e == 0 && !withhold) red_release_gpu_add(count, 1u);
      return true;
    };
    unsigned rx_use[2] = {0u, 0u};
    const uint32_t crank = cluster_ctarank();
    const int setb = a.share_rx ? 0 : 1;

    RingPos pa, pb;  // accumulator regions of the next items
    constexpr int kRounds = GP == 4 ? CW / 8 : 1;
    static_assert(kRounds == 1, "one round of cells per thread and item");
    constexpr uint32_t dg = NT * (MB ? 2 : 1), seg = GP * dg;  // columns of a gate's accumulator, of a depth segment
    // c_{t-1} of this thread's cells: with one stream tile and no intermediate depths in registers across
    // the steps, otherwise in memory, by the parity of t (the depths of step t - 1 run during step t)
    const bool keep_c = nb <= 1 && ndep == 0;
    const bool defer = a.defer_depths != 0 && ndep > 0 && nb > 0;  // a step's depths run during the next step
    float cp[CPT];
    // (c_{-1} = c0: the full depth reads it from the caller and keeps a copy for the depths that run after the
    // step's outputs are written, because the caller may pass one buffer as c0 and as an output)
    auto load_c = [&](int t, int n0, bool depths) {
      const float* src = (t & 1) ? a.c_state1 : (t > 0 || depths) ? a.c_state : a.c0;
#pragma unroll
      for (int c = 0; c < CPT; ++c) cp[c] = (unit_ok && n0 + c < B && src != nullptr) ? src[(n0 + c) * H + j] : 0.f;
    };
    auto store_depth = [&](int jj, int t, int n0, const float (&h)[CPT], const float (&c)[CPT], unsigned skip) {
      if (!unit_ok) return;
      const long long o = (long long)jj * a.ck_stride + ((long long)t * B + n0) * H + j;
      if (a.ckpt_h) {
#pragma unroll
        for (int i = 0; i < CPT; ++i)
          if (n0 + i < B && (skip >> i & 1u) == 0u) a.ckpt_h[o + i * H] = h[i];
      }
      if (a.ckpt_c) {
#pragma unroll
        for (int i = 0; i < CPT; ++i)
          if (n0 + i < B && (skip >> i & 1u) == 0u) a.ckpt_c[o + i * H] = c[i];
      }
    };
    // Depths inside a 16-term slice (SD): the products of the slice's terms past the depth have a zero
    // of U, and a tau' of such a term that is not finite makes them NaN (its pair's lo half is one even for an
    // infinity).  The full depth's sums are then NaN too, in all units of the stream.  So: cells (bits) whose sums
    // are NaN get their depths from depth_cell at the full depth of the step, while tau'_t is still in memory
    // (its next value waits for this CTA's h_t), and the depths' own pass leaves out what is NaN there.
    auto any_nan = [&](const float (&y)[4][CPT]) -> bool {
      uint64_t s2 = f32x2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < CPT; c += 2)
#pragma unroll
        for (int g = 0; g < 4; ++g) s2 = add2(s2, f32x2(y[g][c], y[g][c + 1]));
      float s0, s1;
      f32x2_split(s2, s0, s1);
      const float sum = s0 + s1;
      return sum != sum;
    };
    auto nan_cells = [&](const float (&y)[4][CPT], int n0) -> unsigned {
      unsigned m = 0u;
#pragma unroll
      for (int c = 0; c < CPT; ++c) {
        const float sum = (y[0][c] + y[1][c]) + (y[2][c] + y[3][c]);
        if (sum != sum && unit_ok && n0 + c < B) m |= 1u << c;
      }
      return m;
    };
    bool nan_seen = false;  // in a full depth of this thread's cells so far
    auto exact_depths = [&](unsigned cells, int t, int s, int n0) {
      unsigned seen;  // (every row tile's tau'_t has been released to this counter)
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.tau_count + 32 * (tb0 + s)) : "memory");
#pragma unroll 1
      for (; cells != 0u; cells &= cells - 1u) {
        const int c = __ffs(cells) - 1;
        float cv = cp[0];
#pragma unroll
        for (int i = 1; i < CPT; ++i) cv = i == c ? cp[i] : cv;
#pragma unroll 1
        for (int d = 0; d < ndep; ++d) {
          const long long o = (long long)d * a.ck_stride + ((long long)t * B + n0 + c) * H + j;
          depth_cell(a.U + (long long)j * a.Ks, (long long)H * a.Ks, a.tau + (long long)(n0 + c) * a.ldt, a.tau_plane,
                     a.Ks, a.cut_k[a.dep_segs[d] - 1], a.bias + j, H, cv, a.ckpt_h ? a.ckpt_h + o : nullptr,
                     a.ckpt_c ? a.ckpt_c + o : nullptr);
        }
      }
    };
    // first stream of this thread's cells of stream tile s
    auto first_stream = [&](int s) { return (tb0 + s) * NT + (GP == 4 ? part * CW : zb * SO + part * CPT); };
    // eight streams' sums of one gate over the segments [0, nseg) from column `col` (both planes' products); the
    // caller's warp is together
    auto load_sums = [&](uint32_t col, int nseg, float (&v)[8]) {
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = 0.f;
#pragma unroll 1
      for (int i = 0; i < nseg; ++i) {
        float vh[8];
        if constexpr (MB) {
          float vl[8];
          tmem_ld8x2_sync<true>(col + i * seg, col + i * seg + NT, vh, vl);
#pragma unroll
          for (int c = 0; c < 8; ++c) vh[c] += vl[c];
        } else {
          tmem_ld8_sync<true>(col + i * seg, vh);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] += vh[c];
      }
    };
    // role B's receive buffer of its exchange number u
    auto receive_buf = [&](uint32_t u) {
      return (setb ? L.rxb : L.rxa) + (u & 1u) * (a.share_rx ? max(a.rxa_bytes, a.rxb_bytes) : a.rxb_bytes);
    };
    auto read_received = [&](uint32_t buf, float (&y)[4][CPT]) {
      const float* rb = reinterpret_cast<const float*>(gb_ + buf) + part * CPT;
#pragma unroll
      for (int g = 0; g < 4; ++g)
#pragma unroll
        for (int c = 0; c < CPT; c += 2) {
          const float2 f = *reinterpret_cast<const float2*>(rb + (g * 128 + lrow) * SO + c);
          y[g][c] = f.x;
          y[g][c + 1] = f.y;
        }
    };
    // the four gates' sums as this CTA holds them: in tensor memory (GP = 4) or in the receive buffer of the last
    // exchange; the caller's warp is together
    auto read_sums = [&](int region, int nseg, float (&y)[4][CPT]) {
      if constexpr (GP == 4) {
        const uint32_t tc0 = trow + a.acc_b + (uint32_t)region * reg_segs * seg + part * CW;
        if (!MB && nseg == 1) {
          tmem_ld8x4_sync<true>(tc0, tc0 + dg, tc0 + 2 * dg, tc0 + 3 * dg, y);
        } else {
#pragma unroll
          for (int g = 0; g < 4; ++g) load_sums(tc0 + g * dg, nseg, y[g]);
        }
      } else {
        read_received(receive_buf(rx_use[setb] - 1u), y);
      }
    };
    // the gate sums y over nseg segments of accumulator region `region`; with several CTAs
    // per unit tile (GP < 4) each sends its gates' sums to the owners of the streams and takes what they
    // sent; `last`: the accumulators are not read again
    auto gate_sums = [&](int region, int nseg, bool last, float (&y)[4][CPT]) -> bool {
      const uint32_t tc0 = trow + a.acc_b + (uint32_t)region * reg_segs * seg + part * CW;
      __syncwarp();
      if constexpr (GP == 4) {
        read_sums(region, nseg, y);
        if (last) {
          tc_fence_before();
          warp_arrive(drain_b + 8u * region);
        }
        return true;
      } else {
        const uint32_t u = rx_use[setb]++;
        const uint32_t rxb = rx0 + 16u * setb + 8u * (u & 1u);
        const uint32_t buf = receive_buf(u);
        if (e == 0) mbar_arrive_expect_tx(rxb, (uint32_t)(4 * 128 * SO * 4));
        __syncwarp();
        bool got = true;
#pragma unroll
        for (int g = 0; g < GP; ++g)
#pragma unroll
          for (int c8 = 0; c8 < CW; c8 += 8) {
            float v[8];
            if (!stream) {
              load_sums(tc0 + g * dg + c8, nseg, v);
            } else {  // (one group of streams, one gate) every segment in its own region
              load_sums(tc0, 1, v);
#pragma unroll 1
              for (int i = 1; i < nseg && got; ++i) {
                tc_fence_before();
                warp_arrive(drain_b + 8u * pb.slot);
                pb.next(regs_b);
                got = __all_sync(0xffffffffu, mbar_wait_bounded<false>(acc_b + 8u * pb.slot, pb.parity, limit, err));
                tc_fence_after();
                float w[8];
                load_sums(trow + a.acc_b + (uint32_t)pb.slot * seg + part * CW, 1, w);
#pragma unroll
                for (int c = 0; c < 8; ++c) v[c] += w[c];
              }
            }
#pragma unroll
            for (int h4 = 0; h4 < 2; ++h4) {
              const int col = part * CW + c8 + 4 * h4, d = col / SO, sp = col - d * SO;
              const uint32_t peer = crank - (uint32_t)zb + (uint32_t)d;
              st_async_v4(mapa_shared(base + buf + (uint32_t)((((GP * zb + g) * 128 + lrow) * SO + sp) * 4), peer),
                          v[4 * h4], v[4 * h4 + 1], v[4 * h4 + 2], v[4 * h4 + 3], mapa_shared(rxb, peer));
            }
          }
        if (last) {
          tc_fence_before();
          warp_arrive(drain_b + 8u * (stream ? pb.slot : region));
        }
        got = __all_sync(0xffffffffu, mbar_wait_bounded<true>(rxb, (u >> 1) & 1u, limit, err)) && got;
        read_received(buf, y);
        return got;
      }
    };
    int reg_first = 0;  // region of the step's first stream tile
    // the depth sets [set0, set1) of step t: set 0 is the full depth (its h_t is what the next step waits
    // for), set i > 0 the intermediate depth i - 1
    auto run_sets = [&](int t, int s, int region, int set0, int set1) -> bool {
      const int n0 = first_stream(s);
      bool fail = false;
#pragma unroll 1
      for (int set = set0; set < set1 && !fail; ++set) {
        float y[4][CPT], hv[CPT], cv[CPT];
        fail = !gate_sums(region, set == 0 ? ncut + 1 : a.dep_segs[set - 1], set == ndep, y);
        if (fail) {
          if (set == 0) publish(true, a.h_count, true);  // the barrier where the block's other warps wait
          break;
        }
        unsigned nans = 0u;
        if constexpr (SD) {
          if (set > 0) {
            if (nan_seen) nans = nan_cells(y, n0);
          } else if (__any_sync(0xffffffffu, any_nan(y))) {
            nans = nan_cells(y, n0);
            nan_seen = nan_seen || nans != 0u;
            exact_depths(nans, t, s, n0);
            __syncwarp();
            read_sums(region, ncut + 1, y);
          }
        }
        lstm_cells_s(y, bias, cp, hv, cv);
        if (set > 0) {
          store_depth(set - 1, t, n0, hv, cv, nans);
          continue;
        }
#pragma unroll
        for (int c = 0; c < CPT; c += 2) store_h2(a.h_bf16, a.ldh, a.h_plane, n0 + c, hv[c], hv[c + 1]);
        if (!publish(false, a.h_count + 32 * (tb0 + s), false)) return false;
        // then what nothing waits for
        for (int jj = ndep; jj < a.ck_n; ++jj) store_depth(jj, t, n0, hv, cv, 0u);  // depths of at least K
        if (a.seq_bf16) {
          __nv_bfloat16* sq = a.seq_bf16 + (long long)t * B * a.ldh;
#pragma unroll
          for (int c = 0; c < CPT; c += 2) store_h2(sq, a.ldh, a.seq_plane, n0 + c, hv[c], hv[c + 1]);
        }
        if (unit_ok) {
          if (a.out_h) {
            float* o = a.out_h + (long long)t * B * H + j;
#pragma unroll
            for (int c = 0; c < CPT; ++c)
              if (n0 + c < B) o[(n0 + c) * H] = hv[c];
          }
          if (defer && t == 0) {
            float* o = a.c_state + j;
#pragma unroll
            for (int c = 0; c < CPT; ++c)
              if (n0 + c < B) o[(n0 + c) * H] = cp[c];
          }
          if (!keep_c) {
            float* o = ((t & 1) ? a.c_state : a.c_state1) + j;
#pragma unroll
            for (int c = 0; c < CPT; ++c)
              if (n0 + c < B) o[(n0 + c) * H] = cv[c];
          }
          if (a.c_last && t == T - 1)
#pragma unroll
            for (int c = 0; c < CPT; ++c)
              if (n0 + c < B) a.c_last[(n0 + c) * H + j] = cv[c];
        }
        if (keep_c) {
#pragma unroll
          for (int c = 0; c < CPT; ++c) cp[c] = cv[c];
        }
      }
      return !fail;
    };
    // the intermediate depths of step t, all stream tiles (every thread leaves together if a wait ran out)
    auto run_depths = [&](int t, int region) -> bool {
      bool fail = false;
#pragma unroll 1
      for (int s = 0; s < nb && !fail; ++s) {
        load_c(t, first_stream(s), true);
        fail = !run_sets(t, s, region, 1, ndep + 1);
        if (++region == regs_b) region = 0;
      }
      return !block_or_named(1, EPI, fail);
    };
    bool ok = true;
    // h_{-1} = h0 (or zero) of this CTA's units and streams
    for (int s = 0; s < nb && ok; ++s) {
      const int n0 = (tb0 + s) * NT + (GP == 4 ? part * CW : zb * SO + part * CPT);
#pragma unroll 1
      for (int c = 0; c < (GP == 4 ? CW : CPT); c += 2) {
        float v[2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
          v[i] = (unit_ok && a.h0 != nullptr && n0 + c + i < B) ? a.h0[(long long)(n0 + c + i) * H + j] : 0.f;
        store_h2(a.h_bf16, a.ldh, a.h_plane, n0 + c, v[0], v[1]);
      }
      ok = publish(false, a.h_count + 32 * (tb0 + s), a.test_stall != 0 && cta == 0);
    }

    for (int t = 0; t < T && ok; ++t) {
      // ---- role A: tau' of this CTA's rows ----
      for (int s = 0; s < na && ok; ++s) {
        const int n0 = (ta0 + s) * NT;
        // P_t of the elements this thread finishes (B ldp < 2^31)
        const float* Pt = a.P + (long long)t * B * a.ldp + fr.srow;
        float pv[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) {
          const int n = n0 + fc0 + c;
          pv[c] = (c < fcn && fr.valid && n < B) ? __ldg(Pt + n * a.ldp) : 0.f;
        }
        bool fail = !__all_sync(0xffffffffu, mbar_wait_bounded<false>(acc_a + 8u * pa.slot, pa.parity, limit, err));
        const uint32_t handed = drain_a + 8u * pa.slot;
        if (!fail) {
          tc_fence_after();
          const uint32_t tc0 = trow + a.acc_a + (uint32_t)pa.slot * 2 * NT + part * CW;
          pa.next(regs_a);
          if (ga == 1) {
#pragma unroll
            for (int c8 = 0; c8 < CW; c8 += 8) {
              float vh[8], vl[8];
              tmem_ld8x2_sync(tc0 + c8, tc0 + NT + c8, vh, vl);
              if (c8 + 8 == CW) {
                tc_fence_before();
                warp_arrive(handed);
              }
#pragma unroll
              for (int c = 0; c < 8; c += 2)
                store_tau2(n0 + fc0 + c8 + c, sig * (vh[c] + vl[c] + pv[c8 + c]),
                           sig * (vh[c + 1] + vl[c + 1] + pv[c8 + c + 1]));
            }
          } else {
            const uint32_t u = rx_use[0]++;
            const uint32_t rxb = rx0 + 8u * (u & 1u);
            const uint32_t buf = L.rxa + (u & 1u) * (a.share_rx ? max(a.rxa_bytes, a.rxb_bytes) : a.rxa_bytes);
            // receive buffer [source][RS rows][NT], the 16-byte pieces of a row swizzled by the row
            constexpr int kP = NT / 4;
            auto piece_off = [&](int row, int p) {
              const int x = kP >= 8 ? (row & 7) : ((row >> 1) & (kP - 1));
              return (uint32_t)((row * kP + (p ^ x)) * 16);
            };
            if (e == 0) mbar_arrive_expect_tx(rxb, (uint32_t)(128 * NT * 4));
            __syncwarp();
            const int owner = lrow / RS;
            const uint32_t peer = crank - (uint32_t)za + (uint32_t)owner;
            const uint32_t dst = mapa_shared(base + buf + (uint32_t)za * RS * NT * 4u, peer);
            const uint32_t dbar = mapa_shared(rxb, peer);
#pragma unroll
            for (int c8 = 0; c8 < CW; c8 += 8) {
              float vh[8], vl[8];
              tmem_ld8x2_sync<true>(tc0 + c8, tc0 + NT + c8, vh, vl);
              if (c8 + 8 == CW) {
                tc_fence_before();
                warp_arrive(handed);
              }
#pragma unroll
              for (int h4 = 0; h4 < 2; ++h4)
                st_async_v4(dst + piece_off(lrow - owner * RS, (part * CW + c8) / 4 + h4), vh[4 * h4] + vl[4 * h4],
                            vh[4 * h4 + 1] + vl[4 * h4 + 1], vh[4 * h4 + 2] + vl[4 * h4 + 2],
                            vh[4 * h4 + 3] + vl[4 * h4 + 3], dbar);
            }
            fail = !__all_sync(0xffffffffu, mbar_wait_bounded<true>(rxb, (u >> 1) & 1u, limit, err));
            if (!fail) {
              // the group's partial sums in rank order (the result does not depend on timing)
              const uint8_t* rb = gb_ + buf;
              const int rr = frow - za * RS;
#pragma unroll
              for (int c = 0; c < CW; c += 2) {
                if (c >= fcn) break;
                const int col = fc0 + c;
                const float* src = reinterpret_cast<const float*>(rb + piece_off(rr, col >> 2) + 4 * (col & 3));
                float s0 = 0.f, s1 = 0.f;
#pragma unroll 2
                for (int i = 0; i < ga; ++i) {
                  const float2 f = *reinterpret_cast<const float2*>(src + i * RS * NT);
                  s0 += f.x;
                  s1 += f.y;
                }
                store_tau2(n0 + col, sig * (s0 + pv[c]), sig * (s1 + pv[c + 1]));
              }
            }
          }
        }
        ok = publish(fail, a.tau_count + 32 * (ta0 + s), false);
      }
      // ---- the intermediate depths of the step before, while tau'_t is on its way ----
      if (ok && defer && t > 0) ok = run_depths(t - 1, reg_first);
      // ---- role B: gate sums, cells ----
      reg_first = pb.slot;
#pragma unroll 1
      for (int s = 0; s < nb && ok; ++s) {
        if (t == 0 || !keep_c) load_c(t, first_stream(s), false);
        const bool got = __all_sync(0xffffffffu, mbar_wait_bounded<false>(acc_b + 8u * pb.slot, pb.parity, limit, err));
        tc_fence_after();
        bool good = got && run_sets(t, s, pb.slot, 0, 1);
        if (!got) good = publish(true, a.h_count, true);
        ok = good;
        if (ok && ndep > 0 && !defer) {
          bool fail = !run_sets(t, s, pb.slot, 1, ndep + 1);
          ok = !block_or_named(1, EPI, fail);
        }
        pb.next(regs_b);
      }
    }
    if (ok && defer && T > 0) ok = run_depths(T - 1, reg_first);
    if (!ok) atomicCAS(a.err, 0, kErrTcTimeout);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // no CTA frees its shared memory while a peer may still write into it
  if (*err != 0) {     // after an abort: let pushes already in flight towards this CTA land
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 50000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  // the last CTA to get here clears the counters for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(a.done, 1u) == gridDim.x - 1) {
      __threadfence();
      for (int i = 0; i < a.ST; ++i) {
        a.h_count[32 * i] = 0u;
        a.tau_count[32 * i] = 0u;
      }
      *a.done = 0u;
    }
  }
}


template <int NT, int GP, bool MB, bool SD>
cudaError_t launch_loop_t(const TcMap& V, const TcMap& U, const TcMap& Hm, const TcMap& Taum, const TcLoopPlan& p,
                          const TcLoopArgs& a, cudaStream_t s, bool* resident) {
  auto kern = tc_loop_kernel<NT, GP, MB, SD>;
  // per thread and device: the shared-memory limit, and the cluster sizes and sizes of grids known to be resident
  static thread_local DeviceSet ready;
  static thread_local struct {
    int dev, cs, ctas;
    size_t smem;
  } seen[16] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = once_per_device(
        &ready, [&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024); });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.ctas);
  cfg.blockDim = dim3(loop_threads(NT));
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attrs[2];
  attrs[0].id = cudaLaunchAttributeClusterDimension;
  attrs[0].val.clusterDim.x = p.cs;
  attrs[0].val.clusterDim.y = 1;
  attrs[0].val.clusterDim.z = 1;
  attrs[1].id = cudaLaunchAttributeCooperative;
  attrs[1].val.cooperative = 1;
  cfg.attrs = attrs;
  cfg.numAttrs = 1;
  bool known = false;
  for (const auto& v : seen) known = known || (v.dev == dev && v.cs == p.cs && v.smem >= p.smem && v.ctas >= p.ctas);
  if (!known) {
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
    if (e != cudaSuccess) return e;
    if (clusters * p.cs < p.ctas) {
      *resident = false;
      return cudaSuccess;
    }
    for (auto& v : seen)
      if (v.cs == 0) {
        v = {dev, p.cs, clusters * p.cs, p.smem};
        break;
      }
  }
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, kern, *reinterpret_cast<const CUtensorMap*>(V.bytes),
                         *reinterpret_cast<const CUtensorMap*>(U.bytes),
                         *reinterpret_cast<const CUtensorMap*>(Hm.bytes),
                         *reinterpret_cast<const CUtensorMap*>(Taum.bytes), a);
  *resident = e != cudaErrorCooperativeLaunchTooLarge;
  if (!*resident) {  // (a process limited to part of the GPU): the per-timestep kernels serve
    cudaGetLastError();
    return cudaSuccess;
  }
  return e;
}

}  // namespace

bool tc_loop_plan(int H, int B, int K, const Checkpoints& ck, bool slower_too, TcLoopPlan* out) {
  if (H < 1 || H > 2048 || K < 1 || K > 1024 || B < 1 || B > kLoopMaxTiles * 16) return false;
  TcLoopPlan p{};
  p.rpg = K <= 16 ? 16 : K <= 32 ? 32 : K <= 64 ? 64 : 128;
  p.ktiles = (K + 127) / 128;
  p.RT = p.rpg <= 32 ? 1 : p.rpg == 64 ? 2 : 4 * p.ktiles;
  const int nkh = (H + 63) / 64, nkb = (K + 63) / 64, nsl = (K + 15) / 16;
  p.ga = H <= 512 ? 1 : H <= 1024 ? 2 : 4;
  p.nka = (nkh + p.ga - 1) / p.ga;
  // all four gates in a CTA where their terms fit beside their accumulators, else one gate per CTA (two
  // gates per CTA for 128 < K <= 256 measured slower: 11.4 against 8.8 us a step at H = 512, B = 256, K = 200)
  p.gp = K <= 128 ? 4 : 1;
  const int gb = 4 / p.gp;
  p.UT = (H + 127) / 128;
  p.cs = p.ga > gb ? p.ga : gb;
  p.share_rx = (p.ga == gb || p.ga == 1 || gb == 1) ? 1 : 0;
  // intermediate depths below K; those inside a 16-term slice split it into one more piece
  int pieces = 0, last_split = -1;
  while (p.ndep < ck.n && ck.k[p.ndep] < K) {
    if (ck.k[p.ndep] % 16 != 0) {
      ++pieces;
      last_split = ck.k[p.ndep] / 16;
    }
    ++p.ndep;
  }
  p.split_depths = pieces > 0 ? 1 : 0;
  // The segments: up to each depth, and for K > 512 no longer than kLoopSegTerms, because the rounding of a
  // long running sum adds up.  Error of h against 64 bits, one accumulator / segments / the two launches (which
  // split K over CTAs): H = 512, B = 16, K = 902 4.5e-6 / 3.3e-6 / 3.4e-6; H = 256, B = 64, K = 1000
  // 5.0e-6 / 4.3e-6 / 4.3e-6; at K = 512 one accumulator 3.35e-6, the two launches 3.40e-6.
  for (int i = 0, at = 0; i <= p.ndep; ++i) {
    const int end = i < p.ndep ? ck.k[i] : K;
    if (K > 512)
      for (int n = (end - at + kLoopSegTerms - 1) / kLoopSegTerms; n > 1; --n)  // n parts of whole slices
        p.cut_k[p.ncut++] = at = (at + (end - at + n - 1) / n + 8) / 16 * 16;
    if (i == p.ndep) break;
    p.cut_k[p.ncut++] = at = end;
    p.dep_segs[i] = p.ncut;
  }
  // without depths to read later, the epilogue adds up the segments as they come, and two accumulators do (H = 2048,
  // B = 64, K = 1024: four left room for tiles of 16 streams only, 18.4 us a step; two 15.3)
  p.stream_segs = p.ncut > 0 && p.ndep == 0;
  const int most = p.cs == 4 ? 144 : 148;  // CTAs in one wave: 36 clusters of 4, 74 of 2
  auto per_cta = [&](int nt, int groups) {  // stream tiles per CTA so that all groups' CTAs fit in one wave (0: none)
    const int ST = (B + nt - 1) / nt;
    for (int n = 1; n <= 8; ++n)
      if ((long long)groups * ((ST + n - 1) / n) <= most) return n;
    return 0;
  };
  // Tiles of 16 streams spread a few streams over more CTAs and have half the sums to read and exchange per
  // item; with many tiles per CTA those of 32 pay each item's latencies less often.  Recurrence, us a step, tiles
  // of 16 / 32 by the stream tiles of 16 per CTA (both roles; one gate per CTA, no depths unless said): 2 (H = 512,
  // B = 64, K = 512) 7.5 / 8.7, (K = 128, all gates) 8.0 / 9.0, (K = 512, two depths, B = 128) 9.2 / 10.9; 3 (H =
  // 512, B = 128, K = 902) 11.6 / 13.3, (H = 1024, B = 64, K = 700, a depth) 12.3 / 13.1; 4 (H = 2048, B = 64,
  // K = 512) 9.5 / 10.5, (H = 512, B = 1024, K = 128, all gates) 9.9 / 9.2, (H = 512, B = 256, K = 512, two depths)
  // 12.1 / 11.4; 5 (H = 512, B = 300, K = 200) 10.9 / 10.0; 8 (H = 512, B = 512, K = 512) 15.0 / 11.4.
  const int few = p.gp == 1 && p.ndep == 0 ? 4 : 3;
  const int sa16 = per_cta(16, p.RT * p.ga), sb16 = per_cta(16, p.UT * gb);
  const int first = sa16 > 0 && sb16 > 0 && sa16 + sb16 <= few ? 16 : 32;
  // A CTA's epilogues take longer than the launches they save once its streams (of both roles together) are many.
  // Measured, this launch / two launches, us a step: 96 streams (two layers of H = 2048, B = 64, K = 1024 with
  // depths) 21 / 33; 128 (H = 1024, B = 1024, K = 128) 11.1 / 14.6; 192 (H = 2048, B = 256, K = 200) 17.1 / 18.9,
  // (H = 2048, B = 180, K = 512) 17.6 / 18.6; 256 (H = 1024, B = 600, K = 200) 22.8 / 15.8.  Where the two launches
  // are at their best, and with several segments of terms, the line lies lower (us a run of 12 steps, D = 64):
  // - one gate per CTA, H <= 1024, no depths: 128 up to K = 448 (H > 512) or 384.  H = 1024, 160 streams (B = 300):
  //   K = 320 203 / 177, 384 207 / 186, 448 214 / 207, 512 217 / 216; 128 (B = 256): K = 320 149 / 243.  H = 512,
  //   160 (B = 600): K = 256 186 / 169, 384 198 / 198, 448 197 / 235; 128 (B = 500): K = 256 133 / 235.
  // - K > 512: 160.  H = 1024, K = 640, B = 256 247 / 298; H = 512, K = 800, B = 400 291 / 345; H = 2048, K = 800,
  //   B = 96 265 / 290; 192 (H = 2048, K = 800, B = 128) 305 / 319; but with H over two CTAs and K > 704, no
  //   depths, 128: H = 1024, K = 800, 160 (B = 160) 293 / 267, 96 (B = 128) 199 / 228.
  // - tiles of 16 in place of 32 for want of room: 128 with depths, else 64.  H = 2048, K = 1000, two depths, 96
  //   (B = 64) 306 / 364, 144 (B = 96) 429 / 406; H = 1024, K = 1000, no depths, 80 (B = 96) 240 / 235, 96 251 / 230.
  int limit = 192;
  if (slower_too)
    limit = 224;
  else if (K > 512)
    limit = p.ga == 2 && K > 704 && p.ndep == 0 ? 128 : 160;
  else if (p.gp == 1 && p.ga <= 2 && p.ndep == 0 && K <= (p.ga == 2 ? 448 : 384))
    limit = 128;
  const int limit16 = first == 16 || slower_too ? limit : p.ndep > 0 ? 128 : 64;
  // fills in the tile width nt with ures 64-term chunks of U in tensor memory; false if it does not fit
  auto fit = [&](int nt, int ures, TcLoopPlan* o) {
    TcLoopPlan c = p;
    c.nt = nt;
    c.ures = ures;
    c.ST = (B + nt - 1) / nt;
    if (c.ST > kLoopMaxTiles) return false;
    c.sa = per_cta(nt, c.RT * c.ga);
    c.sb = per_cta(nt, c.UT * gb);
    if (c.sa == 0 || c.sb == 0 || (c.sa + c.sb) * nt > (nt == 16 ? limit16 : limit)) return false;
    c.nA = c.RT * c.ga * ((c.ST + c.sa - 1) / c.sa);
    c.nB = c.UT * gb * ((c.ST + c.sb - 1) / c.sb);
    const int n = c.nA > c.nB ? c.nA : c.nB;
    c.ctas = (n + c.cs - 1) / c.cs * c.cs;
    if (c.ctas > most) return false;
    // tensor memory: U, then the accumulators
    const int slices = 4 * ures < nsl ? 4 * ures : nsl;
    if (last_split >= slices) return false;  // pieces of a slice are in tensor memory
    c.ux_chunks = c.gp * (nkb - ures);
    c.acc_a = ((slices + pieces) * c.gp * 8 + 31) / 32 * 32;
    const int seg = (c.stream_segs ? 1 : c.ncut + 1) * c.gp * nt;  // role B's accumulators of one region, one plane's columns
    int room = 512 - c.acc_a;
    if (room < seg || room < 2 * nt) return false;
    c.shared_acc = room < seg + 2 * nt ? 1 : 0;
    c.acc_b = c.shared_acc ? c.acc_a : c.acc_a + 2 * nt;
    room = 512 - c.acc_b;
    // Regions: a second one lets the next item's MMAs run while the epilogue reads this one's sums (with
    // intermediate depths it reads them late), and comes before both planes in one MMA (half the MMAs, but
    // twice the columns).
    const int want = c.sb > 1 || c.ndep > 0 || c.stream_segs ? 2 : 1;
    c.mb = room >= 2 * seg * want ? 1 : 0;
    c.rb_regions = room / (seg * (1 + c.mb));
    if (c.rb_regions > kMaxRegions) c.rb_regions = kMaxRegions;
    if (c.rb_regions > want && c.rb_regions > c.sb) c.rb_regions = want > c.sb ? want : c.sb;
    // the intermediate depths wait for the next step's tau' where their accumulators can stay that long
    c.defer_depths = (c.ndep > 0 && !c.shared_acc && c.rb_regions >= c.sb) ? 1 : 0;
    c.ra_regions = 1;
    if (c.shared_acc) {
      c.ra_regions = room / (2 * nt) < 2 ? room / (2 * nt) : 2;
    } else if (c.sa > 1 && room - c.rb_regions * seg * (1 + c.mb) >= 2 * nt) {
      c.ra_regions = 2;
      c.acc_b += 2 * nt;
    }
    c.rxa_bytes = c.ga > 1 ? 128 * nt * 4 : 0;
    c.rxb_bytes = gb > 1 ? 4 * 128 * (nt / gb) * 4 : 0;
    const uint32_t fixed = loop_layout(nt, c.nka, c.ux_chunks, 0, c.rxa_bytes, c.rxb_bytes, c.share_rx != 0).total;
    if (fixed > 227u * 1024u) return false;
    int stages = (int)((227u * 1024u - fixed) / (nt * 256u));
    if (stages > kMaxStages) stages = kMaxStages;
    if (stages * nt < 4 * 32) return false;  // at least 32 KB in flight
    c.stages = stages;
    c.smem = loop_layout(nt, c.nka, c.ux_chunks, stages, c.rxa_bytes, c.rxb_bytes, c.share_rx != 0).total;
    if (c.smem < 116u * 1024u) c.smem = 116u * 1024u;  // alone on its SM (tensor memory)
    *o = c;
    return true;
  };
  // Among the ways to hold U: separate accumulators for the two roles first, then as much of U as possible in
  // tensor memory.
  TcLoopPlan c;
  // (tiles of 16 in place of 32 for want of room do not make more streams fit)
  if (first == 32 && (per_cta(32, p.RT * p.ga) + per_cta(32, p.UT * gb)) * 32 > limit) return false;
  for (int nt : {first, 48 - first})
    for (int shared = 0; shared < 2; ++shared)
      for (int ures = nkb; ures >= 0; --ures)
        if (fit(nt, ures, &c) && c.shared_acc == shared) {
          *out = c;
          return true;
        }
  return false;
}

cudaError_t launch_tc_loop(const TcMap& V, const TcMap& U, const TcMap& Hm, const TcMap& Taum, const TcLoopPlan& p,
                           const TcLoopArgs& args, cudaStream_t s, bool* resident) {
  TcLoopArgs a = args;
  static_cast<TcLoopPlan&>(a) = p;
#define LA_LOOP(NT_, GP_, MB_)                                                                         \
  if (p.nt == NT_ && p.gp == GP_ && (p.mb != 0) == MB_)                                               \
    return p.split_depths ? launch_loop_t<NT_, GP_, MB_, true>(V, U, Hm, Taum, p, a, s, resident)     \
                          : launch_loop_t<NT_, GP_, MB_, false>(V, U, Hm, Taum, p, a, s, resident);
  LA_LOOP(16, 4, false) LA_LOOP(16, 1, false) LA_LOOP(32, 4, false) LA_LOOP(32, 1, false)
  LA_LOOP(16, 4, true) LA_LOOP(16, 1, true) LA_LOOP(32, 4, true) LA_LOOP(32, 1, true)
#undef LA_LOOP
  return cudaErrorInvalidValue;
}

}  // namespace lstm_approx_impl
