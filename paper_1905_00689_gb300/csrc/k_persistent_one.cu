// Smallest persistent kernel (fp32 factors): one CTA per stream runs all T
// timesteps, its factors in registers, and where the input is small computes
// the hoisted input projection itself, so that a whole call is one launch
// (Eq. 1 for the four gates, then the cell update of Sec. II).
//
// The cluster kernels (k_persistent.cu, k_persistent_ag.cu) spend a step on
// cluster exchanges: about 3000 cycles at H = 64.  Where both factors' h parts
// fit one CTA's registers (at most 512 threads x 16 values each) there is
// nothing to exchange: a step is two block barriers, two short dot products
// and the cell, bound by their latency chain (shared-memory reads, FMAs,
// shuffles, special functions) and by instruction issue.  The fewest threads
// that hold the factors with 16 values each are taken: the work per thread
// that does not depend on the values (addresses, shuffles, the cell) is what
// more threads repeat.
//
//   phase A  LA lanes share a coefficient row (g, k): each holds VQ quads of
//            V_h, quads l, l + LA, ... of the row, multiplies them with h from
//            shared memory; the lanes' sums are added by shuffles,
//            tau' = sigma (sum + P_t) goes to shared memory.
//   phase B  LB lanes share a gate row (unit j, gate g), the four gates of a
//            unit next to each other in one warp: each holds VQ quads of u;
//            the full depth and every intermediate depth (a masked sum of the
//            same values) are a depth set each, and the lanes of gate i
//            gather set i's four gate sums and runs its cell, so that
//            a round of four sets' cells runs at once.
//
// The projection: the LA lanes of row (g, k) read its x part (dense quads, or
// the kept entries of a compressed row) once for eight timesteps at a time, x
// being staged in shared memory.
//
// Measured (whole call, back to back): D = 64, H = 64, T = 8, K = 16 with two
// intermediate depths 24.2 (cluster of 4 and a projection launch) -> 10.7 us;
// D = 8256, H = 64, T = 1, K = 16, 130 kept entries 8.2 -> 5.8 us.  A step is
// about 2000 cycles with two depths (phase A 500, the full sums 300, the
// depths' sums and the transposition 850, cells 280): some 300 instructions
// per warp at six cycles each, two warps per scheduler.  512 threads instead
// of 256 took 2600 cycles a step.
#include "internal.h"
#include "ptx.cuh"

namespace lstm_approx_impl {
namespace {

using namespace lstm_approx_dev;

constexpr int kMaxThreads = 512;
constexpr int kMaxQuads = 4;      // quads of either factor per thread
constexpr int kStepsPerPass = 8;  // timesteps per read of a row's x part

struct OneDev {
  int LA, LB;  // lanes per coefficient row, per gate row (powers of two)
  int KP;      // stride of a gate's tau' in shared memory; the last quad stays zero
  int HP;      // h buffer length; the last quad stays zero
};

// Sum over the 2^lg lanes that differ in the low lg bits of the lane index.
__device__ __forceinline__ float lanes_sum(float v, int lg) {
  if (lg > 4) v += __shfl_xor_sync(0xffffffffu, v, 16);
  if (lg > 3) v += __shfl_xor_sync(0xffffffffu, v, 8);
  if (lg > 2) v += __shfl_xor_sync(0xffffffffu, v, 4);
  if (lg > 1) v += __shfl_xor_sync(0xffffffffu, v, 2);
  if (lg > 0) v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v;
}

template <int NTH, int VQ>
__global__ void __launch_bounds__(NTH, 1) persistent_one_kernel(PersistentArgs a, OneDev p, OneProj pr) {
  extern __shared__ __align__(16) float sm[];
  constexpr int kEntries = NTH == 512 ? 16 : 8;  // entries of a compressed row in flight per lane
  const int H = a.H, K = a.K, R = 4 * K, J = a.ck.n, T = a.T, B = a.B;
  float* h_s = sm;                    // [2][HP]
  float* tau_s = h_s + 2 * p.HP;      // [4][KP]
  float* P_s = tau_s + 4 * p.KP;      // [T][R] with the projection inside
  float* x_s = P_s + (pr.mode != 0 ? (T * R + 3) / 4 * 4 : 0);  // [T][XD]
  const int XD = (pr.D + 3) & ~3, VXS = XD + 4;
  float* vx_s = x_s + T * XD;  // [R][VXS] dense x rows
  const int tid = threadIdx.x, lane = tid & 31;
  const int b = blockIdx.x;

  const int lga = 31 - __clz(p.LA), lgb = 31 - __clz(p.LB);
  griddep_launch_dependents();
  // ---- factors into registers (they do not depend on earlier kernels) ----
  const int la = tid & (p.LA - 1), r = tid / p.LA;
  const bool row_ok = r < R;
  const int g_a = row_ok ? r / K : 0, k_a = row_ok ? r - g_a * K : 0;
  const long long srow = (long long)g_a * a.Ks + k_a;
  // compressed x rows: this lane's first entries
  int e0 = 0, e1 = 0;
  if (pr.mode == 2 && row_ok) {
    e0 = __ldg(pr.sparse.off[g_a] + k_a) + la;
    e1 = __ldg(pr.sparse.off[g_a] + k_a + 1);
  }
  const int HQ = (H + 3) >> 2;
  float4 va[VQ];
#pragma unroll
  for (int i = 0; i < VQ; ++i) {
    const int q = la + p.LA * i;
    va[i] = (row_ok && q < HQ) ? __ldg(reinterpret_cast<const float4*>(a.Vh + srow * a.ldh) + q)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const float sig = row_ok ? a.sigma[srow] : 0.f;
  const int lb = tid & (p.LB - 1), g_b = (tid / p.LB) & 3, j = tid / (4 * p.LB);
  const bool unit_ok = j < H;
  float4 ub[VQ];
#pragma unroll
  for (int i = 0; i < VQ; ++i) {
    const int k0 = 4 * (lb + p.LB * i);
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (unit_ok && k0 < K) {
      f = __ldg(reinterpret_cast<const float4*>(a.U + ((long long)g_b * H + j) * a.Ks + k0));
      if (k0 + 1 >= K) f.y = 0.f;
      if (k0 + 2 >= K) f.z = 0.f;
      if (k0 + 3 >= K) f.w = 0.f;
    }
    ub[i] = f;
  }
  float bias[4] = {0.f, 0.f, 0.f, 0.f};
  if (unit_ok)
#pragma unroll
    for (int g = 0; g < 4; ++g) bias[g] = a.bias[g * H + j];
  for (int i = tid; i < 2 * p.HP + 4 * p.KP; i += NTH) sm[i] = 0.f;
  int col[kEntries];
  float val[kEntries];
  if (pr.mode == 2) {
#pragma unroll
    for (int i = 0; i < kEntries; ++i) {
      const int e = e0 + p.LA * i;
      col[i] = e < e1 ? __ldg(pr.sparse.idx[g_a] + e) : 0;
      val[i] = e < e1 ? __ldg(pr.sparse.val[g_a] + e) : 0.f;
    }
  }
  if (pr.mode == 1) {  // (columns D .. ldx - 1 of the stored rows are zero)
    const int XQ = XD >> 2;
#pragma unroll 1
    for (int i = tid; i < R * XQ; i += NTH) {
      const int rr = i / XQ, q = i - rr * XQ, g = rr / K;
      const float* src = pr.Vx + ((long long)g * a.Ks + rr - g * K) * pr.ldx + 4 * q;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(vx_s + rr * VXS + 4 * q)), "l"(src)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  griddep_wait();  // x, P and the state may come from the kernels before this one
  __syncthreads();
  float c = 0.f;
  if (unit_ok && a.c0 != nullptr) c = a.c0[(long long)b * H + j];
  for (int i = tid; i < H; i += NTH) h_s[i] = a.h0 != nullptr ? a.h0[(long long)b * H + i] : 0.f;

  // ---- input projection P[t][r] (a1) ----
  // (compact loops: this code runs once per call, so its instructions come from L2)
  if (pr.mode != 0) {
    const int D = pr.D;
    const float* xb = pr.x + (long long)b * D;  // x_t of this stream at t * B * D; a row's tail is zero
    const long long xt = (long long)B * D;
    if ((D & 3) == 0 && (reinterpret_cast<uintptr_t>(pr.x) & 15u) == 0) {
      const int DQ = D >> 2;
#pragma unroll 4
      for (int i = tid; i < T * DQ; i += NTH) {
        const int t = i / DQ, q = i - t * DQ;
        reinterpret_cast<float4*>(x_s)[i] = __ldg(reinterpret_cast<const float4*>(xb + t * xt) + q);
      }
    } else {
#pragma unroll 4
      for (int i = tid; i < T * XD; i += NTH) {
        const int t = i / XD, d = i - t * XD;
        x_s[i] = d < D ? __ldg(xb + t * xt + d) : 0.f;
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (pr.mode == 1) {
      const float* vr = vx_s + (row_ok ? r : 0) * VXS;
#pragma unroll 1
      for (int t0 = 0; t0 < T; t0 += kStepsPerPass) {
        const float* xp = x_s + t0 * XD;
        float acc[kStepsPerPass];
#pragma unroll
        for (int s = 0; s < kStepsPerPass; ++s) acc[s] = 0.f;
#pragma unroll 1
        for (int q = 4 * la; q < XD; q += 4 * p.LA) {
          const float4 v = *reinterpret_cast<const float4*>(vr + q);
#pragma unroll
          for (int s = 0; s < kStepsPerPass; ++s) {
            const float4 xq = *reinterpret_cast<const float4*>(xp + min(s, T - 1 - t0) * XD + q);
            acc[s] = fmaf(v.x, xq.x, fmaf(v.y, xq.y, fmaf(v.z, xq.z, fmaf(v.w, xq.w, acc[s]))));
          }
        }
#pragma unroll
        for (int s = 0; s < kStepsPerPass; ++s) {
          const float v = lanes_sum(acc[s], lga);
          if (row_ok && la == 0 && t0 + s < T) P_s[(t0 + s) * R + r] = v;
        }
      }
    } else {
#pragma unroll 1
      for (int t = 0; t < T; ++t) {
        const float* xp = x_s + t * XD;
        float acc = 0.f;
#pragma unroll
        for (int i = 0; i < kEntries; ++i)
          if (e0 + p.LA * i < e1) acc = fmaf(val[i], xp[col[i]], acc);
#pragma unroll 4
        for (int e = e0 + p.LA * kEntries; e < e1; e += p.LA)
          acc = fmaf(__ldg(pr.sparse.val[g_a] + e), xp[__ldg(pr.sparse.idx[g_a] + e)], acc);
        __syncwarp();
        acc = lanes_sum(acc, lga);
        if (row_ok && la == 0) P_s[t * R + r] = acc;
      }
    }
  }
  __syncthreads();

  // ---- timesteps ----
  const long long p_stride = 4LL * a.Ks;
  const float* Pg = a.P + (long long)b * p_stride + srow;  // (projection by an earlier kernel)
  float p_next = 0.f;
  if (row_ok && la == 0) p_next = pr.mode != 0 ? P_s[r] : __ldcg(Pg);
  const int base = lane & ~(4 * p.LB - 1);  // the first of the unit's 4 LB lanes
  // shared-memory offsets of this lane's quads of h and tau'; past the row they read the zero quad (the lane's
  // factor values are zero there, but zero times an infinity is not)
  int qa[VQ], qb[VQ];
#pragma unroll
  for (int i = 0; i < VQ; ++i) {
    qa[i] = la + p.LA * i < HQ ? 4 * (la + p.LA * i) : p.HP - 4;
    qb[i] = g_b * p.KP + (4 * (lb + p.LB * i) < K ? 4 * (lb + p.LB * i) : p.KP - 4);
  }
  int kcut[4];  // the first round's depths (K: the full sums)
#pragma unroll
  for (int i = 0; i < 4; ++i) kcut[i] = i > 0 && i <= J ? a.ck.k[i - 1] : K;
  float* tau_w = tau_s + g_a * p.KP + k_a;
  for (int t = 0; t < T; ++t) {
    const float* h = h_s + (t & 1) * p.HP;
    const float pt = p_next;
    // ---- phase A: tau' = sigma (V_h h_{t-1} + P_t) ----
    {
      float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
      for (int i = 0; i < VQ; ++i) {
        const float4 hq = *reinterpret_cast<const float4*>(h + qa[i]);
        s0 = fmaf(va[i].x, hq.x, s0);
        s1 = fmaf(va[i].y, hq.y, s1);
        s2 = fmaf(va[i].z, hq.z, s2);
        s3 = fmaf(va[i].w, hq.w, s3);
      }
      const float s = lanes_sum((s0 + s1) + (s2 + s3), lga);
      if (row_ok && la == 0) {
        *tau_w = sig * (s + pt);
        if (t + 1 < T) p_next = pr.mode != 0 ? P_s[(t + 1) * R + r] : __ldcg(Pg + (long long)(t + 1) * B * p_stride);
      }
    }
    __syncthreads();
    // ---- phase B: gate sums and cells of every depth set (a3, a4, a6) ----
    float4 tq[VQ];
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll
    for (int i = 0; i < VQ; ++i) {
      tq[i] = *reinterpret_cast<const float4*>(tau_s + qb[i]);
      s0 = fmaf(ub[i].x, tq[i].x, s0);
      s1 = fmaf(ub[i].y, tq[i].y, s1);
      s2 = fmaf(ub[i].z, tq[i].z, s2);
      s3 = fmaf(ub[i].w, tq[i].w, s3);
    }
    const float full = lanes_sum((s0 + s1) + (s2 + s3), lgb);
    float c_new = c;
    const long long o = ((long long)t * B + b) * H + j;
    for (int n0 = 0; n0 <= J; n0 += 4) {  // four depth sets per round
      float s[4] = {full, full, full, full};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int n = n0 + i;
        const int kj = n0 == 0 ? kcut[i] : n <= J ? a.ck.k[n - 1] : K;
        if (kj < K) {  // the same products cut at k_j
          float m = 0.f;
#pragma unroll
          for (int v = 0; v < VQ; ++v) {
            if (4 * p.LB * v >= kj) break;  // no lane has terms below k_j from here on
            const int k0 = 4 * (lb + p.LB * v);
            if (4 * p.LB * (v + 1) <= kj) {  // all lanes' terms are below it
              m = fmaf(ub[v].x, tq[v].x, m);
              m = fmaf(ub[v].y, tq[v].y, m);
              m = fmaf(ub[v].z, tq[v].z, m);
              m = fmaf(ub[v].w, tq[v].w, m);
            } else {
              if (k0 < kj) m = fmaf(ub[v].x, tq[v].x, m);
              if (k0 + 1 < kj) m = fmaf(ub[v].y, tq[v].y, m);
              if (k0 + 2 < kj) m = fmaf(ub[v].z, tq[v].z, m);
              if (k0 + 3 < kj) m = fmaf(ub[v].w, tq[v].w, m);
            }
          }
          s[i] = lanes_sum(m, lgb);
        }
      }
      // transpose over the unit's four gates: lane (gate g) held gate g's sums of four sets, and takes set
      // n0 + g's four gates (the pairs exchanged are LB and 2 LB lanes apart)
      float y[4];
      {
        const bool o1 = (g_b & 1) != 0, o2 = (g_b & 2) != 0;
        const float r0 = __shfl_xor_sync(0xffffffffu, o1 ? s[0] : s[1], p.LB);
        const float r1 = __shfl_xor_sync(0xffffffffu, o1 ? s[2] : s[3], p.LB);
        const float a0 = o1 ? r0 : s[0], a1 = o1 ? s[1] : r0;  // gates (g & 2) + 0, + 1 of set (g & 1)
        const float b0 = o1 ? r1 : s[2], b1 = o1 ? s[3] : r1;  // the same of set 2 + (g & 1)
        const float q0 = __shfl_xor_sync(0xffffffffu, o2 ? a0 : b0, 2 * p.LB);
        const float q1 = __shfl_xor_sync(0xffffffffu, o2 ? a1 : b1, 2 * p.LB);
        y[0] = (o2 ? q0 : a0) + bias[0];
        y[1] = (o2 ? q1 : a1) + bias[1];
        y[2] = (o2 ? b0 : q0) + bias[2];
        y[3] = (o2 ? b1 : q1) + bias[3];
      }
      float hh, cc;
      lstm_cell_f(y[0], y[1], y[2], y[3], c, hh, cc);
      const int set = n0 + g_b;
      if (n0 == 0) c_new = __shfl_sync(0xffffffffu, cc, base);
      if (unit_ok && lb == 0) {
        if (set == 0) {
          h_s[((t + 1) & 1) * p.HP + j] = hh;
          a.out_h[o] = hh;
        } else if (set <= J) {
          const long long on = (long long)(set - 1) * T * B * H + o;
          if (a.ckpt_h) a.ckpt_h[on] = hh;
          if (a.ckpt_c) a.ckpt_c[on] = cc;
        }
      }
    }
    c = c_new;
    __syncthreads();
  }
  if (unit_ok && lb == 0 && g_b == 0 && a.c_last != nullptr) a.c_last[(long long)b * H + j] = c;
}

int pow2_at_most(int v) {
  int p = 1;
  while (2 * p <= v) p *= 2;
  return p;
}

}  // namespace

bool plan_persistent_one(int H, int K, int T, const Checkpoints& ck, bool gathers, PersistentOnePlan* out) {
  if (H < 1 || H > 128 || K < 1 || K > 128) return false;
  // The fewest threads that hold the factors in 4 quads each; 512 where compressed rows of x are gathered (entries
  // in flight).  With 8 quads a step takes longer than the one-exchange cluster kernel's and the set-up as long:
  // T = 32, H = 64, K = 64 55.7 us against 49.7, H = 128, K = 32 57.8 / 45.6, H = 32, K = 96 60.0 / 47.7; with 4
  // H = 64, K = 16 31.2 / 41.3, H = 32, K = 32 32.3 / 41.5 (256 threads; 512: below).
  PersistentOnePlan p;
  for (int nth = 128; nth <= kMaxThreads; nth *= 2) {
    if (4 * K > nth || 4 * H > nth || (gathers && nth < kMaxThreads)) continue;
    p.threads = nth;
    p.LA = pow2_at_most(nth / (4 * K));
    if (p.LA > 32) p.LA = 32;
    p.LB = pow2_at_most(nth / (4 * H));
    if (p.LB > 8) p.LB = 8;
    const int qa = ((H + 3) / 4 + p.LA - 1) / p.LA, qb = ((K + 3) / 4 + p.LB - 1) / p.LB;
    const int q = qa > qb ? qa : qb;
    p.VQ = q <= 1 ? 1 : q <= 2 ? 2 : q <= kMaxQuads ? kMaxQuads : 0;
    if (p.VQ != 0) goto found;
  }
  return false;
found:
  // With 512 threads of 16 values each a step without intermediate depths takes longer than the cluster kernel's
  // (1.32 us against 1.03 at H = 64, K = 32, 1.18 at H = 128, K = 16; with a depth 1.5 / 2 or less), and only the
  // set-up is shorter (4 us against 8.5).  Calls back to back and single calls, us, this kernel / cluster kernel:
  // H = 64, K = 32 T = 8 13.4 / 16.7 and 28.6 / 28.5, T = 12 20.0 / 20.9 and 36.1 / 32.6, T = 20 30.8 / 29.2 and
  // 47.4 / 40.7, T = 32 46.1 / 41.6; H = 128, K = 16 T = 20 27.3 / 29.1 and 43.4 / 40.2, T = 32 41.3 / 41.4 and 56.7 /
  // 53.1, T = 64 80.0 / 74.3.
  // (H = 8, K = 96 T = 32 43.3 / 45.5.)
  if (p.threads == 512 && p.VQ == kMaxQuads && H >= 32 && !gathers && T > (K > 16 ? 12 : 20) &&
      (ck.n == 0 || ck.k[0] >= K))
    return false;
  p.HP = (H + 3) / 4 * 4 + 4;
  // the four gates' rows eight banks apart, so that the 16-byte reads of a unit's lanes do not collide
  p.KP = ((K + 3) / 4 * 4 + 4 + 23) / 32 * 32 + 8;
  *out = p;
  return true;
}

size_t persistent_one_smem(const PersistentOnePlan& p, int T, int K, const OneProj& pr) {
  size_t f = 2ull * p.HP + 4ull * p.KP;
  const size_t XD = ((size_t)pr.D + 3) & ~(size_t)3;
  if (pr.mode != 0) f += ((size_t)T * 4 * K + 3) / 4 * 4 + (size_t)T * XD;
  if (pr.mode == 1) f += 4ull * K * (XD + 4);
  return f * sizeof(float);
}

// Whether the projection belongs inside: x of one stream, P and (dense) the rows' x parts in shared memory,
// and little enough to read for one CTA (64 KB of dense rows, or 28 K kept entries over up to 8 timesteps: a
// separate grid reads more in the time of a launch: D = 1000, T = 4, K = 32, 25.6 K entries 8.9 us inside, 10.9
// by its own launch; D = 2000, T = 2, K = 40, 32 K 13.1 / 10.5; D = 500, T = 16, K = 16, 26 K 23.0 / 19.0).
int persistent_one_projection(int K, int T, int D, long long kept_x, bool sparse) {
  if ((long long)T * D > 16 * 1024 || (long long)T * 4 * K > 12 * 1024) return 0;
  if (sparse) return T <= 8 && kept_x * T <= 28 * 1024 ? 2 : 0;
  return 4LL * K * D <= 16 * 1024 && 4LL * K * (D + 8) <= 20 * 1024 ? 1 : 0;
}

namespace {

template <int NTH, int VQ>
cudaError_t launch_one_t(const PersistentOnePlan& p, const PersistentArgs& a, const OneProj& pr, cudaStream_t s) {
  auto kern = persistent_one_kernel<NTH, VQ>;
  static thread_local DeviceSet ready;
  const cudaError_t ea = once_per_device(
      &ready, [&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024); });
  if (ea != cudaSuccess) return ea;
  OneDev d;
  d.LA = p.LA;
  d.LB = p.LB;
  d.KP = p.KP;
  d.HP = p.HP;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.B);
  cfg.blockDim = dim3(NTH);
  cfg.dynamicSmemBytes = persistent_one_smem(p, a.T, a.K, pr);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, d, pr);
}

}  // namespace

cudaError_t launch_persistent_one(const PersistentOnePlan& p, const PersistentArgs& a, const OneProj& pr,
                                  cudaStream_t s) {
#define LA_ONE(N_, V_) \
  if (p.threads == N_ && p.VQ == V_) return launch_one_t<N_, V_>(p, a, pr, s);
  LA_ONE(128, 1) LA_ONE(128, 2) LA_ONE(128, 4)
  LA_ONE(256, 1) LA_ONE(256, 2) LA_ONE(256, 4)
  LA_ONE(512, 1) LA_ONE(512, 2) LA_ONE(512, 4)
#undef LA_ONE
  return cudaErrorInvalidValue;
}

}  // namespace lstm_approx_impl
