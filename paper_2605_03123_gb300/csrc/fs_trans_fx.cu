// The reductions of a complex128 reverse sweep whose rotations ran on the
// tensor cores (fs_sweep_fx.cu): the transition sums T[p][q] = <g| E_pq |psi>
// of one spin, and the pass that writes W = Im(conj(g) psi) and applies the
// diagonal gate to both states.
#include <algorithm>

#include "fs_fx.cuh"
#include "fs_common.cuh"
#include "fs_internal.h"

namespace fs {
namespace fx {

constexpr int kTThreads = 256;
constexpr int kTWarps = kTThreads / 32;
constexpr int kTUnits = 4;  // units per pass

// Cells of a slab: what the sums below are bounded for (an SM holds 7200).
constexpr int kMaxVec = 64, kMaxCells = 8191;

// A slab's products are held relative to the product of its two norms.  Where
// no vector of it comes within 2^-kApart of that (psi and g in different
// vectors), or one of its vectors was rotated in FP64, the slab is summed in
// FP64: the integers keep 2^-59 of the norms, FP64 2^-53 of the amplitudes that
// meet.  (KV equal vectors are 2^-8 apart at most, for KV = 64.)
constexpr int kApart = 10;

struct TransArgs {
  const double2* st[2];  // psi, g
  int64_t d_b;
  int dir, d, nvec, KV, npass, norb;
  const int* scale;  // per state and vector, from launch_sweep_fx
  const TPassDev* tpass;
  const TRecord* trec;
  double* T;
};

// An amplitude as integers: each part X = hi 2^27 + lo, |X| < 2^58 (the
// slab's 2-norm is below 2^58 / 1.001), lo balanced.
__device__ __forceinline__ int4 split_amp(double2 x, int eb) {
  const long long a = from_double(x.x, eb + 4), b = from_double(x.y, eb + 4);
  const int al = (int)((uint32_t)a << 5) >> 5, bl = (int)((uint32_t)b << 5) >> 5;
  return make_int4((int)((a - al) >> 27), al, (int)((b - bl) >> 27), bl);
}
__host__ __device__ constexpr int popc4(int x) {
  return (x & 1) + ((x >> 1) & 1) + ((x >> 2) & 1) + ((x >> 3) & 1);
}
__host__ __device__ constexpr int sub_mask(int M, int k) {  // k-th 4-bit mask with M bits
  for (int x = 0; x < 16; ++x)
    if (popc4(x) == M && k-- == 0) return x;
  return -1;
}
__host__ __device__ constexpr int sub_index(int M, int mask) {
  int k = 0;
  for (int x = 0; x < mask; ++x) k += popc4(x) == M;
  return k;
}
__host__ __device__ constexpr int sub_count(int M) { return M == 2 ? 6 : M == 4 ? 1 : 4; }

// Sums of one warp unit: per local slot and part, the products of the high
// halves and the cross products of high and low halves.  The low-low ones are
// left out: with low halves of either sign some 2^-59 of the norms' product, as
// much as the rounding of X.  Neither sum can pass 2^63, by Cauchy-Schwarz with
// a norm of 2^31 of the high and 2^26 sqrt(2 T) of the low halves of T amplitudes:
// the first stays below 2^62, and the second, 2^58 sqrt(2 T), below 2^62.8 for a
// lane's at most 3 (kMaxCells / 128 + kMaxVec) amplitudes a slot (a record holds
// three of them at most), and below 2^62 for a slab's kMaxCells once every lane
// has divided it by 8.
struct Sums {
  long long hh[16][2], cr[16][2];
};
__device__ __forceinline__ void mac(long long& hh, long long& cr, int ph, int pl, int gh, int gl) {
  hh += (long long)ph * gh;
  cr += (long long)ph * gl;
  cr += (long long)pl * gh;
}
// Slot (a, b) of string S: conj(g[S']) psi[S], S' = S - b + a.
template <int M, int J, bool DIAG, int NS>
__device__ __forceinline__ void term(const int4 (&ps)[NS], const int4 (&pg)[NS], Sums& t) {
  constexpr int k = J / 16, a = (J / 4) % 4, b = J % 4;
  if constexpr (k < NS) {
    constexpr int S = sub_mask(M, k), slot = a * 4 + b;
    if constexpr (((S >> b) & 1) && (a == b ? DIAG : !((S >> a) & 1))) {
      constexpr int k2 = a == b ? k : sub_index(M, (S & ~(1 << b)) | (1 << a));
      constexpr int lo = a < b ? a : b, hi = a < b ? b : a;
      constexpr int sg = a != b && (popc4(S & ((1 << hi) - 1) & ~((2 << lo) - 1)) & 1) ? -1 : 1;
      const int ph = sg * ps[k].x, pl = sg * ps[k].y, qh = sg * ps[k].z, ql = sg * ps[k].w;
      const int4 g = pg[k2];
      mac(t.hh[slot][0], t.cr[slot][0], ph, pl, g.x, g.y);    // Re g Re psi
      mac(t.hh[slot][0], t.cr[slot][0], qh, ql, g.z, g.w);    // Im g Im psi
      mac(t.hh[slot][1], t.cr[slot][1], qh, ql, g.x, g.y);    // Re g Im psi
      mac(t.hh[slot][1], t.cr[slot][1], ph, pl, -g.z, -g.w);  // -Im g Re psi
    }
  }
}
template <int M, bool DIAG, int NS, int... J>
__device__ __forceinline__ void terms(const int4 (&ps)[NS], const int4 (&pg)[NS], Sums& t,
                                      std::integer_sequence<int, J...>) {
  (term<M, J, DIAG, NS>(ps, pg, t), ...);
}
__device__ __forceinline__ int4 flip(int4 x, int m) {  // m = 0 or -1
  return make_int4((x.x ^ m) - m, (x.y ^ m) - m, (x.z ^ m) - m, (x.w ^ m) - m);
}
template <int M, bool DIAG>
__device__ __forceinline__ void record(const TRecord& rc, const int4* psi, const int4* g, Sums& t) {
  constexpr int NS = sub_count(M);
  int4 ps[NS], pg[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const int m = -(int)((rc.flips >> k) & 1u);
    ps[k] = flip(psi[rc.addr[k]], m);
    pg[k] = flip(g[rc.addr[k]], m);
  }
  terms<M, DIAG, NS>(ps, pg, t, std::make_integer_sequence<int, 6 * 16>{});
}
template <bool DIAG>
__device__ __forceinline__ void unit(const TransArgs& a, const TPassDev& pd, int q, int nv,
                                     const int4* psi, const int4* g, int lane, Sums& t) {
  const int nrec = (pd.rec1 - pd.rec0) >> 5, nch = nrec * nv;
  for (int ch = q; ch < nch; ch += kTUnits) {
    const int kv = ch / nrec, oc = ch - kv * nrec;
    TRecord rc;
    *reinterpret_cast<uint4*>(&rc) =
        __ldg(reinterpret_cast<const uint4*>(a.trec + pd.rec0 + (oc << 5) + lane));
    const int4* p0 = psi + (size_t)kv * a.d;
    const int4* g0 = g + (size_t)kv * a.d;
    switch (rc.m) {
      case 1: record<1, DIAG>(rc, p0, g0, t); break;
      case 2: record<2, DIAG>(rc, p0, g0, t); break;
      case 3: record<3, DIAG>(rc, p0, g0, t); break;
      case 4: if constexpr (DIAG) record<4, DIAG>(rc, p0, g0, t); break;
      default: break;
    }
  }
}

// The same of a slab in FP64: its cells hold the amplitudes, `sum` ([npass][32]
// [2]) takes each slot's parts as doubles.
template <int M, int J, bool DIAG, int NS>
__device__ __forceinline__ void term64(const double2 (&ps)[NS], const double2 (&pg)[NS],
                                       double (&t)[32]) {
  constexpr int k = J / 16, a = (J / 4) % 4, b = J % 4;
  if constexpr (k < NS) {
    constexpr int S = sub_mask(M, k), slot = a * 4 + b;
    if constexpr (((S >> b) & 1) && (a == b ? DIAG : !((S >> a) & 1))) {
      constexpr int k2 = a == b ? k : sub_index(M, (S & ~(1 << b)) | (1 << a));
      constexpr int lo = a < b ? a : b, hi = a < b ? b : a;
      constexpr double sg = a != b && (popc4(S & ((1 << hi) - 1) & ~((2 << lo) - 1)) & 1) ? -1 : 1;
      const double2 g = pg[k2], p = ps[k];
      t[2 * slot] = fma(sg * g.x, p.x, fma(sg * g.y, p.y, t[2 * slot]));
      t[2 * slot + 1] = fma(sg * g.x, p.y, fma(-sg * g.y, p.x, t[2 * slot + 1]));
    }
  }
}
template <int M, bool DIAG, int NS, int... J>
__device__ __forceinline__ void terms64(const double2 (&ps)[NS], const double2 (&pg)[NS],
                                        double (&t)[32], std::integer_sequence<int, J...>) {
  (term64<M, J, DIAG, NS>(ps, pg, t), ...);
}
template <int M, bool DIAG>
__device__ __forceinline__ void record64(const TRecord& rc, const double2* psi, const double2* g,
                                         double (&t)[32]) {
  constexpr int NS = sub_count(M);
  double2 ps[NS], pg[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double f = (rc.flips >> k) & 1u ? -1.0 : 1.0;
    ps[k] = psi[rc.addr[k]];
    pg[k] = g[rc.addr[k]];
    ps[k].x *= f;
    ps[k].y *= f;
    pg[k].x *= f;
    pg[k].y *= f;
  }
  terms64<M, DIAG, NS>(ps, pg, t, std::make_integer_sequence<int, 6 * 16>{});
}
template <bool DIAG>
__device__ __noinline__ void unit64(const TransArgs& a, const TPassDev& pd, int q, int nv,
                                    const double2* psi, const double2* g, int lane,
                                    unsigned long long* sum) {
  double t[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) t[i] = 0;
  const int nrec = (pd.rec1 - pd.rec0) >> 5, nch = nrec * nv;
  for (int ch = q; ch < nch; ch += kTUnits) {
    const int kv = ch / nrec, oc = ch - kv * nrec;
    TRecord rc;
    *reinterpret_cast<uint4*>(&rc) =
        __ldg(reinterpret_cast<const uint4*>(a.trec + pd.rec0 + (oc << 5) + lane));
    const double2* p0 = psi + (size_t)kv * a.d;
    const double2* g0 = g + (size_t)kv * a.d;
    switch (rc.m) {
      case 1: record64<1, DIAG>(rc, p0, g0, t); break;
      case 2: record64<2, DIAG>(rc, p0, g0, t); break;
      case 3: record64<3, DIAG>(rc, p0, g0, t); break;
      case 4: if constexpr (DIAG) record64<4, DIAG>(rc, p0, g0, t); break;
      default: break;
    }
  }
  // after the halving lane l holds the warp's sum of value l
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const bool up = lane & s;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const double send = up ? t[i] : t[i + s], keep = up ? t[i + s] : t[i];
      t[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, s);
    }
  }
  if (pd.keep & (1u << (lane >> 1))) atomicAdd(reinterpret_cast<double*>(sum + 2 * lane), t[0]);
}

// One CTA per slab of KV vectors of both states.  The multiply-adds of the
// sums (12 wide integer ones per complex product; FP64 would need 4, but
// GB300 issues two of those per clock and SM) bound it: N = 12 (6,6) 0.18 ms
// a spin, where the FP64 reduction took 1.0.  Passes, records and
// local slots are those of the FP64 sweep's reduction (tpass_tables_host); a
// warp takes whole units (pass, every fourth chunk of 32 records) and reduces
// once per unit.  The sums are integers, so a slab's result does not depend
// on the order of its warps.
__global__ void __launch_bounds__(kTThreads, 1)
    k_trans_fx(const __grid_constant__ TransArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ uint32_t s_max[2][kTWarps];
  __shared__ float s_sum[2][kTWarps];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int v0 = blockIdx.x * a.KV, nv = min(a.KV, a.nvec - v0), n = nv * a.d;
  int4* cell = reinterpret_cast<int4*>(smraw);  // psi, then g (KV d cells each)
  unsigned long long* tsm =
      reinterpret_cast<unsigned long long*>(cell + 2 * (size_t)a.KV * a.d);  // [npass][32][2]
  for (int i = tid; i < a.npass * 64; i += kTThreads) tsm[i] = 0;
  // load; the slab's scale per state (see k_sweep_fx)
  for (int s = 0; s < 2; ++s) {
    double2* raw = reinterpret_cast<double2*>(cell + (size_t)s * a.KV * a.d);
    uint32_t mx = 1;
    if (a.dir == 1) {
      for (int kv = 0; kv < nv; ++kv) {
        const double2* src = a.st[s] + (int64_t)(v0 + kv) * a.d_b;
#pragma unroll 4
        for (int e = tid; e < a.d; e += kTThreads) {
          const double2 x = src[e];
          raw[(size_t)kv * a.d + e] = x;
          mx = max(mx, (uint32_t)max(exp_field(x.x), exp_field(x.y)));
        }
      }
    } else {
#pragma unroll 4
      for (int i = tid; i < n; i += kTThreads) {
        const int e = i / nv, kv = i - e * nv;
        const double2 x = a.st[s][(int64_t)e * a.d_b + v0 + kv];
        raw[(size_t)kv * a.d + e] = x;
        mx = max(mx, (uint32_t)max(exp_field(x.x), exp_field(x.y)));
      }
    }
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if (lane == 0) s_max[s][warp] = mx;
  }
  __syncthreads();
  uint32_t fm[2];
  for (int s = 0; s < 2; ++s) {
    fm[s] = 1;
    for (int w = 0; w < kTWarps; ++w) fm[s] = max(fm[s], s_max[s][w]);
    const double2* raw = reinterpret_cast<const double2*>(cell + (size_t)s * a.KV * a.d);
    float q = 0.f;
#pragma unroll 4
    for (int i = tid; i < n; i += kTThreads) {
      const double2 x = raw[i];
      const float u = rel_abs(x.x, (int)fm[s]), v = rel_abs(x.y, (int)fm[s]);
      q = fmaf(u, u, fmaf(v, v, q));
    }
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) q += __shfl_xor_sync(0xFFFFFFFFu, q, k);
    if (lane == 0) s_sum[s][warp] = q;
  }
  __syncthreads();
  int eb[2];
  for (int s = 0; s < 2; ++s) {
    float q = 0.f;
    for (int w = 0; w < kTWarps; ++w) q += s_sum[s][w];
    eb[s] = norm_exponent((int)fm[s], q);
  }
  // (the sweep sent every vector that is not finite to FP64)
  bool apart = false;
  int most = 0;
  for (int kv = lane; kv < nv; kv += 32) {
    const int p = a.scale[v0 + kv], c = a.scale[a.nvec + v0 + kv];
    apart = apart || p < 0 || c < 0;
    most = max(most, p + c);
  }
  most = __reduce_max_sync(0xFFFFFFFFu, most);
  apart = __any_sync(0xFFFFFFFFu, apart) || most + kApart < eb[0] + eb[1];
  for (int s = 0; s < 2 && !apart; ++s) {
    double2* raw = reinterpret_cast<double2*>(cell + (size_t)s * a.KV * a.d);
    int4* c = cell + (size_t)s * a.KV * a.d;
#pragma unroll 4
    for (int i = tid; i < n; i += kTThreads) c[i] = split_amp(raw[i], eb[s]);
  }
  __syncthreads();
  const int4* psi = cell;
  const int4* g = cell + (size_t)a.KV * a.d;
  if (apart) {
    for (int u = warp; u < a.npass * kTUnits; u += kTWarps) {
      const int ip = u / kTUnits, q = u - ip * kTUnits;
      const TPassDev pd = a.tpass[ip];
      const double2* p = reinterpret_cast<const double2*>(psi);
      const double2* c = reinterpret_cast<const double2*>(g);
      if (pd.keep & 0x8421u)
        unit64<true>(a, pd, q, nv, p, c, lane, tsm + ip * 64);
      else
        unit64<false>(a, pd, q, nv, p, c, lane, tsm + ip * 64);
    }
  } else {
    for (int u = warp; u < a.npass * kTUnits; u += kTWarps) {
      const int ip = u / kTUnits, q = u - ip * kTUnits;
      const TPassDev pd = a.tpass[ip];
      Sums t;
#pragma unroll
      for (int i = 0; i < 16; ++i)
        for (int r = 0; r < 2; ++r) t.hh[i][r] = t.cr[i][r] = 0;
      if (pd.keep & 0x8421u)
        unit<true>(a, pd, q, nv, psi, g, lane, t);
      else
        unit<false>(a, pd, q, nv, psi, g, lane, t);
      // value 4 slot + 2 part + {high, cross}: after the halving lane l holds
      // the warp's sums of values 2 l and 2 l + 1
      long long v[64];
#pragma unroll
      for (int i = 0; i < 16; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          v[4 * i + 2 * r] = t.hh[i][r];
          v[4 * i + 2 * r + 1] = (t.cr[i][r] + 4) >> 3;
        }
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) {
        const bool up = lane & s;
#pragma unroll
        for (int i = 0; i < 2 * s; ++i) {
          const long long send = up ? v[i] : v[i + 2 * s], keep = up ? v[i + 2 * s] : v[i];
          v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, s);
        }
      }
      if (pd.keep & (1u << (lane >> 1))) {
        atomicAdd(tsm + (ip * 32 + lane) * 2, (unsigned long long)v[0]);
        atomicAdd(tsm + (ip * 32 + lane) * 2 + 1, (unsigned long long)v[1]);
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < a.npass * 32; i += kTThreads) {
    const TPassDev pd = a.tpass[i >> 5];
    const int slot = (i & 31) >> 1;
    if (!(pd.keep & (1u << slot))) continue;
    // hh 2^54 + cr 2^30 in units of 2^(E_psi + E_g - 116)
    const double s = (double)(long long)tsm[2 * i] + ldexp((double)(long long)tsm[2 * i + 1], -24);
    const double x = apart ? __longlong_as_double((long long)tsm[2 * i])
                           : scalbn(s, eb[0] + eb[1] - 2 * 1023 - 62);
    const int p = pd.q[slot >> 2], q = pd.q[slot & 3];
    atomicAdd(a.T + 2 * (p * a.norb + q) + (i & 1), x);
  }
}

static size_t trans_smem(const Space* sp, int KV, int npass) {
  return (size_t)KV * sp->dim * 32 + (size_t)npass * 64 * 8;
}

}  // namespace fx

bool trans_fx_supported(const Ctx* ctx, const Space* sthis) {
  return sthis->npass > 0 && sthis->dim <= fx::kMaxCells &&
         fx::trans_smem(sthis, 1, sthis->npass) <= (size_t)ctx->prop.sharedMemPerBlockOptin - 1024;
}

void launch_trans_fx(Ctx* ctx, const Space* sa, const Space* sb, int dir, const void* psi,
                     const void* g, const int* scale, double* T, cudaStream_t st) {
  const Space* sthis = dir == 0 ? sa : sb;
  const Space* sother = dir == 0 ? sb : sa;
  fx::TransArgs a{};
  a.st[0] = (const double2*)psi;
  a.st[1] = (const double2*)g;
  a.d_b = sb->dim;
  a.dir = dir;
  a.d = (int)sthis->dim;
  a.nvec = (int)sother->dim;
  a.npass = sthis->npass;
  a.norb = sthis->norb;
  a.tpass = sthis->tpass;
  a.trec = sthis->trec;
  a.scale = scale;
  a.T = T;
  // vectors per slab: the least modelled time, a wave of slabs costing its
  // vectors and what a slab costs by itself (its reductions and scale, worth 400
  // strings).  Measured, one spin: N = 12 (6,6) 7 vectors 180 us (chosen), 4
  // 219, 2 242, 6 296; N = 11 (6,5) 4 72 (chosen), 2 87, 1 127, 8 121; N = 9
  // (4,5) 1 25 (chosen), 2 30, 8 76.
  const size_t avail = (size_t)ctx->prop.sharedMemPerBlockOptin - 1024;
  const int sms = ctx->prop.multiProcessorCount;
  double best = 0;
  for (int kv = 1; kv <= fx::kMaxVec && (int64_t)kv * a.d <= fx::kMaxCells &&
                   fx::trans_smem(sthis, kv, a.npass) <= avail;
       ++kv) {
    const int slabs = (a.nvec + kv - 1) / kv;
    const double c = ((slabs + sms - 1) / sms) * (kv + 400.0 / a.d);
    if (kv == 1 || c < best) {
      best = c;
      a.KV = kv;
    }
  }
  const size_t smem = fx::trans_smem(sthis, a.KV, a.npass);
  allow_shared_memory(fx::k_trans_fx);
  ProfScope ps(dir == 0 ? "trans_alpha_fx" : "trans_beta_fx", st);
  fx::k_trans_fx<<<(a.nvec + a.KV - 1) / a.KV, fx::kTThreads, smem, st>>>(a);
  FS_CUDA(cudaGetLastError());
}

}  // namespace fs
