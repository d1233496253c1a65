// Complex128 orbital-rotation sweeps of small spaces: one CTA per vector,
// rotation by rotation.
//
// On vectors of up to a few hundred strings a window step leaves most lanes
// idle (an orbit per lane, ten of them at N = 8) and a tensor-core tile most
// rows, so both kinds of sweep are chains of latencies.  Here a CTA keeps a
// vector, the coefficients and the pair lists in shared memory and applies
// each Givens rotation (§3.2.3) to its pairs.  GB300 takes some 64 clocks for
// an FP64 instruction of a warp, however few of its lanes work, so the four
// real components of a pair's update go to four lanes: three multiply-adds
// in a row per rotation instead of twelve.  Bound by that chain: some 300
// clocks a rotation at N = 8, of which two are barriers.  A rotation of both
// spins at N = 8 (4,4): 50 us (FP64 window sweeps 91, digits on the tensor
// cores 79); N = 9 (4,5): 49 us (digits 87); N = 4 (2,2): 38 us (window sweeps
// 42).
#include <algorithm>

#include "fs_fx.cuh"
#include "fs_common.cuh"
#include "fs_internal.h"

namespace fs {
namespace pairs {

struct Args {
  double2* st;
  int64_t d_b;
  int dir, d, nvec, npp, m, norb, nchunk, has_x, has_d;
  const uint32_t* list;  // adjacent pair lists
  const uint32_t *masks_this, *masks_other;
  const double2 *ea_this, *ea_other;
  int64_t lin[kMaxOrb];  // has_d: angle of each orbital's diagonal phase, in turns
  double c[kMaxM], sr[kMaxM], si[kMaxM];
  int8_t p[kMaxM];
};

static size_t smem_bytes(const Args& a) {
  const size_t tab = a.has_x ? (size_t)(a.nchunk * 256 + 32 + 32 * a.nchunk) * 16 : 0;
  return (size_t)a.d * 16 + (size_t)a.m * 24 + tab + (size_t)(a.norb - 1) * a.npp * 4;
}

__global__ void __launch_bounds__(256)
    k_sweep_pairs(const __grid_constant__ Args g, const __grid_constant__ Mat X) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ uint32_t bad_x;
  const int tid = threadIdx.x, nt = blockDim.x, d = g.d, v = blockIdx.x;
  double2* x = reinterpret_cast<double2*>(smraw);
  longlong2* tab = reinterpret_cast<longlong2*>(x + d);
  longlong2* work = tab + (g.has_x ? g.nchunk * 256 : 0);
  double* coef = reinterpret_cast<double*>(work + (g.has_x ? 32 + 32 * g.nchunk : 0));
  uint32_t* list = reinterpret_cast<uint32_t*>(coef + 3 * g.m);
  const int64_t es = g.dir == 1 ? 1 : g.d_b;
  double2* vec = g.st + (g.dir == 1 ? (int64_t)v * g.d_b : (int64_t)v);
  for (int e = tid; e < d; e += nt) x[e] = vec[e * es];
  for (int k = tid; k < g.m; k += nt) {
    coef[3 * k] = g.c[k];
    coef[3 * k + 1] = g.sr[k];
    coef[3 * k + 2] = g.si[k];
  }
  for (int i = tid; i < (g.norb - 1) * g.npp; i += nt) list[i] = __ldg(g.list + i);
  __syncthreads();
  // lane component q of a pair (x, y): Re x, Im x, Re y, Im y; each becomes
  // c a + (p b + r e) with b, e the parts of the other amplitude (givens2)
  const int q = tid & 3, own = q >> 1;
  double* xs = reinterpret_cast<double*>(x);
  const int per = nt >> 2;
  for (int k = 0; k < g.m; ++k) {
    const double c = coef[3 * k], sr = coef[3 * k + 1], si = coef[3 * k + 2];
    const double p = q == 3 ? si : q == 2 ? -sr : sr;
    const double r = q == 1 ? si : q == 3 ? -sr : -si;
    const uint32_t* l = list + g.p[k] * g.npp;
    for (int i0 = 0; i0 < g.npp; i0 += per) {  // a pair's four lanes share a warp
      const int i = i0 + (tid >> 2);
      double out = 0;
      int at = 0;
      if (i < g.npp) {
        const uint32_t pr = l[i];
        const int ci = own ? pr >> 16 : pr & 0xFFFFu, co = own ? pr & 0xFFFFu : pr >> 16;
        at = 2 * ci + (q & 1);
        const double a = xs[at], z0 = xs[2 * co], z1 = xs[2 * co + 1];
        const double b = q == 1 ? z1 : z0, e = q == 1 ? z0 : z1;
        out = fma(c, a, fma(p, b, r * e));
      }
      __syncwarp();
      if (i < g.npp) xs[at] = out;
    }
    __syncthreads();
  }
  if (g.has_x)
    fx::cross_tables(g.masks_other, g.dir, g.norb, g.nchunk, X, v, 1, tab, work, &bad_x, tid, nt,
                     [] { __syncthreads(); });
  for (int e = tid; e < d; e += nt) {
    double2 z = make_double2(1.0, 0.0);
    bool bad = false;
    const uint32_t m = __ldg(g.masks_this + e);
    if (g.has_d) {
      uint64_t turn = 0;
      for (uint32_t b = m; b; b &= b - 1) turn += (uint64_t)g.lin[__ffs(b) - 1];
      sincos((double)(int64_t)turn * 3.4061215800865545e-19, &z.y, &z.x);  // 2 pi / 2^64
    }
    if (g.ea_this) z = cmul<double>(z, __ldg(g.ea_this + e));
    if (g.ea_other) z = cmul<double>(z, __ldg(g.ea_other + v));
    if (g.has_x) {
      longlong2 f = tab[m & 255];
      for (int k = 1; k < g.nchunk; ++k) f = fx::phase_mul(f, tab[k * 256 + ((m >> (8 * k)) & 255)]);
      bad = (m & bad_x) != 0;
      z = cmul<double>(z, fx::phase_to(f));
    }
    vec[e * es] = bad ? fx::nan2() : cmul<double>(z, x[e]);
  }
}

}  // namespace pairs

bool pairs_supported(const Ctx* ctx, const Space* sthis, const Space* sother, int dtype,
                     const RotProgram& rp) {
  if (dtype != FS_C128 || ctx->sweep_engine != FS_SWEEP_AUTO) return false;
  if (sthis->dim < 2 || sthis->dim > 512 || (int)rp.g.size() > pairs::kMaxM || rp.g.empty())
    return false;
  // the diagonal layer is held as angles in integers
  if (sother->dim > 65535 || !rp.finite()) return false;
  // modelled clocks: a rotation is a chain of about 350, or the FP64 issue of
  // its components on four units for the vectors of an SM.  The digit sweep
  // is flat at about 60 us with its images up to a few hundred vectors; the
  // two meet near 36000: N = 10 (5,5) models 39000 and takes 136 us here
  // against 135 both spins, N = 10 (2,5) 19000 and 72 against 106, N = 12
  // (2,3) 23000 and 78.
  const int sms = ctx->prop.multiProcessorCount;
  const int64_t vecs = (sother->dim + sms - 1) / sms;
  const double t = (double)rp.g.size() *
                   std::max<double>(350.0, (sthis->npp + 7) / 8 * 48.0 * (double)vecs);
  return t <= 36000.0;
}

void launch_sweep_pairs(Ctx*, const Space* sa, const Space* sb, int dir, void* vec,
                        const RotProgram& rp, bool diag, const PhaseDev& ph, cudaStream_t st) {
  const Space* sthis = dir == 0 ? sa : sb;
  const Space* sother = dir == 0 ? sb : sa;
  pairs::Args g{};
  g.st = (double2*)vec;
  g.d_b = sb->dim;
  g.dir = dir;
  g.d = (int)sthis->dim;
  g.nvec = (int)sother->dim;
  g.npp = sthis->npp;
  g.m = (int)rp.g.size();
  g.norb = sthis->norb;
  g.nchunk = (sthis->norb + 7) / 8;
  g.has_x = ph.has_x;
  g.list = sthis->pairs;
  g.masks_this = sthis->masks;
  g.masks_other = sother->masks;
  g.ea_this = (const double2*)(dir == 0 ? ph.ea_a : ph.ea_b);
  g.ea_other = (const double2*)(dir == 0 ? ph.ea_b : ph.ea_a);
  g.has_d = diag;
  for (int p = 0; diag && p < g.norb; ++p) g.lin[p] = angle_turns(std::arg(rp.phase[p]));
  for (int k = 0; k < g.m; ++k) {
    g.p[k] = (int8_t)rp.g[k].p;
    g.c[k] = rp.g[k].c;
    g.sr[k] = rp.g[k].s.real();
    g.si[k] = rp.g[k].s.imag();
  }
  const size_t smem = pairs::smem_bytes(g);
  allow_shared_memory(pairs::k_sweep_pairs);
  const int nt = std::min(256, std::max(64, (4 * g.npp + 31) / 32 * 32));
  ProfScope ps(dir == 0 ? "sweep_alpha_pairs" : "sweep_beta_pairs", st);
  pairs::k_sweep_pairs<<<(unsigned)g.nvec, nt, smem, st>>>(g, ph.X);
  FS_CUDA(cudaGetLastError());
}

}  // namespace fs
