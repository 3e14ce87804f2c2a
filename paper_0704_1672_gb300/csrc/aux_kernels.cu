// Kernels around the moment pass:
//   a3  cross-tile reduction of the moment partials in double, fixed order, plus the
//       deferred normalisation F_lm a^l                                  (Eq. (multipole))
//   the contraction's pair items (frame of R0, Euler record) from runs of items
//   the rotation of moment sets (tcm_rotate_moments)
#include <cuda_runtime.h>

#include "contract.h"

namespace tcm {

namespace {

// Degrees l <= kLowLmax of one job from its system's low-degree sums (system pass 2, reduced over
// the system's tiles by its last tile): the Cartesian sums are rotated by the job's rotation R
// (P' = R P, T' = R T R^T, p = R d) and turned into the packed Q_lm, l <= 2, with
//   Q_00 = S,  Q_10 = P'_z,  Q_11 = -(P'_x + i P'_y)/sqrt(2),
//   Q_20 = T'_zz - (T'_xx + T'_yy)/2,  Q_21 = -sqrt(3/2) (T'_xz + i T'_yz),
//   Q_22 = sqrt(3/8) (T'_xx - T'_yy + 2 i T'_xy),
// the regular solid harmonics r^l sqrt(4 pi/(2l+1)) Y_lm of Eq. (multipole) written out in x, y, z.
constexpr int kLowComps = (kLowLmax + 1) * (kLowLmax + 1);
__device__ void low_degrees(const MomJob& job, const double* __restrict__ syspart, double* s_low) {
  if (threadIdx.x < kLowSums) s_low[threadIdx.x] = __ldcg(syspart + (long long)job.low_base * kSysPart + kSysPartLow + threadIdx.x);
  __syncthreads();
  const int k = threadIdx.x;  // packed output slot, one thread each
  if (k >= (job.L + 1) * (job.L + 1) || k >= kLowComps) return;
  const double* R = job.rot;
  const double P[3] = {s_low[1], s_low[2], s_low[3]};
  const double T[3][3] = {{s_low[4], s_low[5], s_low[6]}, {s_low[5], s_low[7], s_low[8]}, {s_low[6], s_low[8], s_low[9]}};
  auto pr = [&](int a) { return R[3 * a] * P[0] + R[3 * a + 1] * P[1] + R[3 * a + 2] * P[2]; };  // (R P)_a
  auto tr = [&](int a, int b) {  // (R T R^T)_ab
    double s = 0.0;
    for (int i = 0; i < 3; ++i) s += R[3 * a + i] * (T[i][0] * R[3 * b] + T[i][1] * R[3 * b + 1] + T[i][2] * R[3 * b + 2]);
    return s;
  };
  const double r2 = 0.70710678118654752440, s32 = 1.22474487139158904910, s38 = 0.61237243569579452455;
  double v;
  switch (k) {
    case 0: v = s_low[0]; break;
    case 1: v = pr(2); break;
    case 2: v = -r2 * pr(0); break;
    case 3: v = -r2 * pr(1); break;
    case 4: v = tr(2, 2) - 0.5 * (tr(0, 0) + tr(1, 1)); break;
    case 5: v = -s32 * tr(0, 2); break;
    case 6: v = -s32 * tr(1, 2); break;
    case 7: v = s38 * (tr(0, 0) - tr(1, 1)); break;
    default: v = s32 * tr(0, 1); break;
  }
  job.out[k] = v;
}

// a3: one CTA per moment job, or gridDim.y CTAs per job with a block of its slots each.  The (chunk,
// slot) entries of the job's partial rows are summed over the job's tiles in double in one order,
// whichever the launch: groups of kSumGroup consecutive tiles in tile order, then the groups in
// order.  F_lm a'^l times the sum goes to the packed component the slot holds; a' is a power of two,
// so a'^l is formed exactly from its exponent.
//
// What bounds it: latency, and for batches of many jobs the read of the partial rows.  A CTA per job
// has each thread walk the tiles of its slot (coalesced rows, a group's loads in flight together).
// A few jobs of many tiles would leave all but a few SMs idle at that (one job of 98 tiles x 800
// slots took 42 us): there kFinSlots slots go to a CTA whose threads take the groups in turn.
constexpr int kFinalizeThreads = 512;
constexpr int kSumGroup = 8;
constexpr int kFinSlots = 64;
constexpr int kFinLanes = kFinalizeThreads / kFinSlots;  // threads per slot of a split launch
constexpr int kFinPass = 4 * kFinLanes;                  // groups summed between two barriers

__device__ __forceinline__ double group_sum(const double* base, int row, int t0, int t1) {
  double s = 0.0;
  if (t1 - t0 == kSumGroup) {
#pragma unroll
    for (int t = 0; t < kSumGroup; ++t) s += __ldcg(base + (long long)(t0 + t) * row);
  } else {
    for (int t = t0; t < t1; ++t) s += __ldcg(base + (long long)t * row);
  }
  return s;
}
__global__ void __launch_bounds__(kFinalizeThreads) k_finalize(const MomJob* __restrict__ jobs,
                                                               const double* __restrict__ partials,
                                                               const SysGeom* __restrict__ geoms,
                                                               const int* __restrict__ imap,
                                                               const double* __restrict__ fmap,
                                                               const int* __restrict__ imap_off,
                                                               const double* __restrict__ syspart) {
  __shared__ double s_low[kLowSums];
  __shared__ double s_grp[kFinPass][kFinSlots];
  pdl_trigger();  // the contraction may be scheduled; it waits for this grid before reading
  pdl_wait();     // the moment kernels' partial rows are complete
  const MomJob& job = jobs[blockIdx.x];
  const int L = job.L;
  const int tpc = job.tiles_per_chunk;
  const int kmax = plan_slots(job.plan, L), row = plan_row(job.plan, L);
  const int* off = imap_off + job.plan * (kLmaxMax + 2);
  const int o = off[L];
  const int nq = off[L + 1] - o;  // nch x kmax
  const double a = geoms[job.geom].a;
  int e = 0;  // a' = scale_radius(a) = 2^e
  if (a > 0.0) frexp(a, &e);
  const bool split = gridDim.y > 1;
  const int per = split ? kFinSlots : kFinalizeThreads;
  const int ngroup = (tpc + kSumGroup - 1) / kSumGroup;
  for (int q0 = split ? blockIdx.y * kFinSlots : 0; q0 < nq; q0 += split ? gridDim.y * kFinSlots : kFinalizeThreads) {
    const int q = q0 + threadIdx.x % per;
    const bool in = q < nq;
    const int p = in ? imap[o + q] : -1;
    const double f = in ? fmap[o + q] : 0.0;
    const int ch = q / kmax, slot = q - ch * kmax;
    const double* base = partials + job.part + (long long)ch * tpc * row + slot;
    double s = 0.0;
    if (!split) {
      if (in)
        for (int g = 0; g < ngroup; ++g) s += group_sum(base, row, g * kSumGroup, min(tpc, (g + 1) * kSumGroup));
    } else {
      const int k = threadIdx.x / kFinSlots;
      for (int g0 = 0; g0 < ngroup; g0 += kFinPass) {
        const int ng = min(kFinPass, ngroup - g0);
        for (int g = k; in && g < ng; g += kFinLanes)
          s_grp[g][threadIdx.x % kFinSlots] =
              group_sum(base, row, (g0 + g) * kSumGroup, min(tpc, (g0 + g + 1) * kSumGroup));
        __syncthreads();
        if (k == 0 && in)
          for (int g = 0; g < ng; ++g) s += s_grp[g][threadIdx.x];
        __syncthreads();
      }
      if (k != 0) continue;
    }
    if (p < 0) continue;
    int l = (int)sqrtf((float)p);
    while (l * l > p) --l;
    while ((l + 1) * (l + 1) <= p) ++l;
    const int ex = e * l;  // a'^l = 2^ex, built from its exponent bits when it is a normal double
    const double al = (ex >= -1022 && ex <= 1023) ? __longlong_as_double((long long)(ex + 1023) << 52) : ldexp(1.0, ex);
    if (job.low_tiles > 0 && p < kLowComps) continue;  // written from the low-degree sums below
    job.out[p] = f * al * s;
  }
  if (blockIdx.y > 0) return;
  if (job.low_tiles > 0) low_degrees(job, syspart, s_low);
}

// Rotation of a moment set, Q'_lm = sum_m' d^l_{m'm}(beta) P_lm', P_lm' = e^{-i m' alpha} Q_lm', without
// forming d^l(beta): two products with the constant matrices D^l = d^l(pi/2) around a diagonal phase
// (the formulas stand at the contraction, contract.cu, which does the same in fixed point).
constexpr int kRotateThreads = 512;  // most threads of a rotation CTA

// ztab (doubles): the rows of D^l = d^l(pi/2), D^l_{km}, 0 <= k, m <= l, at dpi2_off(l) + k dpi2_stride(l)
// + m (contract.h).  The row stride is odd (rows of even length get one zero), so that the lanes of a
// warp reading one entry of consecutive rows hit distinct shared-memory banks; shared memory holds the
// same layout.

__device__ __forceinline__ double flip(double x, int odd) {  // (-1)^odd x without an FP64 op
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)(odd & 1) << 63));
}

// i^n z for any integer n, by exchanging and negating the parts (no FP64 operation).
__device__ __forceinline__ double2 mul_ipow(double2 z, int n) {
  const int r = n & 3;
  const double2 s = (r & 1) ? make_double2(z.y, z.x) : z;
  return make_double2(flip(s.x, r == 1 || r == 2), flip(s.y, r >= 2));
}

// Row product with a parity split: (sum over j = par (mod 2) of row[j] Re x_j, sum over the other
// j of row[j] Im x_j), j = 0..l.  One multiply-add per entry.
__device__ __forceinline__ double2 row_split(const double* row, const double2* x, int l, int par) {
  const double* xs = reinterpret_cast<const double*>(x);
  double a = 0.0, b = 0.0;  // even j, odd j
  int j = 0;
  for (; j + 1 <= l; j += 2) {
    a = fma(row[j], xs[2 * j + par], a);
    b = fma(row[j + 1], xs[2 * j + 3 - par], b);
  }
  if (j == l) a = fma(row[j], xs[2 * j + par], a);
  return par ? make_double2(b, a) : make_double2(a, b);
}

// Copies the rows of D^l for l <= L into shared memory (a constant table: no dependence on the
// kernels before, so it is read ahead of griddepcontrol.wait).
__device__ void load_dpi2(double* Ds, const double* __restrict__ ztab, int L) {
  const double* src = ztab;
  const int n = dpi2_off(L + 1);
  for (int i = threadIdx.x; i < n; i += blockDim.x) Ds[i] = __ldg(src + i);
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// z^lane in every lane of the calling warp (lane <= 31): an inclusive product scan of
// (1, z, z, ...), five steps of one complex multiplication each.
__device__ __forceinline__ double2 warp_pow_scan(double2 z, int lane) {
  double2 r = lane == 0 ? make_double2(1.0, 0.0) : z;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const double2 u = make_double2(__shfl_up_sync(0xffffffffu, r.x, s), __shfl_up_sync(0xffffffffu, r.y, s));
    if (lane >= s) r = cmul(r, u);
  }
  return r;
}
// The phase factors of one rotation R_z(-gamma) R_y(-beta) R_z(-alpha), one warp per table,
// entry m = lane <= L:
//   in:   (-i)^m e^{-i m alpha}, doubled for m >= 1       (from e^{i alpha})
//   beta: e^{i k beta}, doubled for k >= 1                (from cos beta, sin beta)
//   out:  i^m e^{-i m gamma}                              (from e^{i gamma})
__device__ __forceinline__ void in_phases(double2* t, double2 e, int L, int lane) {
  const double2 z = mul_ipow(warp_pow_scan(make_double2(e.x, -e.y), lane), -lane);
  if (lane <= L) t[lane] = lane > 0 ? make_double2(2.0 * z.x, 2.0 * z.y) : z;
}
__device__ __forceinline__ void beta_phases(double2* t, double cb, double sb, int L, int lane) {
  const double2 z = warp_pow_scan(make_double2(cb, sb), lane);
  if (lane <= L) t[lane] = lane > 0 ? make_double2(2.0 * z.x, 2.0 * z.y) : z;
}
__device__ __forceinline__ void out_phases(double2* t, double2 e, int L, int lane) {
  const double2 z = mul_ipow(warp_pow_scan(make_double2(e.x, -e.y), lane), lane);
  if (lane <= L) t[lane] = z;
}

// First product of a rotation, item k = (l, kk) of the triangle: p~_kk from v~ (the moments
// times the input phases) of degree l.
__device__ __forceinline__ double2 rot_first(const double* Ds, const double2* v, const double2* eb, int k) {
  const int l = tri_l(k);
  const int kk = k - l * (l + 1) / 2;
  const double2 p = row_split(Ds + dpi2_off(l) + kk * dpi2_stride(l), v + l * (l + 1) / 2, l, (l + kk) & 1);
  return cmul(eb[kk], p);
}
// Second product, item k = (l, m): S_m times the output phase.
__device__ __forceinline__ double2 rot_second(const double* Ds, const double2* p, const double2* phout, int k) {
  const int l = tri_l(k);
  const int m = k - l * (l + 1) / 2;
  const double2 a = row_split(Ds + dpi2_off(l) + m * dpi2_stride(l), p + l * (l + 1) / 2, l, (l + m) & 1);
  return cmul(phout[m], make_double2(flip(a.x, l), flip(a.y, l + 1)));
}

// Moments of a system rotated by M about its centre, from its lab-frame moments: the Wigner
// rotation R_z(-gamma) R_y(-beta) R_z(-alpha) = M applied degree by degree (one CTA per set),
// by the two products with d^l(pi/2) above.
__global__ void __launch_bounds__(kRotateThreads) k_rotate_moments(const RotDesc* __restrict__ sets,
                                                                     const double* __restrict__ ztab) {
  extern __shared__ double2 sm2[];
  __shared__ EulerZYZ g_e;
  const RotDesc d = sets[blockIdx.x];
  const int L = d.L;
  const int nq = (L + 1) * (L + 2) / 2;
  const int n1 = L + 1;
  double2* q = sm2;
  double2* t = q + nq;
  double2* pha = t + nq;
  double2* ebB = pha + n1;
  double2* phg = ebB + n1;
  double* Ds = reinterpret_cast<double*>(phg + n1);
  load_dpi2(Ds, ztab, L);
  if (threadIdx.x == 0) g_e = euler_zyz(sets[blockIdx.x].M);
  for (int k = threadIdx.x; k < nq; k += blockDim.x) {
    const int l = tri_l(k);
    const int m = k - l * (l + 1) / 2;
    q[k] = m == 0 ? make_double2(d.in[l * l], 0.0) : make_double2(d.in[l * l + 2 * m - 1], d.in[l * l + 2 * m]);
  }
  __syncthreads();
  for (int tt = threadIdx.x >> 5; tt < 3; tt += blockDim.x >> 5) {
    const int lane = threadIdx.x & 31;
    if (tt == 0) in_phases(pha, make_double2(g_e.ea[0], g_e.ea[1]), L, lane);
    else if (tt == 1) beta_phases(ebB, g_e.cb, g_e.sb, L, lane);
    else out_phases(phg, make_double2(g_e.eg[0], g_e.eg[1]), L, lane);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nq; k += blockDim.x) {
    const int l = tri_l(k);
    q[k] = cmul(pha[k - l * (l + 1) / 2], q[k]);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nq; k += blockDim.x) t[k] = rot_first(Ds, q, ebB, k);
  __syncthreads();
  for (int k = threadIdx.x; k < nq; k += blockDim.x) {
    const int l = tri_l(k);
    const int m = k - l * (l + 1) / 2;
    const double2 r = rot_second(Ds, t, phg, k);
    if (m == 0) {
      d.out[l * l] = r.x;
    } else {
      d.out[l * l + 2 * m - 1] = r.x;
      d.out[l * l + 2 * m] = r.y;
    }
  }
}

}  // namespace

// Threads of a rotation CTA: about one per component, at least 64; a few hundred sets at high degree take
// 512, so that the products run in one round.
static int rotate_threads(int L, long long n_sets) {
  const int n = (L + 1) * (L + 1);
  if (n <= 64) return 64;
  if (n <= 128) return 128;
  return (n > 256 && n_sets < 1024) ? kRotateThreads : 256;
}

int rotate_smem_bytes(int L) {
  const int nq = (L + 1) * (L + 2) / 2;
  return (2 * nq + 3 * (L + 1)) * (int)sizeof(double2) + dpi2_off(L + 1) * (int)sizeof(double);
}

// The dynamic shared-memory limit of a kernel: above 48 KB of dynamic plus static shared memory
// a launch needs the raised limit.  These kernels hold at most 8 KB of static shared memory, so
// the limit is set whenever the dynamic part passes 40 KB (on every such launch: the attribute
// is per device, and a call costs far less than the kernels it precedes).
template <typename F>
int raise_smem_limit(F kernel, int dyn) {
  if (dyn <= 40 * 1024) return 0;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) == cudaSuccess ? 0 : -1;
}

int launch_rotate_moments(const RotDesc* sets, int n_sets, int Lmax_sets, const double* ztab, cudaStream_t s) {
  if (n_sets <= 0) return 0;
  const int smem = rotate_smem_bytes(Lmax_sets);
  if (raise_smem_limit(k_rotate_moments, smem) != 0) return -1;
  k_rotate_moments<<<n_sets, rotate_threads(Lmax_sets, n_sets), smem, s>>>(sets, ztab);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

int launch_finalize(const MomJob* jobs, int n_jobs, const double* partials, const SysGeom* geoms, const int* imap,
                    const double* fmap, const int* imap_off, const double* syspart, int n_split, cudaStream_t s) {
  if (n_jobs <= 0) return 0;
  return launch_pdl(k_finalize, dim3(n_jobs, n_split), dim3(kFinalizeThreads), 0, s, jobs, partials, geoms, imap, fmap,
                    imap_off, syspart) == cudaSuccess
             ? 0
             : -1;
}

int finalize_split(int n_jobs, int max_tiles, int max_slots) {
  if (n_jobs > 64 || max_tiles <= 2 * kSumGroup) return 1;  // enough CTAs, or little to sum
  return (max_slots + kFinSlots - 1) / kFinSlots;
}

namespace {
// One thread per item: about 15 double square roots and divisions for a rotated one, which cost the
// host 100 to 150 ns an item (108,360 items of a surface scan: 2.6 ms of planning) and this kernel about
// 20 us for all of them.  A thread finds its item's run by bisection.
__global__ void __launch_bounds__(128) k_frames(const PairRun* __restrict__ runs, int n_runs,
                                                const double* __restrict__ R0, int n_items, int n_computed,
                                                const double* __restrict__ rotB, PairDesc* __restrict__ items,
                                                EulerZYZ* __restrict__ rots) {
  pdl_trigger();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n_items) return;
  int lo = 0, hi = n_runs;  // runs[lo].first <= k < runs[hi].first
  if (n_runs == n_items) {
    lo = k;
  } else {
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (runs[mid].first <= k) lo = mid;
      else hi = mid;
    }
  }
  PairDesc d;
  make_pair(runs[lo], k, R0 + 3LL * k, n_computed, rotB, d, rots);
  items[k] = d;
}
}  // namespace

int launch_frames(const PairRun* runs, int n_runs, const double* R0, int n_items, int n_computed, const double* rotB,
                  PairDesc* items, EulerZYZ* rots, cudaStream_t s) {
  k_frames<<<(n_items + 127) / 128, 128, 0, s>>>(runs, n_runs, R0, n_items, n_computed, rotB, items, rots);
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace tcm
