// Moment kernel of the double path, Eq. (multipole) (formulation: tcm_internal.h).
//
// What bounds it: the FP64 pipe, 2 lanes per clock and SM (one warp instruction holds its SMSP's
// pipe for 64 cycles, as long as 64 float instructions).  Nothing else is scarce: there is time for
// shared-memory accumulators, runtime loops over degree and order and warps that specialise, so the
// kernel is arranged to issue as few FP64 instructions as it can and one code serves every degree:
//   - an atom's set-up (centring, rotation, reciprocal square root: about 30 instructions) and its
//     tables u^m, q rho^l (5 per degree) are made once per atom, by three producer warps, and
//     handed to the consumers through a ring of three rows of 32 atoms in shared memory;
//   - the columns m of one row run on consumer warps, columns p and L - p on warp p (L + 2 steps of
//     5 instructions for every warp), each lane one atom; the accumulators of a component stay in
//     shared memory, 32 lanes wide, owned by one warp;
//   - at the end of a tile every thread adds the 32 lanes of a component.
// Column chunks of 80 accumulators in registers, the form before, repeated the set-up in each of up
// to 10 chunks and left a small system to one warp per chunk and 1,024 atoms.  Calls of tcm_moments,
// before and now: 100,003 atoms at degree 24 635 and 320 us (the FP64 instructions it cannot do
// without take 252); 3,260 and 2,587 atoms at degree 10, with their energy, 554 and 170 us; 257 sets
// of 20,000 atoms at degree 20 14.5 and 13.1 ms.
//
// Row j of a tile uses ring slot j mod 3 and producer j mod 3.  Named barriers 1 + slot (row full)
// and 4 + slot (row empty) pair one producer warp with the P consumer warps of a group; with few
// columns (P <= 4) three groups of consumers take the rows in turn, each with its own accumulators.
#include <cuda_runtime.h>

#include "tcm_internal.h"

namespace tcm {

namespace {

constexpr int kRing = 3;
constexpr int kRowAtoms = 32;

// Signed recurrence coefficient of step j >= 2 along column m: H_j = k c H_{j-1} + H_{j-2}.
struct K64 {
  double k[kLmaxMax + 1][kLmaxMax + 1];
  constexpr K64() : k() {
    for (int m = 0; m <= kLmaxMax; ++m)
      for (int j = 2; m + j <= kLmaxMax; ++j) k[m][j] = ((j - 1) & 1) ? -kcoef(m + j - 1, m) : kcoef(m + j - 1, m);
  }
};
__constant__ K64 c_k64 = K64();

__host__ __device__ constexpr int f64_pairs(int L) { return L / 2 + 1; }
__host__ __device__ constexpr int f64_groups(int L) { return f64_pairs(L) <= 4 ? kRing : 1; }
__host__ __device__ constexpr int f64_threads(int L) { return 32 * (f64_pairs(L) * f64_groups(L) + kRing); }
__host__ __device__ constexpr int f64_slot_doubles(int L) { return kRowAtoms * (3 * (L + 1) + 1); }
__host__ __device__ constexpr int f64_smem(int L) {
  return 8 * (f64_groups(L) * (L + 1) * (L + 1) * kRowAtoms + kRing * f64_slot_doubles(L));
}
static_assert(f64_smem(kLmaxMax) <= 227 * 1024, "the accumulators and the ring must fit one SM");
static_assert(f64_threads(kLmaxMax) <= 512, "launch bounds");

__device__ __forceinline__ void bar_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int n) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// The per-tile transform: centring and rot / a'.
struct X64 {
  double c[3], M[9];
};
__device__ __forceinline__ double inv_scale(double a) {  // 1 / scale_radius(a), a power of two
  int e = 0;
  if (a > 0.0) frexp(a, &e);
  return ldexp(1.0, -e);
}

// One atom's set-up and tables; lane stride 1 in every array.
__device__ __forceinline__ void produce(const MomJob& job, const X64& xf, long long i, bool in, double2* u, double* W,
                                        double* cs, int L, int lane) {
  double x[3] = {xf.c[0], xf.c[1], xf.c[2]}, q = 0.0;  // a padding atom: the centre, no charge
  if (in) {
    if (job.dtype == TCM_F32) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(job.xyzq) + i);
      x[0] = v.x;
      x[1] = v.y;
      x[2] = v.z;
      q = v.w;
    } else {
      const double2 a = __ldg(reinterpret_cast<const double2*>(job.xyzq) + 2 * i);
      const double2 b = __ldg(reinterpret_cast<const double2*>(job.xyzq) + 2 * i + 1);
      x[0] = a.x;
      x[1] = a.y;
      x[2] = b.x;
      q = b.y;
    }
  }
  const double d0 = x[0] - xf.c[0], d1 = x[1] - xf.c[1], d2 = x[2] - xf.c[2];
  const double px = fma(xf.M[0], d0, fma(xf.M[1], d1, xf.M[2] * d2));
  const double py = fma(xf.M[3], d0, fma(xf.M[4], d1, xf.M[5] * d2));
  const double pz = fma(xf.M[6], d0, fma(xf.M[7], d1, xf.M[8] * d2));
  const double r2 = fma(px, px, fma(py, py, pz * pz));
  const double rinv = r2 > 0.0 ? rsqrt(r2) : 0.0;
  const double ux = px * rinv, uy = py * rinv, rho = r2 * rinv;
  cs[lane] = pz * rinv;
  double pr = 1.0, pi = 0.0;
  for (int m = 0;; ++m) {
    u[m * kRowAtoms + lane] = make_double2(pr, pi);
    W[m * kRowAtoms + lane] = q;
    if (m == L) break;
    const double nr = pr * ux - pi * uy;
    pi = pr * uy + pi * ux;
    pr = nr;
    q *= rho;
  }
}

__device__ __forceinline__ void add(double* a, double w, double g) { *a = fma(w, g, *a); }

// Column m of one row: the recurrence along l and the sums of q rho^l H.
__device__ __forceinline__ void column(const double2* u, const double* W, double c, double* acc, int L, int m, int lane) {
  const double* k = c_k64.k[m];
  const int n = L - m;
  W += m * kRowAtoms + lane;
  if (m == 0) {  // real
    double* a = acc + lane;
    double g = c, p = 1.0;
    a[0] += W[0];
    if (n >= 1) add(a + kRowAtoms, W[kRowAtoms], g);
    for (int j = 2; j <= n; ++j) {
      const double t = fma(k[j] * c, g, p);
      p = g;
      g = t;
      add(a + j * kRowAtoms, W[j * kRowAtoms], g);
    }
    return;
  }
  // slots of column m: after the L + 1 reals and the complex columns 1 .. m - 1
  double* a = acc + ((L + 1) + (m - 1) * (2 * L + 2 - m)) * kRowAtoms + lane;
  double2 g = u[m * kRowAtoms + lane], p = g;
  add(a, W[0], g.x);
  add(a + kRowAtoms, W[0], g.y);
  if (n == 0) return;
  g = make_double2(c * g.x, c * g.y);
  add(a + 2 * kRowAtoms, W[kRowAtoms], g.x);
  add(a + 3 * kRowAtoms, W[kRowAtoms], g.y);
#pragma unroll 2
  for (int j = 2; j <= n; ++j) {
    const double t = k[j] * c;
    const double2 h = make_double2(fma(t, g.x, p.x), fma(t, g.y, p.y));
    p = g;
    g = h;
    const double w = W[j * kRowAtoms];
    add(a + (2 * j) * kRowAtoms, w, g.x);
    add(a + (2 * j + 1) * kRowAtoms, w, g.y);
  }
}

// Persistent CTAs over tiles of one degree; counter[0] is the work counter and counter[32] the exit
// ticket, both zero on entry and left zero.
__global__ void __launch_bounds__(512, 2)
    k_moments_f64(const MomJob* __restrict__ jobs, const MomTile* __restrict__ tiles, int n_tiles,
                  int* __restrict__ counter, const SysGeom* __restrict__ geoms, double* __restrict__ partials, int L) {
  extern __shared__ __align__(16) double sm64[];
  __shared__ X64 xf;
  __shared__ int s_tile[2];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int P = f64_pairs(L), ng = f64_groups(L), ncomp = (L + 1) * (L + 1);
  double* acc = sm64;
  double* ring = acc + ng * ncomp * kRowAtoms;
  const int slot_doubles = f64_slot_doubles(L);
  const int bar_n = 32 * (P + 1);
  for (int k = threadIdx.x; k < ng * ncomp * kRowAtoms; k += blockDim.x) acc[k] = 0.0;
  pdl_wait();  // the centres and radii of the launch before are complete
  if (threadIdx.x == 0) s_tile[0] = atomicAdd(counter, 1);
  __syncthreads();
  for (int it = 0;; ++it) {
    const int ti = s_tile[it & 1];
    if (ti >= n_tiles) break;
    const MomTile tile = tiles[ti];
    const MomJob& job = jobs[tile.job];
    if (threadIdx.x == 0) s_tile[(it + 1) & 1] = atomicAdd(counter, 1);
    if (threadIdx.x < 9) xf.M[threadIdx.x] = job.rot[threadIdx.x] * inv_scale(geoms[job.geom].a);
    if (threadIdx.x < 3) xf.c[threadIdx.x] = geoms[job.geom].c[threadIdx.x];
    const long long i0 = (long long)tile.t * job.atoms_per_tile;
    const long long i1 = min(job.n, i0 + (long long)job.atoms_per_tile);
    const int nrows = (int)((i1 - i0 + kRowAtoms - 1) / kRowAtoms);
    __syncthreads();
    if (w >= P * ng) {  // producer
      const int s = w - P * ng;
      double2* u = reinterpret_cast<double2*>(ring + s * slot_doubles);
      double* W = reinterpret_cast<double*>(u + (L + 1) * kRowAtoms);
      double* cs = W + (L + 1) * kRowAtoms;
      for (int j = s; j < nrows; j += kRing) {
        const long long i = i0 + (long long)j * kRowAtoms + lane;
        if (j >= kRing) bar_sync(4 + s, bar_n);  // row j - 3 has been used
        produce(job, xf, i, i < i1, u, W, cs, L, lane);
        bar_arrive(1 + s, bar_n);
      }
    } else {
      const int p = w % P, gr = w / P;
      double* a = acc + gr * ncomp * kRowAtoms;
      for (int j = gr; j < nrows; j += ng) {
        const int s = j % kRing;
        const double2* u = reinterpret_cast<const double2*>(ring + s * slot_doubles);
        const double* W = reinterpret_cast<const double*>(u + (L + 1) * kRowAtoms);
        bar_sync(1 + s, bar_n);
        const double c = W[(L + 1) * kRowAtoms + lane];
        column(u, W, c, a, L, p, lane);
        if (L - p != p) column(u, W, c, a, L, L - p, lane);
        if (j + kRing < nrows) bar_arrive(4 + s, bar_n);
      }
    }
    __syncthreads();
    double* row = partials + job.part + (long long)tile.t * ncomp;
    for (int k = threadIdx.x; k < ncomp; k += blockDim.x) {
      double v = 0.0;
      for (int gr = 0; gr < ng; ++gr) {
        double* a = acc + (gr * ncomp + k) * kRowAtoms;
#pragma unroll 8
        for (int i = 0; i < kRowAtoms; ++i) {  // neighbouring threads start at neighbouring banks
          double* e = a + ((i + k) & 31);
          v += *e;
          *e = 0.0;
        }
      }
      row[k] = v;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && atomicAdd(counter + 32, 1) == (int)gridDim.x - 1) {
    atomicExch(counter, 0);
    atomicExch(counter + 32, 0);
  }
}

}  // namespace

int launch_moments_f64(int L, const MomJob* jobs, const MomTile* tiles, int n_tiles, int* counter, const SysGeom* geoms,
                       double* partials, int grid, cudaStream_t s) {
  // the limit of every degree: it does not change under a captured launch
  if (cudaFuncSetAttribute(k_moments_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, f64_smem(kLmaxMax)) != cudaSuccess)
    return -1;
  return launch_pdl(k_moments_f64, dim3(grid), dim3(f64_threads(L)), f64_smem(L), s, jobs, tiles, n_tiles, counter, geoms,
                    partials, L) == cudaSuccess
             ? 0
             : -1;
}

}  // namespace tcm
