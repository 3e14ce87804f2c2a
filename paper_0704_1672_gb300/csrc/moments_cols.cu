// Float moment kernel for calls with little work: the lane sums of moments_kernel.cuh, bit for bit (but for
// the degrees l <= 2, which come from the system pass: nothing reads what either kernel leaves there),
// with one column m per warp instead of a chunk of columns.
//
// A warp tile of 64 atoms per lane and a chunk of up to 160 accumulators keeps its warp busy for about
// 25 us (a chain of dependent float instructions, two warps per SMSP at most), whatever else is idle:
// one system of 20,000 atoms at degree 20 is 30 such tiles.  Here a CTA takes four columns of a tile's
// chunk, so that system is 60 CTAs of warps with a third of the work and less:
//   - the four warps set up one row of 32 atoms each (centring, rotation, reciprocal square root) and
//     share the result through shared memory, four rows at a time, double-buffered;
//   - a lane runs the four rows' recurrences side by side (independent chains) and adds them to its
//     accumulators in row order, as the chunk kernel's lane does;
//   - seeds u^m and weights q rho^l are formed by the chunk kernel's own sequence of roundings (the
//     chunk's u^m0 by squaring, then one multiplication per column; q rho^l by l multiplications).
// Per atom and column that costs about twice the chunk kernel's instructions, so it pays as long as
// the chunk kernel would leave most of the GPU idle (moments_use_cols).  Measured, before and now: the
// pass over 20,000 atoms at degree 20 56 and 20 us, over 2 x 200 atoms at degree 10 25 and 8.5 us; a
// call of tcm_moments on the former 102 and 86 us.
#include <cuda_runtime.h>

#include <algorithm>

#include "moments_kernel.cuh"

namespace tcm {

namespace {

constexpr int kColWarps = 4;           // columns per CTA, and rows set up at once
constexpr int kColThreads = 32 * kColWarps;
constexpr int kColSteps = kLmaxMax + 1;

struct ColTables {
  float k[kLmaxMax + 1][kLmaxMax + 1];                        // [m][j]: signed coefficient of step j >= 2
  unsigned char m0[kNumPlans][kLmaxMax + 1][kLmaxMax + 2];    // first column of each chunk (float plans)
  constexpr ColTables() : k(), m0() {
    for (int m = 0; m <= kLmaxMax; ++m)
      for (int j = 2; m + j <= kLmaxMax; ++j)
        k[m][j] = (float)(((j - 1) & 1) ? -kcoef(m + j - 1, m) : kcoef(m + j - 1, m));
    for (int p = 1; p < kNumPlans; ++p)
      for (int L = 0; L <= kLmaxMax; ++L) {
        const int n = plan_nch(L, plan_kmax(p));
        for (int c = 0; c <= n; ++c) m0[p][L][c] = (unsigned char)plan_m0(L, plan_kmax(p), n, c);
      }
  }
};
__constant__ ColTables c_cols = ColTables();

// u^E of every row by the squarings of upow (moments_kernel.cuh), E >= 1 at run time.
__device__ __forceinline__ void upow_rows(int E, const float* ux, const float* uy, float* pr, float* pi) {
#pragma unroll
  for (int r = 0; r < kColWarps; ++r) {
    pr[r] = ux[r];
    pi[r] = uy[r];
  }
  for (int b = 30 - __clz(E); b >= 0; --b) {
#pragma unroll
    for (int r = 0; r < kColWarps; ++r) {
      const float hr = pr[r], hi = pi[r];
      pr[r] = __fmaf_rn(hr, hr, -(hi * hi));
      pi[r] = 2.0f * hr * hi;
    }
    if ((E >> b) & 1)
#pragma unroll
      for (int r = 0; r < kColWarps; ++r) {
        const float sr = pr[r], si = pi[r];
        pr[r] = __fmaf_rn(sr, ux[r], -(si * uy[r]));
        pi[r] = __fmaf_rn(sr, uy[r], si * ux[r]);
      }
  }
}

__global__ void __launch_bounds__(kColThreads)
    k_moments_cols(const MomJob* __restrict__ jobs, const MomTile* __restrict__ tiles,
                   const SysGeom* __restrict__ geoms, double* __restrict__ partials) {
  constexpr int S = MomTraits<float>::stride;
  __shared__ Xform<float> xf;
  __shared__ float4 s_u[2][kColWarps][32];  // u_x, u_y, c, rho
  __shared__ float s_q[2][kColWarps][32];
  __shared__ __align__(16) float s_row[kColWarps][2 * kColSteps * S];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  pdl_wait();  // the centres and radii of the launch before are complete
  const MomTile tile = tiles[blockIdx.x];
  const MomJob& job = jobs[tile.job];
  const int L = job.L;
  const int m0 = c_cols.m0[job.plan][L][tile.chunk], m1 = c_cols.m0[job.plan][L][tile.chunk + 1];
  const int mb = m0 + blockIdx.y * kColWarps;
  if (mb >= m1) return;
  const int m = mb + w;
  const bool active = m < m1;
  const int n = L - m;
  const SysGeom& g = geoms[job.geom];
  if (w == 0) make_xform<float>(job, g, lane, &xf);
  const double cd[3] = {g.c[0], g.c[1], g.c[2]};
  const long long i0 = (long long)tile.t * job.atoms_per_tile;
  const long long i1 = min(job.n, i0 + (long long)job.atoms_per_tile);
  const int rows = (int)((i1 - i0 + 31) / 32);
  const bool f32 = job.dtype == TCM_F32;
  auto load = [&](int r, float4& v, Rec64& v64) {
    const long long i = i0 + 32LL * r + lane;
    const bool in = i < i1;
    if (f32) {
      v = in ? load_rec(reinterpret_cast<const float4*>(job.xyzq), i) : make_float4(g.chi[0], g.chi[1], g.chi[2], 0.0f);
    } else {
      v64 = in ? load_rec(reinterpret_cast<const Rec64*>(job.xyzq), i)
               : Rec64{make_double2(cd[0], cd[1]), make_double2(cd[2], 0.0)};
    }
  };
  float4 v;
  Rec64 v64;
  load(w, v, v64);
  __syncthreads();
  float ar[kColSteps], ai[kColSteps], kc[kColSteps];
#pragma unroll
  for (int j = 0; j < kColSteps; ++j) {
    ar[j] = ai[j] = 0.0f;
    kc[j] = active ? c_cols.k[m][j] : 0.0f;
  }
  for (int r0 = 0; r0 < rows; r0 += kColWarps) {
    const int buf = (r0 / kColWarps) & 1;
    {
      float d0, d1, d2, q, ux, uy, cz, rho;
      if (f32)
        centre<float>(v, xf, cd, d0, d1, d2, q);
      else
        centre<float>(v64, xf, cd, d0, d1, d2, q);
      setup<float>(d0, d1, d2, xf, ux, uy, cz, rho);
      s_u[buf][w][lane] = make_float4(ux, uy, cz, rho);
      s_q[buf][w][lane] = q;
    }
    if (r0 + kColWarps < rows) load(r0 + kColWarps + w, v, v64);
    __syncthreads();
    if (!active) continue;
    float c[kColWarps], rho[kColWarps], wt[kColWarps], gr[kColWarps], gi[kColWarps], pr[kColWarps], pi[kColWarps];
    float ux[kColWarps], uy[kColWarps];
#pragma unroll
    for (int r = 0; r < kColWarps; ++r) {
      const float4 u = s_u[buf][r][lane];
      ux[r] = u.x;
      uy[r] = u.y;
      c[r] = u.z;
      rho[r] = u.w;
      wt[r] = s_q[buf][r][lane];
      gr[r] = 1.0f;
      gi[r] = 0.0f;
    }
    if (m0 > 0) upow_rows(m0, ux, uy, gr, gi);
    for (int k = m0; k < m; ++k)
#pragma unroll
      for (int r = 0; r < kColWarps; ++r) {
        const float nr = __fmaf_rn(gr[r], ux[r], -(gi[r] * uy[r])), ni = __fmaf_rn(gr[r], uy[r], gi[r] * ux[r]);
        gr[r] = nr;
        gi[r] = ni;
      }
    for (int k = 0; k < m; ++k)
#pragma unroll
      for (int r = 0; r < kColWarps; ++r) wt[r] *= rho[r];
#pragma unroll
    for (int j = 0; j < kColSteps; ++j) {
      if (j > n) break;
#pragma unroll
      for (int r = 0; r < kColWarps; ++r) {
        if (j == 1) {
          pr[r] = gr[r];
          pi[r] = gi[r];
          gr[r] *= c[r];
          gi[r] *= c[r];
        } else if (j > 1) {
          const float t = c[r] * kc[j];
          const float nr = __fmaf_rn(t, gr[r], pr[r]), ni = __fmaf_rn(t, gi[r], pi[r]);
          pr[r] = gr[r];
          pi[r] = gi[r];
          gr[r] = nr;
          gi[r] = ni;
        }
        ar[j] = __fmaf_rn(wt[r], gr[r], ar[j]);
        ai[j] = __fmaf_rn(wt[r], gi[r], ai[j]);
        wt[r] *= rho[r];
      }
    }
  }
  if (!active) return;
  // the 32 lanes of each component, in the chunk kernel's order of summation
  float* wb = s_row[w];
#pragma unroll
  for (int j = 0; j < kColSteps; ++j) {
    if (j > n) break;
    wb[2 * j * S + lane] = ar[j];
    wb[(2 * j + 1) * S + lane] = ai[j];
  }
  __syncwarp();
  double* out = partials + (long long)tile.id * MomTraits<float>::row;
  for (int r = lane; r < 2 * (n + 1); r += 32) {
    const int l = m + (r >> 1), part = r & 1;
    if (m > 0 || part == 0) out[acc_slot(L, m0, m1, l, m, part)] = row_sum32(wb + r * S);
  }
}

}  // namespace

// The column kernel's warps finish a tile sooner at twice the instructions: taken while the chunk kernel
// would have no more than one warp per SM.  Moment pass of one system of 10, 30, 60, 100, 130 and 152 tiles, by
// columns and by chunks: 20, 20, 22, 24, 28, 27 and 36 us throughout at degree 20; 16, 16, 18, 18, 22, 22 and 22 to
// 24 at degree 8; 16 to 18 and 18 to 20 at degree 4; 22 to 28 and 34 at degree 24; a scan of 129 tiles at degree 8
// 18 and 22, of 102 at degree 16 24 and 32: no slower anywhere up to the line.
bool moments_use_cols(int n_tiles, int num_sms) { return n_tiles <= num_sms; }

// Largest number of columns in a chunk of degree L.
int moments_max_cols(int plan, int L) {
  int mx = 0;
  for (int c = 0; c < moments_nchunks(plan, L); ++c)
    mx = std::max(mx, moments_chunk_m0(plan, L, c + 1) - moments_chunk_m0(plan, L, c));
  return mx;
}

int launch_moments_cols(const MomJob* jobs, const MomTile* tiles, int n_tiles, int max_cols, const SysGeom* geoms,
                        double* partials, cudaStream_t s) {
  if (n_tiles <= 0) return 0;
  return launch_pdl(k_moments_cols, dim3(n_tiles, (max_cols + kColWarps - 1) / kColWarps), dim3(kColThreads), 0, s, jobs,
                    tiles, geoms, partials) == cudaSuccess
             ? 0
             : -1;
}

}  // namespace tcm
