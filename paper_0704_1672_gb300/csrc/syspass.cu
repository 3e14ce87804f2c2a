// The pass over each system's atoms before the moment pass (step a1 and the mixed path's
// low-degree sums):
//   - the centroid, for systems without a given centre (Section II: the centres may be any point; the
//     centroid of the positions by default);
//   - the radius a = max |x - c| (exact in double) and, for the mixed path, the low-degree sums
//     S = sum q, P_k = sum q d_k, T_kl = sum q d_k d_l (d = x - c) from which k_finalize forms
//     Q_lm, l <= 2, of every moment job of the system (Eq. (multipole) in Cartesian form).
//
// Which kernel a system takes depends on its own atom count only, so its results do not depend on
// the batch it is in:
//   up to 8,192 atoms     one CTA per system (k_sys_one<1>), centroid and second pass in one kernel
//                         (double records, whose FP64 instructions one SM issues at 2 lanes per clock:
//                         up to 1,024);
//   up to 65,536 atoms    one cluster of 8 CTAs per system (k_sys_one<8>), which exchange their sums
//                         through distributed shared memory;
//   above                 warp tiles of 1,024 atoms, all systems' tiles in one launch per pass
//                         (k_sys_centroid, k_sys_radius_low); the last tile of a system to finish (a
//                         ticket) reduces its tile rows in tile order.
// What bounds it: for small calls the chain of dependent steps: a tile list, and a launch, a ticket and
// a last tile per pass, took 28 us for one system of 20,000 atoms and 27 for two of 200; one kernel takes
// 17 and 13.  For batches the instructions, 141 float operations an atom for the float-float sums (two to a
// packed f32x2 instruction), and the reads of the coordinates: 2,048 uneven systems took 423 us with single
// instructions, 397 packed, 348 with 32-bit indices, full batches without predicates and the radius's
// candidates kept from the one scan instead of found by another.  The limits: at 2,048 atoms for one CTA
// the batch paid for clusters with an atom or two per thread (462 us before; at 4,096 419 against 406);
// double records of 3,260 atoms take 21 us on one CTA, 15 on a cluster.
//
// Per-atom arithmetic is float for float records: error-free two-sums for the centroid, float-float
// (two-sum and fma-based two-product) for the low-degree sums, and a float filter for the radius: each
// thread keeps its farthest atom, and only those within a relative 4e-6 of the float maximum are
// recomputed in double (if a thread's second farthest is as near, the atoms are scanned again).  Every
// reduction runs in a fixed order.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "tcm_internal.h"

namespace tcm {

namespace {

struct FF {  // unevaluated sum h + l of two floats
  float h, l;
};

// s + e += x: Knuth's two-sum of s and x.h; its rounding error, x.l and the running error go to e.
__device__ __forceinline__ void ff_acc(float& s, float& e, FF x) {
  const float t = s + x.h;
  const float bb = t - s;
  e += ((s - (t - bb)) + (x.h - bb)) + x.l;
  s = t;
}

// Product of two FF values to about 2^-46 relative: the exact product of the high parts (fma
// error term) plus the two cross terms.
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = a.h * b.h;
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return FF{p, e};
}

// x - (hi + lo) as an FF pair: exact two-sum of x and -hi, then -lo into the error term.
__device__ __forceinline__ FF ff_sub_split(float x, float hi, float lo) {
  const float s = x - hi;
  const float bb = s - x;
  const float e = (x - (s - bb)) + (-hi - bb);
  return FF{s, e - lo};
}

// The same operations on two independent values at once, packed f32x2 instructions with the roundings of
// the single ones (a - b as b (-1) + a, rounded once).
struct FF2 {
  float2 h, l;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ void ff_acc2(float2& s, float2& e, FF2 x) {
  const float2 t = __fadd2_rn(s, x.h);
  const float2 bb = sub2(t, s);
  e = __fadd2_rn(e, __fadd2_rn(__fadd2_rn(sub2(s, sub2(t, bb)), sub2(x.h, bb)), x.l));
  s = t;
}
__device__ __forceinline__ FF2 ff_mul2(FF2 a, FF2 b) {
  const float2 p = __fmul2_rn(a.h, b.h);
  float2 e = __ffma2_rn(a.h, b.h, make_float2(-p.x, -p.y));
  e = __ffma2_rn(a.h, b.l, e);
  e = __ffma2_rn(a.l, b.h, e);
  return FF2{p, e};
}
__device__ __forceinline__ FF2 ff_sub_split2(float2 x, float2 hi, float2 lo) {
  const float2 s = sub2(x, hi);
  const float2 bb = sub2(s, x);
  const float2 e = __fadd2_rn(sub2(x, sub2(s, bb)), sub2(make_float2(-hi.x, -hi.y), bb));
  return FF2{s, sub2(e, lo)};
}

// |x - c|^2 in plain float, d_k = (x_k - c_hi,k) - c_lo,k: each difference within 2^-23 of its
// value, the square within about 7 x 2^-24 (4.2e-7), far inside the radius filter's margin of 4e-6:
// the atom of the exact maximum is always among the candidates.
__device__ __forceinline__ float r2_plain(const float4& v, const float* chi, const float* clo) {
  const float x = (v.x - chi[0]) - clo[0], y = (v.y - chi[1]) - clo[1], z = (v.z - chi[2]) - clo[2];
  return __fmaf_rn(x, x, __fmaf_rn(y, y, z * z));
}

// Product of a float q (exact) and an FF value: the exact product of the high parts plus q times
// the low part.
__device__ __forceinline__ FF ff_mul_f(float q, FF b) {
  const float p = q * b.h;
  float e = __fmaf_rn(q, b.h, -p);
  e = __fmaf_rn(q, b.l, e);
  return FF{p, e};
}

__device__ __forceinline__ void ff_warp_sum(float& s, float& e) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
    const float e2 = __shfl_xor_sync(0xffffffffu, e, o);
    ff_acc(s, e, FF{s2, e2});
  }
}

// Reduce-scatter of N float-float sums over the 32 lanes of a warp: at each level (lane offset
// O = 16, 8, ..., 1) a lane keeps the first ceil(n/2) of its n sums if its O bit is clear, the
// rest (padded with zeros) if it is set, and adds in its partner's values of the sums it keeps,
// so each level moves half the values of the previous one (one butterfly per sum would move all
// of them at every level).  A fixed pattern: the same inputs give the same sums in every run.
// For N = 10, lane l ends with the whole of sum 5 b4 + 3 b3 + 2 b2 + b1 in (s[0], e[0]), where
// b_i is bit i of l, if bit l of kRs10Lanes is set (ten lanes; the others hold zeros).
constexpr unsigned kRs10Lanes = 0x05150515u;
template <int N, int O>
__device__ __forceinline__ void ff_reduce_scatter(float* s, float* e, int lane) {
  if constexpr (O > 0) {
    constexpr int K = (N + 1) / 2;
    const bool hi = (lane & O) != 0;
    float ns[K], ne[K];
#pragma unroll
    for (int j = 0; j < K; ++j) {
      const float gs = K + j < N ? s[K + j] : 0.f, ge = K + j < N ? e[K + j] : 0.f;
      const float send_s = hi ? s[j] : gs, send_e = hi ? e[j] : ge;
      float a = hi ? gs : s[j], b = hi ? ge : e[j];
      const float rs = __shfl_xor_sync(0xffffffffu, send_s, O), re = __shfl_xor_sync(0xffffffffu, send_e, O);
      ff_acc(a, b, FF{rs, re});
      ns[j] = a;
      ne[j] = b;
    }
#pragma unroll
    for (int j = 0; j < K; ++j) {
      s[j] = ns[j];
      e[j] = ne[j];
    }
    ff_reduce_scatter<K, O / 2>(s, e, lane);
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Warp maximum of non-negative doubles through their bit patterns (they order like the integers),
// so that the comparisons stay off the FP64 pipe.
__device__ __forceinline__ double warp_max_d(double v) {
  long long b = __double_as_longlong(v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
  return __longlong_as_double(b);
}

// Float-float sums of N consecutive (hi, lo) pairs over n tile rows (stride in floats, p and the
// stride 16-byte aligned): lane l adds rows l, l + 32, ... (all N pairs of a row loaded
// together), then the lanes' pairs are added in a fixed tree, so the same rows give the same
// results in every run.  Float instructions only.  Rows are read through L2 (written by other
// CTAs).  With kR2, also the maximum of the double at float offset r2_off of each row.
template <int N, bool kR2>
__device__ __forceinline__ void ordered_ff_sums(const float* p, int n, int stride, int lane, double* out,
                                                int r2_off = 0, double* r2max = nullptr) {
  float s[N], e[N];
#pragma unroll
  for (int k = 0; k < N; ++k) s[k] = e[k] = 0.f;
  long long b2 = 0;
  for (int r = lane; r < n; r += 32) {
    const float* row = p + (long long)r * stride;
    float4 v[N / 2];
    float2 v1 = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) v[k] = __ldcg(reinterpret_cast<const float4*>(row) + k);
    if (N % 2) v1 = __ldcg(reinterpret_cast<const float2*>(row) + N - 1);
    if (kR2) b2 = max(b2, __ldcg(reinterpret_cast<const long long*>(row + r2_off)));
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      ff_acc(s[2 * k], e[2 * k], FF{v[k].x, v[k].y});
      ff_acc(s[2 * k + 1], e[2 * k + 1], FF{v[k].z, v[k].w});
    }
    if (N % 2) ff_acc(s[N - 1], e[N - 1], FF{v1.x, v1.y});
  }
#pragma unroll
  for (int k = 0; k < N; ++k) {
    ff_warp_sum(s[k], e[k]);
    out[k] = (double)s[k] + (double)e[k];
  }
  if (kR2) {  // non-negative doubles order like their bit patterns
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) b2 = max(b2, __shfl_xor_sync(0xffffffffu, b2, o));
    *r2max = __longlong_as_double(b2);
  }
}

// Tile rows hold their sums as (hi, lo) float pairs: no per-tile double arithmetic, which on GB300
// runs at 1/64 of the float rate.  Float offsets within a row:
constexpr int kRowFloats = 2 * kSysPart;
constexpr int kRowCen = 0;                 // centroid sums, 3 pairs
constexpr int kRowLow = 2 * kSysPartLow;   // low-degree sums, kLowSums pairs

constexpr int kSysWarps = kSysThreads / 32;

// Last tile of a job to finish (after its partial rows are written and fenced): lane 0 takes the
// ticket; the result is broadcast to the warp.  The last one resets the ticket for the next use.
__device__ __forceinline__ bool last_tile(int* ticket, int n_tiles, int lane) {
  __threadfence();  // every lane's partial-row writes, before the ticket
  __syncwarp();
  int last = 0;
  if (lane == 0) {
    last = atomicAdd(ticket, 1) == n_tiles - 1;
    if (last) *ticket = 0;
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last) __threadfence();
  return last;
}

// Atoms per lane whose loads are issued together before any of their arithmetic (the per-atom
// work is short, so a lane must keep several loads in flight to cover the memory latency).
constexpr int kSysBatch = 4;  // centroid
constexpr int kLowBatch = 2;  // radius and low-degree sums: more arithmetic per load, more registers

__device__ __forceinline__ FF2 q_times2(FF q, FF2 d) { return ff_mul2(FF2{make_float2(q.h, q.h), make_float2(q.l, q.l)}, d); }
__device__ __forceinline__ FF q_times(FF q, FF d) { return ff_mul(q, d); }
__device__ __forceinline__ FF2 q_times2(float q, FF2 d) {
  const float2 q2 = make_float2(q, q), p = __fmul2_rn(q2, d.h);
  return FF2{p, __ffma2_rn(q2, d.l, __ffma2_rn(q2, d.h, make_float2(-p.x, -p.y)))};
}
__device__ __forceinline__ FF q_times(float q, FF d) { return ff_mul_f(q, d); }
__device__ __forceinline__ FF as_ff(FF q) { return q; }
__device__ __forceinline__ FF as_ff(float q) { return FF{q, 0.f}; }

// The ten low-degree sums of a lane, two to a packed accumulator: (S, P_z), (P_x, P_y), (T_xx, T_yy),
// (T_xz, T_yz), (T_xy, T_zz).  Packed, an atom takes about 90 issue slots instead of 141.
struct LowAcc {
  float2 s[5], e[5];
  __device__ __forceinline__ LowAcc() {
#pragma unroll
    for (int k = 0; k < 5; ++k) s[k] = e[k] = make_float2(0.f, 0.f);
  }
  // q is a float (float records: the charge is exact) or an FF pair (double records).
  template <typename Q>
  __device__ __forceinline__ void add(Q q, FF2 d01, FF d2) {
    const FF2 qd01 = q_times2(q, d01);
    const FF qd2 = q_times(q, d2), qq = as_ff(q);
    ff_acc2(s[0], e[0], FF2{make_float2(qq.h, qd2.h), make_float2(qq.l, qd2.l)});
    ff_acc2(s[1], e[1], qd01);
    ff_acc2(s[2], e[2], ff_mul2(qd01, d01));
    ff_acc2(s[3], e[3], ff_mul2(qd01, FF2{make_float2(d2.h, d2.h), make_float2(d2.l, d2.l)}));
    ff_acc2(s[4], e[4], ff_mul2(FF2{make_float2(qd01.h.x, qd2.h), make_float2(qd01.l.x, qd2.l)},
                                FF2{make_float2(d01.h.y, d2.h), make_float2(d01.l.y, d2.l)}));
  }
  // in the order S, P_x, P_y, P_z, T_xx, T_xy, T_xz, T_yy, T_yz, T_zz
  __device__ __forceinline__ void get(float* so, float* eo) const {
    auto put = [&](const float2* v, float* o) {
      o[0] = v[0].x; o[1] = v[1].x; o[2] = v[1].y; o[3] = v[0].y; o[4] = v[2].x;
      o[5] = v[4].x; o[6] = v[3].x; o[7] = v[2].y; o[8] = v[3].y; o[9] = v[4].y;
    };
    put(s, so);
    put(e, eo);
  }
};

// Float-float sums of the positions of atoms i, i + step, ... < n (float records).
__device__ __forceinline__ void sum_f32(const float4* X, int n, int i, int step, float2& s2, float2& e2, float& sz, float& ez) {
  auto one = [&](const float4& v) {
    ff_acc2(s2, e2, FF2{make_float2(v.x, v.y), make_float2(0.f, 0.f)});
    ff_acc(sz, ez, FF{v.z, 0.f});
  };
  for (; i + (kSysBatch - 1) * step < n; i += kSysBatch * step) {
    float4 v[kSysBatch];
#pragma unroll
    for (int u = 0; u < kSysBatch; ++u) v[u] = __ldg(X + i + u * step);
#pragma unroll
    for (int u = 0; u < kSysBatch; ++u) one(v[u]);
  }
#pragma unroll 1
  for (; i < n; i += step) one(__ldg(X + i));
}

__global__ void __launch_bounds__(kSysThreads) k_sys_centroid(const SysJob* __restrict__ jobs,
                                                              const SysTile* __restrict__ tiles, int n_tiles,
                                                              double* __restrict__ part, int* __restrict__ tickets,
                                                              SysGeom* __restrict__ geoms) {
  const int w = blockIdx.x * kSysWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= n_tiles) return;
  const SysTile tl = tiles[w];
  const SysJob j = jobs[tl.job];
  const long long i0 = (long long)tl.t * j.atoms_per_tile;
  const long long i1 = min(j.n, i0 + (long long)j.atoms_per_tile);
  FF pair[3];
  if (j.dtype == TCM_F32) {
    const float4* X = reinterpret_cast<const float4*>(j.xyzq);
    float s[3] = {0.f, 0.f, 0.f}, e[3] = {0.f, 0.f, 0.f};
    float2 s2 = make_float2(0.f, 0.f), e2 = make_float2(0.f, 0.f);
    sum_f32(X + i0, (int)(i1 - i0), lane, 32, s2, e2, s[2], e[2]);
    s[0] = s2.x, s[1] = s2.y, e[0] = e2.x, e[1] = e2.y;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ff_warp_sum(s[k], e[k]);
      pair[k] = FF{s[k], e[k]};
    }
  } else {
    const double2* X = reinterpret_cast<const double2*>(j.xyzq);
    double s[3] = {0.0, 0.0, 0.0};
    for (long long i = i0 + lane; i < i1; i += 32 * kSysBatch) {
      double2 a[kSysBatch], b[kSysBatch];
#pragma unroll
      for (int u = 0; u < kSysBatch; ++u) {
        const bool ok = i + 32 * u < i1;
        a[u] = ok ? __ldg(X + 2 * (i + 32 * u)) : make_double2(0.0, 0.0);
        b[u] = ok ? __ldg(X + 2 * (i + 32 * u) + 1) : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int u = 0; u < kSysBatch; ++u) {
        s[0] += a[u].x;
        s[1] += a[u].y;
        s[2] += b[u].x;
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // double records: the tile's double sum as a float pair
      const double t = warp_sum_d(s[k]);
      const float h = (float)t;
      pair[k] = FF{h, (float)(t - (double)h)};
    }
  }
  float* row = reinterpret_cast<float*>(part + (long long)(j.tile_base + tl.t) * kSysPart);
  if (lane < 6) row[kRowCen + lane] = (lane & 1) ? pair[lane >> 1].l : pair[lane >> 1].h;
  if (!last_tile(&tickets[2 * tl.job], j.n_tiles, lane)) return;
  const float* p0 = reinterpret_cast<const float*>(part + (long long)j.tile_base * kSysPart);
  const double inv = j.n > 0 ? 1.0 / (double)j.n : 0.0;
  double cs[3];
  ordered_ff_sums<3, false>(p0 + kRowCen, j.n_tiles, kRowFloats, lane, cs);
  if (lane < 3) {  // the centre and its split into float parts
    const double c = (lane == 0 ? cs[0] : (lane == 1 ? cs[1] : cs[2])) * inv;
    const float hi = (float)c;
    geoms[j.geom].c[lane] = c;
    geoms[j.geom].chi[lane] = hi;
    geoms[j.geom].clo[lane] = (float)(c - (double)hi);
  }
}

// A thread's two largest |x - c|^2 in float and the atom of the largest: what the radius filter needs
// to name its candidates without a second scan of the atoms.
struct Farthest {
  float m1 = -1.f, m2 = -1.f;
  int at = 0;
  __device__ __forceinline__ void add(float r, int i) {
    if (r > m1) at = i;
    m2 = fmaxf(m2, fminf(m1, r));
    m1 = fmaxf(m1, r);
  }
};

// Float records: low-degree sums over atoms i, i + step, ... < n of X and the farthest of them.
template <bool kLow>
__device__ __forceinline__ void scan_f32(const float4* X, int n, int i, int step, const float* chi, const float* clo,
                                         LowAcc& acc, Farthest& far) {
  const float2 hi2 = make_float2(chi[0], chi[1]), lo2 = make_float2(clo[0], clo[1]);
  auto one = [&](const float4& v, int at) {
    const FF2 d01 = ff_sub_split2(make_float2(v.x, v.y), hi2, lo2);
    const FF d2 = ff_sub_split(v.z, chi[2], clo[2]);
    const float2 xy = sub2(sub2(make_float2(v.x, v.y), hi2), lo2);  // r2_plain
    const float z = (v.z - chi[2]) - clo[2];
    far.add(__fmaf_rn(xy.x, xy.x, __fmaf_rn(xy.y, xy.y, z * z)), at);
    if (kLow) acc.add(v.w, d01, d2);
  };
  for (; i + (kLowBatch - 1) * step < n; i += kLowBatch * step) {
    float4 v[kLowBatch];
#pragma unroll
    for (int u = 0; u < kLowBatch; ++u) v[u] = __ldg(X + i + u * step);
#pragma unroll
    for (int u = 0; u < kLowBatch; ++u) one(v[u], i + u * step);
  }
  for (; i < n; i += step) one(__ldg(X + i), i);
}

// The same of double records; rmax: the exact largest |x - c|^2.
template <bool kLow>
__device__ __forceinline__ void scan_f64(const double2* X, int n, int i0, int step, const double* c, LowAcc& acc, double& rmax) {
  for (int i = i0; i < n; i += step * kLowBatch) {
    double2 a[kLowBatch], b[kLowBatch];
#pragma unroll
    for (int u = 0; u < kLowBatch; ++u) {
      const bool ok = i + step * u < n;
      a[u] = ok ? __ldg(X + 2 * (i + step * u)) : make_double2(c[0], c[1]);
      b[u] = ok ? __ldg(X + 2 * (i + step * u) + 1) : make_double2(c[2], 0.0);  // padding: d = 0, q = 0
    }
#pragma unroll
    for (int u = 0; u < kLowBatch; ++u) {
      const double dd[4] = {a[u].x - c[0], a[u].y - c[1], b[u].x - c[2], b[u].y};
      rmax = fmax(rmax, dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2]);
      if (kLow) {
        FF t[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float h = (float)dd[k];
          t[k] = FF{h, (float)(dd[k] - (double)h)};
        }
        acc.add(t[3], FF2{make_float2(t[0].h, t[1].h), make_float2(t[0].l, t[1].l)}, t[2]);
      }
    }
  }
}

// The exact largest |x - c|^2 of a warp's atoms (float records) among those within a relative 4e-6 of
// the float maximum mf: each lane's farthest; if a lane's second is within it too, every atom in
// question is looked at.  The candidates are taken one at a time, in a loop whose trip count is the
// warp's candidate count: a predicated double block would occupy the 1/64-rate FP64 pipe every time.
// Lane l's atoms are i0 + l, i0 + l + step, ... < n.
__device__ __forceinline__ double exact_r2(const float4* X, int n, int i0, int step, int lane, const double* c,
                                           const float* chi, const float* clo, const Farthest& far, float mf) {
  const float thr = mf * (1.0f - 4e-6f);
  double rmax = 0.0;
  auto exact = [&](int i) {
    const float4 v = __ldg(X + i);
    const double ex = (double)v.x - c[0], ey = (double)v.y - c[1], ez = (double)v.z - c[2];
    rmax = fmax(rmax, ex * ex + ey * ey + ez * ez);  // the same value in every lane
  };
  if (!__any_sync(0xffffffffu, far.m2 >= thr)) {
    for (unsigned m = __ballot_sync(0xffffffffu, far.m1 >= thr); m; m &= m - 1)
      exact(__shfl_sync(0xffffffffu, far.at, __ffs(m) - 1));
    return rmax;
  }
  for (int iw = i0; iw < n; iw += step) {  // warp-uniform trip count
    const bool cand = iw + lane < n && r2_plain(__ldg(X + iw + lane), chi, clo) >= thr;
    for (unsigned m = __ballot_sync(0xffffffffu, cand); m; m &= m - 1) exact(iw + __ffs(m) - 1);
  }
  return rmax;
}

__global__ void __launch_bounds__(kSysThreads, 3) k_sys_radius_low(const SysJob* __restrict__ jobs,
                                                                const SysTile* __restrict__ tiles, int n_tiles,
                                                                double* __restrict__ part, int* __restrict__ tickets,
                                                                SysGeom* __restrict__ geoms, bool trigger) {
  const int w = blockIdx.x * kSysWarps + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (trigger) pdl_trigger();
  if (w >= n_tiles) return;
  // the centroids of pass 1 are complete; with given centres there is no pass 1, and the kernel before is
  // the one that wrote the tiles and jobs (a long tile list, the fixed scratch's descriptors)
  pdl_wait();
  const SysTile tl = tiles[w];
  const SysJob j = jobs[tl.job];
  const SysGeom g = geoms[j.geom];
  const long long i0 = (long long)tl.t * j.atoms_per_tile;
  const long long i1 = min(j.n, i0 + (long long)j.atoms_per_tile);
  double rmax = 0.0;  // exact max |x - c|^2 of the tile's atoms
  LowAcc acc;
  const int cnt = (int)(i1 - i0);
  if (j.dtype == TCM_F32) {
    const float4* X = reinterpret_cast<const float4*>(j.xyzq) + i0;
    Farthest far;
    if (j.need_low)
      scan_f32<true>(X, cnt, lane, 32, g.chi, g.clo, acc, far);
    else
      scan_f32<false>(X, cnt, lane, 32, g.chi, g.clo, acc, far);
    if (j.need_radius) {
      float mf = far.m1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
      rmax = exact_r2(X, cnt, 0, 32, lane, g.c, g.chi, g.clo, far, mf);
    }
  } else {
    const double2* X = reinterpret_cast<const double2*>(j.xyzq) + 2 * i0;
    if (j.need_low)
      scan_f64<true>(X, cnt, lane, 32, g.c, acc, rmax);
    else
      scan_f64<false>(X, cnt, lane, 32, g.c, acc, rmax);
  }
  rmax = warp_max_d(rmax);
  double* row = part + (long long)(j.tile_base + tl.t) * kSysPart;
  if (j.need_low) {
    static_assert(kLowSums == 10, "the lane map of the reduce-scatter is for ten sums");
    float s[kLowSums], e[kLowSums];
    acc.get(s, e);
    ff_reduce_scatter<kLowSums, 16>(s, e, lane);
    if ((kRs10Lanes >> lane) & 1u) {  // the lane holding sum k writes its (hi, lo) pair
      const int k = 5 * ((lane >> 4) & 1) + 3 * ((lane >> 3) & 1) + 2 * ((lane >> 2) & 1) + ((lane >> 1) & 1);
      reinterpret_cast<float2*>(reinterpret_cast<float*>(row) + kRowLow)[k] = make_float2(s[0], e[0]);
    }
  }
  if (lane == 0) row[kSysPartR2] = rmax;
  if (!last_tile(&tickets[2 * tl.job + 1], j.n_tiles, lane)) return;
  // the last tile of the system: its radius and its low-degree sums over all tiles (tile order),
  // written once to the system's sum row, which every moment job of the system reads
  const double* p0 = part + (long long)j.tile_base * kSysPart;
  if (j.need_low) {  // one pass over the tile rows: the ten sums and the radius together
    double* sr = part + (long long)j.sum_row * kSysPart;
    double low[kLowSums], m = 0.0;
    ordered_ff_sums<kLowSums, true>(reinterpret_cast<const float*>(p0) + kRowLow, j.n_tiles, kRowFloats, lane, low,
                                    2 * (kSysPartR2 - kSysPartLow), &m);
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < kLowSums; ++k) sr[kSysPartLow + k] = low[k];
      if (j.need_radius) geoms[j.geom].a = sqrt(m);
    }
  } else if (j.need_radius) {
    double m = 0.0;
    for (int r = lane; r < j.n_tiles; r += 32) m = fmax(m, __ldcg(p0 + (long long)r * kSysPart + kSysPartR2));
    m = warp_max_d(m);
    if (lane == 0) geoms[j.geom].a = sqrt(m);
  }
}

// The two halves of a cluster barrier: every thread of the cluster arrives, and waits for all.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// One system per cluster of CL CTAs; atom i belongs to thread i mod (CL kSysThreads).
template <int CL>
struct OneShared {
  float2 wlow[kSysWarps][kLowSums];  // each warp's sums
  double wcen[kSysWarps][3], wr2[kSysWarps];
  float wmf[kSysWarps];
  double cen[CL][3];                 // each CTA's centroid sums (in every CTA)
  float2 low[CL][kLowSums];          // each CTA's low-degree sums and maximum (in CTA 0)
  double r2[CL];
  double c[3];
  float chi[3], clo[3];
};

template <int CL>
__global__ void __launch_bounds__(kSysThreads, 4) k_sys_one(const SysJob* __restrict__ jobs, double* __restrict__ part,
                                                            SysGeom* __restrict__ geoms, bool trigger) {
  namespace cg = cooperative_groups;
  __shared__ OneShared<CL> sh;
  if (trigger) pdl_trigger();
  if constexpr (CL > 1) cluster_arrive();  // (its wait: others_started)
  const SysJob j = jobs[blockIdx.x / CL];
  const int rank = blockIdx.x % CL;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int n = (int)j.n;  // at most kSysClusterMax
  constexpr int step = CL * kSysThreads;
  const int i0 = rank * kSysThreads + t;
  auto sync = [] {
    if constexpr (CL > 1)
      cg::this_cluster().sync();
    else
      __syncthreads();
  };
  // Ahead of a CTA's first access to another's shared memory: every CTA of the cluster has started (one
  // that owns no atoms would store within a microsecond of its own start).  The barrier was entered at the
  // top, so the wait is over by the time the scan of the atoms is.
  auto others_started = [] {
    if constexpr (CL > 1) cluster_wait();
  };
  auto of_rank = [&](auto* p, int r) {  // the same variable in CTA r of the cluster
    if constexpr (CL > 1) return cg::this_cluster().map_shared_rank(p, r);
    else return p;
  };
  if (j.need_center) {
    double cs[3] = {0.0, 0.0, 0.0};
    if (j.dtype == TCM_F32) {
      const float4* X = reinterpret_cast<const float4*>(j.xyzq);
      float s[3] = {0.f, 0.f, 0.f}, e[3] = {0.f, 0.f, 0.f};
      float2 s2 = make_float2(0.f, 0.f), e2 = make_float2(0.f, 0.f);
      sum_f32(X, n, i0, step, s2, e2, s[2], e[2]);
      s[0] = s2.x, s[1] = s2.y, e[0] = e2.x, e[1] = e2.y;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        ff_warp_sum(s[k], e[k]);
        cs[k] = (double)s[k] + (double)e[k];
      }
    } else {
      const double2* X = reinterpret_cast<const double2*>(j.xyzq);
      for (int i = i0; i < n; i += step) {
        const double2 a = __ldg(X + 2 * i), b = __ldg(X + 2 * i + 1);
        cs[0] += a.x;
        cs[1] += a.y;
        cs[2] += b.x;
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) cs[k] = warp_sum_d(cs[k]);
    }
    if (lane < 3) sh.wcen[w][lane] = lane == 0 ? cs[0] : (lane == 1 ? cs[1] : cs[2]);
    others_started();
    __syncthreads();
    if (t < 3) {
      double v = 0.0;
#pragma unroll
      for (int k = 0; k < kSysWarps; ++k) v += sh.wcen[k][t];
#pragma unroll
      for (int r = 0; r < CL; ++r) of_rank(&sh.cen[0][0], r)[3 * rank + t] = v;
    }
    sync();
    if (t < 3) {  // the centre and its split into float parts
      double v = 0.0;
#pragma unroll
      for (int r = 0; r < CL; ++r) v += sh.cen[r][t];
      const double c = v * (j.n > 0 ? 1.0 / (double)j.n : 0.0);
      const float hi = (float)c;
      const float lo = (float)(c - (double)hi);
      sh.c[t] = c;
      sh.chi[t] = hi;
      sh.clo[t] = lo;
      if (rank == 0) {
        geoms[j.geom].c[t] = c;
        geoms[j.geom].chi[t] = hi;
        geoms[j.geom].clo[t] = lo;
      }
    }
  } else if (t < 3) {
    sh.c[t] = geoms[j.geom].c[t];
    sh.chi[t] = geoms[j.geom].chi[t];
    sh.clo[t] = geoms[j.geom].clo[t];
  }
  __syncthreads();
  if (!j.need_radius && !j.need_low) {  // the whole cluster
    if (!j.need_center) others_started();
    pdl_wait();
    return;
  }
  const double c[3] = {sh.c[0], sh.c[1], sh.c[2]};
  const float chi[3] = {sh.chi[0], sh.chi[1], sh.chi[2]}, clo[3] = {sh.clo[0], sh.clo[1], sh.clo[2]};
  LowAcc acc;
  Farthest far;
  double rmax = 0.0;
  const float4* X4 = reinterpret_cast<const float4*>(j.xyzq);
  const double2* X8 = reinterpret_cast<const double2*>(j.xyzq);
  if (j.need_low) {
    if (j.dtype == TCM_F32)
      scan_f32<true>(X4, n, i0, step, chi, clo, acc, far);
    else
      scan_f64<true>(X8, n, i0, step, c, acc, rmax);
    float s[kLowSums], e[kLowSums];
    acc.get(s, e);
    ff_reduce_scatter<kLowSums, 16>(s, e, lane);
    if ((kRs10Lanes >> lane) & 1u)
      sh.wlow[w][5 * ((lane >> 4) & 1) + 3 * ((lane >> 3) & 1) + 2 * ((lane >> 2) & 1) + ((lane >> 1) & 1)] =
          make_float2(s[0], e[0]);
  } else if (j.dtype == TCM_F32) {
    scan_f32<false>(X4, n, i0, step, chi, clo, acc, far);
  } else {
    scan_f64<false>(X8, n, i0, step, c, acc, rmax);
  }
  if (j.need_radius && j.dtype == TCM_F32) {
    float mf = far.m1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
    if (lane == 0) sh.wmf[w] = mf;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSysWarps; ++k) mf = fmaxf(mf, sh.wmf[k]);
    rmax = exact_r2(X4, n, i0 - lane, step, lane, c, chi, clo, far, mf);
  }
  rmax = warp_max_d(rmax);
  if (lane == 0) sh.wr2[w] = rmax;
  if (!j.need_center) others_started();
  __syncthreads();
  if (t < kLowSums && j.need_low) {
    FF v{0.f, 0.f};
#pragma unroll
    for (int k = 0; k < kSysWarps; ++k) ff_acc(v.h, v.l, FF{sh.wlow[k][t].x, sh.wlow[k][t].y});
    of_rank(&sh.low[0][0], 0)[rank * kLowSums + t] = make_float2(v.h, v.l);
  }
  if (t == 32) {
    double m = 0.0;
#pragma unroll
    for (int k = 0; k < kSysWarps; ++k) m = fmax(m, sh.wr2[k]);
    of_rank(&sh.r2[0], 0)[rank] = m;
  }
  sync();
  pdl_wait();  // this grid's completion implies that of the kernels it overlaps
  if (rank != 0) return;
  if (t < kLowSums && j.need_low) {
    FF v{0.f, 0.f};
#pragma unroll
    for (int r = 0; r < CL; ++r) ff_acc(v.h, v.l, FF{sh.low[r][t].x, sh.low[r][t].y});
    part[(long long)j.sum_row * kSysPart + kSysPartLow + t] = (double)v.h + (double)v.l;
  }
  if (t == 32 && j.need_radius) {
    double m = 0.0;
#pragma unroll
    for (int r = 0; r < CL; ++r) m = fmax(m, sh.r2[r]);
    geoms[j.geom].a = sqrt(m);
  }
}

}  // namespace

int sys_class(long long n, int dtype) {
  return n <= (dtype == TCM_F32 ? kSysOneMaxF32 : kSysOneMaxF64) ? 0 : (n <= kSysClusterMax ? 1 : 2);
}

int sys_tile_atoms(long long) { return 1024; }

// Largest systems first.  The kernels of different classes do not depend on each other: all but the
// last trigger their successor on entry, and each of those waits for its predecessors before it ends
// (in sequence, each with its own tail, they took 462 us for 2,048 uneven systems).
int launch_sys(const SysJob* jobs, const SysCount& n, const SysTile* t1, const SysTile* t2, double* part, int* tickets,
               SysGeom* geoms, bool pdl, cudaStream_t s) {
  if (n.tiles1 > 0) {
    k_sys_centroid<<<(n.tiles1 + kSysWarps - 1) / kSysWarps, kSysThreads, 0, s>>>(jobs, t1, n.tiles1, part, tickets, geoms);
    if (cudaPeekAtLastError() != cudaSuccess) return -1;
  }
  if (n.tiles2 > 0 && launch_pdl(k_sys_radius_low, dim3((n.tiles2 + kSysWarps - 1) / kSysWarps), dim3(kSysThreads), 0, s,
                                 jobs, t2, n.tiles2, part, tickets, geoms, n.cluster + n.one > 0) != cudaSuccess)
    return -1;
  // (a centroid always comes with its radius, and k_sys_radius_low waits before it reads anything)
  const bool overlap = pdl || n.tiles2 > 0;
  if (n.cluster > 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n.cluster * kSysClusterSize);
    cfg.blockDim = dim3(kSysThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kSysClusterSize;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, k_sys_one<kSysClusterSize>, jobs + n.one, part, geoms, n.one > 0) != cudaSuccess)
      return -1;
  }
  if (n.one > 0) {
    if (n.cluster > 0 || overlap) {
      if (launch_pdl(k_sys_one<1>, dim3(n.one), dim3(kSysThreads), 0, s, jobs, part, geoms, false) != cudaSuccess) return -1;
    } else {
      k_sys_one<1><<<n.one, kSysThreads, 0, s>>>(jobs, part, geoms, false);
      if (cudaPeekAtLastError() != cudaSuccess) return -1;
    }
  }
  return 0;
}

int sys_launches(const SysCount& n) { return (n.one > 0) + (n.cluster > 0) + (n.tiles1 > 0) + (n.tiles2 > 0); }

}  // namespace tcm
