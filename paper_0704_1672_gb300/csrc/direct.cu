// Step a6: the exact pairwise Coulomb sum, Eq. (Coulomb), for a batch of placements of B.
//
// Each CTA takes one item, a block of A's atoms (one per thread) and a range of B's atoms, which
// it stages through shared memory already rotated and translated: b' = R0 + rot (x_b - c_B).
//
// Two forms of the pair loop:
//
//   fixed point: positions, 1/r and the sum in 64-bit integers.  The FP64 pipe takes 2 lanes per
//   clock and SM, the integer multiply-add with a 64-bit sum (IMAD.WIDE) 32 to 64, and the pair loop is
//   nothing but arithmetic on registers: 12 FP64 instructions of a pair held an SMSP for 770 cycles; the
//   57 instructions of the fixed-point pair (13 IMAD.WIDE) take it 109, the integer multiplier 0.8 busy.
//   double: the plain loop, for placements whose systems come close or overlap, for
//   values that fixed point cannot hold (not finite, or outside the radii), and for extreme scales.
//
// Fixed point, for separated systems (r_min = R - a_A - a_B > 0, D = R + a_A + a_B):
//   positions in units of 1/f, f the power of two with 2^61 <= D f < 2^62, as two signed 31-bit
//   limbs X = 2^31 h + l; differences of limbs need no carries:
//     T = sum dh^2 + 2^-30 sum dh dl  =  r^2 f^2 / 2^62      (the three dl^2, below one unit each, enter by
//                                                              their mean)
//   1/r from the float reciprocal square root of T, as the integer Y = 2^55 / sqrt(T), and one
//   third-order correction: with p = T Y^2 / 2^32 mod 2^64 = -2^78 e (the residual e of
//   Y, |e| < 2^-21.1 from the bounds of rsqrt.approx and the roundings of its argument and of Y, is all that the modulus leaves of the product),
//     y = 2^32 Y (1 + e/2 + 3/8 e^2)  =  2^118 / (f r),   good to about 2^-54 of 1/sqrt(T);
//   charges as 53-bit integers on the scale of the range's largest, and three integer sums of limb
//   products, which are exact; the sum itself rounds only when it leaves the loop.  Errors against 64-bit
//   positions: T to 0.42 units rms, 3 at most (one unit is 2^-62 to 2^-60 D^2), so 1/r to 0.21 / T rms;
//   the double loop rounds b' to 2^-53 of itself, so 1/r to 2^-53 |b'| / r.  The closest pairs decide.  With
//   all charges on the facing surfaces, rms of 1/r in fixed point and in double (against 113-bit arithmetic):
//   9.4e-16 and 7.0e-16 at r_min f = 2^55 and D / r_min = 62, 4.3e-16 and 3.9e-16 at 2^56 and 36, 2.7e-16 and
//   2.7e-16 at 2^57 and 24, and sums of such pairs 2.3e-17 and 2.4e-17 of their magnitude.  From there on
//   fixed point is the more exact, so the limit stands at 2^57.
// Measured (2,587 x 3,260 atoms, 256 placements): 47.9 ms in double, 5.37 ms in fixed point; error
// against 64-bit torch 4.0e-14 before, 1.3e-14 now (net-zero charges: of the cancelled sum).  Two atoms
// of A per thread were slower (116 cycles a pair at 128 registers); so were the same steps left to the
// compiler as 64-bit expressions (125: it spends the multiplier on register moves).
// Bounds: r_min f >= 2^57 (r_min / D above 1/32 to 1/16) keeps T above 2^52 and Y below 2^29, D f < 2^62 (with
// room for the limbs' rounding) dh below 2^31 and Y above 2^24.
#include <cuda_runtime.h>

#include "contract.h"

namespace tcm {

namespace {

constexpr int kDirectThreads = 256;
constexpr int kDirectTile = 256;  // atoms of B staged at once, one per thread

struct alignas(16) FixAtom {  // a staged atom of B: position limbs, charge limbs
  int h[3];
  int qh;
  int l[3];
  int ql;
};
struct alignas(32) Atom4 {  // the same for the double loop
  double x, y, z, w;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
// Fixed-order block sum; result valid in thread 0.
__device__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    r = lane < nw ? sh[lane] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;
}
__device__ __forceinline__ void load_xyz(const void* p, int dtype, long long i, double* x, double& q) {
  if (dtype == TCM_F32) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p) + i);
    x[0] = v.x;
    x[1] = v.y;
    x[2] = v.z;
    q = v.w;
  } else {
    const double2 a = __ldg(reinterpret_cast<const double2*>(p) + 2 * i);
    const double2 b = __ldg(reinterpret_cast<const double2*>(p) + 2 * i + 1);
    x[0] = a.x;
    x[1] = a.y;
    x[2] = b.x;
    q = b.y;
  }
}
__device__ __forceinline__ double load_q(const void* p, int dtype, long long i) {
  return dtype == TCM_F32 ? (double)__ldg(reinterpret_cast<const float*>(p) + 4 * i + 3)
                          : __ldg(reinterpret_cast<const double*>(p) + 4 * i + 3);
}

__device__ __forceinline__ int exponent(double v) { return (int)((__double2hiint(v) >> 20) & 0x7ff) - 1022; }
constexpr int kNoCharge = -1022;  // of a range without charge
__device__ __forceinline__ int charge_exponent(double q) { return q == 0.0 ? kNoCharge : max(exponent(q), kNoCharge + 1); }
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// The item's transform: centres, rotation, separation.
struct Place {
  double cA[3], cB[3], rot[9], R0[3];
};

// Atom of B in the frame of A: rotated offset from its centre in d, b' = R0 + d.
__device__ __forceinline__ void place_b(const Place& g, const double* x, double* d) {
  const double v[3] = {x[0] - g.cB[0], x[1] - g.cB[1], x[2] - g.cB[2]};
#pragma unroll
  for (int k = 0; k < 3; ++k) d[k] = g.rot[3 * k] * v[0] + g.rot[3 * k + 1] * v[1] + g.rot[3 * k + 2] * v[2];
}

__device__ __forceinline__ void split31(double x, double f, int& h, int& l) {
  const long long X = __double2ll_rn(x * f);
  h = (int)((X + (1LL << 30)) >> 31);
  l = (int)(X - ((long long)h << 31));
}

__device__ __forceinline__ long long madw(int a, int b, long long c) {
  return (long long)a * (long long)b + c;
}
// 2^118 / (f r) of one pair (see the head of the file).
__device__ __forceinline__ int2 inv_r(const int* ah, const int* al, const int4 bh, const int4 bl) {
  const int h0 = bh.x - ah[0], h1 = bh.y - ah[1], h2 = bh.z - ah[2];
  const int l0 = bl.x - al[0], l1 = bl.y - al[1], l2 = bl.z - al[2];
  const long long s = madw(h2, h2, madw(h1, h1, (long long)h0 * h0));
  // 2^30: half a unit for the shift's floor, half for the mean of sum dl^2
  const long long c = madw(h2, l2, madw(h1, l1, madw(h0, l0, 1LL << 30)));
  unsigned Th, Tl;  // T = s + (c >> 30)
  asm("{ .reg .u32 a, b, x, y;\n\t"
      "mov.b64 {a, b}, %2;\n\tmov.b64 {x, y}, %3;\n\t"
      "shf.r.wrap.b32 x, x, y, 30;\n\tshr.s32 y, y, 30;\n\t"
      "add.cc.u32 %0, a, x;\n\taddc.u32 %1, b, y; }"
      : "=r"(Tl), "=r"(Th)
      : "l"(s), "l"(c));
  float y0;  // within 2^-22.9
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(fmaf((float)Th, 4294967296.0f, (float)Tl)));
  const int Y = __float2int_rn(y0 * 36028797018963968.0f);  // 2^55
  const unsigned long long U = (unsigned long long)(unsigned)Y * (unsigned)Y;
  const unsigned Uh = (unsigned)(U >> 32), Ul = (unsigned)U;
  // p = T U / 2^32 mod 2^64 (its multiple of 2^78 drops out), |p| < 2^57; the product of the low
  // words by their upper halves
  const unsigned long long w = (unsigned long long)Tl * Uh + (unsigned long long)Th * Ul;
  unsigned pl, ph;
  asm("{ .reg .u32 a, b;\n\t"
      "mov.b64 {a, b}, %2;\n\tadd.cc.u32 %0, a, %3;\n\taddc.u32 b, b, 0;\n\tmad.lo.u32 %1, %4, %5, b; }"
      : "=r"(pl), "=r"(ph)
      : "l"(w), "r"((Tl >> 16) * (Ul >> 16)), "r"(Th), "r"(Uh));
  const float t = (float)(int)ph;
  // p / 2^26 with the second-order term, 3/8 e^2 2^53
  const int q = (int)__funnelshift_r(pl, ph, 26) - __float2int_rn(t * t * (0.375f / 549755813888.0f));
  const long long M = (long long)Y * q;
  int lo, hi;
  asm("sub.cc.u32 %0, 0, %2;\n\tsubc.u32 %1, %3, %4;"  // 2^32 Y - (M >> 21)
      : "=r"(lo), "=r"(hi)
      : "r"(__funnelshift_r((unsigned)M, (unsigned)(M >> 32), 21)), "r"(Y), "r"((int)(M >> 32) >> 21));
  return make_int2(lo, hi);
}

// One atom of A against the staged atoms: sums of q y in three limb products, 32 pairs at a time
// (26 + 31 + 5 bits), each folded into a pair of wide sums.
struct FixSum {
  long long hi[3] = {0, 0, 0};
  unsigned long long lo[3] = {0, 0, 0};
  __device__ __forceinline__ void fold(const long long* a) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      hi[k] += a[k] >> 32;
      lo[k] += (unsigned)a[k];
    }
  }
  __device__ __forceinline__ double value(double scale) const {
    double v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = fma((double)hi[k], 4294967296.0, (double)lo[k]);
    // weights 2^59 (qh yh), 2^27 (qh yl), 2^32 (ql yh)
    return fma(v[0], 134217728.0, fma(v[2], 1.0, v[1] * (1.0 / 32.0))) * scale;
  }
};

struct Fixed {  // the scales of one CTA's fixed-point loop
  double f;     // positions
  double rA2, rB2;  // largest |x|^2 of an atom of A, of B about its centre
  bool ok;
};

__device__ __forceinline__ Fixed fixed_scales(const Place& g, double aA, double aB) {
  Fixed s;
  const double R = sqrt(g.R0[0] * g.R0[0] + g.R0[1] * g.R0[1] + g.R0[2] * g.R0[2]);
  aA *= 1.0 + 1e-9;  // room for the rounding of the rotated offsets
  aB *= 1.0 + 1e-9;
  const double D = (R + aA + aB) * (1.0 + 1e-9);  // (and for the limbs)
  const int e = exponent(D);  // D < 2^e
  s.rA2 = aA * aA;
  s.rB2 = aB * aB;
  s.ok = D > 0.0 && e > -400 && e < 400;
  s.f = pow2(s.ok ? 62 - e : 0);
  s.ok = s.ok && (R - aA - aB) * s.f >= 0x1p57;
  return s;
}

__global__ void __launch_bounds__(kDirectThreads, 4)
    k_direct(const void* __restrict__ a, long long na, int dta, const void* __restrict__ b, long long nb, int dtb,
             const SysGeom* __restrict__ geo, const double* __restrict__ xf, int ablocks, int chunk,
             double* __restrict__ part) {
  __shared__ union {
    FixAtom fix[kDirectTile];
    Atom4 dbl[kDirectTile];
  } sb;
  __shared__ Place g;
  __shared__ double sh[32];
  __shared__ int s_exp;
  const int t = threadIdx.x;
  const double* item = xf + 12LL * blockIdx.y;  // this item's rotation of B and separation
  if (t < 9) g.rot[t] = item[t];
  if (t < 3) {
    g.R0[t] = item[9 + t];
    g.cA[t] = geo[0].c[t];
    g.cB[t] = geo[1].c[t];
  }
  if (t == 0) s_exp = 0;
  __syncthreads();
  const int ab = blockIdx.x % ablocks, bb = blockIdx.x / ablocks;
  const long long j0 = (long long)bb * chunk, j1 = min(nb, j0 + (long long)chunk);
  const Fixed fs = fixed_scales(g, geo[0].a, geo[1].a);
  const long long i = (long long)ab * kDirectThreads + t;
  double pos[3] = {0.0, 0.0, 0.0}, qa = 0.0;  // a padding atom: A's centre, no charge
  bool bad = !fs.ok;
  if (i < na) {
    load_xyz(a, dta, i, pos, qa);
    double r2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      pos[k] -= g.cA[k];
      r2 += pos[k] * pos[k];
    }
    bad = bad || !(r2 <= fs.rA2);
  }
  const bool warp_idle = __all_sync(0xffffffffu, i >= na);
  double acc = 0.0;
  bool fixed = false;
  if (!__syncthreads_or(bad)) {
    // the range's largest charge sets the scale of the charges; every staged atom lies within the radius
    int qe = kNoCharge;
    for (long long j = j0 + t; j < j1; j += kDirectThreads) qe = max(qe, charge_exponent(load_q(b, dtb, j)));
    qe = __reduce_max_sync(0xffffffffu, qe);
    if ((t & 31) == 0) atomicMax(&s_exp, qe + 1022);
    __syncthreads();
    qe = s_exp - 1022;
    // (not finite: 1025); under 2^-500 the scale of the sum would leave the normal numbers
    fixed = qe < 900 && (qe >= -500 || qe == kNoCharge);
    if (qe == kNoCharge) qe = 0;
    const double gq = pow2(26 - qe);  // |q| gq < 2^26
    int ah[3], al[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) split31(pos[k], fs.f, ah[k], al[k]);
    FixSum sum;
    for (long long jt = j0; fixed && jt < j1; jt += kDirectTile) {
      FixAtom v;
      double d[3] = {0.0, 0.0, 0.0}, q = 0.0;  // a padding atom: B's centre, no charge
      if (jt + t < j1) {
        double x[3];
        load_xyz(b, dtb, jt + t, x, q);
        place_b(g, x, d);
      }
      bad = !(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] <= fs.rB2);
#pragma unroll
      for (int k = 0; k < 3; ++k) split31(g.R0[k] + d[k], fs.f, v.h[k], v.l[k]);
      const long long Q = __double2ll_rn(q * gq * 134217728.0);  // 2^27
      v.qh = (int)((Q + (1LL << 26)) >> 27);
      v.ql = (int)(Q - ((long long)v.qh << 27));
      fixed = !__syncthreads_or(bad);  // (also: every thread is done with the tile before)
      sb.fix[t] = v;
      __syncthreads();
      if (warp_idle || !fixed) continue;
      const int cnt = (int)min((long long)kDirectTile, j1 - jt);
      for (int k0 = 0; k0 < cnt; k0 += 32) {
        long long s[3] = {};
#pragma unroll 2
        for (int k = k0; k < k0 + 32; ++k) {
          const int4 bh = *reinterpret_cast<const int4*>(sb.fix[k].h), bl = *reinterpret_cast<const int4*>(sb.fix[k].l);
          const int2 y = inv_r(ah, al, bh, bl);
          const int yh = y.y + (int)((unsigned)y.x >> 31);  // y = 2^32 yh + yl, yl signed
          s[0] = madw(bh.w, yh, s[0]);
          s[1] = madw(bh.w, y.x, s[1]);
          s[2] = madw(bl.w, yh, s[2]);
        }
        sum.fold(s);
      }
    }
    if (fixed) {
      // q / r = 2^-118 f y / (2^27 gq) q's integer; FixSum::value leaves a weight of 2^32
      const double scale = fs.f * pow2(-118 - 27 + 32) * pow2(qe - 26);
      acc = sum.value(scale);
    }
  }
  if (!fixed) {
    for (long long jt = j0; jt < j1; jt += kDirectTile) {
      Atom4 v{1e300, 1e300, 1e300, 0.0};
      if (jt + t < j1) {
        double x[3], d[3], q;
        load_xyz(b, dtb, jt + t, x, q);
        place_b(g, x, d);
        v = Atom4{g.R0[0] + d[0], g.R0[1] + d[1], g.R0[2] + d[2], q};
      }
      __syncthreads();
      sb.dbl[t] = v;
      __syncthreads();
      if (warp_idle) continue;
      const int cnt = (int)min((long long)kDirectTile, j1 - jt);
      for (int k = 0; k < cnt; ++k) {
        const Atom4 w = sb.dbl[k];
        const double dx = w.x - pos[0], dy = w.y - pos[1], dz = w.z - pos[2];
        acc += w.w * rsqrt(dx * dx + dy * dy + dz * dz);
      }
    }
  }
  const double v = block_sum(i < na ? acc * qa : 0.0, sh);
  if (t == 0) part[(long long)blockIdx.y * gridDim.x + blockIdx.x] = v;
}

// One CTA per item: each thread sums a contiguous stripe of the item's partials, then a
// fixed-order block sum.
__global__ void k_direct_final(const double* __restrict__ part, int nblk, double* __restrict__ E) {
  __shared__ double sh[32];
  part += (long long)blockIdx.x * nblk;
  double s = 0.0;
  const int per = (nblk + blockDim.x - 1) / blockDim.x;
  const int b0 = threadIdx.x * per;
  for (int k = b0; k < min(nblk, b0 + per); ++k) s += part[k];
  s = block_sum(s, sh);
  if (threadIdx.x == 0) E[blockIdx.x] = s;
}

}  // namespace

// The split of one item, from the atom counts alone (so that an item's energy does not depend on
// the batch it is in): A in blocks of 256 atoms, B in as many ranges as bring an item to
// about 64 CTAs while each range keeps at least 512 atoms (a CTA's set-up is then about a tenth of
// its work).
DirectSplit direct_split(long long na, long long nb) {
  DirectSplit d;
  const long long nA = (na + kDirectThreads - 1) / kDirectThreads;
  long long nB = nA > 0 ? (64 + nA - 1) / nA : 1;
  nB = std::max<long long>(1, std::min<long long>(nB, nb / 512));
  d.ablocks = (int)nA;
  d.chunk = (int)std::max<long long>(32, ((nb + nB - 1) / nB + 31) / 32 * 32);
  d.parts = (int)(nA * std::max<long long>(1, (nb + d.chunk - 1) / d.chunk));
  // items whose partial sums fit the buffer at once; one launch's grid holds at most 65,535
  d.slab = (int)std::max<long long>(1, std::min<long long>(65535, (1LL << 24) / std::max(d.parts, 1)));
  return d;
}

int launch_direct(const void* a, long long na, int dta, const void* b, long long nb, int dtb, const SysGeom* geo,
                  const double* xf, int n_items, double* part, const DirectSplit& d, double* E, cudaStream_t s) {
  for (int i0 = 0; i0 < n_items; i0 += d.slab) {  // the slabs reuse the partial sums in stream order
    const int n = std::min(d.slab, n_items - i0);
    if (d.parts > 0)
      k_direct<<<dim3(d.parts, n), kDirectThreads, 0, s>>>(a, na, dta, b, nb, dtb, geo, xf + 12LL * i0, d.ablocks, d.chunk, part);
    k_direct_final<<<n, 128, 0, s>>>(part, d.parts, E + i0);
  }
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace tcm
