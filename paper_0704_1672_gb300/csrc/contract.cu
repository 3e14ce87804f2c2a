// a4 + a5: the two-center contraction, Eq. (Formula), in the frame where R0hat is the z axis, and its
// derivatives.
//
// With the stretched 3j symbol (L = l1 + l2) Eq. (Formula) reads
//   U = sum (-1)^l2 Qhat^A_l1m1 Qhat^B_l2m2 J_{l1+l2, m1+m2},
//   Qhat_lm = Q_lm / sqrt((l+m)!(l-m)!),  J_LM = sqrt((L+M)!(L-M)!) sqrt(4pi/(2L+1)) Y*_LM(R0hat) / R^{L+1}.
// U does not change when A, B and R0 rotate together.  In the frame W = R_y(-beta) R_z(-alpha)
// that takes R0hat = (sin b cos a, sin b sin a, cos b) to z, J_LM = delta_M0 L! / R^{L+1}, so
//   U = sum_{l1,l2} (-1)^l2 (l1+l2)! / R^{l1+l2+1}
//         [Qhat'^A_l1,0 Qhat'^B_l2,0 + 2 sum_{m>=1} (-1)^m Re(Qhat'^A_l1m conj(Qhat'^B_l2m))]
// (real charges: Q_l,-m = (-1)^m conj(Q_lm)).  Moments enter in the rotated frame: those of B
// either come from the moment kernels with W folded into the atom transform (mode kBInFrame),
// or, like those of A, are rotated here (kBLab by W; kBRotate by W rotB from a lab-frame set):
//   Q'_lm = sum_m' d^l_{m'm}(beta) P_lm',  P_lm' = e^{-i m' alpha} Q_lm'.
// The Wigner matrix d^l(beta) is never formed.  A rotation about y is a rotation about z
// between two rotations by pi/2 about x, which for the constant matrices D^l = d^l(pi/2) gives
//   d^l_{m'm}(beta) = i^(m-m') sum_k D^l_{km'} D^l_{km} e^{i k beta},
// so Q' follows from two products with D^l around a diagonal phase:
//   p_k = sum_m' D^l_{km'} v_m',  v_m' = (-i)^m' P_lm';   Q'_lm = i^m sum_k D^l_{km} e^{i k beta} p_k.
// For real charges v_-m' = (-1)^m' conj(v_m') and p_-k = (-1)^k conj(p_k); with
// D^l_{k,-m'} = (-1)^(l+k) D^l_{km'} and D^l_{km} = (-1)^(k-m) D^l_{mk} the terms of m' and -m'
// (and of k and -k) combine into one real product, which leaves, for k, m >= 0,
//   Re p_k = sum_{m' = l+k (mod 2)} D^l_{km'} Re v~_m',   Im p_k = sum_{other m'} D^l_{km'} Im v~_m',
//   S_m = (-1)^l [sum_{k = l+m (mod 2)} D^l_{mk} Re p~_k - i sum_{other k} D^l_{mk} Im p~_k],  Q'_lm = i^m S_m,
// with p~_k = e^{i k beta} p_k and the entries of indices >= 1 counted twice (the table's columns):
// (l+1)^2 real multiply-adds per product and degree, no table of d^l(beta) per energy.
//
// What bounds it, and why the rotations are in fixed point: in double the kernel was bound by the FP64 pipe
// (a warp instruction holds its SMSP for 64 cycles; 400 of them per energy at degree 10), most of it the
// phases and the two products.  Their quantities are bounded (|D| <= 1, phases of modulus 1, rotations keep a
// degree's norm), so they are held as 60-bit integers on a scale per degree and side and multiplied in
// 30-bit limbs: three IMAD.WIDE of about four cycles each instead of an FP64 instruction.  A rotation
// spreads the rounding of a degree's largest component over all of them, in double as here: a value
// in fixed point is off by a few 2^-57 of that component, in double by a few 2^-53 of the partial sums.
// From there on the components are far apart: l!/sqrt((l+m)!(l-m)!) falls to 2e-7 at l = m = 24, and a pair
// stacked on a common axis may have nothing but its highest orders.  So the factor, the products of A's and
// B's components and every sum of them are double.  (With the products in fixed point too, rounded on the
// scale of the degree's largest component, two coaxial rings of 12 alternating charges lost five
// digits, of 48 fourteen.)  B's moments in mode kBInFrame need no rotation and stay double throughout.
// Error of an energy (rms, of sum |U_l1l2|, 40 random pairs at degrees 1 to 24; against 113-bit
// arithmetic): 1.5e-16 to 8.9e-16, the all-double kernel's 1.5e-16 to 8.9e-16; forces and torques alike.
// Measured (us), all in double, with the products in fixed point too, and now: 108,360 energies at degrees 1 to
// 10 1,340, 298, 328; 2,048 at degrees 8 to 24 (B rotated) 140, 64, 76; 256 at degree 20 24, 16, 20; forces
// and torques of 512 at degree 12 92, 25, 42 (49 with products by m instead of partial sums).  What bounds it now: the
// FP64 pipe in the (l1, l2) phase (busy 0.54 over the kernel at degree 24) between phases separated by barriers.
// A CTA takes a group of items of one degree side by side (contract_group), so that its lanes are full
// at low degrees too, one lane column per item.  The group size, and with it the order of every sum,
// depends on the degree alone: an item's result does not depend on its batch.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "contract.h"

namespace tcm {

namespace {

constexpr int kCT = 256;  // threads of a contraction CTA
constexpr int kMaxGroup = 16;
// X = Q 2^(kMomBits - e), parts of Q_lm below 2^e: the norm of a degree, at most sqrt(97) 2^e, and with it
// every value on the way is below 2^60.3, so that a high limb stays below 2^30.3, the high-limb sums (a table
// row has norm 1, the orders m and -m share it) below 2^61.3 and the cross sums of 13 products below 2^61.5.
constexpr int kMomBits = 57;

__host__ __device__ constexpr int group_of(int L) {
  const int g = 512 / ((L + 1) * (L + 2));
  return g < 1 ? 1 : (g > kMaxGroup ? kMaxGroup : g);
}
__host__ __device__ constexpr int tri(int l) { return l * (l + 1) / 2; }

// Shared memory of a group (bytes): int4 arrays qa, qb, ta, tb (and qm) of tri(L + 1) entries and five
// phase tables of L + 1, doubles R^-(k+1), k <= 2 L + 1, ints of the degrees' exponents; per item.
constexpr int item_bytes(int L, bool grad) {
  return 16 * ((grad ? 5 : 4) * tri(L + 1) + 5 * (L + 1)) + 8 * (2 * L + 2) + 8 * (L + 1);
}
int smem_bytes(int Lmax, bool grad) {
  int mx = 0;
  for (int L = 0; L <= Lmax; ++L) mx = std::max(mx, group_of(L) * item_bytes(L, grad));
  return 8 * ((dpi2_off(Lmax + 1) + 1) & ~1) + mx;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double flip(double x, int odd) {  // (-1)^odd x without an FP64 op
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)(odd & 1) << 63));
}

// ---- fixed point
struct Acc {  // a sum of products: 2^60 h + 2^30 m (the low limbs' product, at most 2^58, is dropped)
  long long h = 0, m = 0;
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
    h += (long long)ah * bh;
    m += (long long)ah * bl;
    m += (long long)al * bh;
  }
  __device__ __forceinline__ void sub(int ah, int al, int bh, int bl) { add(-ah, -al, bh, bl); }
  __device__ __forceinline__ long long value60() const { return h + ((m + (1 << 29)) >> 30); }        // / 2^60
  __device__ __forceinline__ long long value59() const { return 2 * h + ((m + (1 << 28)) >> 29); }    // / 2^59
};
__device__ __forceinline__ Fx split30(long long x) {
  Fx f;
  f.h = (int)((x + (1 << 29)) >> 30);
  f.l = (int)((unsigned)x - ((unsigned)f.h << 30));
  return f;
}
__device__ __forceinline__ int4 pack(Fx r, Fx i) { return make_int4(r.h, r.l, i.h, i.l); }
struct Wide {  // a complex number before its parts are split into limbs
  long long x, y;
};
__device__ __forceinline__ int4 pack(Wide z) { return pack(split30(z.x), split30(z.y)); }
__device__ __forceinline__ Wide cmulw(int4 a, int4 b) {  // one factor on the scale 2^60
  Acc r, i;
  r.add(a.x, a.y, b.x, b.y);
  r.sub(a.z, a.w, b.z, b.w);
  i.add(a.x, a.y, b.z, b.w);
  i.add(a.z, a.w, b.x, b.y);
  return Wide{r.value60(), i.value60()};
}
__device__ __forceinline__ int4 cmulf(int4 a, int4 b) { return pack(cmulw(a, b)); }
__device__ __forceinline__ int4 ipow(int4 z, int n) {  // i^n z
  const int r = n & 3;
  const int4 s = (r & 1) ? make_int4(z.z, z.w, z.x, z.y) : z;
  return make_int4((r == 1 || r == 2) ? -s.x : s.x, (r == 1 || r == 2) ? -s.y : s.y, r >= 2 ? -s.z : s.z,
                   r >= 2 ? -s.w : s.w);
}
__device__ __forceinline__ Wide ipow(Wide z, int n) {
  const int r = n & 3;
  const Wide s = (r & 1) ? Wide{z.y, z.x} : z;
  return Wide{(r == 1 || r == 2) ? -s.x : s.x, r >= 2 ? -s.y : s.y};
}
__device__ __forceinline__ double2 times(Wide z, double f) { return make_double2((double)z.x * f, (double)z.y * f); }
__device__ __forceinline__ int4 unit(double x, double y) {  // a complex number of modulus <= 1 on the scale 2^60
  return pack(split30(__double2ll_rn(x * 1152921504606846976.0)), split30(__double2ll_rn(y * 1152921504606846976.0)));
}
__device__ __forceinline__ int4 zpow(int4 z, int n) {  // z^n by squaring
  int4 r = make_int4(1 << 30, 0, 0, 0);
  if (n == 0) return r;
  r = z;
  for (int b = 30 - __clz(n); b >= 0; --b) {
    r = cmulf(r, r);
    if ((n >> b) & 1) r = cmulf(r, z);
  }
  return r;
}

__device__ __forceinline__ bool finite(double v) { return ((__double2hiint(v) >> 20) & 0x7ff) != 0x7ff; }
__device__ __forceinline__ int exponent(double v) { return ((__double2hiint(v) >> 20) & 0x7ff) - 1022; }  // |v| < 2^e
// v 2^(kMomBits - e), |v| < 2^e, to the nearest integer: integer instructions only
__device__ __forceinline__ long long to_fixed(double v, int e) {
  const long long b = __double_as_longlong(v);
  int ex = (int)((b >> 52) & 0x7ff);
  long long m = b & 0xfffffffffffffLL;
  if (ex > 0) m |= 1LL << 52;
  else ex = 1;
  const int sh = ex - 1075 + kMomBits - e;  // at most 4
  m = sh >= 0 ? m << sh : (sh > -63 ? ((m >> (-sh - 1)) + 1) >> 1 : 0);
  return b < 0 ? -m : m;
}
__device__ __forceinline__ double scale2(double c, int n) {  // c 2^n
  const int ex = ((__double2hiint(c) >> 20) & 0x7ff) + n;
  if (ex >= 1 && ex <= 2046 && ex - n >= 1 && ex - n <= 2046) return __longlong_as_double(__double_as_longlong(c) + ((long long)n << 52));
  return ldexp(c, n);
}
__device__ __forceinline__ double rpow(double x, int n) {
  double r = 1.0;
  while (n) {
    if (n & 1) r *= x;
    x *= x;
    n >>= 1;
  }
  return r;
}

// Row product with a parity split: (sum over j = par (mod 2) of row[j] Re x_j, sum over the other j of
// row[j] Im x_j), j = 0..l, of one item's column of x (stride G).
__device__ __forceinline__ Wide row_split(const Fx* row, const int4* x, int G, int l, int par) {
  const int2* xs = reinterpret_cast<const int2*>(x);
  Acc a, b;  // even j, odd j
  int j = 0;
  for (; j + 1 <= l; j += 2) {
    const Fx r0 = row[j], r1 = row[j + 1];
    const int2 x0 = xs[2 * j * G + par], x1 = xs[2 * (j + 1) * G + 1 - par];
    a.add(r0.h, r0.l, x0.x, x0.y);
    b.add(r1.h, r1.l, x1.x, x1.y);
  }
  if (j == l) {
    const Fx r0 = row[j];
    const int2 x0 = xs[2 * j * G + par];
    a.add(r0.h, r0.l, x0.x, x0.y);
  }
  const long long va = a.value59(), vb = b.value59();
  return par ? Wide{vb, va} : Wide{va, vb};
}

// Eq. (Formula) for one (pair, orientation) per column of a CTA.  With kGrad also, per item, the force on
// B (-grad_R0 E) and the torques on A and on B about their centres, from the same frame moments:
//   in the frame, with c = (-1)^l2 L!/R^(L+1), c' = (-1)^l2 (L+1)!/R^(L+2), L = l1 + l2,
//   T0 = sum_m Qa_m Qb_-m,  S+ = sum_{m1+m2=1} Qa_m1 Qb_m2,  P = sum_{m1+m2=1} (l2+m2) Qa_m1 Qb_m2,
//   Z = sum_{m>=1} (-1)^m 2m Im(Qa_m conj Qb_m)  (Qhat normalisation throughout):
//   grad E = -sum c' (Re S+, Im S+, T0)       (only J_L,0 and J_L,+-1 have a first-order
//                                                derivative on the z axis);
//   tau_B = sum c (Im P, -Re P, -Z),  tau_A = sum c (Im P', -Re P', Z),  P' = (L+1) S+ - P
//   (infinitesimal rotations act on Qhat_lm through L_z and the ladder operators with the
//   integer weights (l+m+1), (l-m+1)).  The vectors go back to the lab frame with W^T.
// A's moments are kept as a_m = (-1)^m Qa_m, so that T0 = Re sum a_m conj(b_m) and so on without signs;
// the sums weighted by m take m a_m.
template <bool kGrad>
__global__ void __launch_bounds__(kCT, kGrad ? 2 : 4)
    k_contract(const PairDesc* __restrict__ items, const int* __restrict__ order, const ContractPlan* __restrict__ plan,
               int n_groups, int Lmax, const MomJob* __restrict__ jobs, const SysGeom* __restrict__ geoms,
               const ContractTables* __restrict__ tab, const EulerZYZ* __restrict__ rots,
               const PairOut* __restrict__ out) {
  extern __shared__ __align__(16) int4 sm4[];
  __shared__ PairDesc s_d[kMaxGroup];
  __shared__ int s_item[kMaxGroup], s_ok[kMaxGroup];  // s_ok: 1 converges, 0 not, -1 moments or phases that are not finite
  __shared__ unsigned short s_lm[(kLmaxMax + 1) * (kLmaxMax + 2) / 2];
  __shared__ double s_sum[kGrad ? 9 : 1][kCT];
  constexpr int kTabs = 5;
  Fx* Ds = reinterpret_cast<Fx*>(sm4);
  int4* base4 = sm4 + ((dpi2_off(Lmax + 1) + 1) >> 1);
  // Before griddepcontrol.wait: everything that depends only on the tables and on descriptors that were
  // uploaded ahead of the kernels.
  for (int i = threadIdx.x; i < dpi2_off(Lmax + 1); i += kCT) Ds[i] = tab->row[i];
  for (int k = threadIdx.x; k < tri(Lmax + 1); k += kCT) {
    const int l = tri_l(k);
    s_lm[k] = (unsigned short)(l << 8 | (k - tri(l)));
  }
  const PairOut o = *out;
  bool waited = false;
  for (int g = blockIdx.x; g < n_groups; g += gridDim.x) {
    int L = 0;
    while (plan->gfirst[L + 1] <= g) ++L;
    const int G = group_of(L), Q = kCT / G;
    const int first = plan->first[L] + (g - plan->gfirst[L]) * G;
    const int cnt = min(G, plan->first[L + 1] - first);
    const int nq = tri(L + 1), n1 = L + 1;
    int4* qa = base4;           // A: moments (double), v (fixed), then a_m in the frame (double)
    int4* qb = qa + nq * G;     // B: the same
    int4* ta = qb + nq * G;     // p~ of A
    int4* tb = ta + nq * G;     // p~ of B
    int4* qm = tb + nq * G;     // kGrad: m a_m (double)
    double2 *da = reinterpret_cast<double2*>(qa), *db = reinterpret_cast<double2*>(qb), *dm = reinterpret_cast<double2*>(qm);
    int4* ph = kGrad ? qm + nq * G : qm;  // input phases of W (alpha of R0); mode kBRotate: 2, 3, 4 of W rotB
    double* rp = reinterpret_cast<double*>(ph + kTabs * n1 * G);  // R^-(k+1), k <= 2 L + 1
    int* ex = reinterpret_cast<int*>(rp + (2 * L + 2) * G);       // exponents of the degrees, A then B
    __syncthreads();  // the group before is done
    if (threadIdx.x < cnt) {
      const int k = order ? order[first + threadIdx.x] : first + threadIdx.x;
      s_item[threadIdx.x] = k;
      s_d[threadIdx.x] = items[k];
    }
    for (int k = threadIdx.x; k < 2 * n1 * G; k += kCT) ex[k] = -1022;
    __syncthreads();
    const int it = threadIdx.x % G, q0 = threadIdx.x / G;
    const bool in = it < cnt && q0 < Q;
    const PairDesc& d = s_d[it < cnt ? it : 0];
    const int bmode = d.b_mode;
    if (in) {
      // the phase tables, one entry per step: (-i)^m e^{-i m alpha}, e^{i k beta} of W; in mode kBRotate
      // those of W rotB and i^m e^{-i m gamma}; then the powers of 1/R (other threads', so side by side)
      const int ntab = bmode == kBRotate ? kTabs : 2;
      for (int q = q0; q < ntab * n1 + 2 * L + 2; q += Q) {
        const int t = q / n1, m = q - t * n1;
        if (t >= ntab) {
          const int k = q - ntab * n1;
          rp[k * G + it] = rpow(d.fr[0], k + 1);
          continue;
        }
        double zx, zy;
        if (t < 2) {
          zx = t == 0 ? d.fr[4] : d.fr[2];
          zy = t == 0 ? -d.fr[5] : d.fr[3];
        } else {
          const EulerZYZ* e = rots + d.rot;
          zx = t == 2 ? e->ea[0] : (t == 3 ? e->cb : e->eg[0]);
          zy = t == 2 ? -e->ea[1] : (t == 3 ? e->sb : -e->eg[1]);
        }
        const int4 z = zpow(unit(zx, zy), m);
        ph[q * G + it] = (t == 0 || t == 2) ? ipow(z, -m) : (t == 4 ? ipow(z, m) : z);
      }
    }
    if (!waited) {
      pdl_wait();  // the moments (and centres and radii) of the launches before are complete
      waited = true;
    }
    if (in) {
      const double* pa = jobs[d.jobA].out;
      const double* pb = jobs[d.jobB].out;
      for (int q = q0; q < nq; q += Q) {
        const int l = s_lm[q] >> 8, m = s_lm[q] & 255;
        const double2 a = m == 0 ? make_double2(pa[l * l], 0.0) : make_double2(pa[l * l + 2 * m - 1], pa[l * l + 2 * m]);
        const double2 b = m == 0 ? make_double2(pb[l * l], 0.0) : make_double2(pb[l * l + 2 * m - 1], pb[l * l + 2 * m]);
        da[q * G + it] = a;
        db[q * G + it] = b;
        atomicMax(&ex[l * G + it], max(exponent(a.x), exponent(a.y)));
        atomicMax(&ex[(n1 + l) * G + it], max(exponent(b.x), exponent(b.y)));
      }
      if (q0 == 0) {
        s_ok[it] = d.fr[1] > geoms[d.geomA].a + geoms[d.geomB].a;  // Eq. (mainCond)
        // phases that are not finite have no fixed-point form (degree 0 has no phase)
        bool ok = L == 0 || (finite(d.fr[2]) && finite(d.fr[3]) && finite(d.fr[4]) && finite(d.fr[5]));
        if (L > 0 && bmode == kBRotate) {
          const EulerZYZ* e = rots + d.rot;
          ok = ok && finite(e->cb) && finite(e->sb) && finite(e->ea[0]) && finite(e->ea[1]) && finite(e->eg[0]) &&
               finite(e->eg[1]);
        }
        if (s_ok[it] && !ok) s_ok[it] = -1;
      }
    }
    __syncthreads();
    const double* hat = &tab->hat[0][0];
    if (in) {  // to fixed point; v = input phases times the moments; mode kBInFrame only scales B (in double)
      for (int q = q0; q < nq; q += Q) {
        const int l = s_lm[q] >> 8, m = s_lm[q] & 255;
        const int ea = ex[l * G + it], eb = ex[(n1 + l) * G + it];
        const double2 a = da[q * G + it];
        double2 b = db[q * G + it];
        if (max(ea, eb) > 1024 && s_ok[it] == 1) s_ok[it] = -1;
        qa[q * G + it] = cmulf(ph[m * G + it], pack(Wide{to_fixed(a.x, ea), to_fixed(a.y, ea)}));
        if (bmode == kBInFrame) {
          int n = kMomBits - eb;
          if (n < -800) {  // (2^n hat would be subnormal)
            b = make_double2(b.x * 0x1p-300, b.y * 0x1p-300);
            n += 300;
          }
          const double f = scale2(hat[l * kZN + m], n);
          db[q * G + it] = make_double2(b.x * f, b.y * f);
        } else {
          qb[q * G + it] = cmulf(ph[((bmode == kBRotate ? 2 * n1 : 0) + m) * G + it],
                                 pack(Wide{to_fixed(b.x, eb), to_fixed(b.y, eb)}));
        }
      }
    }
    __syncthreads();
    if (in) {  // first product: p~_kk from v of degree l
      const int4* eb = ph + ((bmode == kBRotate ? 3 : 1) * n1) * G;
      for (int q = q0; q < nq; q += Q) {
        const int l = s_lm[q] >> 8, kk = s_lm[q] & 255;
        const Fx* row = Ds + dpi2_off(l) + kk * dpi2_stride(l);
        ta[q * G + it] = cmulf(ph[(n1 + kk) * G + it], pack(row_split(row, qa + tri(l) * G + it, G, l, (l + kk) & 1)));
        if (bmode != kBInFrame)
          tb[q * G + it] = cmulf(eb[kk * G + it], pack(row_split(row, qb + tri(l) * G + it, G, l, (l + kk) & 1)));
      }
    }
    __syncthreads();
    if (in) {  // second product: S_m, times i^m (or the output phase) and, in double, the hat factor
      for (int q = q0; q < nq; q += Q) {
        const int l = s_lm[q] >> 8, m = s_lm[q] & 255;
        const Fx* row = Ds + dpi2_off(l) + m * dpi2_stride(l);
        const double f = hat[l * kZN + m];
        auto signs = [&](Wide p) { return (l & 1) ? Wide{-p.x, p.y} : Wide{p.x, -p.y}; };
        Wide S = signs(row_split(row, ta + tri(l) * G + it, G, l, (l + m) & 1));
        const double2 a = times(ipow(S, m + 2 * m), f);  // (-1)^m i^m
        da[q * G + it] = a;
        if (kGrad) dm[q * G + it] = make_double2((double)m * a.x, (double)m * a.y);
        if (bmode != kBInFrame) {
          S = signs(row_split(row, tb + tri(l) * G + it, G, l, (l + m) & 1));
          db[q * G + it] = times(bmode == kBRotate ? cmulw(ph[(4 * n1 + m) * G + it], pack(S)) : ipow(S, m), f);
        }
      }
    }
    __syncthreads();
    // z-axis contraction: one (l1, l2) per step.  The pairs are taken in shells of equal s = min(l1, l2),
    // s = L first: the (L - s)^2 pairs before shell s are those of the larger shells, and shell s lists
    // (s, s), (s, s+1), (s+1, s), (s, s+2), ...  Neighbouring lanes then run their m loops to nearly the
    // same length.
    double sum[kGrad ? 9 : 1];
#pragma unroll
    for (int k = 0; k < (kGrad ? 9 : 1); ++k) sum[k] = 0.0;
    if (in) {
      for (int p = q0; p < n1 * n1; p += Q) {
        int u = (int)sqrtf((float)p);  // u = L - s = floor(sqrt(p))
        while (u * u > p) --u;
        while ((u + 1) * (u + 1) <= p) ++u;
        const int s = L - u, j = p - u * u;
        const int l1 = (j & 1) ? s : s + (j >> 1);
        const int l2 = (j & 1) ? s + ((j + 1) >> 1) : s;
        const double2* a = da + tri(l1) * G + it;
        const double2* b = db + tri(l2) * G + it;
        double es = 0.0;
        for (int m = 1; m <= s; ++m) {
          const double2 x = a[m * G], y = b[m * G];
          es = fma(x.x, y.x, es);
          es = fma(x.y, y.y, es);
        }
        const double T = fma(a[0].x, b[0].x, es + es);
        const int n = l1 + l2;
        const int sh = ex[l1 * G + it] + ex[(n1 + l2) * G + it];
        const double bi = tab->binom[l1][l2];
        const double c = flip(scale2(bi * rp[n * G + it], sh), l2);
        sum[0] = fma(c, T, sum[0]);
        if (kGrad) {
          const double2* am = dm + tri(l1) * G + it;
          // the sums weighted by m as sums of partial sums, from the highest m down: an addition each
          // instead of two multiply-adds
          double sr = 0.0, si = 0.0, tr = 0.0, ti = 0.0, wr = 0.0, wi = 0.0, z = 0.0;
          for (int m = min(l1, l2 + 1); m >= 1; --m) {  // (m, 1 - m): -a_m conj(b_(m-1)), weight l2 + 1 - m
            const double2 x = a[m * G], y = b[(m - 1) * G];
            sr = fma(-x.x, y.x, sr);
            sr = fma(-x.y, y.y, sr);
            si = fma(-x.y, y.x, si);
            si = fma(x.x, y.y, si);
            wr -= sr;
            wi -= si;
          }
          for (int m = min(l1, l2 - 1); m >= 0; --m) {  // (-m, m + 1): conj(a_m) b_(m+1), weight l2 + 1 + m
            const double2 x = a[m * G], y = b[(m + 1) * G];
            tr = fma(x.x, y.x, tr);
            tr = fma(x.y, y.y, tr);
            ti = fma(x.x, y.y, ti);
            ti = fma(-x.y, y.x, ti);
            if (m == 0) break;
            wr += tr;
            wi += ti;
          }
          sr += tr;
          si += ti;
          for (int m = 1; m <= s; ++m) {
            const double2 xm = am[m * G], y = b[m * G];
            z = fma(xm.y, y.x, z);
            z = fma(-xm.x, y.y, z);
          }
          const double w1 = (double)(l2 + 1);
          const double Pr = fma(w1, sr, wr), Pi = fma(w1, si, wi);
          const double Z = z + z;
          const double L1 = (double)(n + 1);
          const double c1 = flip(scale2(bi * L1 * rp[(n + 1) * G + it], sh), l2);
          sum[1] = fma(-c1, sr, sum[1]);
          sum[2] = fma(-c1, si, sum[2]);
          sum[3] = fma(-c1, T, sum[3]);
          sum[4] = fma(c, Pi, sum[4]);
          sum[5] = fma(-c, Pr, sum[5]);
          sum[6] = fma(-c, Z, sum[6]);
          sum[7] = fma(c, fma(L1, si, -Pi), sum[7]);
          sum[8] = fma(-c, fma(L1, sr, -Pr), sum[8]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < (kGrad ? 9 : 1); ++k) s_sum[k][threadIdx.x] = sum[k];
    __syncthreads();
    // one warp per item adds its column: lane c adds entries c, c + 32, ... in order, then a fixed tree
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < cnt; i += kCT / 32) {
      double v[kGrad ? 9 : 1];
#pragma unroll
      for (int k = 0; k < (kGrad ? 9 : 1); ++k) {
        double t = 0.0;
        for (int q = lane; q < Q; q += 32) t += s_sum[k][q * G + i];
        v[k] = warp_sum(t);
      }
      if (lane != 0) continue;
      const int item = s_item[i];
      const double nan = __longlong_as_double(0x7ff8000000000000LL);
      if (s_ok[i] == 1) {
        o.E[item] = v[0];
      } else if (s_ok[i] == 0) {  // the expansion does not converge
        o.E[item] = nan;
      } else {  // moments or phases that are not finite: only Lmax = 0 has a product of its own
        const PairDesc& e = s_d[i];
        o.E[item] = L == 0 ? jobs[e.jobA].out[0] * jobs[e.jobB].out[0] * e.fr[0] : nan;
      }
      if (o.status) o.status[item] = s_ok[i] == 0 ? TCM_ENOTCONV : TCM_OK;
      if (kGrad) {
        double* w = o.G + 9LL * item;
        if (s_ok[i] != 1) {
          for (int k = 0; k < 9; ++k) w[k] = nan;
          continue;
        }
        const double* fr = s_d[i].fr;
        const double cb = fr[2], sb = fr[3], ca = fr[4], sa = fr[5];
        const double W[9] = {cb * ca, cb * sa, -sb, -sa, ca, 0.0, sb * ca, sb * sa, cb};  // R_y(-b) R_z(-a)
        // frame -> lab: v_lab = W^T v_frame; force = -grad; tau_A,z = -tau_B,z
        const double f[3] = {-v[1], -v[2], -v[3]};
        const double tA[3] = {v[7], v[8], -v[6]};
        const double tB[3] = {v[4], v[5], v[6]};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          w[k] = W[k] * f[0] + W[3 + k] * f[1] + W[6 + k] * f[2];
          w[3 + k] = W[k] * tA[0] + W[3 + k] * tA[1] + W[6 + k] * tA[2];
          w[6 + k] = W[k] * tB[0] + W[3 + k] * tB[1] + W[6 + k] * tB[2];
        }
      }
    }
  }
  if (!waited) pdl_wait();
}

}  // namespace

int contract_group(int L) { return group_of(L); }

int launch_contract(const PairDesc* items, const int* order, const ContractPlan* plan, int n_groups, int Lmax_items,
                    const MomJob* jobs, const SysGeom* geoms, const ContractTables* tab, const EulerZYZ* rots,
                    const PairOut* out, bool grad, bool pdl, int num_sms, cudaStream_t s) {
  if (n_groups <= 0) return 0;
  const int smem = smem_bytes(Lmax_items, grad);
  auto k = grad ? k_contract<true> : k_contract<false>;
  // the limit of every degree: it does not change under a captured launch
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(kLmaxMax, grad)) != cudaSuccess)
    return -1;
  // CTAs stay resident and walk the groups (the tables are loaded once per CTA)
  const int per_sm = std::max(1, std::min(grad ? 2 : 4, 227 * 1024 / (smem + (grad ? 23 : 6) * 1024)));
  const int grid = std::min(n_groups, per_sm * num_sms);
  if (!pdl)
    k<<<grid, kCT, smem, s>>>(items, order, plan, n_groups, Lmax_items, jobs, geoms, tab, rots, out);
  else if (launch_pdl(k, dim3(grid), dim3(kCT), smem, s, items, order, plan, n_groups, Lmax_items, jobs, geoms, tab, rots,
                      out) != cudaSuccess)
    return -1;
  return cudaPeekAtLastError() == cudaSuccess ? 0 : -1;
}

namespace {
// d^l_{km}(pi/2) for 0 <= k, m <= l: at beta = pi/2 both half-angle factors are 2^(-1/2), so
//   d^l_{km}(pi/2) = 2^-l sqrt((l+k)!(l-k)! / ((l+m)!(l-m)!)) sum_s (-1)^(k-m+s) C(l+m, s) C(l-m, l-k-s),
// an exact integer sum (at most C(2l, l-k) in magnitude) times one square root.
long double dpi2_entry(int l, int k, int m, const long long (*C)[2 * kZN + 1], const long double* fact) {
  long long S = 0;
  for (int s = (m > k ? m - k : 0); s <= l + m && s <= l - k; ++s) {
    const long long t = C[l + m][s] * C[l - m][l - k - s];
    S += ((k - m + s) & 1) ? -t : t;
  }
  const long double r = sqrtl(fact[l + k] * fact[l - k] / (fact[l + m] * fact[l - m]));
  return ldexpl((long double)S * r, -l);
}
Fx split_host(long double x) {
  const long long v = llrintl(x);
  const int h = (int)((v + (1LL << 29)) >> 30);
  return Fx{h, (int)(v - ((long long)h << 30))};
}
void build_tables(ContractTables& t) {
  long double fact[2 * kZN + 2];
  fact[0] = 1.0L;
  for (int k = 1; k < 2 * kZN + 2; ++k) fact[k] = fact[k - 1] * (long double)k;
  static long long C[2 * kZN + 1][2 * kZN + 1];  // binomials up to C(2 kLmaxMax, .), exact
  for (int n = 0; n <= 2 * kZN; ++n) {
    C[n][0] = 1;
    for (int k = 1; k <= 2 * kZN; ++k) C[n][k] = n == 0 ? 0 : C[n - 1][k - 1] + C[n - 1][k];
  }
  for (int l = 0; l < kZN; ++l) {
    for (int m = 0; m <= l; ++m) t.hat[l][m] = (double)ldexpl(fact[l] / sqrtl(fact[l + m] * fact[l - m]), -kMomBits);
    for (int k = 0; k < kZN; ++k) t.binom[l][k] = (double)C[l + k][l];
    for (int k = 0; k <= l; ++k)
      for (int m = 0; m <= l; ++m) {
        const long double d = dpi2_entry(l, k, m, C, fact);
        t.dpi2[dpi2_off(l) + k * dpi2_stride(l) + m] = (double)d;
        t.row[dpi2_off(l) + k * dpi2_stride(l) + m] = split_host(ldexpl(d, m > 0 ? 60 : 59));
      }
  }
}
}  // namespace

const ContractTables& contract_tables() {
  static const ContractTables* t = [] {
    ContractTables* p = new ContractTables();
    build_tables(*p);
    return p;
  }();
  return *t;
}

}  // namespace tcm
