// Descriptors and launchers of the kernels after the moment pass: the contraction (Eq. (Formula)
// in the frame where R0hat = z), the Wigner rotation of cached moments, and the direct sum
// (Eq. (Coulomb)).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "tcm_internal.h"

namespace tcm {

// How the contraction receives B's moments.
constexpr int kBLab = 0;      // lab frame: rotated by the frame rotation W (R0hat -> z) like A's
constexpr int kBInFrame = 1;  // already in the frame (the rotation was applied to B's atoms)
constexpr int kBRotate = 2;   // lab frame, rotated by Mb = W rotB with the Wigner D in the kernel

struct PairDesc {  // one energy: moments of jobA and jobB at lmax L, separation R0
  int jobA, jobB;
  int geomA, geomB;
  int L;
  int b_mode;      // kBLab, kBInFrame or kBRotate
  long long rot;   // kBRotate: index of the Euler record (EulerZYZ) of Mb = W rotB, which takes
                   // B's lab-frame moments into the frame, in the call's rotation array
  double fr[6];    // R0 by its frame W = R_y(-b) R_z(-a) (r0_frame): 1/R, R, cos b, sin b, cos a, sin a
};

// What the host writes for the items of a batch: runs of consecutive items of one pair, degree and mode
// (a scan is one run), and each item's R0.  The descriptors are made from them on the host for small
// batches, by k_frames for large ones, with the same roundings (frame arithmetic below).
struct PairRun {
  int first;         // its first item
  int jobA, jobB;    // computed sets; ~k: the k-th cached set, which follow the computed ones
  int geomA, geomB;
  short L, b_mode;
  int rot;           // kBRotate: rotation of the first item; the others follow
};                   // kBInFrame: jobB of the first item; the others follow

// Where a batched call's results go (device; status and G may be null).
struct PairOut {
  double* E;
  int32_t* status;
  double* G;
};

// Frame arithmetic: every operation rounded by itself, on the device as on the host (where the build
// does not contract either), so that an item's frame does not depend on where it is made.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ double xmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double xadd(double a, double b) { return __dadd_rn(a, b); }
#else
inline double xmul(double a, double b) { return a * b; }
inline double xadd(double a, double b) { return a + b; }
#endif

// The frame record of R0: 1/R, R, cos b = z/R, sin b = rho/R, e^{ia} = (x + iy)/rho (1 on the z axis).
__host__ __device__ inline void r0_frame(const double* R0, double* fr) {
  const double x = R0[0], y = R0[1], z = R0[2];
  const double rho2 = xadd(xmul(x, x), xmul(y, y));
  const double rho = sqrt(rho2), R = sqrt(xadd(rho2, xmul(z, z)));
  fr[0] = 1.0 / R;
  fr[1] = R;
  fr[2] = z / R;
  fr[3] = rho / R;
  fr[4] = rho > 0.0 ? x / rho : 1.0;
  fr[5] = rho > 0.0 ? y / rho : 0.0;
}
// W rot of a frame record: W = R_y(-b) R_z(-a) takes R0hat to the z axis (row-major).
__host__ __device__ inline void frame_times(const double* fr, const double* rot, double* M) {
  const double cb = fr[2], sb = fr[3], ca = fr[4], sa = fr[5];
  const double W[9] = {xmul(cb, ca), xmul(cb, sa), -sb, -sa, ca, 0.0, xmul(sb, ca), xmul(sb, sa), cb};
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j)
      M[3 * i + j] = xadd(xadd(xmul(W[3 * i], rot[j]), xmul(W[3 * i + 1], rot[3 + j])), xmul(W[3 * i + 2], rot[6 + j]));
}

// A rotation M = R_z(-gamma) R_y(-beta) R_z(-alpha), beta in [0, pi], as (cos beta, sin beta,
// e^{i alpha}, e^{i gamma}).
struct EulerZYZ {
  double cb, sb;
  double ea[2], eg[2];
};

// Euler record of a rotation matrix (row-major) through its unit quaternion (largest-component
// extraction): with q = (w, x, y, z),
//   cos(beta/2) = |(w, z)|,  sin(beta/2) = |(x, y)|,
//   e^{i(alpha+gamma)/2} = (w - i z) / cos(beta/2),  e^{i(alpha-gamma)/2} = (-y + i x) / sin(beta/2),
// which stays accurate near beta = 0 and pi (where only alpha+gamma, resp. alpha-gamma, matters).
__host__ __device__ inline EulerZYZ euler_zyz(const double* M) {
  const double t = xadd(xadd(M[0], M[4]), M[8]);
  double w, x, y, z;
  if (t > 0.0) {
    const double s = xmul(2.0, sqrt(xadd(t, 1.0)));
    w = xmul(0.25, s); x = xadd(M[7], -M[5]) / s; y = xadd(M[2], -M[6]) / s; z = xadd(M[3], -M[1]) / s;
  } else if (M[0] > M[4] && M[0] > M[8]) {
    const double s = xmul(2.0, sqrt(xadd(xadd(xadd(1.0, M[0]), -M[4]), -M[8])));
    w = xadd(M[7], -M[5]) / s; x = xmul(0.25, s); y = xadd(M[1], M[3]) / s; z = xadd(M[2], M[6]) / s;
  } else if (M[4] > M[8]) {
    const double s = xmul(2.0, sqrt(xadd(xadd(xadd(1.0, M[4]), -M[0]), -M[8])));
    w = xadd(M[2], -M[6]) / s; x = xadd(M[1], M[3]) / s; y = xmul(0.25, s); z = xadd(M[5], M[7]) / s;
  } else {
    const double s = xmul(2.0, sqrt(xadd(xadd(xadd(1.0, M[8]), -M[0]), -M[4])));
    w = xadd(M[3], -M[1]) / s; x = xadd(M[2], M[6]) / s; y = xadd(M[5], M[7]) / s; z = xmul(0.25, s);
  }
  const double c2 = xadd(xmul(w, w), xmul(z, z)), s2 = xadd(xmul(x, x), xmul(y, y));
  const double n = 1.0 / sqrt(xadd(c2, s2));
  w = xmul(w, n); x = xmul(x, n); y = xmul(y, n); z = xmul(z, n);
  const double ch = sqrt(xadd(xmul(w, w), xmul(z, z))), sh = sqrt(xadd(xmul(x, x), xmul(y, y)));
  const double pr = ch > 0.0 ? w / ch : 1.0, pi = ch > 0.0 ? -z / ch : 0.0;   // p = e^{i(alpha+gamma)/2}
  const double qr = sh > 0.0 ? -y / sh : 1.0, qi = sh > 0.0 ? x / sh : 0.0;   // q = e^{i(alpha-gamma)/2}
  EulerZYZ e;
  e.cb = xmul(xadd(ch, -sh), xadd(ch, sh));
  e.sb = xmul(xmul(2.0, ch), sh);
  e.ea[0] = xadd(xmul(pr, qr), -xmul(pi, qi));  // p q
  e.ea[1] = xadd(xmul(pr, qi), xmul(pi, qr));
  e.eg[0] = xadd(xmul(pr, qr), xmul(pi, qi));  // p conj(q)
  e.eg[1] = xadd(xmul(pi, qr), -xmul(pr, qi));
  return e;
}

// The descriptor of item k of run r at separation R0; rotB: the rotations of the kBRotate items.
__host__ __device__ inline void make_pair(const PairRun& r, int k, const double* R0, int n_computed, const double* rotB,
                                          PairDesc& d, EulerZYZ* e) {
  const int i = k - r.first;
  const int jobB = r.b_mode == kBInFrame ? r.jobB + i : r.jobB;
  d.jobA = r.jobA >= 0 ? r.jobA : n_computed + ~r.jobA;
  d.jobB = jobB >= 0 ? jobB : n_computed + ~jobB;
  d.geomA = r.geomA;
  d.geomB = r.geomB;
  d.L = r.L;
  d.b_mode = r.b_mode;
  d.rot = r.b_mode == kBRotate ? r.rot + i : 0;
  r0_frame(R0, d.fr);
  if (r.b_mode == kBRotate) {
    double M[9];
    frame_times(d.fr, rotB + 9 * d.rot, M);
    e[d.rot] = euler_zyz(M);
  }
}

struct RotDesc {  // one moment set rotated about its centre: out = moments of (M x) from in
  const double* in;
  double* out;
  int L, pad_;
  double M[9];
};

// Tables of the contraction and of the rotation, built once per process.
constexpr int kZN = kLmaxMax + 1;
__host__ __device__ constexpr int dpi2_stride(int l) { return (l + 1) | 1; }
__host__ __device__ constexpr int dpi2_off(int l) {  // sum over l' < l of (l'+1) dpi2_stride(l')
  return l * (l + 1) * (2 * l + 1) / 6 + (l / 2) * (l / 2 + 1);
}
struct Fx {  // fixed point: 2^30 h + l, |l| <= 2^29
  int h, l;
};
struct ContractTables {
  double dpi2[dpi2_off(kZN)];  // rows of d^l(pi/2)
  Fx row[dpi2_off(kZN)];       // the same times 2^59, columns m >= 1 doubled (contract.cu)
  double hat[kZN][kZN];        // [l][m]: 2^-kMomBits l!/sqrt((l+m)!(l-m)!)
  double binom[kZN][kZN];      // [l1][l2]: C(l1 + l2, l1)
};
const ContractTables& contract_tables();
// The order in which a call's items are contracted: by degree, so that a CTA takes contract_group(L)
// items of one degree L at a time.  Items of degree L are order[first[L]] .. order[first[L + 1] - 1]
// (order null: in place), groups gfirst[L] .. gfirst[L + 1] - 1.
struct ContractPlan {
  int first[kLmaxMax + 2], gfirst[kLmaxMax + 2];
};
int contract_group(int L);
// out (device): where the results go; grad: also G, 9 doubles per item: force on B, torque on A, torque
// on B (lab frame).  rots: device, one EulerZYZ per kBRotate item (PairDesc.rot), or null when there is
// none.  pdl: the descriptors are complete before the kernel before this one.
int launch_contract(const PairDesc* items, const int* order, const ContractPlan* plan, int n_groups, int Lmax_items,
                    const MomJob* jobs, const SysGeom* geoms, const ContractTables* tab, const EulerZYZ* rots,
                    const PairOut* out, bool grad, bool pdl, int num_sms, cudaStream_t s);
// Descriptors of a large batch from its runs and separations.  Its successor on the stream may start at
// once (and waits for it before it ends).
int launch_frames(const PairRun* runs, int n_runs, const double* R0, int n_items, int n_computed, const double* rotB,
                  PairDesc* items, EulerZYZ* rots, cudaStream_t s);
int rotate_smem_bytes(int L);
int launch_rotate_moments(const RotDesc* sets, int n_sets, int Lmax_sets, const double* ztab, cudaStream_t s);

__device__ __forceinline__ int tri_l(int k) {  // l with l(l+1)/2 <= k < (l+1)(l+2)/2
  int l = (int)((sqrtf(8.0f * k + 1.0f) - 1.0f) * 0.5f);
  while (l * (l + 1) / 2 > k) --l;
  while ((l + 1) * (l + 2) / 2 <= k) ++l;
  return l;
}

// How the direct sum of one item is cut into CTAs (direct_split): parts = A blocks x B ranges of
// chunk atoms; slab: items per launch (slab x parts partial sums).
struct DirectSplit {
  int ablocks, chunk, parts, slab;
};
DirectSplit direct_split(long long na, long long nb);
int launch_direct(const void* a, long long na, int dta, const void* b, long long nb, int dtb,
                  const SysGeom* geo /* device: [A, B] centres and radii */,
                  const double* xf /* device: per item rot[9], R0[3] */, int n_items,
                  double* part /* min(n_items, slab) x parts */, const DirectSplit& d, double* E /* device, n_items */,
                  cudaStream_t s);

// Sets the calling thread's tcm_last_error() message; returns code.
int record_error(int code, const char* msg);

}  // namespace tcm
