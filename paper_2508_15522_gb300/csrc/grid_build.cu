// Substrate grid construction on the GPU (Sec. 3, 4, 5 of the paper):
//   node values of V^C (3D Ewald, slab dipole correction), V^P, V^L
//   -> exact cubic B-spline coefficients (separable 1D line solves)
//   -> padded float4 records read by the interpolation kernels.
// Everything before the final packing runs in FP64.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "internal.h"
#include "trace.h"

namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr double kKe = 14.399645;  // eV*A/e^2

struct alignas(32) D4 {   // x, y, z, charge
  double x, y, z, w;
};

// One lattice image of a substrate atom that comes within a cutoff of the
// grid box: position, charge and the weights of the two Morse channels,
// L = wL e^{-alpha d}, P = wP (e^{-alpha d})^2 with wL = eps e^{alpha R} and
// wP = eps e^{2 alpha R}; R and eps for the form without the table.
struct alignas(32) SubImage {
  double x, y, z, q, wL, wP, R, eps;
};

struct BuildParams {
  int nx, ny, nz;
  double x0, y0, z0, dx, dy, dz;
  double alpha, rcut2, ercut2, beta;
  int morse;                        // compute V^P, V^L
  int coulomb;                      // compute V^C
  int slotP, slotL, slotC;          // output channel slots (-1 = absent)
  double bg;                        // -pi Q / (beta^2 V)
  double dip;                       // 4 pi M_z / V
};

// --------------------------------------------------------------------------
// reciprocal space
// --------------------------------------------------------------------------
// In-plane vectors k2 = m1 B1 + m2 B2 of one half plane (the potential is
// real, so -k2 adds the complex conjugate of k2's term) and m3 = -M3 .. M3
// along z.  The phase e^{-i k.r} of an atom is the product of an in-plane
// phase and one of 2 M3 + 1 phases along z, and the latter are shared by all
// k2: one table EZ[m3][atom] (and EL[m3][plane] for the node planes) replaces
// a sine and a cosine per (k, atom), 2.6 ms of a 384-ion build before.

// E[t][i] = e^{i sign kz z_i}, kz = (t - M3) B3z
__global__ void z_phase_kernel(const double* __restrict__ z, int zstride, int n, double z0, double dz, int M3,
                               double B3z, double sign, double2* __restrict__ E) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n * (2 * M3 + 1)) return;
  const int t = idx / n, i = idx % n;
  double s, c;
  sincos(sign * (t - M3) * B3z * (z ? z[(size_t)i * zstride] : z0 + i * dz), &s, &c);
  E[idx] = make_double2(c, s);
}

// AS[k2][m3] = A_k S(k), A_k = 4 pi e^{-k^2/4b^2}/(V k^2), S(k) = sum_j q_j
// e^{-i k.r_j}; zero outside the sphere |k| < kmax or at k = 0.  One block
// per k2; keep[k2] = some |S(k)| exceeds s_min, the rounding error of S (a
// supercell of a perfect crystal has structure factors at the few vectors
// of the primitive lattice only: 10 of 595 in an 8 x 8 rock-salt slab).
constexpr int kStructThreads = 128;
__global__ void __launch_bounds__(kStructThreads)
k_struct_kernel(const D4* __restrict__ atoms, int n_atoms, const double2* __restrict__ kvec,
                const double2* __restrict__ EZ, int M3, double B3z, double kmax2, double beta, double vol,
                double s_min2, double2* __restrict__ AS, int* __restrict__ keep) {
  __shared__ double2 s_p[kStructThreads];
  __shared__ int s_keep;
  const int nm3 = 2 * M3 + 1;
  const double kx = kvec[blockIdx.x].x, ky = kvec[blockIdx.x].y, kp2 = kx * kx + ky * ky;
  if (threadIdx.x == 0) s_keep = 0;
  for (int t0 = 0; t0 < nm3; t0 += kStructThreads) {
    const int t = t0 + threadIdx.x;
    double re = 0.0, im = 0.0;
    for (int j0 = 0; j0 < n_atoms; j0 += kStructThreads) {
      __syncthreads();
      if (j0 + (int)threadIdx.x < n_atoms) {
        const D4 a = atoms[j0 + threadIdx.x];
        double s, c;
        sincos(kx * a.x + ky * a.y, &s, &c);
        s_p[threadIdx.x] = make_double2(a.w * c, -a.w * s);
      }
      __syncthreads();
      const int cnt = min(kStructThreads, n_atoms - j0);
      if (t < nm3)
        for (int j = 0; j < cnt; ++j) {
          const double2 p = s_p[j], e = EZ[(size_t)t * n_atoms + j0 + j];
          re += p.x * e.x - p.y * e.y;
          im += p.x * e.y + p.y * e.x;
        }
    }
    if (t < nm3) {
      const double kz = (t - M3) * B3z, k2n = kp2 + kz * kz;
      double2 out = make_double2(0.0, 0.0);
      if (k2n > 0.0 && k2n < kmax2) {
        const double A = 4.0 * kPi / vol * exp(-k2n / (4.0 * beta * beta)) / k2n;
        out = make_double2(A * re, A * im);
        if (re * re + im * im > s_min2) s_keep = 1;
      }
      AS[(size_t)blockIdx.x * nm3 + t] = out;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) keep[blockIdx.x] = s_keep;
}

// list = the kept k2 in increasing order, n_list[0] their count (one warp).
__global__ void k_select_kernel(const int* __restrict__ keep, int n_k2, int* __restrict__ list,
                                int* __restrict__ n_list) {
  int base = 0;
  for (int k0 = 0; k0 < n_k2; k0 += 32) {
    const int k = k0 + threadIdx.x;
    const unsigned b = __ballot_sync(0xffffffffu, k < n_k2 && keep[k]);
    if ((b >> threadIdx.x) & 1u) list[base + __popc(b & ((1u << threadIdx.x) - 1u))] = k;
    base += __popc(b);
  }
  if (threadIdx.x == 0) n_list[0] = base;
}

// G[i][l] = w sum_m3 AS[list[i]][m3] e^{i kz(m3) z_l}, w = 2 for the half
// plane's vectors and 1 for k2 = 0 (vector 0).
__global__ void k_zsum_kernel(const double2* __restrict__ AS, const double2* __restrict__ EL,
                              const int* __restrict__ list, const int* __restrict__ n_list, int M3, int nz,
                              double2* __restrict__ G) {
  const int nm3 = 2 * M3 + 1;
  const int n = n_list[0] * nz;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
    const int k2 = list[idx / nz], l = idx % nz;
    double re = 0.0, im = 0.0;
    for (int t = 0; t < nm3; ++t) {
      const double2 as = AS[(size_t)k2 * nm3 + t], e = EL[(size_t)t * nz + l];
      re += as.x * e.x - as.y * e.y;
      im += as.x * e.y + as.y * e.x;
    }
    const double w = k2 == 0 ? 1.0 : 2.0;
    G[idx] = make_double2(w * re, w * im);
  }
}

// --------------------------------------------------------------------------
// radial functions as piecewise polynomials in u = d^2
// --------------------------------------------------------------------------
// f(u) = e^{-alpha sqrt(u)} and g(u) = erfc(beta sqrt(u)) / sqrt(u) on the
// intervals that share u's exponent and first 7 mantissa bits (relative
// width 2^-7): degree 7 and 5 around the interval's centre, the Taylor
// series of the functions' differential equations
//   4 u f'' + 2 f' = alpha^2 f,   u g' = -g/2 - (beta/sqrt(pi)) E,  E' = -beta^2 E
// economised by Chebyshev polynomials.  The relative truncation error of f is
// (alpha d 2^-9)^8 / (8! 2^7), 7e-18 at alpha d = 25.5; that of g is below
// 1e-16 wherever g exceeds 1e-6 of its value at 1 A.  No square root, no
// exponential and no erfc per pair: 9 FP64 instructions for f and 6 for g
// where the library functions take about 40 and 60, and the FP64 pipe (two
// lanes per SM and cycle) is what bounds the sums.
constexpr int kTabBits = 7;
constexpr int kTabLoExp = -2;                              // the table begins at u = 2^-2 (d = 0.5 A)
constexpr int kFCoef = 8, kGCoef = 6;
__host__ __device__ inline int tab_index(int hi) { return (hi >> (20 - kTabBits)) - ((1023 + kTabLoExp) << kTabBits); }

// tab: float64 pairs, f: [kFCoef / 2][n_f], then g: [kGCoef / 2][n_g].
__global__ void radial_table_kernel(int n_f, int n_g, double alpha, double beta, double2* __restrict__ tab) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_f && i >= n_g) return;
  const int hi = ((i + ((1023 + kTabLoExp) << kTabBits)) << (20 - kTabBits)) | (1 << (19 - kTabBits));
  const double u0 = __hiloint2double(hi, 0);                             // centre
  const double w = ldexp(1.0, (hi >> 20) - 1023 - kTabBits - 1);         // half width
  double a[11];
  auto economise = [&](int deg) {
    // drop tau^10, tau^9, ... down to tau^(deg + 1), tau = (u - u0) / w
    for (int k = 1; k <= 10; ++k) a[k] *= ldexp(1.0, k * ilogb(w));
    if (deg < 10) {
      const double c = a[10] / 512;
      a[8] += 1280 * c, a[6] -= 1120 * c, a[4] += 400 * c, a[2] -= 50 * c, a[0] += c;
    }
    if (deg < 9) {
      const double c = a[9] / 256;
      a[7] += 576 * c, a[5] -= 432 * c, a[3] += 120 * c, a[1] -= 9 * c;
    }
    if (deg < 8) {
      const double c = a[8] / 128;
      a[6] += 256 * c, a[4] -= 160 * c, a[2] += 32 * c, a[0] -= c;
    }
    if (deg < 7) {
      const double c = a[7] / 64;
      a[5] += 112 * c, a[3] -= 56 * c, a[1] += 7 * c;
    }
    if (deg < 6) {
      const double c = a[6] / 32;
      a[4] += 48 * c, a[2] -= 18 * c, a[0] += c;
    }
    for (int k = 1; k <= deg; ++k) a[k] *= ldexp(1.0, -k * ilogb(w));
  };
  const double d0 = sqrt(u0);
  if (i < n_f) {
    a[0] = exp(-alpha * d0);
    a[1] = -alpha / (2.0 * d0) * a[0];
    for (int k = 0; k + 2 <= 10; ++k)
      a[k + 2] = (alpha * alpha * a[k] - (4.0 * k + 2.0) * (k + 1) * a[k + 1]) / (4.0 * u0 * (k + 2) * (k + 1));
    economise(kFCoef - 1);
    for (int k = 0; k < kFCoef; k += 2) tab[(size_t)(k / 2) * n_f + i] = make_double2(a[k], a[k + 1]);
  }
  if (i < n_g) {
    a[0] = erfc(beta * d0) / d0;
    double e = beta * 0.56418958354775628695 * exp(-beta * beta * u0);   // 1 / sqrt(pi)
    for (int k = 0; k + 1 <= 10; ++k) {
      a[k + 1] = -((k + 0.5) * a[k] + e) / (u0 * (k + 1));
      e *= -beta * beta / (k + 1);
    }
    economise(kGCoef - 1);
    double2* t = tab + (size_t)(kFCoef / 2) * n_f;
    for (int k = 0; k < kGCoef; k += 2) t[(size_t)(k / 2) * n_g + i] = make_double2(a[k], a[k + 1]);
  }
}

// --------------------------------------------------------------------------
// node values
// --------------------------------------------------------------------------
// A warp computes COLS neighbouring columns (consecutive y, one x) x 32
// consecutive z: 4 columns with the table, 1 without it, where a pair costs about
// ten times as much.  A warp's first item is fixed, spread over the SMs; the
// others come from a counter, lowest z first (they have the most atoms in range).
// A small grid has fewer items than the chip has warps: 75 x 75 x 27 nodes with a
// cutoff of 25 A, 1425 items of 4 columns from a counter alone, left 63 of 152 SMs
// without work (14.1 ms, now 2.6).  Its lanes first test 32 images at a time
// against the item's box and compute the squared in-plane distances to the
// four columns; then the images that can reach it are taken one by one, their
// distances broadcast, one lane per z.  Bound by the FP64 pipe: per pair in
// range 12 FP64 instructions for the Morse channels, 7 for the Coulomb one.
// One block of 16 warps per SM, the radial table in its shared memory.
// 8 x 8 x 3 rock-salt slab, 113 x 113 x 208 nodes: 12.7 ms (659 ms with a
// thread per node over every image of every atom and the library functions).
constexpr int kNodeWarps = 16;
constexpr int kTableCols = 4;

struct NodeTables {
  const double2* tab;          // radial table (TABLE)
  int n_f, n_g;
  const SubImage* img;
  int n_img;
  const int* k_list;           // kept in-plane vectors
  const int* n_k;
  const double2* kvec;
  const double2* G;            // [n_k][nz]
};

__device__ __forceinline__ double bcast(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }

template <bool TABLE, int COLS>
__global__ void __launch_bounds__(32 * kNodeWarps, 1)
node_values_kernel(BuildParams p, NodeTables nt, int* __restrict__ next, double* __restrict__ vals) {
  extern __shared__ __align__(16) double2 s_tab[];
  const int lane = threadIdx.x & 31;
  const double2* const s_g = s_tab + (size_t)(kFCoef / 2) * nt.n_f;
  if (TABLE) {
    const int n = (kFCoef / 2) * nt.n_f + (kGCoef / 2) * nt.n_g;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s_tab[i] = nt.tab[i];
    __syncthreads();
  }
  const int ng = (p.ny + COLS - 1) / COLS, nzc = (p.nz + 31) / 32;
  const size_t n_nodes = (size_t)p.nx * p.ny * p.nz;
  const double cut2 = fmax(p.morse ? p.rcut2 : 0.0, p.coulomb ? p.ercut2 : 0.0);
  // distances are compared as integers (non-negative doubles order like their
  // bit patterns), which keeps the comparisons off the FP64 pipe
  const unsigned long long rc2 = (unsigned long long)__double_as_longlong(p.morse ? p.rcut2 : 0.0);
  const unsigned long long ec2 = (unsigned long long)__double_as_longlong(p.coulomb ? p.ercut2 : 0.0);
  const int n_k = p.coulomb ? nt.n_k[0] : 0;
  int item = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  for (;; item = gridDim.x * kNodeWarps + __shfl_sync(0xffffffffu, lane == 0 ? atomicAdd(next, 1) : 0, 0)) {
    if (item >= p.nx * ng * nzc) break;
    const int zc = item / (p.nx * ng), ix = (item / ng) % p.nx, iy0 = (item % ng) * COLS;
    const int iz = zc * 32 + lane;
    const double x = p.x0 + ix * p.dx, z = p.z0 + min(iz, p.nz - 1) * p.dz;
    const double zlo = p.z0 + zc * 32 * p.dz, zhi = p.z0 + min(zc * 32 + 31, p.nz - 1) * p.dz;
    double y[COLS], vP[COLS], vL[COLS], phi[COLS];
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
      y[c] = p.y0 + (iy0 + c) * p.dy;      // columns past ny are computed and not stored
      vP[c] = vL[c] = phi[c] = 0.0;
    }
    double z_prev = 0.0, dz2 = 0.0;
    bool have = false;
    for (int j0 = 0; j0 < nt.n_img; j0 += 32) {
      const int j = j0 + lane;
      double rho2[COLS];
      bool near = false;
      if (j < nt.n_img) {
        const SubImage* im = nt.img + j;
        const double ddx = x - im->x, yj = im->y, zj = im->z;
        double least = 1e300;
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
          const double ddy = y[c] - yj;
          rho2[c] = ddx * ddx + ddy * ddy;
          least = fmin(least, rho2[c]);
        }
        const double gap = fmax(0.0, fmax(zlo - zj, zj - zhi));
        near = least + gap * gap < cut2;
      }
      unsigned hits = __ballot_sync(0xffffffffu, near);
      while (hits) {
        const int src = __ffs(hits) - 1;
        hits &= hits - 1;
        const SubImage* im = nt.img + j0 + src;
        const double zj = __ldg(&im->z), q = __ldg(&im->q), wL = __ldg(&im->wL), wP = __ldg(&im->wP);
        if (!have || zj != z_prev) {       // images come sorted by height: few changes
          const double ddz = z - zj;
          dz2 = ddz * ddz;
          z_prev = zj;
          have = true;
        }
        double u[COLS];
#pragma unroll
        for (int c = 0; c < COLS; ++c) u[c] = bcast(rho2[c], src) + dz2;
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
          const unsigned long long ub = (unsigned long long)__double_as_longlong(u[c]);
          if (ub >= rc2 && ub >= ec2) continue;
          const int hi = (int)(ub >> 32), idx = tab_index(hi);
          if (TABLE && idx >= 0) {
            const double t = u[c] - __hiloint2double((hi & ~((1 << (20 - kTabBits)) - 1)) | (1 << (19 - kTabBits)), 0);
            if (ub < rc2) {
              const double2 c0 = s_tab[idx], c1 = s_tab[nt.n_f + idx], c2 = s_tab[2 * nt.n_f + idx],
                            c3 = s_tab[3 * nt.n_f + idx];
              const double e = fma(fma(fma(fma(fma(fma(fma(c3.y, t, c3.x), t, c2.y), t, c2.x), t, c1.y), t, c1.x), t,
                                       c0.y), t, c0.x);
              vL[c] = fma(wL, e, vL[c]);
              vP[c] = fma(wP, e * e, vP[c]);
            }
            if (ub < ec2) {
              const double2 c0 = s_g[idx], c1 = s_g[nt.n_g + idx], c2 = s_g[2 * nt.n_g + idx];
              phi[c] = fma(q, fma(fma(fma(fma(fma(c2.y, t, c2.x), t, c1.y), t, c1.x), t, c0.y), t, c0.x), phi[c]);
            }
          } else {   // closer than 0.5 A, or parameters outside the table's range
            if (ub < rc2) {
              const double e = exp(-p.alpha * (sqrt(u[c]) - __ldg(&im->R))), eps = __ldg(&im->eps);
              vL[c] += eps * e;
              vP[c] += eps * e * e;
            }
            if (ub < ec2 && q != 0.0) {
              const double d = sqrt(u[c]);
              phi[c] += q * erfc(p.beta * d) / d;
            }
          }
        }
      }
    }
    // reciprocal part: lanes compute the phases e^{i k.rho} of 32 vectors,
    // then every vector's G(z) is added with the broadcast phases
    for (int k0 = 0; k0 < n_k; k0 += 32) {
      double pc[COLS], ps[COLS];
      if (k0 + lane < n_k) {
        const double2 kv = nt.kvec[nt.k_list[k0 + lane]];
#pragma unroll
        for (int c = 0; c < COLS; ++c) sincos(kv.x * x + kv.y * y[c], &ps[c], &pc[c]);
      }
      const int cnt = min(32, n_k - k0);
      for (int t = 0; t < cnt; ++t) {
        const double2 g = nt.G[(size_t)(k0 + t) * p.nz + min(iz, p.nz - 1)];
#pragma unroll
        for (int c = 0; c < COLS; ++c) phi[c] += g.x * bcast(pc[c], t) - g.y * bcast(ps[c], t);
      }
    }
    if (iz < p.nz) {
#pragma unroll
      for (int c = 0; c < COLS; ++c) {
        if (iy0 + c >= p.ny) break;
        const size_t node = ((size_t)ix * p.ny + iy0 + c) * p.nz + iz;
        if (p.coulomb) vals[(size_t)p.slotC * n_nodes + node] = kKe * (phi[c] + p.bg + p.dip * z);
        if (p.morse) {
          vals[(size_t)p.slotP * n_nodes + node] = vP[c];
          vals[(size_t)p.slotL * n_nodes + node] = vL[c];
        }
      }
    }
  }
}

// --------------------------------------------------------------------------
// B-spline line solves (FP64, in place)
// --------------------------------------------------------------------------
// Tridiagonal matrix with constant off-diagonals 1/6 and diagonal bd[k]:
// forward sweep d'_k = (d_k - d'_{k-1}/6) inv[k], back substitution
// y_k = d'_k - cp[k] y_{k+1}.  Cyclic systems add the Sherman-Morrison
// correction x = y - fac (y_0 + (1/6)/gamma y_{n-1}) zc.
struct LineTables {
  const double* inv;
  const double* cp;
  const double* zc;      // nullptr: not cyclic
  double fac, a_over_gamma;
};

__global__ void line_solve_kernel(double* __restrict__ data, int n, long long stride,
                                  long long n_lines, int inner, long long inner_stride,
                                  long long outer_stride, LineTables t) {
  long long line = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (line >= n_lines) return;
  long long o = line / inner, i = line % inner;
  double* d = data + o * outer_stride + i * inner_stride;
  const double a = 1.0 / 6.0;
  double prev = 0.0;
  for (int k = 0; k < n; ++k) {
    double v = (d[k * stride] - a * prev) * t.inv[k];
    d[k * stride] = v;
    prev = v;
  }
  double next = d[(long long)(n - 1) * stride];
  for (int k = n - 2; k >= 0; --k) {
    double v = d[k * stride] - t.cp[k] * next;
    d[k * stride] = v;
    next = v;
  }
  if (t.zc) {
    double s = t.fac * (d[0] + t.a_over_gamma * d[(long long)(n - 1) * stride]);
    for (int k = 0; k < n; ++k) d[k * stride] -= s * t.zc[k];
  }
}

void host_tables(int n, bool cyclic, std::vector<double>& out, double& fac, double& aog) {
  const double a = 1.0 / 6.0, c = 1.0 / 6.0, b = 2.0 / 3.0;
  std::vector<double> bd(n, b);
  double gamma = -b;
  if (cyclic) {
    bd[0] = b - gamma;
    bd[n - 1] = b - a * c / gamma;
  } else {
    bd[0] = b + a;        // clamped end: the index -1 reads b_0
    bd[n - 1] = b + c;    // index n reads b_{n-1}
  }
  std::vector<double> inv(n), cp(n);
  inv[0] = 1.0 / bd[0];
  cp[0] = c * inv[0];
  for (int k = 1; k < n; ++k) {
    double den = bd[k] - a * cp[k - 1];
    inv[k] = 1.0 / den;
    cp[k] = c * inv[k];
  }
  std::vector<double> zc(n, 0.0);
  fac = 0.0;
  aog = 0.0;
  if (cyclic) {
    std::vector<double> u(n, 0.0);
    u[0] = gamma;
    u[n - 1] = c;
    double prev = 0.0;
    for (int k = 0; k < n; ++k) {
      zc[k] = (u[k] - a * prev) * inv[k];
      prev = zc[k];
    }
    for (int k = n - 2; k >= 0; --k) zc[k] -= cp[k] * zc[k + 1];
    aog = a / gamma;
    fac = 1.0 / (1.0 + zc[0] + aog * zc[n - 1]);
  }
  out.clear();
  out.insert(out.end(), inv.begin(), inv.end());
  out.insert(out.end(), cp.begin(), cp.end());
  out.insert(out.end(), zc.begin(), zc.end());
}

// --------------------------------------------------------------------------
// packing into padded records
// --------------------------------------------------------------------------
// Round x to the nearest value with `bits` significant bits (ties to even),
// quantum at least 2^min_exp: the value an FP16 (11, -24) or BF16 (8, -133)
// number nearest to x has; computed exactly in FP64 (x / q is exact for a
// power of two q, rint rounds to even).
__device__ double round_sig(double x, int bits, int min_exp) {
  if (x == 0.0 || !isfinite(x)) return x;
  int e;
  frexp(x, &e);
  const int qe = e - bits > min_exp ? e - bits : min_exp;
  const double q = ldexp(1.0, qe);
  return rint(x / q) * q;
}

template <int KIND>
__global__ void pack_kernel(const double* __restrict__ coefs, int nx, int ny, int nz, int nyp, int nzp,
                            long long n_rec, int slotC, int slotP, int slotL, double iC, double iP, double iL,
                            void* __restrict__ out) {
  long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n_rec) return;
  int pz = (int)(r % nzp);
  int py = (int)((r / nzp) % nyp);
  int px = (int)(r / ((long long)nzp * nyp));
  int ix = (px - 1 + nx) % nx, iy = (py - 1 + ny) % ny;
  int iz = min(max(pz - 1, 0), nz - 1);
  size_t n_nodes = (size_t)nx * ny * nz;
  size_t node = ((size_t)ix * ny + iy) * nz + iz;
  // coefficient / scale (the scales are powers of two: exact)
  const double c = slotC >= 0 ? coefs[(size_t)slotC * n_nodes + node] * iC : 0.0;
  const double p = slotP >= 0 ? coefs[(size_t)slotP * n_nodes + node] * iP : 0.0;
  const double l = slotL >= 0 ? coefs[(size_t)slotL * n_nodes + node] * iL : 0.0;
  if (KIND == REC_F32x4) {
    ((float4*)out)[r] = make_float4((float)c, (float)p, (float)l, 0.f);
  } else if (KIND == REC_F32x2) {
    ((float2*)out)[r] = make_float2((float)p, (float)l);
  } else if (KIND == REC_F16x4 || KIND == REC_F16x2) {
    const __half hc = __double2half(round_sig(c, 11, -24)), hp = __double2half(round_sig(p, 11, -24));
    const __half hl = __double2half(round_sig(l, 11, -24));
    if (KIND == REC_F16x4) {
      ((__half2*)out)[2 * r] = __halves2half2(hc, hp);
      ((__half2*)out)[2 * r + 1] = __halves2half2(hl, __double2half(0.0));
    } else {
      ((__half2*)out)[r] = __halves2half2(hp, hl);
    }
  } else {
    const __nv_bfloat16 bc = __double2bfloat16(round_sig(c, 8, -133));
    const __nv_bfloat16 bp = __double2bfloat16(round_sig(p, 8, -133));
    const __nv_bfloat16 bl = __double2bfloat16(round_sig(l, 8, -133));
    if (KIND == REC_BF16x4) {
      ((__nv_bfloat162*)out)[2 * r] = __halves2bfloat162(bc, bp);
      ((__nv_bfloat162*)out)[2 * r + 1] = __halves2bfloat162(bl, __double2bfloat16(0.0));
    } else {
      ((__nv_bfloat162*)out)[r] = __halves2bfloat162(bp, bl);
    }
  }
}

// max |coefficient| of each channel (bit patterns of non-negative doubles
// order like the values)
__global__ void absmax_kernel(const double* __restrict__ coefs, size_t n_nodes, int n_ch,
                              unsigned long long* __restrict__ out) {
  for (int ch = 0; ch < n_ch; ++ch) {
    double m = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes; i += (size_t)gridDim.x * blockDim.x)
      m = fmax(m, fabs(coefs[(size_t)ch * n_nodes + i]));
    if (m > 0.0) atomicMax(&out[ch], (unsigned long long)__double_as_longlong(m));
  }
}

struct DevFree {
  std::vector<void*> ptrs;
  ~DevFree() {
    for (void* p : ptrs) cudaFree(p);
  }
  template <class T>
  cudaError_t alloc(T** p, size_t bytes) {
    cudaError_t e = cudaMalloc((void**)p, bytes);
    if (e == cudaSuccess) ptrs.push_back(*p);
    return e;
  }
  void release(void* p) { ptrs.erase(std::remove(ptrs.begin(), ptrs.end(), p), ptrs.end()); }
};

void channel_slots(int channels, int& sC, int& sP, int& sL, int& n_ch) {
  n_ch = 0;
  sC = sP = sL = -1;
  if (channels & GRIDFF_CH_C) sC = n_ch++;
  if (channels & GRIDFF_CH_P) sP = n_ch++;
  if (channels & GRIDFF_CH_L) sL = n_ch++;
}

// Allocate grid->rec for the grid's storage layout and pack FP64
// coefficients ([C][nx][ny][nz], device) into it.  FP16/BF16: per-channel
// scale 2^(e - 15) with max |coef| < 2^e, so that |coef| / scale < 2^15.
gridff_status pack_records(gridff_ctx* ctx, gridff_grid* g, const double* data) {
  int nx = g->dims[0], ny = g->dims[1], nz = g->dims[2];
  cudaStream_t s = ctx->stream;
  g->nxp = nx + 3;
  g->nyp = ny + 3;
  g->nzp = nz + 2;
  int sC, sP, sL, nch;
  channel_slots(g->channels, sC, sP, sL, nch);
  const bool two = sC < 0;     // no Coulomb channel: {P, L} records
  g->kind = g->storage == GRIDFF_STORE_F16 ? (two ? REC_F16x2 : REC_F16x4)
          : g->storage == GRIDFF_STORE_BF16 ? (two ? REC_BF16x2 : REC_BF16x4)
                                            : (two ? REC_F32x2 : REC_F32x4);
  double inv[3] = {1.0, 1.0, 1.0};
  g->scale[0] = g->scale[1] = g->scale[2] = 1.f;
  if (g->storage != GRIDFF_STORE_F32) {
    unsigned long long* mx = nullptr;
    GRIDFF_CUDA(ctx, scratch_alloc(ctx, &mx, 3 * sizeof(unsigned long long)));
    cudaError_t e = cudaMemsetAsync(mx, 0, 3 * sizeof(unsigned long long), s);
    if (e == cudaSuccess) {
      absmax_kernel<<<4 * ctx->n_sm, 256, 0, s>>>(data, (size_t)nx * ny * nz, nch, mx);
      e = cudaGetLastError();
    }
    unsigned long long h[3] = {0, 0, 0};
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, mx, 3 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s);
    cudaFreeAsync(mx, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return set_err(ctx, GRIDFF_ECUDA, "channel maxima: %s", cudaGetErrorString(e));
    const int slot_of[3] = {sC, sP, sL};
    for (int c = 0; c < 3; ++c) {
      if (slot_of[c] < 0) continue;
      double m;
      memcpy(&m, &h[slot_of[c]], sizeof(double));
      int ex = 0;
      if (m > 0.0) frexp(m, &ex);
      g->scale[c] = (float)ldexp(1.0, ex - 15);
      inv[c] = ldexp(1.0, 15 - ex);
    }
  }
  long long n_rec = (long long)g->nxp * g->nyp * g->nzp;
  g->rec_bytes = (size_t)n_rec * rec_bytes_of(g->kind);
  GRIDFF_CUDA(ctx, cudaMalloc(&g->rec, g->rec_bytes));
  const unsigned blocks = (unsigned)((n_rec + 255) / 256);
#define GRIDFF_PACK(K)                                                                                \
  pack_kernel<K><<<blocks, 256, 0, s>>>(data, nx, ny, nz, g->nyp, g->nzp, n_rec, sC, sP, sL, inv[0], \
                                         inv[1], inv[2], g->rec)
  switch (g->kind) {
    case REC_F32x4: GRIDFF_PACK(REC_F32x4); break;
    case REC_F32x2: GRIDFF_PACK(REC_F32x2); break;
    case REC_F16x4: GRIDFF_PACK(REC_F16x4); break;
    case REC_F16x2: GRIDFF_PACK(REC_F16x2); break;
    case REC_BF16x4: GRIDFF_PACK(REC_BF16x4); break;
    default: GRIDFF_PACK(REC_BF16x2); break;
  }
#undef GRIDFF_PACK
  GRIDFF_CUDA(ctx, cudaGetLastError());
  return GRIDFF_OK;
}

bool storage_ok(int st) {
  return st == GRIDFF_STORE_F32 || st == GRIDFF_STORE_F16 || st == GRIDFF_STORE_BF16;
}

// Fit coefficients in place (3 passes) and pack them into grid->rec.
gridff_status fit_and_pack(gridff_ctx* ctx, gridff_grid* g, double* data, DevFree& df) {
  int nx = g->dims[0], ny = g->dims[1], nz = g->dims[2];
  int n_ch = g->n_ch;
  cudaStream_t s = ctx->stream;
  // tables for the three axes
  std::vector<double> tz, ty, tx;
  double fz, ay, fy, ax, fx, az;
  host_tables(nz, false, tz, fz, az);
  host_tables(ny, true, ty, fy, ay);
  host_tables(nx, true, tx, fx, ax);
  std::vector<double> all;
  all.insert(all.end(), tz.begin(), tz.end());
  all.insert(all.end(), ty.begin(), ty.end());
  all.insert(all.end(), tx.begin(), tx.end());
  double* dt = nullptr;
  GRIDFF_CUDA(ctx, df.alloc(&dt, all.size() * sizeof(double)));
  GRIDFF_CUDA(ctx, cudaMemcpyAsync(dt, all.data(), all.size() * sizeof(double),
                                   cudaMemcpyHostToDevice, s));
  double* pz = dt;
  double* py = dt + tz.size();
  double* px = py + ty.size();
  long long N = (long long)nx * ny * nz;
  const int TB = 128;
  // z: lines (c, ix, iy), contiguous
  {
    LineTables t{pz, pz + nz, nullptr, 0.0, 0.0};
    long long lines = (long long)n_ch * nx * ny;
    line_solve_kernel<<<(unsigned)((lines + TB - 1) / TB), TB, 0, s>>>(data, nz, 1, lines, 1, 0,
                                                                      nz, t);
  }
  // y: lines (c, ix, iz): outer = c*nx + ix (stride ny*nz), inner = iz
  {
    LineTables t{py, py + ny, py + 2 * ny, fy, ay};
    long long lines = (long long)n_ch * nx * nz;
    line_solve_kernel<<<(unsigned)((lines + TB - 1) / TB), TB, 0, s>>>(
        data, ny, nz, lines, nz, 1, (long long)ny * nz, t);
  }
  // x: lines (c, iy, iz): outer = c (stride N), inner = iy*nz + iz
  {
    LineTables t{px, px + nx, px + 2 * nx, fx, ax};
    long long lines = (long long)n_ch * ny * nz;
    line_solve_kernel<<<(unsigned)((lines + TB - 1) / TB), TB, 0, s>>>(
        data, nx, (long long)ny * nz, lines, ny * nz, 1, N, t);
  }
  GRIDFF_CUDA(ctx, cudaGetLastError());
  return pack_records(ctx, g, data);
}

bool dims_ok(const int* d) { return d[0] >= 4 && d[1] >= 4 && d[2] >= 4; }

// --------------------------------------------------------------------------
// Allocation-free coefficient fit (gridff_fit_coefs_noalloc)
// --------------------------------------------------------------------------
// The per-axis line-solve tables live in this file-scope device array
// instead of memory allocated per call.  Layout per axis a (0 = x, 1 = y,
// 2 = z): inv[n], cp[n], zc[n], then fac and a_over_gamma, at a * kNoAllocStride.
constexpr int kNoAllocMaxN = 4096;
constexpr int kNoAllocStride = 3 * kNoAllocMaxN + 2;
__device__ __align__(256) double g_noalloc_tables[3 * kNoAllocStride];

// One thread per axis builds that axis' tables (same recurrences as host_tables).
__global__ void noalloc_tables_kernel(double* tab, int nx, int ny, int nz) {
  int a = threadIdx.x;
  if (a > 2) return;
  int n = a == 0 ? nx : a == 1 ? ny : nz;
  bool cyclic = a < 2;
  double* inv = tab + (size_t)a * kNoAllocStride;
  double* cp = inv + kNoAllocMaxN;
  double* zc = cp + kNoAllocMaxN;
  double* scal = zc + kNoAllocMaxN;
  const double lo = 1.0 / 6.0, up = 1.0 / 6.0, b = 2.0 / 3.0, gamma = -b;
  for (int k = 0; k < n; ++k) {
    double bd = b;
    if (k == 0) bd = cyclic ? b - gamma : b + lo;
    if (k == n - 1) bd = cyclic ? b - lo * up / gamma : b + up;
    double den = k == 0 ? bd : bd - lo * cp[k - 1];
    inv[k] = 1.0 / den;
    cp[k] = up * inv[k];
  }
  scal[0] = 0.0;
  scal[1] = 0.0;
  if (cyclic) {
    double prev = 0.0;
    for (int k = 0; k < n; ++k) {
      double u = k == 0 ? gamma : (k == n - 1 ? up : 0.0);
      zc[k] = (u - lo * prev) * inv[k];
      prev = zc[k];
    }
    for (int k = n - 2; k >= 0; --k) zc[k] -= cp[k] * zc[k + 1];
    scal[1] = lo / gamma;
    scal[0] = 1.0 / (1.0 + zc[0] + scal[1] * zc[n - 1]);
  }
}

// Line solve that reads its tables (and the cyclic correction scalars) from
// device memory; `cyclic` selects the Sherman-Morrison correction.
__global__ void noalloc_line_kernel(double* __restrict__ data, int n, long long stride, long long n_lines,
                                    int inner, long long inner_stride, long long outer_stride,
                                    const double* __restrict__ tab, int cyclic) {
  long long line = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (line >= n_lines) return;
  const double* inv = tab;
  const double* cp = tab + kNoAllocMaxN;
  const double* zc = cp + kNoAllocMaxN;
  const double* scal = zc + kNoAllocMaxN;
  long long o = line / inner, i = line % inner;
  double* d = data + o * outer_stride + i * inner_stride;
  const double a = 1.0 / 6.0;
  double prev = 0.0;
  for (int k = 0; k < n; ++k) {
    double v = (d[k * stride] - a * prev) * inv[k];
    d[k * stride] = v;
    prev = v;
  }
  double next = d[(long long)(n - 1) * stride];
  for (int k = n - 2; k >= 0; --k) {
    double v = d[k * stride] - cp[k] * next;
    d[k * stride] = v;
    next = v;
  }
  if (cyclic) {
    double s = scal[0] * (d[0] + scal[1] * d[(long long)(n - 1) * stride]);
    for (int k = 0; k < n; ++k) d[k * stride] -= s * zc[k];
  }
}

// Device address of g_noalloc_tables, looked up once per device (the host
// symbol g_noalloc_tables is only a stand-in, never a device address).
double* noalloc_tables_address(int device, cudaError_t* err) {
  static std::mutex mu;
  static double* addr[64] = {nullptr};
  *err = cudaSuccess;
  if (device < 0 || device >= 64) {
    *err = cudaErrorInvalidDevice;
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[device]) {
    void* p = nullptr;
    *err = cudaGetSymbolAddress(&p, g_noalloc_tables);
    if (*err != cudaSuccess) return nullptr;
    addr[device] = (double*)p;
  }
  return addr[device];
}

}  // namespace

GridView gridff_grid::view() const {
  GridView v;
  v.rec = rec;
  v.kind = kind;
  v.sC = scale[0];
  v.sP = scale[1];
  v.sL = scale[2];
  v.nx = dims[0];
  v.ny = dims[1];
  v.nz = dims[2];
  v.nyp = nyp;
  v.nzp = nzp;
  v.sx = (long long)nyp * nzp;
  v.x0 = (float)origin[0];
  v.y0 = (float)origin[1];
  v.z0 = (float)origin[2];
  v.inv_dx = (float)(1.0 / spacing[0]);
  v.inv_dy = (float)(1.0 / spacing[1]);
  v.inv_dz = (float)(1.0 / spacing[2]);
  v.Lx = (float)(spacing[0] * dims[0]);
  v.Ly = (float)(spacing[1] * dims[1]);
  v.inv_Lx = (float)(1.0 / (spacing[0] * dims[0]));
  v.inv_Ly = (float)(1.0 / (spacing[1] * dims[1]));
  v.uzf = (float)ghost;
  return v;
}

extern "C" {

gridff_status gridff_build_grid(gridff_ctx* ctx, const gridff_substrate* sub,
                                const gridff_grid_opts* opts, gridff_grid** out) {
  NvtxRange nvtx_range("gridff_build_grid");
  if (!ctx || !sub || !opts || !out) return set_err(ctx, GRIDFF_EINVAL, "null argument");
  *out = nullptr;
  if (sub->n_atoms <= 0 || !sub->xyz || !sub->q || !sub->R || !sub->eps)
    return set_err(ctx, GRIDFF_EINVAL, "substrate needs n_atoms > 0 and all arrays");
  if (!storage_ok(opts->storage)) return set_err(ctx, GRIDFF_ENOTSUP, "storage not supported");
  if (!(opts->spacing > 0) || !(opts->length[0] > 0) || !(opts->length[1] > 0) ||
      !(opts->length[2] > 0))
    return set_err(ctx, GRIDFF_EINVAL, "grid box lengths and spacing must be > 0");
  const double* C = sub->cell;
  if (C[2] != 0.0 || C[5] != 0.0 || C[6] != 0.0 || C[7] != 0.0 || !(C[8] > 0))
    return set_err(ctx, GRIDFF_EINVAL, "cell rows must be A1, A2 in-plane and A3 = (0, 0, Lz)");
  double area = C[0] * C[4] - C[1] * C[3];
  if (!(fabs(area) > 1e-6)) return set_err(ctx, GRIDFF_EINVAL, "degenerate in-plane cell");
  GRIDFF_CUDA(ctx, cudaSetDevice(ctx->device));

  gridff_grid* g = new gridff_grid();
  g->ctx = ctx;
  g->device = ctx->device;
  g->storage = opts->storage;
  bool charged = false;
  double Qtot = 0.0, Mz = 0.0;
  double zmin = 1e300, zmax = -1e300;
  for (int j = 0; j < sub->n_atoms; ++j) {
    charged |= sub->q[j] != 0.0;
    Qtot += sub->q[j];
    Mz += sub->q[j] * sub->xyz[3 * j + 2];
    zmin = std::min(zmin, sub->xyz[3 * j + 2]);
    zmax = std::max(zmax, sub->xyz[3 * j + 2]);
  }
  int chans = opts->channels ? opts->channels : (GRIDFF_CH_C | GRIDFF_CH_P | GRIDFF_CH_L);
  if (!charged) chans &= ~GRIDFF_CH_C;
  if (!(chans & (GRIDFF_CH_P | GRIDFF_CH_L)) && !(chans & GRIDFF_CH_C)) {
    delete g;
    return set_err(ctx, GRIDFF_EINVAL, "no channel to build");
  }
  // Morse channels come in pairs
  if (chans & (GRIDFF_CH_P | GRIDFF_CH_L)) chans |= GRIDFF_CH_P | GRIDFF_CH_L;
  g->channels = chans;
  int sC, sP, sL;
  channel_slots(chans, sC, sP, sL, g->n_ch);
  if (opts->ghost_below < 0 || opts->ghost_below > 64) {
    delete g;
    return set_err(ctx, GRIDFF_EINVAL, "ghost_below = %d outside 0..64", opts->ghost_below);
  }
  for (int a = 0; a < 3; ++a) {
    g->dims[a] = (int)ceil(opts->length[a] / opts->spacing - 1e-9);
    g->spacing[a] = opts->length[a] / g->dims[a];
    g->origin[a] = opts->origin[a];
  }
  // ghost planes: nodes also below the box; the floor stays at its face
  g->ghost = opts->ghost_below;
  g->floor_z = opts->origin[2];
  g->dims[2] += g->ghost;
  g->origin[2] = opts->origin[2] - g->ghost * g->spacing[2];
  if (!dims_ok(g->dims)) {
    delete g;
    return set_err(ctx, GRIDFF_EINVAL, "grid needs at least 4 nodes per axis");
  }
  if (g->ghost > 0 && !(g->origin[2] > zmax + 0.1)) {
    const double low = g->origin[2];
    delete g;
    return set_err(ctx, GRIDFF_EINVAL,
                   "ghost planes reach z = %g, not above the substrate's highest atom (z = %g) by 0.1 A", low, zmax);
  }
  double alpha = opts->alpha > 0 ? opts->alpha : 1.5;
  double rcut = opts->rcut > 0 ? opts->rcut : 17.0;
  double tol = opts->ewald_tol > 0 ? opts->ewald_tol : 1e-10;
  double ercut = opts->ewald_rcut > 0 ? opts->ewald_rcut : 12.0;
  double s_tol = sqrt(-log(tol));
  double beta = s_tol / ercut;
  double kmax = 2.0 * beta * s_tol;
  double Lz = C[8];
  double ztop = g->origin[2] + g->spacing[2] * (g->dims[2] - 1);
  double zspan = std::max(ztop, zmax) - std::min(g->origin[2], zmin);
  if (charged && Lz - zspan < ercut) {
    delete g;
    return set_err(ctx, GRIDFF_EINVAL,
                   "Ewald height Lz = %g too small: needs >= %g (z span %g + real-space cutoff)",
                   Lz, zspan + ercut, zspan);
  }

  DevFree df;
  cudaStream_t s = ctx->stream;
  size_t n_nodes = (size_t)g->dims[0] * g->dims[1] * g->dims[2];
  double* vals = nullptr;
  const size_t vals_bytes = n_nodes * g->n_ch * sizeof(double);
  if (df.alloc(&vals, vals_bytes) != cudaSuccess) {
    delete g;
    return set_err(ctx, GRIDFF_ENOMEM, "cannot allocate %zu bytes of node values", vals_bytes);
  }
  auto bail = [&](gridff_status st) {
    gridff_grid_destroy(g);
    return st;
  };
  BuildParams p{};
  p.nx = g->dims[0];
  p.ny = g->dims[1];
  p.nz = g->dims[2];
  p.x0 = g->origin[0];
  p.y0 = g->origin[1];
  p.z0 = g->origin[2];
  p.dx = g->spacing[0];
  p.dy = g->spacing[1];
  p.dz = g->spacing[2];
  p.alpha = alpha;
  p.rcut2 = rcut * rcut;
  p.ercut2 = ercut * ercut;
  p.beta = beta;
  p.morse = (chans & GRIDFF_CH_P) ? 1 : 0;
  p.coulomb = (chans & GRIDFF_CH_C) ? 1 : 0;
  p.slotC = sC;
  p.slotP = sP;
  p.slotL = sL;
  double vol = fabs(area) * Lz;
  p.bg = -kPi * Qtot / (beta * beta * vol);
  p.dip = 4.0 * kPi * Mz / vol;

  // lattice images that come within a cutoff of the grid box, by height
  const double cut = std::max(p.morse ? rcut : 0.0, p.coulomb ? ercut : 0.0);
  std::vector<SubImage> h_img;
  double a_R = 0.0;
  {
    std::vector<int> by_z(sub->n_atoms);
    for (int j = 0; j < sub->n_atoms; ++j) by_z[j] = j;
    std::stable_sort(by_z.begin(), by_z.end(), [&](int a, int b) { return sub->xyz[3 * a + 2] < sub->xyz[3 * b + 2]; });
    const double xe = g->origin[0] + opts->length[0], ye = g->origin[1] + opts->length[1];
    const double xs[2] = {g->origin[0], xe}, ys[2] = {g->origin[1], ye};
    double dmax = 0.0;
    for (int j = 0; j < sub->n_atoms; ++j)
      for (double xx : xs)
        for (double yy : ys) dmax = std::max(dmax, hypot(xx - sub->xyz[3 * j], yy - sub->xyz[3 * j + 1]));
    const double h1 = fabs(area) / hypot(C[3], C[4]);   // distance between A1 lattice lines
    const double h2 = fabs(area) / hypot(C[0], C[1]);
    const int n1 = (int)ceil((dmax + cut) / h1), n2 = (int)ceil((dmax + cut) / h2);
    for (int j : by_z) {
      const double* r = sub->xyz + 3 * j;
      const double gz = std::max(0.0, std::max(g->origin[2] - r[2], r[2] - ztop));
      a_R = std::max(a_R, alpha * sub->R[j]);
      SubImage im{0, 0, r[2], sub->q[j], sub->eps[j] * exp(alpha * sub->R[j]), sub->eps[j] * exp(2 * alpha * sub->R[j]),
                  sub->R[j], sub->eps[j]};
      for (int i1 = -n1; i1 <= n1; ++i1)
        for (int i2 = -n2; i2 <= n2; ++i2) {
          im.x = r[0] + i1 * C[0] + i2 * C[3];
          im.y = r[1] + i1 * C[1] + i2 * C[4];
          const double gx = std::max(0.0, std::max(g->origin[0] - im.x, im.x - xe));
          const double gy = std::max(0.0, std::max(g->origin[1] - im.y, im.y - ye));
          if (gx * gx + gy * gy + gz * gz < cut * cut) h_img.push_back(im);
        }
    }
  }
  NodeTables nt{};
  nt.n_img = (int)h_img.size();
  SubImage* d_img = nullptr;
  int* d_next = nullptr;
  if (df.alloc(&d_img, std::max<size_t>(1, h_img.size()) * sizeof(SubImage)) != cudaSuccess ||
      df.alloc(&d_next, sizeof(int)) != cudaSuccess)
    return bail(set_err(ctx, GRIDFF_ENOMEM, "substrate upload"));
  if ((nt.n_img > 0 && cudaMemcpyAsync(d_img, h_img.data(), h_img.size() * sizeof(SubImage), cudaMemcpyHostToDevice, s)) ||
      cudaMemsetAsync(d_next, 0, sizeof(int), s))
    return bail(set_err(ctx, GRIDFF_ECUDA, "substrate upload failed"));
  nt.img = d_img;

  std::vector<D4> h_at;
  std::vector<double2> kvec;
  if (p.coulomb) {
    // reciprocal lattice: B = 2 pi inv(cell)^T; for this cell B3 = (0, 0, 2 pi / Lz)
    const double inv_area = 1.0 / area;
    const double B1x = 2 * kPi * C[4] * inv_area, B1y = -2 * kPi * C[3] * inv_area;
    const double B2x = -2 * kPi * C[1] * inv_area, B2y = 2 * kPi * C[0] * inv_area;
    const double B3z = 2 * kPi / Lz;
    const int M1 = (int)ceil(kmax * hypot(C[0], C[1]) / (2 * kPi)) + 1;
    const int M2 = (int)ceil(kmax * hypot(C[3], C[4]) / (2 * kPi)) + 1;
    const int M3 = (int)ceil(kmax * Lz / (2 * kPi)) + 1;
    for (int m1 = 0; m1 <= M1; ++m1)      // half plane, k2 = 0 first
      for (int m2 = m1 == 0 ? 0 : -M2; m2 <= M2; ++m2) {
        const double kx = m1 * B1x + m2 * B2x, ky = m1 * B1y + m2 * B2y;
        if (kx * kx + ky * ky < kmax * kmax) kvec.push_back(make_double2(kx, ky));
      }
    const int n_k2 = (int)kvec.size(), nm3 = 2 * M3 + 1, na = sub->n_atoms;
    double q_abs = 0.0;
    for (int j = 0; j < na; ++j) {
      h_at.push_back(D4{sub->xyz[3 * j], sub->xyz[3 * j + 1], sub->xyz[3 * j + 2], sub->q[j]});
      q_abs += fabs(sub->q[j]);
    }
    D4* d_at = nullptr;
    double2 *d_kvec = nullptr, *d_EZ = nullptr, *d_EL = nullptr, *d_AS = nullptr, *d_G = nullptr;
    int* d_sel = nullptr;     // keep flags, list, count
    if (df.alloc(&d_at, na * sizeof(D4)) != cudaSuccess || df.alloc(&d_kvec, n_k2 * sizeof(double2)) != cudaSuccess ||
        df.alloc(&d_EZ, (size_t)na * nm3 * sizeof(double2)) != cudaSuccess ||
        df.alloc(&d_EL, (size_t)p.nz * nm3 * sizeof(double2)) != cudaSuccess ||
        df.alloc(&d_AS, (size_t)n_k2 * nm3 * sizeof(double2)) != cudaSuccess ||
        df.alloc(&d_G, (size_t)n_k2 * p.nz * sizeof(double2)) != cudaSuccess ||
        df.alloc(&d_sel, (2 * (size_t)n_k2 + 1) * sizeof(int)) != cudaSuccess)
      return bail(set_err(ctx, GRIDFF_ENOMEM, "reciprocal tables"));
    if (cudaMemcpyAsync(d_at, h_at.data(), na * sizeof(D4), cudaMemcpyHostToDevice, s) ||
        cudaMemcpyAsync(d_kvec, kvec.data(), n_k2 * sizeof(double2), cudaMemcpyHostToDevice, s))
      return bail(set_err(ctx, GRIDFF_ECUDA, "table upload"));
    const double s_min = ldexp(q_abs, -46);
    z_phase_kernel<<<(unsigned)(((size_t)na * nm3 + 127) / 128), 128, 0, s>>>(&d_at->z, 4, na, 0.0, 0.0, M3, B3z, -1.0,
                                                                             d_EZ);
    z_phase_kernel<<<(unsigned)(((size_t)p.nz * nm3 + 127) / 128), 128, 0, s>>>(nullptr, 0, p.nz, p.z0, p.dz, M3, B3z,
                                                                               1.0, d_EL);
    k_struct_kernel<<<n_k2, kStructThreads, 0, s>>>(d_at, na, d_kvec, d_EZ, M3, B3z, kmax * kmax, beta, vol,
                                                    s_min * s_min, d_AS, d_sel);
    k_select_kernel<<<1, 32, 0, s>>>(d_sel, n_k2, d_sel + n_k2, d_sel + 2 * n_k2);
    k_zsum_kernel<<<4 * ctx->n_sm, 128, 0, s>>>(d_AS, d_EL, d_sel + n_k2, d_sel + 2 * n_k2, M3, p.nz, d_G);
    if (cudaGetLastError() != cudaSuccess) return bail(set_err(ctx, GRIDFF_ECUDA, "reciprocal kernels"));
    nt.k_list = d_sel + n_k2;
    nt.n_k = d_sel + 2 * n_k2;
    nt.kvec = d_kvec;
    nt.G = d_G;
  }
  // The radial table holds its error bound up to alpha d = 30 (measured: no
  // larger than the direct form's) and must fit the shared memory of an SM;
  // beyond (long cutoffs, steep exponents) the functions are called directly.
  auto intervals = [](double u) {
    long long bits;
    memcpy(&bits, &u, sizeof(bits));
    return std::max(1, tab_index((int)(bits >> 32)) + 1);
  };
  nt.n_f = p.morse ? intervals(p.rcut2) : 1;
  nt.n_g = p.coulomb ? intervals(p.ercut2) : 1;
  const size_t tab_bytes = ((kFCoef / 2) * (size_t)nt.n_f + (kGCoef / 2) * (size_t)nt.n_g) * sizeof(double2);
  const bool table = alpha * rcut <= 30.0 && s_tol <= 6.0 && a_R <= 100.0 && tab_bytes <= 200 * 1024;
    if (table) {
    double2* d_tab = nullptr;
    if (df.alloc(&d_tab, tab_bytes) != cudaSuccess) return bail(set_err(ctx, GRIDFF_ENOMEM, "radial table"));
    radial_table_kernel<<<(std::max(nt.n_f, nt.n_g) + 63) / 64, 64, 0, s>>>(nt.n_f, nt.n_g, alpha, beta, d_tab);
    nt.tab = d_tab;
    if (allow_dyn_smem((const void*)node_values_kernel<true, kTableCols>, tab_bytes) != cudaSuccess)
      return bail(set_err(ctx, GRIDFF_ECUDA, "radial table of %zu bytes", tab_bytes));
    node_values_kernel<true, kTableCols><<<ctx->n_sm, 32 * kNodeWarps, tab_bytes, s>>>(p, nt, d_next, vals);
  } else {
    node_values_kernel<false, 1><<<ctx->n_sm, 32 * kNodeWarps, 0, s>>>(p, nt, d_next, vals);
  }
  if (cudaGetLastError() != cudaSuccess) return bail(set_err(ctx, GRIDFF_ECUDA, "node kernel launch"));
  if (opts->keep_f64) {
    if (cudaMalloc(&g->f64_values, n_nodes * g->n_ch * sizeof(double)) != cudaSuccess)
      return bail(set_err(ctx, GRIDFF_ENOMEM, "kept node values"));
    if (cudaMemcpyAsync(g->f64_values, vals, n_nodes * g->n_ch * sizeof(double),
                        cudaMemcpyDeviceToDevice, s))
      return bail(set_err(ctx, GRIDFF_ECUDA, "copy of node values"));
  }
  gridff_status st = fit_and_pack(ctx, g, vals, df);
  if (st != GRIDFF_OK) return bail(st);
  if (opts->keep_f64) {
    g->f64_coefs = vals;
    df.release(vals);
  }
  cudaError_t e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return bail(set_err(ctx, GRIDFF_ECUDA, "grid build: %s", cudaGetErrorString(e)));
  *out = g;
  return GRIDFF_OK;
}

gridff_status gridff_grid_from_coefs(gridff_ctx* ctx, const double origin[3], const double spacing[3],
                                     const int32_t dims[3], int32_t channels, const double* coefs,
                                     int32_t storage, gridff_grid** out) {
  NvtxRange nvtx_range("gridff_grid_from_coefs");
  if (!ctx || !origin || !spacing || !dims || !coefs || !out)
    return set_err(ctx, GRIDFF_EINVAL, "null argument");
  *out = nullptr;
  if (!storage_ok(storage)) return set_err(ctx, GRIDFF_ENOTSUP, "storage not supported");
  if (!dims_ok(dims)) return set_err(ctx, GRIDFF_EINVAL, "grid needs at least 4 nodes per axis");
  if (!(channels & 7) || (channels & ~7)) return set_err(ctx, GRIDFF_EINVAL, "bad channel mask");
  for (int a = 0; a < 3; ++a)
    if (!(spacing[a] > 0)) return set_err(ctx, GRIDFF_EINVAL, "spacing must be > 0");
  GRIDFF_CUDA(ctx, cudaSetDevice(ctx->device));
  gridff_grid* g = new gridff_grid();
  g->ctx = ctx;
  g->device = ctx->device;
  g->channels = channels;
  g->storage = storage;
  int sC, sP, sL;
  channel_slots(channels, sC, sP, sL, g->n_ch);
  for (int a = 0; a < 3; ++a) {
    g->dims[a] = dims[a];
    g->origin[a] = origin[a];
    g->spacing[a] = spacing[a];
  }
  g->floor_z = origin[2];
  size_t n = (size_t)dims[0] * dims[1] * dims[2] * g->n_ch;
  DevFree df;
  double* d = nullptr;
  if (df.alloc(&d, n * sizeof(double)) != cudaSuccess) {
    delete g;
    return set_err(ctx, GRIDFF_ENOMEM, "coefficient upload");
  }
  if (cudaMemcpyAsync(d, coefs, n * sizeof(double), cudaMemcpyHostToDevice, ctx->stream) != cudaSuccess) {
    delete g;
    return set_err(ctx, GRIDFF_ECUDA, "coefficient upload");
  }
  // reuse the packing step only (coefficients are given)
  gridff_status pst = pack_records(ctx, g, d);
  if (pst != GRIDFF_OK) {
    gridff_grid_destroy(g);
    return pst;
  }
  cudaError_t e = cudaStreamSynchronize(ctx->stream);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) {
    gridff_grid_destroy(g);
    return set_err(ctx, GRIDFF_ECUDA, "pack: %s", cudaGetErrorString(e));
  }
  *out = g;
  return GRIDFF_OK;
}

gridff_status gridff_fit_coefs_noalloc(gridff_ctx* ctx, const double* values, double* coefs,
                                       const int32_t dims[3], int32_t n_channels, int flags) {
  NvtxRange nvtx_range("gridff_fit_coefs_noalloc");
  if (!ctx || !values || !coefs || !dims) return set_err(ctx, GRIDFF_EINVAL, "null argument");
  if (n_channels < 1) return set_err(ctx, GRIDFF_EINVAL, "n_channels must be >= 1");
  for (int a = 0; a < 3; ++a)
    if (dims[a] < 4 || dims[a] > kNoAllocMaxN)
      return set_err(ctx, GRIDFF_EINVAL,
                     "gridff_fit_coefs_noalloc: dims[%d] = %d outside 4..%d (the size of its fixed "
                     "device table)", a, dims[a], kNoAllocMaxN);
  GRIDFF_CUDA(ctx, cudaSetDevice(ctx->device));
  const size_t bytes = (size_t)dims[0] * dims[1] * dims[2] * n_channels * sizeof(double);
  // both arrays must be memory of this context's device (a host pointer
  // handed to the line-solve kernels would be an out-of-bounds access)
  for (const void* p : {(const void*)values, (const void*)coefs}) {
    cudaPointerAttributes pa{};
    const cudaError_t pe = cudaPointerGetAttributes(&pa, p);
    if (pe != cudaSuccess) cudaGetLastError();
    if (pe != cudaSuccess || (pa.type != cudaMemoryTypeDevice && pa.type != cudaMemoryTypeManaged) ||
        (pa.type == cudaMemoryTypeDevice && pa.device != ctx->device))
      return set_err(ctx, GRIDFF_EINVAL, "gridff_fit_coefs_noalloc: %s is not memory of device %d",
                     p == (const void*)values ? "values" : "coefs", ctx->device);
  }
  {
    // in place (equal pointers) is allowed; partly overlapping ranges are not
    const char *v0 = (const char*)values, *c0 = (const char*)coefs;
    if (v0 != c0 && v0 < c0 + bytes && c0 < v0 + bytes)
      return set_err(ctx, GRIDFF_EINVAL, "gridff_fit_coefs_noalloc: values and coefs overlap without being equal");
  }
  cudaError_t e;
  double* tab = noalloc_tables_address(ctx->device, &e);
  if (!tab) return set_err(ctx, GRIDFF_ECUDA, "cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
  cudaStream_t s = ctx->stream;
  int nx = dims[0], ny = dims[1], nz = dims[2];
  long long N = (long long)nx * ny * nz;
  if (values != coefs)
    GRIDFF_CUDA(ctx, cudaMemcpyAsync(coefs, values, (size_t)N * n_channels * sizeof(double),
                                     cudaMemcpyDeviceToDevice, s));
  noalloc_tables_kernel<<<1, 32, 0, s>>>(tab, nx, ny, nz);
  const int TB = 128;
  long long lines = (long long)n_channels * nx * ny;   // z: contiguous lines
  noalloc_line_kernel<<<(unsigned)((lines + TB - 1) / TB), TB, 0, s>>>(
      coefs, nz, 1, lines, 1, 0, nz, tab + 2 * kNoAllocStride, 0);
  lines = (long long)n_channels * nx * nz;             // y
  noalloc_line_kernel<<<(unsigned)((lines + TB - 1) / TB), TB, 0, s>>>(
      coefs, ny, nz, lines, nz, 1, (long long)ny * nz, tab + kNoAllocStride, 1);
  lines = (long long)n_channels * ny * nz;             // x
  noalloc_line_kernel<<<(unsigned)((lines + TB - 1) / TB), TB, 0, s>>>(
      coefs, nx, (long long)ny * nz, lines, ny * nz, 1, N, tab, 1);
  GRIDFF_CUDA(ctx, cudaGetLastError());
  if (!(flags & GRIDFF_ASYNC)) GRIDFF_CUDA(ctx, cudaStreamSynchronize(s));
  return GRIDFF_OK;
}

gridff_status gridff_grid_floor(const gridff_grid* g, double* z_floor) {
  if (!g || !z_floor) return GRIDFF_EINVAL;
  *z_floor = g->floor_z;
  return GRIDFF_OK;
}

gridff_status gridff_grid_storage(const gridff_grid* g, int32_t* storage, float scales[3]) {
  if (!g) return GRIDFF_EINVAL;
  if (storage) *storage = g->storage;
  if (scales)
    for (int c = 0; c < 3; ++c) scales[c] = g->scale[c];
  return GRIDFF_OK;
}

gridff_status gridff_grid_info(const gridff_grid* g, int32_t dims[3], double origin[3],
                               double spacing[3], int32_t* channels, size_t* device_bytes) {
  if (!g) return GRIDFF_EINVAL;
  for (int a = 0; a < 3; ++a) {
    if (dims) dims[a] = g->dims[a];
    if (origin) origin[a] = g->origin[a];
    if (spacing) spacing[a] = g->spacing[a];
  }
  if (channels) *channels = g->channels;
  if (device_bytes) *device_bytes = g->rec_bytes;
  return GRIDFF_OK;
}

gridff_status gridff_grid_download_f64(const gridff_grid* g, int what, double* host_out) {
  if (!g || !host_out) return GRIDFF_EINVAL;
  const double* src = what == 0 ? g->f64_values : what == 1 ? g->f64_coefs : nullptr;
  if (!src) return set_err(g->ctx, GRIDFF_EINVAL, "FP64 data not kept (set keep_f64 at build)");
  size_t n = (size_t)g->dims[0] * g->dims[1] * g->dims[2] * g->n_ch;
  GRIDFF_CUDA(g->ctx, cudaSetDevice(g->ctx->device));
  GRIDFF_CUDA(g->ctx, cudaMemcpyAsync(host_out, src, n * sizeof(double), cudaMemcpyDeviceToHost,
                                      g->ctx->stream));
  GRIDFF_CUDA(g->ctx, cudaStreamSynchronize(g->ctx->stream));
  return GRIDFF_OK;
}

void gridff_grid_destroy(gridff_grid* g) {
  if (!g) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(g->device);
  if (g->rec) cudaFree(g->rec);
  if (g->f64_values) cudaFree(g->f64_values);
  if (g->f64_coefs) cudaFree(g->f64_coefs);
  cudaSetDevice(prev);
  cudaGetLastError();   // leave no error of this teardown behind
  delete g;
}

}  // extern "C"
