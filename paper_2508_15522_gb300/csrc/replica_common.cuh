// Device code shared by the kernels that evaluate replicas (dynamics.cu,
// flex_team.cu): launch parameters, warp sums, the stencil cache and the
// grid term of one atom by a quad of lanes.
#pragma once

#include <math.h>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "internal.h"
#include "interp.cuh"

namespace {

constexpr int kQuads = 8;                 // atoms evaluated per warp at a time
constexpr int kMaxA = GRIDFF_MAX_ATOMS;
constexpr unsigned kFull = 0xffffffffu;

struct FireP {
  float dt_start, dt_max, f_inc, f_dec, alpha_start, f_alpha, d_max, f_conv2;
  int n_min;
};

struct Control {
  const volatile int* abort_flag;   // host-mapped
  unsigned long long budget_ns;     // 0 = none
  DevResult* res;
};

__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Stop bits of a team (abort flag, clock budget; one thread calls it, every 32
// steps).  The budget counts from the call's start: the result record holds it in a
// split call, whose warp kernel runs first (mark_start_kernel), else the
// first look at the clock sets it.
__device__ __forceinline__ int call_stop_bits(const Control& ctl) {
  int b = *ctl.abort_flag ? GRIDFF_REP_ABORTED : 0;
  if (ctl.budget_ns) {
    const unsigned long long now = gtimer(), first = atomicCAS(&ctl.res->t0, 0ull, now);
    if (first && now > first && now - first > ctl.budget_ns) b |= GRIDFF_REP_STEPLIMIT;
  }
  return b;
}

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ float qsum(float v) {
  v += __shfl_xor_sync(kFull, v, 1);
  v += __shfl_xor_sync(kFull, v, 2);
  return v;
}

// Per-warp stencil cache in shared memory.  Slot i (i < S) holds, for the
// atom evaluated by a quad, the 64 node values c = Q b^C + P b^P + L b^L
// of its 4x4x4 stencil (combined with that atom's fixed factors) and the
// cell they belong to.  Between consecutive steps an atom usually stays in
// its cell, so the gather is served from shared memory; it goes to global
// memory only when the cell changes.  Layout: lane q of the quad holds the
// 16 values of node z+q-1 for the 16 (x, y) runs, as 4 float4; float4 j of
// lane q of slot i sits at index (j * S + i) * 4 + q, so a warp access to 8
// consecutive slots is contiguous (no bank conflicts).
struct StencilCache {
  float4* val;   // [4 * S * 4]
  int* key;      // [S] packed cell index, -1 = empty
  int S;
};

// Channel-combined values c = Q C + P P + L L of the 16 (x, y) runs at one
// z-node: records base + a sx + b nzp, run m = 4a + b, for the grid's record
// kind (channel scales folded into the atom's factors; the branch is
// uniform over the warp).
// KIND >= 0: the record kind is known at compile time (no other code is
// generated); KIND < 0: dispatch on g.kind.
template <int KIND = -1>
__device__ __forceinline__ void gather_runs(const GridView& g, long long base, float4 par, float cv[16]) {
  const float fc = par.x * g.sC, fp = par.y * g.sP, fl = par.z * g.sL;
  switch (KIND >= 0 ? KIND : g.kind) {
    case REC_F32x4: {
      const float4* p = (const float4*)g.rec + base;
      float4 r[16];
#pragma unroll
      for (int m = 0; m < 16; ++m) r[m] = __ldg(p + (m >> 2) * g.sx + (m & 3) * g.nzp);
#pragma unroll
      for (int m = 0; m < 16; ++m) cv[m] = fmaf(fc, r[m].x, fmaf(fp, r[m].y, fl * r[m].z));
      break;
    }
    case REC_F32x2: {
      const float2* p = (const float2*)g.rec + base;
      float2 r[16];
#pragma unroll
      for (int m = 0; m < 16; ++m) r[m] = __ldg(p + (m >> 2) * g.sx + (m & 3) * g.nzp);
#pragma unroll
      for (int m = 0; m < 16; ++m) cv[m] = fmaf(fp, r[m].x, fl * r[m].y);
      break;
    }
    case REC_F16x4:
    case REC_BF16x4: {
      const uint2* p = (const uint2*)g.rec + base;
      uint2 r[16];
#pragma unroll
      for (int m = 0; m < 16; ++m) r[m] = __ldg(p + (m >> 2) * g.sx + (m & 3) * g.nzp);
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        float2 a, b;
        if (g.kind == REC_F16x4) {
          a = __half22float2(*reinterpret_cast<const __half2*>(&r[m].x));
          b = __half22float2(*reinterpret_cast<const __half2*>(&r[m].y));
        } else {
          a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r[m].x));
          b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r[m].y));
        }
        cv[m] = fmaf(fc, a.x, fmaf(fp, a.y, fl * b.x));
      }
      break;
    }
    default: {   // REC_F16x2, REC_BF16x2
      const unsigned* p = (const unsigned*)g.rec + base;
      unsigned r[16];
#pragma unroll
      for (int m = 0; m < 16; ++m) r[m] = __ldg(p + (m >> 2) * g.sx + (m & 3) * g.nzp);
#pragma unroll
      for (int m = 0; m < 16; ++m) {
        const float2 a = g.kind == REC_F16x2 ? __half22float2(*reinterpret_cast<const __half2*>(&r[m]))
                                             : __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r[m]));
        cv[m] = fmaf(fp, a.x, fl * a.y);
      }
      break;
    }
  }
}

// Energy and force of one atom in the substrate field (Eqs. E, E_Coulomb,
// E_Morse), evaluated by the 4 lanes of a quad (q = lane & 3); every lane of
// the quad returns the full result.  Lane q gathers record q of each of
// the 16 z-runs (one warp load fetches 8 whole 64-byte runs), combines the
// channels with the atom's factors (Q, P, L), accumulates the x/y-weighted
// sums for node z+q-1, applies its own z weight, and the quad sums.  The
// force is minus the analytic gradient of the interpolant (Sec. 5).
// `act` false: the quad has no atom (it still takes part in the shuffles).
// `slot` >= 0: the atom may use stencil-cache slot `slot`.
// kPartial: return this lane's share (the 4 shares of a quad sum to the
// atom's value) instead of the quad sum.
template <bool kPartial = false, int KIND = -1>
__device__ __forceinline__ void grid_quad(const GridView& g, int q, bool act, float x, float y, float z,
                                          float4 par, float& e, float& fx, float& fy, float& fz, int& flags,
                                          const StencilCache& sc, int slot) {
  const Cell cl = locate(g, act, x, y, z, flags);
  float wx[4], dwx[4], wy[4], dwy[4], wz[4], dwz[4];
  bspline_weights(cl.tx, wx, dwx);
  bspline_weights(cl.ty, wy, dwy);
  bspline_weights(cl.tz, wz, dwz);
  float cv[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) cv[j] = 0.f;
  if (cl.inside) {
    const int key = (cl.ix * g.ny + cl.iy) * g.nz + cl.iz;
    const bool cached = slot >= 0 && slot < sc.S;
    if (cached && sc.key[slot] == key) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float4 v = sc.val[(j * sc.S + slot) * 4 + q];
        cv[4 * j] = v.x;
        cv[4 * j + 1] = v.y;
        cv[4 * j + 2] = v.z;
        cv[4 * j + 3] = v.w;
      }
    } else {
      gather_runs<KIND>(g, ((long long)cl.ix * g.nyp + cl.iy) * g.nzp + cl.iz + q, par, cv);
      if (cached) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          sc.val[(j * sc.S + slot) * 4 + q] = make_float4(cv[4 * j], cv[4 * j + 1], cv[4 * j + 2], cv[4 * j + 3]);
        if (q == 0) sc.key[slot] = key;
      }
    }
  }
  float S0 = 0.f, Sx = 0.f, Sy = 0.f;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    float s = 0.f, sy = 0.f;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      s = fmaf(wy[b], cv[4 * a + b], s);
      sy = fmaf(dwy[b], cv[4 * a + b], sy);
    }
    S0 = fmaf(wx[a], s, S0);
    Sx = fmaf(dwx[a], s, Sx);
    Sy = fmaf(wx[a], sy, Sy);
  }
  const float wq = q == 0 ? wz[0] : q == 1 ? wz[1] : q == 2 ? wz[2] : wz[3];
  const float dwq = q == 0 ? dwz[0] : q == 1 ? dwz[1] : q == 2 ? dwz[2] : dwz[3];
  e = wq * S0;
  fx = -wq * Sx * g.inv_dx;
  fy = -wq * Sy * g.inv_dy;
  fz = -dwq * S0 * g.inv_dz;
  if (!kPartial) {
    e = qsum(e);
    fx = qsum(fx);
    fy = qsum(fy);
    fz = qsum(fz);
  }
}

// Entry of the rigid kernels' refill list: record index of the stencil's first
// node, atom slot (8 bits) and sub-warp (2).  WIDE: 54 bits of index, for grids of
// more than 2^32 records (17 GB of 16-bit pairs); else 32, which is 1.4 to 2.4 % of a
// relaxation's or a run's time faster (the index is in every gather's address).
template <bool WIDE>
__host__ __device__ __forceinline__ int2 refill_entry(long long record, int slot, int sw) {
  const unsigned high = WIDE ? (unsigned)(record >> 32) << 10 : 0u;
  return make_int2((int)(unsigned)record, (int)(high | (unsigned)sw << 8 | (unsigned)slot));
}
template <bool WIDE>
__host__ __device__ __forceinline__ long long refill_record(int2 e) {
  return WIDE ? (long long)((unsigned long long)((unsigned)e.y >> 10) << 32 | (unsigned)e.x) : (long long)(unsigned)e.x;
}
__host__ __device__ __forceinline__ int refill_slot(int2 e) { return e.y & 0xff; }
template <bool WIDE>
__host__ __device__ __forceinline__ int refill_sub(int2 e) { return WIDE ? (e.y >> 8) & 3 : e.y >> 8; }

// Bytes of one warp's cache with S slots (a multiple of 16).
__host__ __device__ constexpr size_t cache_bytes(int S) { return (size_t)S * 256 + (((size_t)S * 4 + 15) & ~size_t(15)); }

__device__ __forceinline__ float3 ld3(const float* s, int i) {
  return make_float3(s[3 * i], s[3 * i + 1], s[3 * i + 2]);
}
__device__ __forceinline__ float3 sub3(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross3(float3 a, float3 b) {
  return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

// cos(n phi) and sin(n phi) from cos phi and sin phi by n rotations in the
// complex plane (exact trigonometry, no angle): (c, s) <- (c, s) e^{i phi}.
__device__ __forceinline__ void multiple_angle(float cphi, float sphi, int n, float& cn, float& sn) {
  cn = 1.f;
  sn = 0.f;
  for (int k = 0; k < n; ++k) {
    const float c2 = fmaf(cn, cphi, -sn * sphi);
    sn = fmaf(sn, cphi, cn * sphi);
    cn = c2;
  }
}

__device__ __forceinline__ bool finite3(float a, float b, float c) {
  return isfinite(a) && isfinite(b) && isfinite(c);
}

__device__ __forceinline__ void report(const Control& ctl, int n, int evals, int st, int steps) {
  atomicAdd(&ctl.res->atom_evals, (unsigned long long)n * (unsigned long long)evals);
  if (st & GRIDFF_REP_CONVERGED) atomicAdd(&ctl.res->n_converged, 1);
  atomicMax(&ctl.res->max_steps, steps);
  int sb = st & (GRIDFF_REP_ABORTED | GRIDFF_REP_STEPLIMIT);
  if (sb) atomicOr(&ctl.res->stop_bits, sb);
}

// 2^x by the PTX instruction ex2.approx.ftz.f32 (relative error about 2^-22).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
constexpr float kLog2e = 1.44269504088896341f;   // log2(e)

// e^{-alpha (r - R_i - R_j)} of a pair: relaxations and Langevin dynamics take the
// factors prepared, b = alpha log2(e) R, and one ex2 (rounding 3e-7 of the
// exponential); evaluations and constant-energy dynamics, which are read as
// results, the difference in FP32 and expf, b = R.  Either way an evaluation of
// 4097 uneven molecules took 106 us (117 with the divisions and FP64 sums below) and
// constant-energy dynamics of 1024 x 47 atoms takes 27 us a step: neither is bound by the
// pairs' instructions.
template <class Acc>
constexpr bool kReadOut = sizeof(Acc) > sizeof(float);
template <bool EX>
__device__ __forceinline__ float pair_exp(float alpha, float a, float r, float bi, float bj) {
  return EX ? expf(-alpha * (r - bi - bj)) : ex2_approx(fmaf(-a, r, bi + bj));
}

// Force factor c (F_i = c d) and stretch dr of a bond of squared length r2; a bond
// of zero length has no direction and no force.  EX as above, with the length by
// sqrtf: r2 rsqrt(r2) is two roundings worse, which a stiff bond turns into most
// of an evaluation's error (relative, of 4097 uneven molecules: 1.3e-6, with sqrtf 1.1e-6,
// in the same time).
template <bool EX>
__device__ __forceinline__ void bond_factor(float r2, float k, float r0, float& c, float& dr) {
  if (EX) {
    const float r = sqrtf(r2);
    dr = r - r0;
    c = r > 0.f ? -2.f * k * dr / r : 0.f;
  } else {
    const float ir = r2 > 0.f ? rsqrtf(r2) : 0.f;
    dr = r2 * ir - r0;
    c = -2.f * k * dr * ir;
  }
}

// One angle (u = x_a - x_b, w = x_c - x_b): gradients ga, gc of cos(theta) with
// respect to atoms a and c (b: minus their sum), dE/dcos; returns the energy.
// EX as above: divisions by u^2 and w^2, elsewhere products of reciprocal square roots.
template <bool EX>
__device__ __forceinline__ float angle_term(float3 u, float3 w, float k, float cos0, float3& ga, float3& gc, float& dEdc) {
  const float u2 = dot3(u, u), w2 = dot3(w, w);
  float inv, c, cu, cw;
  if (EX) {
    inv = rsqrtf(u2 * w2);
    c = dot3(u, w) * inv;
    cu = c / u2;
    cw = c / w2;
  } else {
    const float ru = rsqrtf(u2), rw = rsqrtf(w2);
    inv = ru * rw;
    c = dot3(u, w) * inv;
    cu = c * (ru * ru);
    cw = c * (rw * rw);
  }
  dEdc = 2.f * k * (c - cos0);
  ga = make_float3(w.x * inv - cu * u.x, w.y * inv - cu * u.y, w.z * inv - cu * u.z);
  gc = make_float3(u.x * inv - cw * w.x, u.y * inv - cw * w.y, u.z * inv - cw * w.z);
  return k * (c - cos0) * (c - cos0);
}

// One torsion: its energy is added to e; add(k, x, y, z) takes the force on its k-th
// atom, in turn.  (Forces of all four at once, alive across the warp pass's atomics, or
// the factors below before multiple_angle's loop cost the uneven batch's relaxation 0.3
// to 0.4 %.)  Collinear atoms (no dihedral) have no torque: no forces are added, or
// (ZEROS) zeros.  EX as above: square root and divisions.  Relative error of an atom's
// force, median: 2.1e-7 by divisions, 2.7e-7 by reciprocal square roots.
template <bool EX, bool ZEROS, class Acc, class Add>
__device__ __forceinline__ void torsion_term(float3 xa, float3 xb, float3 xc, float3 xd, const TorsionRec& T, Acc& e,
                                             Add add) {
  const float3 F = sub3(xa, xb), G = sub3(xb, xc), H = sub3(xd, xc);
  const float3 A = cross3(F, G), B = cross3(H, G);
  const float A2 = dot3(A, A), B2 = dot3(B, B), G2 = dot3(G, G);
  if (A2 < 1e-12f || B2 < 1e-12f || G2 < 1e-12f) {
    if (ZEROS)
      for (int k = 0; k < 4; ++k) add(k, 0.f, 0.f, 0.f);
    return;
  }
  float sn, cn, dEdphi, FG, HG, ca, cd;
  if (EX) {
    const float Gn = sqrtf(G2), iAB = rsqrtf(A2 * B2);
    multiple_angle(dot3(A, B) * iAB, dot3(cross3(B, A), G) * iAB / Gn, T.n, cn, sn);
    dEdphi = 0.5f * T.V * T.cn0 * T.n * sn;
    FG = dot3(F, G) / (A2 * Gn);
    HG = dot3(H, G) / (B2 * Gn);
    ca = -Gn / A2;
    cd = Gn / B2;
  } else {
    const float rA = rsqrtf(A2), rB = rsqrtf(B2), rG = rsqrtf(G2);
    const float iA2 = rA * rA, iB2 = rB * rB, Gn = G2 * rG, iAB = rA * rB;
    multiple_angle(dot3(A, B) * iAB, dot3(cross3(B, A), G) * iAB * rG, T.n, cn, sn);
    dEdphi = 0.5f * T.V * T.cn0 * T.n * sn;
    FG = dot3(F, G) * iA2 * rG;
    HG = dot3(H, G) * iB2 * rG;
    ca = -Gn * iA2;
    cd = Gn * iB2;
  }
  const float a1 = -ca + FG, b1 = -cd + HG;
  // gradients of phi with respect to the four atoms, times -dE/dphi
  const float m0 = -dEdphi * ca, m3 = -dEdphi * cd, m1 = -dEdphi * a1, m2 = -dEdphi * b1;
  const float h1 = dEdphi * HG, h2 = dEdphi * FG;
  add(0, m0 * A.x, m0 * A.y, m0 * A.z);
  add(1, m1 * A.x + h1 * B.x, m1 * A.y + h1 * B.y, m1 * A.z + h1 * B.z);
  add(2, m2 * B.x + h2 * A.x, m2 * B.y + h2 * A.y, m2 * B.z + h2 * A.z);
  add(3, m3 * B.x, m3 * B.y, m3 * B.z);
  e += (Acc)(0.5f * T.V * (1.f - T.cn0 * cn));
}

}  // namespace
