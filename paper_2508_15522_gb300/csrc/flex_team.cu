// Flexible replicas by teams: one block of NW warps per replica, for batches
// that leave warps of the chip without a replica.  Force evaluation, FIRE
// relaxation (Sec. 6), NVE and Langevin dynamics (Sec. 7) with the same
// arithmetic per term and the same updates as the warp-per-replica kernels.
//
// A step of one replica on one warp is a chain of dependent phases (a 22-atom
// molecule: 10.5 us, of which 2.1 the grid term, 1.6 the pairs, 4.6 the bonded
// terms with their shared-memory float atomics, and 1.6 the update with the
// velocities in global memory), and a batch that fits the chip once pays that
// latency whatever its size.  Here the team's warps share every phase:
//   1. grid term by quads of lanes over the atoms, stencils cached in shared
//      memory; nonbonded pairs, the steps of the pair rings split evenly over
//      the warps, each with force sums of its own; bonded terms one per
//      thread, their forces written to slots (no atomics);
//   2. after a barrier, a quad per atom gathers that atom's force: the grid's,
//      the warps' sums and the slots that name the atom (a list per template);
//   3. sums over the team, the update, a barrier.
// Bound by that chain's latency: 22 atoms 3.4 us a step on 4 warps (grid 0.6,
// pairs 0.4, bonded 0.8, the rest sums, barriers and update); 120 atoms 10 us on
// 8 warps (60.8 on one), more than half of it pairs.
#include <type_traits>

#include "replica_common.cuh"

namespace {

enum TeamMode { TEAM_RELAX, TEAM_LANGEVIN, TEAM_NVE, TEAM_EVAL };

struct TeamArgs {
  const int* rep_tmpl;
  const int* rep_off;
  const int* order;
  int n_rep, N, S, n_slots;     // N: atoms per team (a multiple of 32), S: stencil-cache slots
  float *xs, *vs;
  float *fdt, *falpha;
  int *fnp, *status, *steps;
  double* energy;
  float *last_x, *last_f;
  int nsteps, use_grid, use_intra;
  // dynamics
  float dt, c1, c2, kT_acc;
  unsigned long long seed;
  long long step0;
  int rec_every;
  double* trace;
  int trace_stride;
  // evaluation
  double* E;
  float *F, *Ea;
  int* st_out;
};

// Shared memory of a team: stencil cache, positions and charges, pair
// factors, inverse masses, velocities, grid (then total) forces, the warps'
// pair forces, bonded slots, reduction words.
struct TeamState {
  StencilCache sc;
  float4* x;        // [N] {x, y, z, q}
  float2* nb;       // [N] {alpha log2(e) R, eps} (TEAM_NVE, TEAM_EVAL: {R, eps})
  float* im;        // [N] 1/m; 1/sqrt(m) (Langevin); dt/2 / m (NVE)
  float* v;         // [3N]
  float* f;         // [3N] grid force, then the total
  float* fw;        // [NW][3N]
  float* slot;      // [3 n_slots]
  double* redd;     // [NW]
  float4* red;      // [NW] {f2, P, v2, flags}
  int* word;        // [1]
};

__host__ __device__ constexpr size_t team_bytes(int NW, int N, int S, int n_slots) {
  return cache_bytes(S) + (size_t)N * (16 + 8 + 4 + 12 + 12) + (size_t)NW * N * 12 + (((size_t)n_slots * 12 + 15) & ~size_t(15)) +
         (size_t)NW * 8 + (size_t)NW * 16 + 16;
}

__device__ __forceinline__ TeamState team_state(unsigned char* p, int NW, int N, int S, int n_slots) {
  TeamState s;
  s.sc.val = (float4*)p;
  s.sc.key = (int*)(p + (size_t)S * 256);
  s.sc.S = S;
  p += cache_bytes(S);
  s.x = (float4*)p;
  p += (size_t)N * 16;
  s.red = (float4*)p;
  p += (size_t)NW * 16;
  s.nb = (float2*)p;
  p += (size_t)N * 8;
  s.redd = (double*)p;
  p += (size_t)NW * 8;
  s.im = (float*)p;
  p += (size_t)N * 4;
  s.v = (float*)p;
  p += (size_t)N * 12;
  s.f = (float*)p;
  p += (size_t)N * 12;
  s.fw = (float*)p;
  p += (size_t)NW * N * 12;
  s.slot = (float*)p;
  p += (size_t)n_slots * 12;
  s.word = (int*)p;
  return s;
}

__device__ __forceinline__ float3 xyz(float4 v) { return make_float3(v.x, v.y, v.z); }
__device__ __forceinline__ void put3(float* p, int i, float x, float y, float z) {
  p[3 * i] = x;
  p[3 * i + 1] = y;
  p[3 * i + 2] = z;
}
__device__ __forceinline__ void add3(float* p, int i, float3 g) {
  p[3 * i] += g.x;
  p[3 * i + 1] += g.y;
  p[3 * i + 2] += g.z;
}

// This warp's part of the nonbonded pairs (steps w T / NW .. (w + 1) T / NW of
// the molecule's T ring steps), forces added to f (this warp's own array,
// zeroed here); returns this lane's share of the energy.
//
// Blocks of 32 atoms, lane l owns atom 32 I + l.  Block pair I < J: partners
// (l + d) mod r of block J, d = 0 .. r - 1, r = 32, or the next power of two of
// a last block of at most 16 atoms; inside a block of m atoms partners
// (l + d) mod m, d = 1 .. m / 2 (d = m / 2 for even m from l < m / 2 only).  At
// a given d the lanes of a ring have distinct partners; the reaction sum G of
// a partner travels with it from lane to lane, so a part of the steps stands
// by itself.
template <int NW, class Acc>
__device__ __forceinline__ Acc team_pairs(const TeamState& s, const TemplateView& tv, int ab, int n, int lane, int w,
                                          float* f) {
  for (int i = lane; i < 3 * n; i += 32) f[i] = 0.f;
  __syncwarp();
  const int nblk = (n + 31) >> 5, ml = n - 32 * (nblk - 1);    // atoms of the last block
  const int rl = ml > 16 ? 32 : ml <= 1 ? 1 : 1 << (32 - __clz(ml - 1));
  // ring steps: inside the blocks, between full blocks, with the last block
  const int T = (nblk - 1) * 16 + (ml >> 1) + ((nblk - 1) * (nblk - 2) / 2) * 32 + (nblk - 1) * rl;
  const int t0 = T * w / NW, t1 = T * (w + 1) / NW;
  const float alpha = tv.alpha, a = alpha * kLog2e;
  Acc e = Acc(0);
  int cum = 0;
  for (int I = 0; I < nblk && cum < t1; ++I)
    for (int J = I; J < nblk && cum < t1; ++J) {
      const bool diag = I == J;
      const int base = 32 * J, m = min(32, n - base);
      const int ring = diag ? m : J == nblk - 1 ? rl : 32, total = diag ? m >> 1 : ring;
      const int lo = max(t0 - cum, 0), hi = min(t1 - cum, total);
      cum += total;
      if (lo >= hi) continue;
      const int i = 32 * I + lane;
      const bool own = i < n;
      const int ii = own ? i : 32 * I;
      const float3 xi = xyz(s.x[ii]);
      const float2 p2 = s.nb[ii];
      const float qi = GRIDFF_KE * s.x[ii].w;
      const uint32_t ok = (m >= 32 ? 0xffffffffu : (1u << m) - 1u) & ~__ldg(&tv.excl[4 * (size_t)(ab + ii) + J]);
      uint32_t act;
      int pos, src;
      if (diag) {
        const int h = m >> 1;
        act = (uint32_t)((((unsigned long long)ok | ((unsigned long long)ok << m)) >> lane) >> 1);   // bit k: d = k + 1
        if (!(m & 1) && lane >= h) act &= ~(1u << (h - 1));
        pos = lane < m ? (lane + 1 + lo) % m : 0;
        src = lane < m ? (lane + 1 == m ? 0 : lane + 1) : lane;
      } else {
        const int lr = lane & (ring - 1);
        act = ring == 32 ? __funnelshift_r(ok, ok, lane) : (ok | (ok << ring)) >> lr;
        pos = (lr + lo) & (ring - 1);
        src = (lane & ~(ring - 1)) | ((lr + 1) & (ring - 1));
      }
      act = own ? act >> lo : 0u;
      float3 fi = make_float3(0.f, 0.f, 0.f), G = fi;
      float ep = 0.f;
      int sl = pos;
#pragma unroll 2
      for (int d = lo; d < hi; ++d) {
        pos = sl;
        const float4 P = s.x[base + sl];
        const float2 Q = s.nb[base + sl];
        sl = sl + 1 == ring ? 0 : sl + 1;
        const float3 dv = sub3(xi, xyz(P));
        const float r2 = dot3(dv, dv);
        const float ir = rsqrtf(r2), r = r2 * ir;
        const float e1 = pair_exp<kReadOut<Acc>>(alpha, a, r, p2.x, Q.x);
        const float ee = p2.y * Q.y, qr = qi * P.w * ir;      // k_e q_i q_j / r
        const bool on = act & 1u;
        act >>= 1;
        const float c = on ? -(2.f * alpha * ee * e1 * (1.f - e1) - qr * ir) * ir : 0.f;
        ep += on ? ee * e1 * (e1 - 2.f) + qr : 0.f;
        fi.x = fmaf(c, dv.x, fi.x);
        fi.y = fmaf(c, dv.y, fi.y);
        fi.z = fmaf(c, dv.z, fi.z);
        G.x = fmaf(-c, dv.x, __shfl_sync(kFull, G.x, src));
        G.y = fmaf(-c, dv.y, __shfl_sync(kFull, G.y, src));
        G.z = fmaf(-c, dv.z, __shfl_sync(kFull, G.z, src));
      }
      e += (Acc)ep;
      if (!diag)
        for (int o = ring; o < 32; o <<= 1) {      // repeated rings met the same partners
          G.x += __shfl_xor_sync(kFull, G.x, o);
          G.y += __shfl_xor_sync(kFull, G.y, o);
          G.z += __shfl_xor_sync(kFull, G.z, o);
        }
      if (lane < ring && base + pos < n) add3(f, base + pos, G);
      __syncwarp();
      if (own) add3(f, i, fi);
      __syncwarp();
    }
  return e;
}

// Bonded terms of template t, one per thread of the team: forces on the term's
// atoms to the term's slots (bonds: the force on atom i; angles: a, b, c;
// torsions: a, b, c, d).  Returns this thread's share of the energy.
template <class Acc>
__device__ __forceinline__ Acc team_bonded(const TeamState& s, const TemplateView& tv, int t, int tid, int threads) {
  const int b0 = tv.ub_off[t], a0 = tv.ua_off[t], k0 = tv.ut_off[t];
  const int nb = tv.ub_off[t + 1] - b0, na = tv.ua_off[t + 1] - a0, nt = tv.ut_off[t + 1] - k0;
  constexpr bool EX = kReadOut<Acc>;
  Acc e = Acc(0);
  for (int k = tid; k < nb + na + nt; k += threads) {
    if (k < nt) {
      const TorsionRec T = tv.ut[k0 + k];
      const int o = nb + 3 * na + 4 * k;
      torsion_term<EX, true>(xyz(s.x[T.a]), xyz(s.x[T.b]), xyz(s.x[T.c]), xyz(s.x[T.d]), T, e,
                             [&](int i, float x, float y, float z) { put3(s.slot, o + i, x, y, z); });
    } else if (k < nt + na) {
      const int j = k - nt, o = nb + 3 * j;
      const AngleRec A = tv.ua[a0 + j];
      const float3 xb = xyz(s.x[A.b]);
      const float3 u = sub3(xyz(s.x[A.a]), xb), w = sub3(xyz(s.x[A.c]), xb);
      float3 ga, gc;
      float dEdc;
      e += (Acc)angle_term<EX>(u, w, A.k, A.cos0, ga, gc, dEdc);
      put3(s.slot, o, -dEdc * ga.x, -dEdc * ga.y, -dEdc * ga.z);
      put3(s.slot, o + 1, dEdc * (ga.x + gc.x), dEdc * (ga.y + gc.y), dEdc * (ga.z + gc.z));
      put3(s.slot, o + 2, -dEdc * gc.x, -dEdc * gc.y, -dEdc * gc.z);
    } else {
      const int j = k - nt - na;
      const BondTerm B = tv.ub[b0 + j];
      const float3 d = sub3(xyz(s.x[B.i]), xyz(s.x[B.j]));
      float c, dr;
      bond_factor<EX>(dot3(d, d), B.k, B.r0, c, dr);
      put3(s.slot, j, c * d.x, c * d.y, c * d.z);
      e += (Acc)(B.k * dr * dr);
    }
  }
  return e;
}

// Forces of the team's replica at s.x: total forces in s.f, sums over this
// thread's atoms of F^2, F.v and v^2; returns this thread's share of the
// energy.  Two phases with a barrier between; the caller's next barrier makes
// s.f visible.
template <int NW, int KIND, class Acc>
__device__ __forceinline__ Acc team_forces(const GridView& g, const TemplateView& tv, const TeamArgs& A, TeamState& s,
                                           int t, int ab, int n, int tid, int& flags, float* Ea, float& f2, float& P,
                                           float& v2) {
  const int lane = tid & 31, w = tid >> 5, q = tid & 3;
  Acc e = Acc(0);
  for (int base = 0; base < n; base += kQuads * NW) {
    const int i = base + (tid >> 2);
    const bool act = i < n;
    float4 p = make_float4(0.f, 0.f, 0.f, 0.f), par = p;
    if (act) {
      p = s.x[i];
      par = __ldg(&tv.par[ab + i]);
      if (!finite3(p.x, p.y, p.z)) flags |= GRIDFF_REP_NONFINITE;
    }
    float eg = 0.f, fx = 0.f, fy = 0.f, fz = 0.f;
    if (A.use_grid) grid_quad<false, KIND>(g, q, act, p.x, p.y, p.z, par, eg, fx, fy, fz, flags, s.sc, i);
    if (act && q == 0) {
      put3(s.f, i, fx, fy, fz);
      if (Ea) Ea[i] = eg;
      e += (Acc)eg;
    }
  }
  float* const fw = s.fw + (size_t)w * 3 * A.N;
  if (A.use_intra) {
    e += team_pairs<NW, Acc>(s, tv, ab, n, lane, w, fw);
    e += team_bonded<Acc>(s, tv, t, tid, 32 * NW);
  }
  __syncthreads();
  f2 = P = v2 = 0.f;
  for (int base = 0; base < n; base += kQuads * NW) {
    const int i = base + (tid >> 2);
    const bool act = i < n;
    float3 F = make_float3(0.f, 0.f, 0.f);
    if (act && A.use_intra) {
      const int g1 = tv.gat_off[ab + i + 1];
      for (int k = tv.gat_off[ab + i] + q; k < g1; k += 4) {
        const int ref = __ldg(&tv.gat[k]);
        const float sg = (ref & 1) ? -1.f : 1.f;
        const float* p = s.slot + 3 * (ref >> 1);
        F.x = fmaf(sg, p[0], F.x);
        F.y = fmaf(sg, p[1], F.y);
        F.z = fmaf(sg, p[2], F.z);
      }
      for (int k = q; k < NW; k += 4) {
        const float* p = s.fw + (size_t)k * 3 * A.N + 3 * i;
        F.x += p[0];
        F.y += p[1];
        F.z += p[2];
      }
    }
    F.x = qsum(F.x);
    F.y = qsum(F.y);
    F.z = qsum(F.z);
    if (act && q == 0) {
      add3(s.f, i, F);
      const float* p = s.f + 3 * i;
      const float* v = s.v + 3 * i;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        f2 = fmaf(p[c], p[c], f2);
        P = fmaf(p[c], v[c], P);
        v2 = fmaf(v[c], v[c], v2);
      }
    }
  }
  return e;
}

// Sums over the team of three values and the union of the flags, in every
// thread; a barrier.  (The words are written again only after another one.)
template <int NW>
__device__ __forceinline__ void team_sum(const TeamState& s, int tid, float& a, float& b, float& c, int& flags) {
  a = wsum(a);
  b = wsum(b);
  c = wsum(c);
  flags = __reduce_or_sync(kFull, flags);
  if ((tid & 31) == 0) s.red[tid >> 5] = make_float4(a, b, c, __int_as_float(flags));
  __syncthreads();
  a = b = c = 0.f;
  flags = 0;
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    const float4 r = s.red[k];
    a += r.x;
    b += r.y;
    c += r.z;
    flags |= __float_as_int(r.w);
  }
}

template <int NW>
__device__ __forceinline__ double team_sum_d(const TeamState& s, int tid, double v) {
  v = wsum(v);
  if ((tid & 31) == 0) s.redd[tid >> 5] = v;
  __syncthreads();
  v = 0.0;
#pragma unroll
  for (int k = 0; k < NW; ++k) v += s.redd[k];
  __syncthreads();
  return v;
}

template <int NW, int KIND, int MODE>
__global__ void __launch_bounds__(32 * NW, 32 / NW) flex_team_kernel(GridView g, TemplateView tv, TeamArgs A, FireP fp,
                                                                     Control ctl) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  using Acc = typename std::conditional<MODE == TEAM_NVE || MODE == TEAM_EVAL, double, float>::type;
  constexpr int kThr = 32 * NW;
  const int tid = threadIdx.x;
  TeamState s = team_state(dyn_smem, NW, A.N, A.S, A.n_slots);
  // stop bits every 32 steps (abort flag, clock budget), the same in every thread
  auto stop = [&]() {
    if (tid == 0) *s.word = call_stop_bits(ctl);
    __syncthreads();
    const int b = *s.word;
    __syncthreads();
    return b;
  };
  // more replicas than teams: a queue, largest molecules first (an evaluation
  // has no queue word of its own and takes every gridDim-th)
  const bool queued = MODE != TEAM_EVAL && gridDim.x < (unsigned)A.n_rep;
  for (int j = blockIdx.x;; j += gridDim.x) {
    int k = j;
    if (queued) {
      if (tid == 0) *s.word = atomicAdd(&ctl.res->team_next, 1);
      __syncthreads();
      k = *s.word;
      __syncthreads();
    }
    if (k >= A.n_rep) break;
    const int r = A.order[k];
    const int t = A.rep_tmpl[r], n = tv.natoms[t], ab = tv.atom_off[t], off = A.rep_off[r];
    for (int i = tid; i < A.S; i += kThr) s.sc.key[i] = -1;
    for (int i = tid; i < A.N; i += kThr) {
      const bool in = i < n;
      const float4 p = in ? __ldg(&tv.nb[ab + i]) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float m = in ? __ldg(&tv.body[ab + i]).w : 1.f;
      const float* x = A.xs + 3 * ((size_t)off + i);
      s.x[i] = in ? make_float4(x[0], x[1], x[2], p.x) : p;
      s.nb[i] = make_float2(kReadOut<Acc> ? p.y : p.y * (tv.alpha * kLog2e), p.z);
      s.im[i] = MODE == TEAM_LANGEVIN ? rsqrtf(m) : MODE == TEAM_NVE ? 0.5f * A.dt * GRIDFF_ACC / m : 1.f / m;
      for (int c = 0; c < 3; ++c) s.v[3 * i + c] = in && MODE != TEAM_EVAL ? A.vs[3 * ((size_t)off + i) + c] : 0.f;
    }
    __syncthreads();
    float f2, P, v2;
    if (MODE == TEAM_RELAX) {
      float dt = A.fdt[r], al = A.falpha[r];
      int np = A.fnp[r], st = A.status[r], evals = 0;
      Acc e = Acc(0);
      for (int it = 0; it < A.nsteps; ++it) {
        if (st & (GRIDFF_REP_CONVERGED | GRIDFF_REP_NONFINITE)) break;
        if ((it & 31) == 0) {
          const int sb = stop();
          if (sb) {
            st |= sb;
            break;
          }
        }
        int flags = 0;
        e = team_forces<NW, KIND, Acc>(g, tv, A, s, t, ab, n, tid, flags, nullptr, f2, P, v2);
        team_sum<NW>(s, tid, f2, P, v2, flags);
        st |= flags;
        ++evals;
        if (it == A.nsteps - 1 || (st & GRIDFF_REP_NONFINITE) || !(f2 >= fp.f_conv2)) {
          for (int i = tid; i < n; i += kThr) {      // the final evaluation's state and forces
            put3(A.last_x, off + i, s.x[i].x, s.x[i].y, s.x[i].z);
            put3(A.last_f, off + i, s.f[3 * i], s.f[3 * i + 1], s.f[3 * i + 2]);
          }
        }
        if ((st & GRIDFF_REP_NONFINITE) || !isfinite(f2)) {
          st |= GRIDFF_REP_NONFINITE;
          break;
        }
        if (f2 < fp.f_conv2) {
          st |= GRIDFF_REP_CONVERGED;
          break;
        }
        float keep, mixf;
        if (P > 0.f) {
          keep = 1.f - al;
          mixf = f2 > 0.f && v2 > 0.f ? al * v2 * rsqrtf(v2) * rsqrtf(f2) : 0.f;   // al |v| / |F|
          if (np > fp.n_min) {
            dt = fminf(dt * fp.f_inc, fp.dt_max);
            al *= fp.f_alpha;
          }
          ++np;
        } else {
          keep = 0.f;
          mixf = 0.f;
          dt *= fp.f_dec;
          al = fp.alpha_start;
          np = 0;
        }
        const float adt = GRIDFF_ACC * dt, dmax2 = fp.d_max * fp.d_max;
        for (int i = tid; i < n; i += kThr) {
          const float im = s.im[i];
          float4 x = s.x[i];
          float d[3];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float f = s.f[3 * i + c];
            float vv = keep * s.v[3 * i + c] + mixf * f;
            vv += adt * im * f;
            s.v[3 * i + c] = vv;
            d[c] = vv * dt;
          }
          const float dn2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
          const float scl = dn2 > dmax2 ? fp.d_max * rsqrtf(dn2) : 1.f;
          x.x += d[0] * scl;
          x.y += d[1] * scl;
          x.z += d[2] * scl;
          s.x[i] = x;
        }
        __syncthreads();
      }
      const double Etot = team_sum_d<NW>(s, tid, (double)e);
      if (evals > 0 && !isfinite(Etot)) st |= GRIDFF_REP_NONFINITE;
      if (tid == 0) {
        A.fdt[r] = dt;
        A.falpha[r] = al;
        A.fnp[r] = np;
        A.status[r] = st;
        const int total = A.steps[r] + evals;
        A.steps[r] = total;
        if (evals > 0) A.energy[r] = Etot;
        report(ctl, n, evals, st, total);
      }
    } else if (MODE == TEAM_LANGEVIN) {
      const unsigned long long key = splitmix64(A.seed ^ splitmix64((unsigned long long)r));
      const float hdt = 0.5f * A.dt, sq_kT = sqrtf(A.kT_acc);
      int st = A.status[r] & ~(GRIDFF_REP_CONVERGED | GRIDFF_REP_ABORTED | GRIDFF_REP_STEPLIMIT);
      int flags = 0, steps_done = 0;
      Acc e = team_forces<NW, KIND, Acc>(g, tv, A, s, t, ab, n, tid, flags, nullptr, f2, P, v2);
      __syncthreads();
      for (int it = 0; it < A.nsteps && !(st & GRIDFF_REP_NONFINITE); ++it) {
        if ((it & 31) == 0) {
          const int sb = stop();
          if (sb) {
            st |= sb;
            break;
          }
        }
        const unsigned long long sstep = (unsigned long long)(A.step0 + it) * 512ull;
        // one component per thread: the noise (a logarithm, a square root and
        // a cosine each) is the update's cost
        for (int m = tid; m < 3 * n; m += kThr) {
          const int i = m / 3;
          float* const xc = (float*)s.x + 4 * i + (m - 3 * i);
          const float rsm = s.im[i];   // 1 / sqrt(m_i)
          float v = s.v[m] + hdt * GRIDFF_ACC * s.f[m] * (rsm * rsm);
          const float x = *xc + hdt * v;
          const float xi = normal_of(splitmix64(key ^ (sstep + (unsigned long long)m)));
          v = A.c1 * v + A.c2 * sq_kT * rsm * xi;
          *xc = x + hdt * v;
          s.v[m] = v;
        }
        __syncthreads();
        e = team_forces<NW, KIND, Acc>(g, tv, A, s, t, ab, n, tid, flags, nullptr, f2, P, v2);
        team_sum<NW>(s, tid, f2, P, v2, flags);
        for (int m = tid; m < 3 * n; m += kThr) {
          const float rsm = s.im[m / 3];
          s.v[m] += hdt * GRIDFF_ACC * s.f[m] * (rsm * rsm);
        }
        st |= flags;
        ++steps_done;
        if (!isfinite(f2)) st |= GRIDFF_REP_NONFINITE;
      }
      const double Etot = team_sum_d<NW>(s, tid, (double)e);
      if (!isfinite(Etot)) st |= GRIDFF_REP_NONFINITE;
      if (tid == 0) {
        A.status[r] = st;
        A.energy[r] = Etot;
        report(ctl, n, steps_done + 1, st, steps_done);
      }
    } else if (MODE == TEAM_NVE) {
      int st = A.status[r] & ~(GRIDFF_REP_ABORTED | GRIDFF_REP_STEPLIMIT);
      int flags = 0, evals = 0;
      Acc e = team_forces<NW, KIND, Acc>(g, tv, A, s, t, ab, n, tid, flags, nullptr, f2, P, v2);
      __syncthreads();
      auto total = [&](Acc epot) {
        double ke = 0.0;
        for (int i = tid; i < n; i += kThr) {
          const double m = __ldg(&tv.body[ab + i]).w;
          const double vx = s.v[3 * i], vy = s.v[3 * i + 1], vz = s.v[3 * i + 2];
          ke += 0.5 * m * (vx * vx + vy * vy + vz * vz);
        }
        return team_sum_d<NW>(s, tid, (double)epot + ke / (double)GRIDFF_ACC);
      };
      if (A.trace) {
        const double E = total(e);
        if (tid == 0) A.trace[r] = E;
      }
      int rec = 1;
      for (int it = 0; it < A.nsteps; ++it) {
        if ((it & 31) == 0) {
          const int sb = stop();
          if (sb) {
            st |= sb;
            break;
          }
        }
        for (int i = tid; i < n; i += kThr) {
          const float h = s.im[i];
          float4 x = s.x[i];
          float* xc = &x.x;
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float vv = s.v[3 * i + c] + h * s.f[3 * i + c];
            s.v[3 * i + c] = vv;
            xc[c] += A.dt * vv;
          }
          s.x[i] = x;
        }
        __syncthreads();
        e = team_forces<NW, KIND, Acc>(g, tv, A, s, t, ab, n, tid, flags, nullptr, f2, P, v2);
        __syncthreads();
        ++evals;
        for (int i = tid; i < n; i += kThr) {
          const float h = s.im[i];
          for (int c = 0; c < 3; ++c) s.v[3 * i + c] += h * s.f[3 * i + c];
        }
        if (A.trace && A.rec_every > 0 && (it + 1) % A.rec_every == 0) {
          const double E = total(e);
          if (tid == 0) A.trace[(size_t)rec * A.trace_stride + r] = E;
          ++rec;
        }
      }
      const double Epot = team_sum_d<NW>(s, tid, (double)e);
      float z = 0.f;
      team_sum<NW>(s, tid, z, z, z, flags);
      if (tid == 0) {
        st |= flags;
        A.status[r] = st;
        A.energy[r] = Epot;
        report(ctl, n, evals, st & ~GRIDFF_REP_CONVERGED, evals);
      }
    } else {
      int flags = 0;
      const Acc e = team_forces<NW, KIND, Acc>(g, tv, A, s, t, ab, n, tid, flags, A.Ea ? A.Ea + off : nullptr, f2, P, v2);
      __syncthreads();
      for (int i = tid; i < n; i += kThr) {
        const float* f = s.f + 3 * i;
        put3(A.F, off + i, f[0], f[1], f[2]);
        if (!finite3(f[0], f[1], f[2])) flags |= GRIDFF_REP_NONFINITE;
      }
      const double E = team_sum_d<NW>(s, tid, (double)e);
      float z = 0.f;
      team_sum<NW>(s, tid, z, z, z, flags);
      if (!isfinite(E)) flags |= GRIDFF_REP_NONFINITE;
      if (tid == 0) {
        A.E[r] = E;
        if (A.st_out) A.st_out[r] = flags;
      }
    }
    __syncthreads();
    if (MODE != TEAM_EVAL)
      for (int i = tid; i < n; i += kThr) {
        put3(A.xs, off + i, s.x[i].x, s.x[i].y, s.x[i].z);
        put3(A.vs, off + i, s.v[3 * i], s.v[3 * i + 1], s.v[3 * i + 2]);
      }
    __syncthreads();
  }
}

using TeamFn = void (*)(GridView, TemplateView, TeamArgs, FireP, Control);
template <int NW, int KIND>
TeamFn team_fn_m(int mode) {
  switch (mode) {
    case TEAM_RELAX: return flex_team_kernel<NW, KIND, TEAM_RELAX>;
    case TEAM_LANGEVIN: return flex_team_kernel<NW, KIND, TEAM_LANGEVIN>;
    case TEAM_NVE: return flex_team_kernel<NW, KIND, TEAM_NVE>;
    default: return flex_team_kernel<4, KIND, TEAM_EVAL>;      // eval_team_width
  }
}
TeamFn team_fn(int NW, int kind, int mode) {
  if (NW == 2) return kind == REC_F32x4 ? team_fn_m<2, REC_F32x4>(mode) : team_fn_m<2, -1>(mode);
  if (NW == 8) return kind == REC_F32x4 ? team_fn_m<8, REC_F32x4>(mode) : team_fn_m<8, -1>(mode);
  return kind == REC_F32x4 ? team_fn_m<4, REC_F32x4>(mode) : team_fn_m<4, -1>(mode);
}

constexpr size_t kTeamMaxSmem = 100 * 1024;   // two teams per SM at least

}  // namespace

static bool team_fits(const gridff_replicas* R, int NW) {
  return team_bytes(NW, (R->max_natoms + 31) & ~31, R->max_natoms, R->max_slots) <= kTeamMaxSmem;
}

// Which replicas go to teams, by the batch's size against the W warps that are
// resident at once and by the largest molecule (n atoms).  us a FIRE step on
// GB300 (W = 4864), a warp per replica against 2 / 4 / 8 warps each:
//   replicas   10 atoms                  22 atoms                   47 atoms                    120 atoms
//        152    7.5   3.7  3.5  3.2      10.4   5.0  3.6  3.7       24.5   9.2   6.0  4.4       60.8   29.7  16.1   9.9
//        608    7.7   4.1  4.2  5.0      10.6   5.7  4.6  5.8       24.8  10.6   7.8  7.9       61.2   32.7  22.2  22.9
//       1216    7.8   5.0  6.0  9.5      10.8   7.0  6.9  11.2      25.1  13.0  12.7  15.4      61.3   65.2  43.8  39.9
//       2432    9.1   8.6 11.4 18.8      13.0  11.9 13.2  22.2      29.0  25.5  24.1  27.8      74.6  129.3  87.3  79.2
//       3648   10.9  11.7                15.2  16.4                 34.5  36.5                  97.3  192.9
// Past W replicas a last round of few replicas costs a whole step latency; where all
// replicas cost about the same (estimated costs within a tenth) it goes to teams, of
// molecules of up to 64 atoms also in the second round.  us a step, all on
// warps / the last round on teams (relaxation; Langevin; NVE):
//                   W + 304                                   2 W + 304
//    22 atoms   33.2 / 24.9  34.6 / 26.9  38.1 / 28.5     49.7 / 44.4   53.8 / 48.6   60.0 / 52.1
//    44..47     56.5 / 48.1  61.5 / 53.4  68.1 / 55.2     89.8 / 85.8   99.8 / 96.8  111.4 / 102.6
//    64         67.8 / 57.0  74.9 / 63.3  82.6 / 66.3    107.7 / 104.1 119.4 / 117.5 134.5 / 124.8
//    96          115 / 96.5   122 / 107    138 / 113      179 / 178     199 / 201     222 / 213
//   113..120     154 / 135    164 / 150    185 / 158      248 / 263     281 / 298     293 / 296
// and, at one round, 120 atoms with all torsions (three teams an SM) 175 / 151, with W + 608
// 178 / 170.  In an uneven batch the queue fills the last round's place with the small
// molecules while the large ones are still at work, and teams only add to that
// (10..120 atoms, 5000 replicas: 96.9 / 108.6 NVE, 10032: 91.4 / 100.7 relaxation).
FlexSplit flex_split(const gridff_ctx* ctx, const gridff_replicas* R) {
  const int n = R->max_natoms, n_rep = R->n_rep, W = 32 * ctx->n_sm;
  if (!team_fits(R, 4)) return {0, n_rep};
  if (n_rep <= W / 2) {
    if (team_fits(R, 8) && (n > 96 ? n_rep <= W / 4 : n > 32 && n_rep <= W / 16)) return {8, 0};
    if (n > 32) return n > 96 && n_rep > W / 4 ? FlexSplit{0, n_rep} : FlexSplit{4, 0};
    return {n_rep <= (n > 16 ? W / 4 : W / 8) ? 4 : 2, 0};
  }
  const int rest = n_rep % W;
  if (n_rep > W && n_rep < (n > 64 ? 2 : 3) * W && rest > 0 && rest <= W / 8 && R->evenness >= 0.9f)
    return {4, n_rep - rest};
  return {0, n_rep};
}

// One evaluation: us a call (with 13 us of launch), a warp per replica against
// 4 warps each: 22 atoms 24.5 / 20.3 at 608, 25.8 / 22.9 at 1216, 28.1 / 32.6 at
// 2432; 120 atoms 72.8 / 43.9 at 608, 77.7 / 73.1 at 1216, 95.6 / 129 at 2432.
int eval_team_width(const gridff_ctx* ctx, const gridff_replicas* R) {
  if (R->rigid || !team_fits(R, 4) || R->n_rep > 8 * ctx->n_sm) return 0;
  return 4;
}

static gridff_status team_launch(gridff_ctx* ctx, const gridff_grid* grid, gridff_replicas* R, int NW, int first,
                                 int mode, TeamArgs& A, const FireP& fp, const Control& ctl) {
  GridView gv{};
  gv.nx = gv.ny = gv.nz = 4;
  if (grid) gv = grid->view();
  A.rep_tmpl = R->rep_tmpl;
  A.rep_off = R->rep_off;
  A.order = R->order + first;
  A.n_rep = R->n_rep - first;
  A.N = (R->max_natoms + 31) & ~31;
  A.S = A.use_grid ? R->max_natoms : 0;
  A.n_slots = R->max_slots;
  A.xs = R->x;
  A.vs = R->v;
  A.fdt = R->fire_dt;
  A.falpha = R->fire_alpha;
  A.fnp = R->fire_nplus;
  A.status = R->status;
  A.steps = R->steps;
  A.energy = R->energy;
  A.last_x = R->last_x;
  A.last_f = R->last_f;
  const TeamFn fn = team_fn(NW, grid ? grid->kind : REC_F32x4, mode);
  const size_t dyn = team_bytes(NW, A.N, A.S, A.n_slots);
  GRIDFF_CUDA(ctx, allow_dyn_smem((const void*)fn, dyn));
  int per_sm = 0;
  GRIDFF_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)fn, 32 * NW, dyn));
  if (per_sm < 1) return set_err(ctx, GRIDFF_EINVAL, "team launch does not fit on an SM");
  const int cap = per_sm * ctx->n_sm;
  fn<<<A.n_rep < cap ? A.n_rep : cap, 32 * NW, dyn, ctx->stream>>>(gv, R->tv, A, fp, ctl);
  GRIDFF_CUDA(ctx, cudaGetLastError());
  return GRIDFF_OK;
}

static Control team_control(const gridff_ctx* ctx, double budget_s) {
  return Control{ctx->ctrl_dev, (unsigned long long)(budget_s > 0 ? budget_s * 1e9 : 0), (DevResult*)ctx->result_dev};
}

gridff_status enqueue_team_relax(gridff_ctx* ctx, const gridff_grid* grid, gridff_replicas* R, FlexSplit sp, int nsteps,
                                 const gridff_fire_params& P, int flags) {
  TeamArgs A{};
  A.nsteps = nsteps;
  A.use_grid = !(flags & GRIDFF_NO_GRID);
  A.use_intra = !(flags & GRIDFF_NO_INTRA);
  const FireP fp{P.dt_start, P.dt_max, P.f_inc, P.f_dec, P.alpha_start, P.f_alpha, P.d_max, P.f_conv * P.f_conv, P.n_min};
  return team_launch(ctx, grid, R, sp.team, sp.n_warp, TEAM_RELAX, A, fp, team_control(ctx, P.clock_budget_s));
}

gridff_status enqueue_team_langevin(gridff_ctx* ctx, const gridff_grid* grid, gridff_replicas* R, FlexSplit sp, int nsteps,
                                    const gridff_langevin_params& P, float c1, float c2, float kT_acc, int flags) {
  TeamArgs A{};
  A.nsteps = nsteps;
  A.use_grid = !(flags & GRIDFF_NO_GRID);
  A.use_intra = !(flags & GRIDFF_NO_INTRA);
  A.dt = P.dt;
  A.c1 = c1;
  A.c2 = c2;
  A.kT_acc = kT_acc;
  A.seed = P.seed;
  A.step0 = P.step0;
  return team_launch(ctx, grid, R, sp.team, sp.n_warp, TEAM_LANGEVIN, A, FireP{}, team_control(ctx, P.clock_budget_s));
}

gridff_status enqueue_team_run(gridff_ctx* ctx, const gridff_grid* grid, gridff_replicas* R, FlexSplit sp, int nsteps,
                               const gridff_md_params& P, double* trace, int flags) {
  TeamArgs A{};
  A.nsteps = nsteps;
  A.use_grid = !(flags & GRIDFF_NO_GRID);
  A.use_intra = !(flags & GRIDFF_NO_INTRA);
  A.dt = P.dt;
  A.rec_every = P.record_every;
  A.trace = trace;
  A.trace_stride = R->n_rep;
  return team_launch(ctx, grid, R, sp.team, sp.n_warp, TEAM_NVE, A, FireP{}, team_control(ctx, P.clock_budget_s));
}

gridff_status enqueue_team_eval(gridff_ctx* ctx, const gridff_grid* grid, gridff_replicas* R, int NW, double* E, float* F,
                                float* Ea, int* st, int flags) {
  TeamArgs A{};
  A.use_grid = !(flags & GRIDFF_NO_GRID);
  A.use_intra = !(flags & GRIDFF_NO_INTRA);
  A.E = E;
  A.F = F;
  A.Ea = Ea;
  A.st_out = st;
  return team_launch(ctx, grid, R, NW, 0, TEAM_EVAL, A, FireP{}, team_control(ctx, 0.0));
}
