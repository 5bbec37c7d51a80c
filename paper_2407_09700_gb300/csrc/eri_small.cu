// Compile-time specialised Rys kernels for the low angular-momentum classes whose
// contracted [e0|f0] block fits a lane's registers (up to 54 values in FP64, 96 in the
// FP32 path of the mixed mode; in integers sums of more than 30 values live in shared
// memory); each runs with one lane per shell quartet.  Following
// Sec. 3's design for small root counts (Alg. 2: unrolled recurrences, intermediates in
// registers, contraction before digestion), every loop here has compile-time bounds: the
// 2D tables I_x, I_y, I_z of one root and the contracted accumulators live in registers
// and the Eq. 1 index map is folded into the code.  Task fetching and screening are the shared
// device functions of eri_device.cuh; the
// transfer relations and the digestion run in registers as well (finish_lane).
#include <type_traits>

#include "eri_device.cuh"
#include "eri_scalar.cuh"

namespace {

template <int I, int N, typename F>
__device__ __forceinline__ void sfor(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    sfor<I + 1, N>(f);
  }
}

__host__ __device__ constexpr int cb(int l) { return l * (l + 1) * (l + 2) / 6; }
__host__ __device__ constexpr int cart_l(int g) {
  int l = 0;
  while (cb(l + 1) <= g) ++l;
  return l;
}
// exponent of axis ax (0 = x, 1 = y, 2 = z) of the Cartesian function with global index g
__host__ __device__ constexpr int cart_e(int g, int ax) {
  const int l = cart_l(g);
  const int pos = g - cb(l);
  int r = 0;
  while ((r + 1) * (r + 2) / 2 <= pos) ++r;
  const int lz = pos - r * (r + 1) / 2;
  return ax == 0 ? l - r : (ax == 1 ? r - lz : lz);
}

template <int LA, int LB, int LC, int LD>
struct Small {
  static constexpr int LE = LA + LB, LF = LC + LD, L1 = LF + 1, NI = (LE + 1) * L1;
  static constexpr int N = (LA + LB + LC + LD) / 2 + 1;
  static constexpr int EB = cb(LA), FB = cb(LC);
  static constexpr int NE = cb(LE + 1) - EB, NF = cb(LF + 1) - FB, NOUT = NE * NF;
  // offset into the 2D table of axis ax for output o = ie * NF + jf
  __host__ __device__ static constexpr int idx(int o, int ax) {
    return cart_e(EB + o / NF, ax) * L1 + cart_e(FB + o % NF, ax);
  }
};

// ---------------------------------------------------------------- transfer and digestion of one lane
// global index of the Cartesian function (x, y, z)
__host__ __device__ constexpr int cart_id(int x, int y, int z) {
  const int l = x + y + z, r = y + z;
  return cb(l) + r * (r + 1) / 2 + z;
}
// axis the relation builds b along (b > 0), b's index one lower along it, a's index one higher
__host__ __device__ constexpr int hrr_axis(int b) { return cart_e(b, 0) > 0 ? 0 : (cart_e(b, 1) > 0 ? 1 : 2); }
__host__ __device__ constexpr int cart_step(int g, int ax, int d) {
  return cart_id(cart_e(g, 0) + (ax == 0 ? d : 0), cart_e(g, 1) + (ax == 1 ? d : 0), cart_e(g, 2) + (ax == 2 ? d : 0));
}

// Transfer relations (a, b + 1_i| = (a + 1_i, b| + (A - B)_i (a, b| from in(e, v), |e| from l0 to
// l0 + l1, to out[(a nb + b) oa + v ov], v < NV; l1 <= 2.
template <int L0, int L1, int NV, int OA, int OV, typename In>
__device__ __forceinline__ void hrr_lane(const In& in, const double AB[3], double* out) {
  static_assert(L1 <= 2, "one or two steps");
  constexpr int base = cb(L0), NA = cb(L0 + 1) - base;
  if constexpr (L1 == 0) {
    sfor<0, NA>([&](auto e) {
      sfor<0, NV>([&](auto v) { out[decltype(e)::value * OA + decltype(v)::value * OV] = in(e, v); });
    });
  } else {
    constexpr int N1 = cb(L0 + L1) - base;          // |a| from l0 to l0 + l1 - 1
    double t1[L1 == 2 ? N1 * 3 * NV : 1];
    sfor<0, N1>([&](auto ac) {
      sfor<0, 3>([&](auto bc) {
        sfor<0, NV>([&](auto v) {
          constexpr int ia = decltype(ac)::value, i = decltype(bc)::value, vv = decltype(v)::value;
          constexpr int up = cart_step(base + ia, i, 1) - base;
          const double r = fma(AB[i], in(ac, v), in(std::integral_constant<int, up>{}, v));
          if constexpr (L1 == 1) out[(ia * 3 + i) * OA + vv * OV] = r;
          else t1[(ia * 3 + i) * NV + vv] = r;
        });
      });
    });
    if constexpr (L1 == 2) {
      sfor<0, NA>([&](auto ac) {
        sfor<0, 6>([&](auto bc) {
          sfor<0, NV>([&](auto v) {
            constexpr int ia = decltype(ac)::value, ib = decltype(bc)::value, vv = decltype(v)::value;
            constexpr int i = hrr_axis(cb(2) + ib), bm = cart_step(cb(2) + ib, i, -1) - cb(1);
            constexpr int up = cart_step(base + ia, i, 1) - base;
            out[(ia * 6 + ib) * OA + vv * OV] = fma(AB[i], t1[(ia * 3 + bm) * NV + vv], t1[(up * 3 + bm) * NV + vv]);
          });
        });
      });
    }
  }
}

// The contracted [e0|f0] values E(o) of one quartet to J~ and K~: the transfer relations and the six
// updates of Alg. 2 with every index a constant, (ab|cd) and the density blocks in registers.
// E carries the quartet's permutation weight.  Through per-lane scratch in global memory (32
// lines per access) this took 2-6 ns a quartet and most of the time of shallow s/p/d shells.
template <int LA, int LB, int LC, int LD, typename Get>
__device__ __forceinline__ void finish_lane(const TaskCtx& tc, const ShellPair* bra, const ShellPair* ket, const Get& E) {
  using S = Small<LA, LB, LC, LD>;
  constexpr int NA = cb(LA + 1) - cb(LA), NB = cb(LB + 1) - cb(LB), NC = cb(LC + 1) - cb(LC), ND = cb(LD + 1) - cb(LD);
  constexpr int NAB = NA * NB, NCD = NC * ND;
  const double AB[3] = {bra->AB[0], bra->AB[1], bra->AB[2]}, CD[3] = {ket->AB[0], ket->AB[1], ket->AB[2]};
  double G[NAB * NCD];
  if constexpr (LB == 0 && LD == 0) {
#pragma unroll
    for (int o = 0; o < NAB * NCD; ++o) G[o] = E(o);
  } else {
    double Y[NAB * S::NF];                          // (ab|f0]
    hrr_lane<LA, LB, S::NF, S::NF, 1>(
        [&](auto e, auto v) { return E(decltype(e)::value * S::NF + decltype(v)::value); }, AB, Y);
    hrr_lane<LC, LD, NAB, 1, NCD>(
        [&](auto f, auto v) { return Y[decltype(v)::value * S::NF + decltype(f)::value]; }, CD, G);
  }
  const int nbf = tc.nbf;
  const size_t p0 = bra->bf0, q0 = bra->bf1, r0 = ket->bf0, s0 = ket->bf1;
  for (int xd = 0; xd < tc.nD; ++xd) {
    const size_t off = (size_t)xd * nbf * nbf;
    const double* D = tc.D + off;
    if (tc.want & 1) {
      double* J = tc.J + off;
      double d[NCD], jcd[NCD];
#pragma unroll
      for (int i = 0; i < NCD; ++i) {
        d[i] = __ldg(D + (r0 + i / ND) * nbf + s0 + i % ND);
        jcd[i] = 0.0;
      }
#pragma unroll
      for (int i = 0; i < NAB; ++i) {
        const size_t at = (p0 + i / NB) * nbf + q0 + i % NB;
        const double dab = __ldg(D + at);
        double t = 0.0;
#pragma unroll
        for (int k = 0; k < NCD; ++k) {
          t = fma(G[i * NCD + k], d[k], t);
          jcd[k] = fma(G[i * NCD + k], dab, jcd[k]);
        }
        atomicAdd(J + at, 2.0 * t);
      }
#pragma unroll
      for (int i = 0; i < NCD; ++i) atomicAdd(J + (r0 + i / ND) * nbf + s0 + i % ND, 2.0 * jcd[i]);
    }
    if (tc.want & 2) {
      double* K = tc.K + off;
      // D_bd and D_bc, D_ad and D_ac against G, one a at a time
      double dbd[NB * ND], dbc[NB * NC], kbd[NB * ND], kbc[NB * NC];
#pragma unroll
      for (int i = 0; i < NB * ND; ++i) {
        dbd[i] = __ldg(D + (q0 + i / ND) * nbf + s0 + i % ND);
        kbd[i] = 0.0;
      }
#pragma unroll
      for (int i = 0; i < NB * NC; ++i) {
        dbc[i] = __ldg(D + (q0 + i / NC) * nbf + r0 + i % NC);
        kbc[i] = 0.0;
      }
#pragma unroll
      for (int ia = 0; ia < NA; ++ia) {
        const size_t row = (p0 + ia) * nbf;
        double dac[NC], dad[ND], kac[NC], kad[ND];
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          dac[i] = __ldg(D + row + r0 + i);
          kac[i] = 0.0;
        }
#pragma unroll
        for (int i = 0; i < ND; ++i) {
          dad[i] = __ldg(D + row + s0 + i);
          kad[i] = 0.0;
        }
#pragma unroll
        for (int ibb = 0; ibb < NB; ++ibb)
#pragma unroll
          for (int ic = 0; ic < NC; ++ic)
#pragma unroll
            for (int id = 0; id < ND; ++id) {
              const double g = G[(ia * NB + ibb) * NCD + ic * ND + id];
              kac[ic] = fma(g, dbd[ibb * ND + id], kac[ic]);
              kad[id] = fma(g, dbc[ibb * NC + ic], kad[id]);
              kbd[ibb * ND + id] = fma(g, dac[ic], kbd[ibb * ND + id]);
              kbc[ibb * NC + ic] = fma(g, dad[id], kbc[ibb * NC + ic]);
            }
#pragma unroll
        for (int i = 0; i < NC; ++i) atomicAdd(K + row + r0 + i, kac[i]);
#pragma unroll
        for (int i = 0; i < ND; ++i) atomicAdd(K + row + s0 + i, kad[i]);
      }
#pragma unroll
      for (int i = 0; i < NB * ND; ++i) atomicAdd(K + (q0 + i / ND) * nbf + s0 + i % ND, kbd[i]);
#pragma unroll
      for (int i = 0; i < NB * NC; ++i) atomicAdd(K + (q0 + i / NC) * nbf + r0 + i % NC, kbc[i]);
    }
  }
}

// log2 of the permutation weight of a unique quartet (0, -1, -2 or -3)
__device__ __forceinline__ int weight_log2(const ShellPair* bra, const ShellPair* ket, int ib, int ik) {
  return -(int)(bra->sh0 == bra->sh1) - (int)(ket->sh0 == ket->sh1) - (int)(ib == ik);
}

// m 2^k rounded to nearest (normal results or m = 0)
__device__ __forceinline__ float round_f(int64_t m, int k) {
  const float f = __ll2float_rn(m);
  return m ? __int_as_float(__float_as_int(f) + (k << 23)) : 0.0f;
}

template <int LA, int LB, int LC, int LD, typename R>
__global__ void __launch_bounds__(TPB, (Small<LA, LB, LC, LD>::NOUT > 32 ? 2 : 3)) eri_small_kernel(const KernelArgs a) {
  using S = Small<LA, LB, LC, LD>;
  constexpr int LE = S::LE, LF = S::LF, L1 = S::L1, NI = S::NI, N = S::N, NOUT = S::NOUT;
  const int lane = threadIdx.x & 31;
  // contracted [e0|f0] and the transfer relations are FP64 in both paths (see eri_kernels.cu)
  const bool listed = a.tlist != nullptr || a.jobs != nullptr;
  const int qs = (a.mode == KMODE_JK && a.qsplit > 1) ? a.qsplit : 1;   // tasks per quartet (primitive ranges)
  const long long ntask = (listed ? (long long)*a.tcount : a.ntask) * qs;
  unsigned long long cnt_q = 0, cnt_p = 0;

  while (true) {
    unsigned long long tbase = 0;
    if (lane == 0) tbase = atomicAdd(a.counter, 32ULL);
    tbase = __shfl_sync(0xffffffffu, tbase, 0);
    if (tbase >= (unsigned long long)ntask) break;
    const long long slot = (long long)tbase + lane;
    bool active = slot < ntask;
    const long long task = slot / qs;
    const int ch = (int)(slot - task * qs);
    int ib = 0, ik = 0;
    TaskCtx tc = single_ctx(a);
    if (active) resolve_task(a, task, listed, tc, ib, ik);
    const ShellPair* bra = tc.pairs + ib;
    const ShellPair* ket = tc.pairs + ik;
    if (active && !listed) {
      const int cat = quartet_category(a, bra, ket, a.prec_sel != 0);
      active = cat != 0 && (a.prec_sel == 0 || cat == a.prec_sel);
    }
    const int npb = active ? bra->nprim : 0;
    const int npk = active ? ket->nprim : 0;
    // primitive quartets [qlo, qlo + nq) of this task (the last range counts the quartet)
    const int nqf = npb * npk;
    const int qlo = (qs > 1) ? (int)((long long)ch * nqf / qs) : 0;
    const int nq = (qs > 1) ? (int)((long long)(ch + 1) * nqf / qs) - qlo : nqf;
    if (nq == 0) active = false;
    const int maxq = warp_max(nq);
    if (active) { cnt_q += (ch == qs - 1) ? 1 : 0; cnt_p += (unsigned long long)nq; }
    const int boff = active ? bra->prim_off : 0, koff = active ? ket->prim_off : 0;

    R acc[NOUT];
#pragma unroll
    for (int o = 0; o < NOUT; ++o) acc[o] = R(0);

    // the primitive quartet's bra and ket records, ket fastest
    int ixp = 0, iyp = 0;
    if (active) {
      ixp = qlo / npk;
      iyp = qlo - ixp * npk;
    }
    for (int q = 0; q < maxq; ++q) {
      if (q < nq) {
        // Gaussian-product scalars: C = PA - uz (P - Q) and so on, in the recurrence type
        R hz, he, rz, re, hs, theta, P0, P1, P2, PA0, PA1, PA2, QC0, QC1, QC2;
        RysAt at;
        SxQuartet s;
        if constexpr (sizeof(R) == 8) {
          const PrimPair* x = tc.prims + boff + ixp;
          const PrimPair* y = tc.prims + koff + iyp;
          const double zeta = x->zeta, eta = y->zeta;
          const double r = rsqrt(zeta + eta);
          P0 = x->P[0] - y->P[0]; P1 = x->P[1] - y->P[1]; P2 = x->P[2] - y->P[2];
          const double inv_s = r * r;
          rz = eta * inv_s;
          re = zeta * inv_s;
          at = rys_locate((zeta * rz) * fma(P0, P0, fma(P1, P1, P2 * P2)), a.rys_tcut_hi);
          hs = 0.5 * inv_s;
          hz = x->hz; he = y->hz;
          theta = x->E * y->E * r;
          PA0 = x->PA[0]; PA1 = x->PA[1]; PA2 = x->PA[2];
          QC0 = y->PA[0]; QC1 = y->PA[1]; QC2 = y->PA[2];
        } else {
          // P - Q, 1/sqrt(zeta + eta), T and the lookup in integers (eri_scalar.cuh), rounded to
          // nearest at the recurrence input
          const PrimFx* xi = tc.prfx + boff + ixp;
          const PrimFx* yi = tc.prfx + koff + iyp;
          const PrimPairF* x = tc.primsf + boff + ixp;
          const PrimPairF* y = tc.primsf + koff + iyp;
          const int64_t P[3] = {xi->P[0], xi->P[1], xi->P[2]}, Q[3] = {yi->P[0], yi->P[1], yi->P[2]};
          sx_quartet((uint64_t)__double_as_longlong(xi->H + yi->H), P, Q, tc.pu, a.rys_tcut4, s);
          P0 = round_f(s.d[0], s.k - 60);
          P1 = round_f(s.d[1], s.k - 60);
          P2 = round_f(s.d[2], s.k - 60);
          const float r = round_f(sx_mulm(sx_mulm(xi->Sm, yi->Sm), s.g << 2), xi->Se + yi->Se + s.ge - 62);
          const float inv_s = r * r;
          rz = y->zeta * inv_s;
          re = x->zeta * inv_s;
          hs = 0.5f * inv_s;
          hz = x->hz; he = y->hz;
          theta = x->E * y->E * r;
          PA0 = x->PA[0]; PA1 = x->PA[1]; PA2 = x->PA[2];
          QC0 = y->PA[0]; QC1 = y->PA[1]; QC2 = y->PA[2];
        }
        if (++iyp == npk) {
          iyp = 0;
          ++ixp;
        }
#pragma unroll
        for (int n = 0; n < N; ++n) {
          R u, w;
          if constexpr (sizeof(R) == 8) {
            rys_root(a.rys_coef, a.rys_au, a.rys_aw, N, at, n, u, w);
          } else {
            int64_t um, wm;
            int ue, we;
            sx_root(a.rys_coef, reinterpret_cast<const longlong2*>(a.rys_asym), N, s, n, um, ue, wm, we);
            u = round_f(um, ue - 62);
            w = round_f(wm, we - 62);
          }
          const R B00 = u * hs;
          const R wt = w * theta;
          R B10, B01, C[3], Cp[3];
          if constexpr (sizeof(R) == 8) {
            // u eta/(zeta+eta) and u zeta/(zeta+eta) once per root: with N <= 3 fewer products than
            // scaling P - Q and the half inverse exponents first
            const R uz = u * rz, ue = u * re;
            B10 = fma(-uz, hz, hz);
            B01 = fma(-ue, he, he);
            C[0] = fma(-uz, P0, PA0); C[1] = fma(-uz, P1, PA1); C[2] = fma(-uz, P2, PA2);
            Cp[0] = fma(ue, P0, QC0); Cp[1] = fma(ue, P1, QC1); Cp[2] = fma(ue, P2, QC2);
          } else {
            B10 = fma(-u, hz * rz, hz);
            B01 = fma(-u, he * re, he);
            C[0] = fma(-u, rz * P0, PA0); C[1] = fma(-u, rz * P1, PA1); C[2] = fma(-u, rz * P2, PA2);
            Cp[0] = fma(u, re * P0, QC0); Cp[1] = fma(u, re * P1, QC1); Cp[2] = fma(u, re * P2, QC2);
          }
          R g[3][NI];
          g[0][0] = R(1);
          g[1][0] = R(1);
          g[2][0] = wt;
          if constexpr (LE >= 1) {
            g[0][L1] = C[0];
            g[1][L1] = C[1];
            g[2][L1] = C[2] * wt;
          }
#pragma unroll
          for (int n2 = 1; n2 < LE; ++n2) {
            const R nb10 = R(n2) * B10;
#pragma unroll
            for (int ax = 0; ax < 3; ++ax)
              g[ax][(n2 + 1) * L1] = fma(C[ax], g[ax][n2 * L1], nb10 * g[ax][(n2 - 1) * L1]);
          }
#pragma unroll
          for (int n2 = 0; n2 <= LE; ++n2) {
            const R nb00 = R(n2) * B00;
#pragma unroll
            for (int m = 0; m < LF; ++m) {
              const R mb01 = R(m) * B01;
#pragma unroll
              for (int ax = 0; ax < 3; ++ax) {
                const int e = n2 * L1 + m;
                R v = Cp[ax] * g[ax][e];
                if (n2 > 0) v = fma(nb00, g[ax][e - L1], v);
                if (m > 0) v = fma(mb01, g[ax][e - 1], v);
                g[ax][e + 1] = v;
              }
            }
          }
          // Eq. 1 products, accumulated over roots and primitives (Eq. 5)
          sfor<0, NOUT>([&](auto oc) {
            constexpr int o = decltype(oc)::value;
            constexpr int i0 = S::idx(o, 0), i1 = S::idx(o, 1), i2 = S::idx(o, 2);
            acc[o] = fma(g[0][i0] * g[1][i1], g[2][i2], acc[o]);
          });
        }
      }
    }
    if (active) {
      const R w = R(1) / R(1 << -weight_log2(bra, ket, ib, ik));
      finish_lane<LA, LB, LC, LD>(tc, bra, ket, [&](int o) { return (double)(w * acc[o]); });
    }
    __syncwarp();
  }
  for (int off = 16; off > 0; off >>= 1) {
    cnt_q += __shfl_xor_sync(0xffffffffu, cnt_q, off);
    cnt_p += __shfl_xor_sync(0xffffffffu, cnt_p, off);
  }
  if (lane == 0 && a.stats) {
    atomicAdd(a.stats + 0, cnt_q);
    atomicAdd(a.stats + 1, cnt_p);
  }
}

// ---------------------------------------------------------------- the same classes in integers
// FP64-accurate launches with the scalars (eri_scalar.cuh), the 2D tables and the products of
// Eq. 1 in fixed point, lengths in units of 2^a (bra) and 2^b (ket) chosen per primitive pair;
// each primitive quartet's sums over the roots return to FP64 (a conversion and an FMA per value)
// at scale Theta 2^(a |e| + b |f|).  Sums of more than 30 values live in shared memory.
// The FP64 kernels above kept the FP64 pipe 85 % busy and the integer pipes 10-15 %.  16-atom
// medium build: (dp|ps) 74.5 -> 49.7 ms, (ds|ps) 47.2 -> 26.4, (ps|ps) 35.3 -> 15.6, (ps|ss) 24.9 ->
// 9.5, (ss|ss) 6.0 -> 2.5; in (dp|ps) the FP64 pipe is then 36 % busy and two warps a scheduler wait
// for dependent integer instructions; J and K are as close to quadruple precision as with FP64 (45 functions
// of 6-31G(d)-like shells: 1.2e-15, 1.6e-15 against 1.3e-15, 1.7e-15 for a small change of the
// density).
template <int LA, int LB, int LC, int LD>
struct SmallFx {
  using S = Small<LA, LB, LC, LD>;
  static constexpr bool SM = S::NOUT > 30;
  static constexpr int blocks = S::NOUT > 16 ? 2 : 3;
  static constexpr int smem = SM ? (int)sizeof(double) * S::NOUT * TPB : 0;
  // total degree above the lowest of bra and ket: the value's scale
  __host__ __device__ static constexpr int group(int o) {
    return (cart_l(S::EB + o / S::NF) - LA) * (LD + 1) + cart_l(S::FB + o % S::NF) - LC;
  }
};

__device__ __forceinline__ PrimFx load_fx(const PrimFx* p) {
  PrimFx r;
  const longlong2* q = reinterpret_cast<const longlong2*>(p);
  longlong2* d = reinterpret_cast<longlong2*>(&r);
#pragma unroll
  for (int i = 0; i < 6; ++i) d[i] = __ldg(q + i);      // without Sm, Se
  return r;
}

// v 2^k for a finite v (0 below the normal range); infinities and NaNs unchanged
__device__ __forceinline__ double scale_pow2(double v, int k) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
  if (e == 0x7ff) return v;
  if (e == 0 || e + k <= 0) return 0.0;
  return __hiloint2double(hi + (k << 20), __double2loint(v));
}

template <int LA, int LB, int LC, int LD>
__global__ void __launch_bounds__(TPB, (SmallFx<LA, LB, LC, LD>::blocks)) eri_small_fx_kernel(const KernelArgs a) {
  using S = Small<LA, LB, LC, LD>;
  using F = SmallFx<LA, LB, LC, LD>;
  constexpr int LE = S::LE, LF = S::LF, L1 = S::L1, NI = S::NI, N = S::N, NOUT = S::NOUT;
  constexpr int NG = (LB + 1) * (LD + 1);
  extern __shared__ double smem[];
  double* sacc = smem + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool listed = a.tlist != nullptr || a.jobs != nullptr;
  const int qs = a.qsplit > 1 ? a.qsplit : 1;
  const long long ntask = (listed ? (long long)*a.tcount : a.ntask) * qs;
  unsigned long long cnt_q = 0, cnt_p = 0;

  while (true) {
    unsigned long long tbase = 0;
    if (lane == 0) tbase = atomicAdd(a.counter, 32ULL);
    tbase = __shfl_sync(0xffffffffu, tbase, 0);
    if (tbase >= (unsigned long long)ntask) break;
    const long long slot = (long long)tbase + lane;
    bool active = slot < ntask;
    const long long task = slot / qs;
    const int ch = (int)(slot - task * qs);
    int ib = 0, ik = 0;
    TaskCtx tc = single_ctx(a);
    if (active) resolve_task(a, task, listed, tc, ib, ik);
    const ShellPair* bra = tc.pairs + ib;
    const ShellPair* ket = tc.pairs + ik;
    if (active && !listed) {
      const int cat = quartet_category(a, bra, ket, a.prec_sel != 0);
      active = cat != 0 && (a.prec_sel == 0 || cat == a.prec_sel);
    }
    const int npb = active ? bra->nprim : 0;
    const int npk = active ? ket->nprim : 0;
    const int nqf = npb * npk;
    const int qlo = (qs > 1) ? (int)((long long)ch * nqf / qs) : 0;
    const int nq = (qs > 1) ? (int)((long long)(ch + 1) * nqf / qs) - qlo : nqf;
    if (nq == 0) active = false;
    const int maxq = warp_max(nq);
    if (active) { cnt_q += (ch == qs - 1) ? 1 : 0; cnt_p += (unsigned long long)nq; }

    double racc[F::SM ? 1 : NOUT];
    if constexpr (F::SM) {
#pragma unroll
      for (int o = 0; o < NOUT; ++o) sacc[o * TPB] = 0.0;
    } else {
#pragma unroll
      for (int o = 0; o < NOUT; ++o) racc[o] = 0.0;
    }
    const int wl = active ? weight_log2(bra, ket, ib, ik) : 0;
    const PrimFx* xp = tc.prfx + (active ? bra->prim_off : 0);
    const PrimFx* yp = tc.prfx + (active ? ket->prim_off : 0);
    int ixp = 0, iyp = 0;
    if (active) {
      ixp = qlo / npk;
      iyp = qlo - ixp * npk;
    }
    for (int q = 0; q < maxq; ++q) {
      if (q < nq) {
        const PrimFx x = load_fx(xp + ixp), y = load_fx(yp + iyp);
        if (++iyp == npk) {
          iyp = 0;
          ++ixp;
        }
        SxQuartet s;
        sx_quartet((uint64_t)__double_as_longlong(x.H + y.H), x.P, y.P, tc.pu, a.rys_tcut4, s);
        // Theta = E E' g
        const double gd = __ll2double_rn(s.g);
        const double theta = x.E * y.E * __hiloint2double(__double2hiint(gd) + ((s.ge - 60) << 20), __double2loint(gd));
        const SxL dl[3] = {sx_limbs(s.d[0]), sx_limbs(s.d[1]), sx_limbs(s.d[2])};
        // eta/(zeta+eta) and zeta/(zeta+eta)
        const int64_t rzm = sx_mulm(x.Hm, s.g2), rem = sx_mulm(y.Hm, s.g2);
        const int rze = x.He + s.g2e, ree = y.He + s.g2e;
        const SxL hzl = sx_limbs(x.hz), hel = sx_limbs(y.hz);
        SxL hs{0, 0};
        if (LE > 0 && LF > 1) {
          // 1 / (2 (zeta + eta)) 2^-(a + b): from the side that needs no left shift
          const bool br = x.a <= y.a;
          const SxL r = sx_limbs(br ? sx_shift(rem, 2 - ree) : sx_shift(rzm, 2 - rze));
          hs = sx_limbs(sx_shift(sx_mul(br ? hzl : hel, r), br ? y.a - x.a : x.a - y.a));
        }
        int64_t acc[NOUT];
        // binary places by which the bra's and the ket's unit of length is finer than 2^a, 2^b
        int sa = 0, sb = 0;
#pragma unroll
        for (int nn = 0; nn < N; ++nn) {
          const int n = N - 1 - nn;                       // the largest root first
          int64_t um, wm;
          int ue, we;
          sx_root(a.rys_coef, reinterpret_cast<const longlong2*>(a.rys_asym), N, s, n, um, ue, wm, we);
          // in units of 2^rTe, about 1/sqrt(T), in the large-T limit: the weight keeps its 60 bits there
          // (as an absolute 2^-60 it lost log2(T) / 2 of them, 2.3e-13 of a repulsion at T = 1e11)
          const int64_t w60 = sx_shift(wm, 2 - (we - s.rTe));
          // u eta/(zeta+eta), u zeta/(zeta+eta)
          const int64_t fz = LE > 0 ? sx_mulm(um, rzm) : 0, fn = LF > 0 ? sx_mulm(um, rem) : 0;
          const int fze = ue + rze, fne = ue + ree;
          int64_t C6[3] = {0, 0, 0}, Cp6[3] = {0, 0, 0}, b10 = 0, b01 = 0, b00 = 0;
          // C is linear in u, so every root's lies between P - A and the largest root's: units in
          // which the larger of them is below 1 and the half inverse exponent below 1/8 (every
          // 2D entry then below 2).  Without this the fourth-degree entries of typical C (a few
          // hundredths of the bound) kept too few bits.
          if (LE > 1) {
            const SxL f = sx_limbs(sx_shift(fz, 2 - (fze + s.k - x.a)));
#pragma unroll
            for (int i = 0; i < 3; ++i) C6[i] = x.PA[i] - sx_mul(f, dl[i]);
            b10 = x.hz - sx_mul(hzl, sx_limbs(sx_shift(fz, 2 - fze)));
            if (N > 1 && nn == 0) sa = sx_places(x.PA, C6, x.hz);
#pragma unroll
            for (int i = 0; i < 3; ++i) C6[i] = (int64_t)((uint64_t)C6[i] << sa);
            b10 = (int64_t)((uint64_t)b10 << (2 * sa));
          }
          if (LF > 1) {
            const SxL f = sx_limbs(sx_shift(fn, 2 - (fne + s.k - y.a)));
#pragma unroll
            for (int i = 0; i < 3; ++i) Cp6[i] = y.PA[i] + sx_mul(f, dl[i]);
            b01 = y.hz - sx_mul(hel, sx_limbs(sx_shift(fn, 2 - fne)));
            if (N > 1 && nn == 0) sb = sx_places(y.PA, Cp6, y.hz);
#pragma unroll
            for (int i = 0; i < 3; ++i) Cp6[i] = (int64_t)((uint64_t)Cp6[i] << sb);
            b01 = (int64_t)((uint64_t)b01 << (2 * sb));
            if (LE > 0) b00 = (int64_t)((uint64_t)sx_mul(hs, sx_limbs(sx_shift(um, 2 - ue))) << (sa + sb));
          }
          // A side of one unit of angular momentum has no half inverse exponent in its entries: its unit goes
          // by C alone, before anything is rounded, so that a dipole keeps its bits at any distance
          // ((ps|ps) of exponents 10 and 1e3 eight bohr apart was off by 2.9e-13 and 3.5e-10)
          if (LE == 1 && nn == 0) sa = sx_places1(x.PA, fz, fze + s.k - x.a);
          if (LF == 1) {
            const int64_t hm = sx_mulm(fz, y.Hm);        // u / (2 (zeta + eta)) = hm 2^(he - 62), units 2^(a + b)
            const int he = fze + y.He - 1 - x.a - y.a;
            if (nn == 0) {
              const int lim = max(0, sx_room(hm, he) - 3);     // places that leave it below 1/8
              if (LE == 1) sa = sa < lim ? sa : lim;
              const int p = sx_places1(y.PA, fn, fne + s.k - y.a), q = lim > sa ? lim - sa : 0;
              sb = p < q ? p : q;
            }
            b00 = sx_shift(hm, 2 - (he + sa + sb));
            const SxL f = sx_limbs(sx_shift(fn, 2 - (fne + s.k - y.a + sb)));
#pragma unroll
            for (int i = 0; i < 3; ++i) Cp6[i] = (int64_t)((uint64_t)y.PA[i] << sb) + sx_mul(f, dl[i]);
          }
          if (LE == 1) {
            const SxL f = sx_limbs(sx_shift(fz, 2 - (fze + s.k - x.a + sa)));
#pragma unroll
            for (int i = 0; i < 3; ++i) C6[i] = (int64_t)((uint64_t)x.PA[i] << sa) - sx_mul(f, dl[i]);
          }
          SxL C[3], Cp[3];
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            C[i] = sx_limbs(C6[i]);
            Cp[i] = sx_limbs(Cp6[i]);
          }
          // 2D tables; entry 0 of x and y is 1 and stays out of the products
          SxL g[3][NI];
          g[2][0] = sx_limbs(w60);
          auto mac = [&](SxSum& t, SxL k, int ax, int e) {
            if (ax < 2 && e == 0) t.d0 += sx_int(k);
            else sx_mac(t, k, g[ax][e]);
          };
#pragma unroll
          for (int n2 = 0; n2 < LE; ++n2) {
            const SxL nb = sx_limbs(n2 * b10);
#pragma unroll
            for (int ax = 0; ax < 3; ++ax) {
              SxSum t;
              mac(t, C[ax], ax, n2 * L1);
              if (n2 > 0) mac(t, nb, ax, (n2 - 1) * L1);
              g[ax][(n2 + 1) * L1] = sx_limbs(sx_value(t));
            }
          }
#pragma unroll
          for (int n2 = 0; n2 <= LE; ++n2) {
            const SxL nb = sx_limbs(n2 * b00);
#pragma unroll
            for (int m = 0; m < LF; ++m) {
              const SxL mb = sx_limbs(m * b01);
#pragma unroll
              for (int ax = 0; ax < 3; ++ax) {
                const int e = n2 * L1 + m;
                SxSum t;
                mac(t, Cp[ax], ax, e);
                if (n2 > 0) mac(t, nb, ax, e - L1);
                if (m > 0) mac(t, mb, ax, e - 1);
                g[ax][e + 1] = sx_limbs(sx_value(t));
              }
            }
          }
          sfor<0, NOUT>([&](auto oc) {
            constexpr int o = decltype(oc)::value;
            constexpr int i0 = S::idx(o, 0), i1 = S::idx(o, 1), i2 = S::idx(o, 2);
            const SxL z = g[2][i2];
            int64_t t;
            if constexpr (i0 == 0 && i1 == 0) t = sx_int(z);
            else if constexpr (i0 == 0) t = sx_mul(g[1][i1], z);
            else if constexpr (i1 == 0) t = sx_mul(g[0][i0], z);
            else t = sx_mul(sx_limbs(sx_mul(g[0][i0], g[1][i1])), z);
            acc[o] = nn == 0 ? t : acc[o] + t;
          });
        }
        double sc[NG];
#pragma unroll
        for (int i = 0; i <= LB; ++i)
#pragma unroll
          for (int j = 0; j <= LD; ++j)
            sc[i * (LD + 1) + j] = scale_pow2(theta, (x.a - sa) * (LA + i) + (y.a - sb) * (LC + j) + s.rTe - 60 + wl);
        sfor<0, NOUT>([&](auto oc) {
          constexpr int o = decltype(oc)::value;
          const double d = __ll2double_rn(acc[o]);
          if constexpr (F::SM) sacc[o * TPB] = fma(d, sc[F::group(o)], sacc[o * TPB]);
          else racc[o] = fma(d, sc[F::group(o)], racc[o]);
        });
      }
    }
    if (active)
      finish_lane<LA, LB, LC, LD>(tc, bra, ket, [&](int o) { return F::SM ? sacc[o * TPB] : racc[F::SM ? 0 : o]; });
    __syncwarp();
  }
  for (int off = 16; off > 0; off >>= 1) {
    cnt_q += __shfl_xor_sync(0xffffffffu, cnt_q, off);
    cnt_p += __shfl_xor_sync(0xffffffffu, cnt_p, off);
  }
  if (lane == 0 && a.stats) {
    atomicAdd(a.stats + 0, cnt_q);
    atomicAdd(a.stats + 1, cnt_p);
  }
}

// (la lb | lc ld) of the specialised classes and their kernels
#define SMALL_CLASSES(X)                                                                       \
  X(0, 0, 0, 0) X(1, 0, 0, 0) X(1, 1, 0, 0) X(2, 0, 0, 0) X(2, 1, 0, 0) X(2, 2, 0, 0)           \
  X(3, 0, 0, 0) X(3, 1, 0, 0) X(4, 0, 0, 0) X(1, 0, 1, 0) X(1, 1, 1, 0) X(2, 0, 1, 0) X(3, 0, 1, 0)      \
  X(2, 1, 1, 0) X(2, 0, 2, 0) X(2, 0, 1, 1)

// classes whose accumulators fit a lane's registers only in FP32: specialised for the FP32
// path of the mixed mode, team kernels for FP64
#define SMALL_CLASSES_F32(X) X(1, 1, 1, 1) X(2, 1, 2, 0) X(2, 2, 1, 0)

const void* small_ptr(int la, int lb, int lc, int ld, int fp32) {
#define SMALL_CASE(A, B, C, D)                                                   \
  if (la == A && lb == B && lc == C && ld == D)                                  \
    return fp32 ? (const void*)eri_small_kernel<A, B, C, D, float>               \
                : (const void*)eri_small_kernel<A, B, C, D, double>;
  SMALL_CLASSES(SMALL_CASE)
#undef SMALL_CASE
#define SMALL_CASE_F32(A, B, C, D)                                               \
  if (fp32 && la == A && lb == B && lc == C && ld == D) return (const void*)eri_small_kernel<A, B, C, D, float>;
  SMALL_CLASSES_F32(SMALL_CASE_F32)
#undef SMALL_CASE_F32
  return nullptr;
}

}  // namespace

extern "C" int erik_upload_cart_tables_small(void) { return (int)upload_cart_table(); }

// 1 if (la lb | lc ld) has a specialised kernel for this precision (fp32 = 1: FP32 path).
extern "C" int erik_small_available(int la, int lb, int lc, int ld, int fp32) {
  return small_ptr(la, lb, lc, ld, fp32) != nullptr;
}

extern "C" int erik_small_blocks_per_sm(int la, int lb, int lc, int ld, int fp32, int* out) {
  const void* k = small_ptr(la, lb, lc, ld, fp32);
  if (!k) return (int)cudaErrorInvalidValue;
  return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, TPB, 0);
}

extern "C" int erik_launch_small(int la, int lb, int lc, int ld, int fp32, const KernelArgs* a, int grid, void* stream) {
  cudaStream_t s = (cudaStream_t)stream;
#define SMALL_LAUNCH(A, B, C, D)                                                              \
  if (la == A && lb == B && lc == C && ld == D) {                                             \
    if (fp32)                                                                                 \
      eri_small_kernel<A, B, C, D, float><<<grid, TPB, 0, s>>>(*a);                           \
    else                                                                                      \
      eri_small_kernel<A, B, C, D, double><<<grid, TPB, 0, s>>>(*a);                          \
    return (int)cudaGetLastError();                                                           \
  }
  SMALL_CLASSES(SMALL_LAUNCH)
#undef SMALL_LAUNCH
#define SMALL_LAUNCH_F32(A, B, C, D)                                                          \
  if (fp32 && la == A && lb == B && lc == C && ld == D) {                                     \
    eri_small_kernel<A, B, C, D, float><<<grid, TPB, 0, s>>>(*a);                             \
    return (int)cudaGetLastError();                                                           \
  }
  SMALL_CLASSES_F32(SMALL_LAUNCH_F32)
#undef SMALL_LAUNCH_F32
  return (int)cudaErrorInvalidValue;
}

extern "C" int erik_small_fx_blocks_per_sm(int la, int lb, int lc, int ld, int* out) {
#define SMALL_FX_BLOCKS(A, B, C, D)                                                                              \
  if (la == A && lb == B && lc == C && ld == D) {                                                                \
    const void* k = (const void*)eri_small_fx_kernel<A, B, C, D>;                                                \
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SmallFx<A, B, C, D>::smem); \
    if (e != cudaSuccess) return (int)e;                                                                         \
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, TPB, SmallFx<A, B, C, D>::smem);           \
  }
  SMALL_CLASSES(SMALL_FX_BLOCKS)
#undef SMALL_FX_BLOCKS
  return (int)cudaErrorInvalidValue;
}

extern "C" int erik_launch_small_fx(int la, int lb, int lc, int ld, const KernelArgs* a, int grid, void* stream) {
#define SMALL_FX_LAUNCH(A, B, C, D)                                                                               \
  if (la == A && lb == B && lc == C && ld == D) {                                                                 \
    eri_small_fx_kernel<A, B, C, D><<<grid, TPB, SmallFx<A, B, C, D>::smem, (cudaStream_t)stream>>>(*a);          \
    return (int)cudaGetLastError();                                                                               \
  }
  SMALL_CLASSES(SMALL_FX_LAUNCH)
#undef SMALL_FX_LAUNCH
  return (int)cudaErrorInvalidValue;
}
