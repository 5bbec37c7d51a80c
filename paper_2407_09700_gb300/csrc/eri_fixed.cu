// FP64-accurate class kernels with the Eq. 1 assembly in block fixed point (eri_fixed.cuh), for
// the classes that run with more than one lane per shell quartet.  Teams, tasks, batches of
// primitive quartets, the transfer relations and the digestion are those of eri_class_kernel
// (see eri_kernels.cu); the 2D recurrences are FP64 as there, the roots and weights FP64 Horner sums
// (rys_root64: in 64-bit integers, as in the class kernel, (dp|pp) took 61 instead of 54 ms).  Per batch:
//   a. primitive-quartet scalars, b. roots and 2D tables (FP64, in shared memory);
//   c. lanes over the table entries: the largest exponent of the entry over the batch's
//      primitives and roots, then the entry's limbs in place of its doubles;
//   d. each lane sums its tiles in 64-bit integers and returns them to FP64.  A tile is two
//      products I_x I_y by two I_z: values whose I_x I_y have the same list of I_z offsets form
//      rectangles, cut into such tiles (5-45 % of the sums are padding, most in small classes),
//      so four sums need four I_x, I_y and two I_z loads and two products.  All tiles have one
//      shape and every team of a warp runs as many steps (missing primitives are zero limbs),
//      so a step is straight-line code: with a branch per slot (lane programs) the same sums
//      left each warp waiting 7 cycles per instruction and the 16-atom medium build took 941 ms
//      against 811 ms with FP64 lane programs.
// Measured on that build (CUDA events, FP64 class kernel -> this): (dd|pp) 43.9 -> 24.9 ms, (dd|dp) 56.3 ->
// 39.0, (dp|dp) 64.8 -> 45.7, (pp|pp) 29.2 -> 18.7, (dp|ds) 71.0 -> 60.7, (dp|pp) 64.0 -> 58.9; all
// nine classes 430 -> 331 ms.  In (dp|dp) the FP64 pipe (recurrences, roots, transfer, digestion)
// is 49 % busy, the issue slots 52 %: the three warps of a scheduler mostly wait for the fixed
// latency of dependent integer instructions.
#include <cuda_runtime.h>
#include <stdint.h>

#include "eri_device.cuh"
#include "eri_fixed.cuh"

namespace {

// TS lanes per quartet, NT tiles per lane and pass.
template <int TS, int NT>
__global__ void __launch_bounds__(TPB, 3) eri_fixed_kernel(const KernelArgs a) {
  extern __shared__ double smem[];
  constexpr int TEAMS_PER_WARP = 32 / TS;
  const int lane = threadIdx.x & 31;
  const int tl = lane % TS;
  const int team_in_block = threadIdx.x / TS;
  const long long gteam = (long long)blockIdx.x * (TPB / TS) + team_in_block;
  const ClassDesc& c = a.c;
  const int N = c.nroots, nI = c.nI, nIs = c.nIs, Le = c.Le, Lf = c.Lf, bp = c.bp;
  const int str = 3 * nIs;                             // entries between steps

  // team region: [bp][NPD] and [bp][NPR] doubles, [bp N][3] tables of nI entries nIs apart (step
  // j N + n: primitive j, root n; doubles, then their limbs), K of the 3 nI entries,
  // the steps' shifts
  Smem<double> sd, sr;
  sd.base = smem + (size_t)team_in_block * c.team_doubles;
  sd.es = 1;
  sr.base = sd.base + bp * NPD;
  sr.es = 1;
  const int S_2D = bp * NPR;
  int2* tab = reinterpret_cast<int2*>(sr.base + S_2D);
  const int ntab = bp * 3 * N * nIs;
  int32_t* Kexp = reinterpret_cast<int32_t*>(tab + ntab);
  int32_t* Kstep = Kexp + 3 * nI;

  double* scr = a.scratch + gteam * c.scratch_per_team;
  double* E0 = scr;
  double* bufA = scr + c.nout;
  double* bufB = bufA + c.hrr_doubles;
  double* part = scr + c.part_off;

  unsigned long long cnt_q = 0, cnt_p = 0;
  const bool listed = a.tlist != nullptr || a.jobs != nullptr;
  const int qs = a.qsplit > 1 ? a.qsplit : 1;
  const long long ntask = (listed ? (long long)*a.tcount : a.ntask) * qs;

  while (true) {
    unsigned long long tbase = 0;
    if (lane == 0) tbase = atomicAdd(a.counter, (unsigned long long)TEAMS_PER_WARP);
    tbase = __shfl_sync(0xffffffffu, tbase, 0);
    if (tbase >= (unsigned long long)ntask) break;
    const long long slot = (long long)tbase + lane / TS;
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
    if (tl == 0 && active) { cnt_q += (ch == qs - 1) ? 1 : 0; cnt_p += (unsigned long long)nq; }
    double AB[3], CD[3];
    if (active) {
      AB[0] = bra->AB[0]; AB[1] = bra->AB[1]; AB[2] = bra->AB[2];
      CD[0] = ket->AB[0]; CD[1] = ket->AB[1]; CD[2] = ket->AB[2];
    }
    const int boff = active ? bra->prim_off : 0, koff = active ? ket->prim_off : 0;

    // a. and b. of one batch (the FP64 steps of eri_class_kernel)
    auto batch_tables = [&](int q0, int nbt, int nstw) {
      for (int j = tl; j < bp; j += TS) {
        if (j < nbt) {
          const int q = qlo + q0 + j;
          // ket primitives up and down in turn, so that neighbours in a batch have like exponents
          const int ibp = q / npk, r = q - ibp * npk;
          const int ix = boff + ibp, iy = koff + ((ibp & 1) ? npk - 1 - r : r);
          const PrimPair* x = tc.prims + ix;
          const PrimPair* y = tc.prims + iy;
          const double zeta = x->zeta, eta = y->zeta;
          const double rd = rsqrt(zeta + eta);
          double PQ0, PQ1, PQ2;
          pair_distance(tc, x, y, ix, iy, PQ0, PQ1, PQ2);
          const double inv_s = rd * rd;
          const double T = zeta * eta * inv_s * fma(PQ0, PQ0, fma(PQ1, PQ1, PQ2 * PQ2));
          rys_put_team(sd, j * NPD, rys_locate(T, a.rys_tcut_hi));
          const double rz = eta * inv_s, re = zeta * inv_s;
          const int o = j * NPR;
          sr[o + 0] = x->PA[0]; sr[o + 1] = x->PA[1]; sr[o + 2] = x->PA[2];
          sr[o + 3] = y->PA[0]; sr[o + 4] = y->PA[1]; sr[o + 5] = y->PA[2];
          sr[o + 6] = rz * PQ0; sr[o + 7] = rz * PQ1; sr[o + 8] = rz * PQ2;
          sr[o + 9] = re * PQ0; sr[o + 10] = re * PQ1; sr[o + 11] = re * PQ2;
          sr[o + 12] = 0.5 * inv_s;
          sr[o + 13] = x->hz * rz;
          sr[o + 14] = y->hz * re;
          sr[o + 15] = x->E * y->E * rd;
          sr[o + 16] = x->hz;
          sr[o + 17] = y->hz;
        }
      }
      team_sync<TS>();
      if (c.split3) {
        for (int tk = tl; tk < bp * N * 3; tk += TS) {
          const int jn = tk / 3, ax = tk - jn * 3;
          const int j = jn / N, n = jn - (jn / N) * N;
          if (j < nbt) {
            const int o = j * NPR;
            double u, w;
            rys_root64(a.rys_coef64, a.rys_au, a.rys_aw, N, rys_get_team(sd, j * NPD), n, u, w);
            const double B00 = u * sr[o + 12];
            const double B10 = fma(-u, sr[o + 13], sr[o + 16]);
            const double B01 = fma(-u, sr[o + 14], sr[o + 17]);
            const double Cax = fma(-u, sr[o + 6 + ax], sr[o + 0 + ax]);
            const double Cpx = fma(u, sr[o + 9 + ax], sr[o + 3 + ax]);
            const double I00 = (ax == 2) ? w * sr[o + 15] : 1.0;
            rys_2d1<double>(sr, S_2D + jn * str + ax * nIs, Le, Lf, I00, Cax, Cpx, B00, B10, B01);
          }
        }
      } else {
        for (int tk = tl; tk < bp * N; tk += TS) {
          const int j = tk / N, n = tk - (tk / N) * N;
          if (j < nbt) {
            const int o = j * NPR;
            double u, w;
            rys_root64(a.rys_coef64, a.rys_au, a.rys_aw, N, rys_get_team(sd, j * NPD), n, u, w);
            const double B00 = u * sr[o + 12];
            const double B10 = fma(-u, sr[o + 13], sr[o + 16]);
            const double B01 = fma(-u, sr[o + 14], sr[o + 17]);
            const double wt = w * sr[o + 15];
            const double C[3] = {fma(-u, sr[o + 6], sr[o + 0]), fma(-u, sr[o + 7], sr[o + 1]),
                                 fma(-u, sr[o + 8], sr[o + 2])};
            const double Cp[3] = {fma(u, sr[o + 9], sr[o + 3]), fma(u, sr[o + 10], sr[o + 4]),
                                  fma(u, sr[o + 11], sr[o + 5])};
            const int g0 = S_2D + tk * str;
            const int og[3] = {g0, g0 + nIs, g0 + 2 * nIs};
            rys_2d3<double>(sr, og, Le, Lf, wt, C, Cp, B00, B10, B01);
          }
        }
      }
      team_sync<TS>();
      // c. limbs in place of the doubles; zeros in the steps past this team's primitives
      const int nst = nbt > 0 ? nbt * N : 0;
      // shift of step st's I_x and I_y (I_z: twice its negative): a third of the binary exponent
      // of I_z(0, 0) = w Theta
      auto kappa = [&](int st) { return fx_third(((tab[st * str + 2 * nIs].y >> 20) & 0x7ff) - 1023); };
      for (int st = tl; st < nst; st += TS) Kstep[st] = kappa(st);
      team_sync<TS>();
      for (int i = tl; i < 3 * nI; i += TS) {
        const int ax = i / nI, o0 = ax * nIs + (i - ax * nI);
        const int mul = ax == 2 ? -2 : 1;
        int emax = -4096;
        bool bad = false;
        for (int st = 0; st < nst; ++st) {
          const int e = (tab[o0 + st * str].y >> 20) & 0x7ff;
          if (e) emax = max(emax, e + mul * Kstep[st]);
          bad |= e == 0x7ff;
        }
        Kexp[i] = bad ? FX_POISON : emax - 1022;
        const int top = fx_top(ax);
#pragma unroll 2
        for (int st = 0; st < nst; ++st) {
          const int2 v = tab[o0 + st * str];
          int32_t l[2];
          fx_split((uint32_t)v.y, (uint32_t)v.x, emax - mul * Kstep[st], top, l);
          tab[o0 + st * str] = make_int2(l[0], l[1]);
        }
        for (int st = nst; st < nstw; ++st) tab[o0 + st * str] = make_int2(0, 0);
      }
      team_sync<TS>();
    };
    auto load = [&](int o, int32_t l[2]) {
      const int2 v = tab[o];
      l[0] = v.x;
      l[1] = v.y;
    };
    // d. one pass: a batch's sums of this lane's tiles, added to the slot-ordered partial sums in
    //    the team's scratch, and to E0 in [e][f] order after the last batch
    auto assemble = [&](int pass, int nbt, int nstw, bool first, bool last) {
      const int t0 = pass * NT * TS + tl;                            // tile k: t0 + k TS
      int ox[NT][2], oy[NT][2], oz[NT][2];
      int64_t acc[NT][4][2];
#pragma unroll
      for (int k = 0; k < NT; ++k) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(c.outidx) + t0 + k * TS);
        ox[k][0] = (int)(w.x & 0xffu);
        oy[k][0] = (int)((w.x >> 8) & 0xffu) + nIs;
        ox[k][1] = (int)((w.x >> 16) & 0xffu);
        oy[k][1] = (int)(w.x >> 24) + nIs;
        oz[k][0] = (int)(w.y & 0xffffu) + 2 * nIs;
        oz[k][1] = (int)(w.y >> 16) + 2 * nIs;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          acc[k][q][0] = acc[k][q][1] = 0;
      }
      for (int st = 0; st < nstw; ++st) {
        const int o = st * str;
#pragma unroll
        for (int k = 0; k < NT; ++k) {
          int32_t x[2], y[2], v0[2], v1[2], z[2];
          load(o + ox[k][0], x);
          load(o + oy[k][0], y);
          fx_mul(x, y, v0);
          load(o + ox[k][1], x);
          load(o + oy[k][1], y);
          fx_mul(x, y, v1);
          load(o + oz[k][0], z);
          fx_mac(v0, z, acc[k][0]);
          fx_mac(v1, z, acc[k][1]);
          load(o + oz[k][1], z);
          fx_mac(v0, z, acc[k][2]);
          fx_mac(v1, z, acc[k][3]);
        }
      }
      if (active) {
#pragma unroll
        for (int k = 0; k < NT; ++k) {
          const uint4 d4 = __ldg(reinterpret_cast<const uint4*>(c.dst) + t0 + k * TS);
          const uint32_t d[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int o = ((pass * NT + k) * 4 + q) * TS + tl;
            double r = first ? 0.0 : part[o];
            if (nbt > 0)
              r = fx_flush(acc[k][q],
                              Kexp[ox[k][q & 1]] + Kexp[oy[k][q & 1] - nIs + nI] + Kexp[oz[k][q >> 1] - 2 * nIs + 2 * nI], r);
            if (!last) part[o] = r;
            else if (d[q] != 0xffffffffu) E0[d[q]] = r;
          }
        }
      }
    };
    const int nbatch = (maxq + bp - 1) / bp;        // uniform
    for (int bi = 0; bi < nbatch; ++bi) {
      const int q0 = bi * bp, nbt = min(bp, nq - q0);   // this team's primitives (may be <= 0)
      const int nstw = min(bp, maxq - q0) * N;          // the warp's steps
      batch_tables(q0, nbt, nstw);
      for (int pass = 0; pass < c.npass; ++pass) assemble(pass, nbt, nstw, bi == 0, bi == nbatch - 1);
      team_sync<TS>();
    }
    finish_quartet<TS, double>(a, tc, c, E0, bufA, bufB, tl, active, AB, CD, bra, ket, ib, ik, task, sd.base,
                               c.team_doubles);
    team_sync<TS>();
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

// instantiated lanes per quartet and tiles per lane and pass
#define FIXED_KERNELS(X) X(16, 2) X(16, 3) X(32, 3)

const void* fixed_ptr(int ts, int tiles) {
#define FIXED_CASE(T, NT) \
  if (ts == T && tiles == NT) return (const void*)eri_fixed_kernel<T, NT>;
  FIXED_KERNELS(FIXED_CASE)
#undef FIXED_CASE
  return nullptr;
}

}  // namespace

extern "C" int erik_upload_cart_tables_fixed(void) { return (int)upload_cart_table(); }

extern "C" int erik_fixed_blocks_per_sm(int ts, int tiles, int smem_bytes, int* out) {
  const void* k = fixed_ptr(ts, tiles);
  if (!k) return (int)cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return (int)e;
  return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k, TPB, smem_bytes);
}

extern "C" int erik_launch_fixed(int ts, int tiles, const KernelArgs* a, int grid, int smem_bytes, void* stream) {
  const void* k = fixed_ptr(ts, tiles);
  if (!k || a->mode != KMODE_JK) return (int)cudaErrorInvalidValue;
  void* args[] = {const_cast<KernelArgs*>(a)};
  return (int)cudaLaunchKernel(k, dim3(grid), dim3(TPB), args, (size_t)smem_bytes, (cudaStream_t)stream);
}
