// Device code of the batched ROS4 chemistry integrator (FP64, sm_103a).
//
// Compiled at run time by NVRTC, once per mechanism and launch configuration, after a
// generated header (chem_host.cpp, emit_mechanism) that defines:
//   NS, NR            species and reactions; the state length is NS ([T, n_1..n_{NS-1}])
//   TEAM, TPB         lanes per cell (1, 4, 8, 16, 32 or TPB) and threads per block
//   MIN_BLOCKS        blocks per SM that the integrator's registers must leave room for
//   CHUNK, NCHUNK     reactions per chunk of the multi-lane reaction loop, number of chunks
//   tables mk_*       NASA-7 coefficients pre-divided for cp and h; rate constants as fixed-point
//                     base-2 logarithms; one record per reaction; gather lists; efficiencies;
//                     falloff data (see emit_mechanism)
// and after fxmath.cuh (exp2, log2 and reciprocals on the integer pipe).
//
// What the kernels compute (Curtis, Niemeyer & Sung):
//   * f(y), Sec. 2.1 Eq. (e:dphidt): concentrations from the unit-mass closure of Eq. (e:n_nsp);
//     NASA-7 thermo; Arrhenius / third-body / Lindemann / Troe forward rates; reverse rates from
//     the equilibrium constant; net production rates; dT/dt from the constant-pressure energy
//     balance;
//   * the analytical Jacobian J = df/dy, Eq. (e:jac), in closed form: the reaction part
//     d(omega)/dC (sparse gather plus the dense third-body efficiency part), then the chain
//     rule to the [T, n] state (the bath-gas column, the volume terms and the temperature row);
//   * the transformed ROS4 step of Sec. 2.3 with partial-pivoting LU of (I/(gamma h) - J), four
//     stage solves (three f evaluations: the Hairer-Wanner set repeats stage 3's argument for
//     stage 4), the embedded error estimate and the step-size controller;
//   * batching (Sec. 2.4.1): a persistent kernel whose teams pull cells from a device work
//     queue, and a plain form that runs one step attempt per launch.
//
// Work decomposition.  A "team" of TEAM threads owns one cell at a time; all of the cell's
// working set (the N x N matrix, stage vectors, thermo and rate scratch) sits in shared memory.
// TEAM == 1: one thread per cell, arrays interleaved across the block's threads (stride TPB)
// so that lane-consecutive accesses hit consecutive banks.  TEAM == 4, 8, 16: several cells per
// warp (sub-warp teams, for small mechanisms whose loops would leave most lanes of a wider team
// idle), contiguous arrays per team, team-masked warp synchronisation and shuffles.  TEAM == 32:
// a warp per cell.  TEAM == TPB (64..256): a block per cell.  Reaction loops give each lane a
// subset of reactions; the team then gathers their rates by species and by Jacobian entry.
// Every device loop is bounded; there is no grid-wide wait.
//
// What sets the time on GB300: an FP64 warp instruction takes 64 clocks of an SM sub-partition (16 of
// the SM) and 64 of latency, an integer multiply 1 to 2, a tensor-core instruction 8.  So whatever is
// not an FP64 sum or product of the state goes elsewhere: exponentials, logarithms and reciprocals
// to the integer pipe, the LU's trailing update to the tensor cores, sums of lists to registers.

#define ELEM 0
#define THIRD 1
#define LIND 2
#define TROE 3

#define R_U 8314.462618
#define INV_R_U (1.0 / 8314.462618)
#define P_ATM 101325.0
#define R_OVER_PATM (8314.462618 / 101325.0)
#define PATM_OVER_R (101325.0 / 8314.462618)
#define LN10 2.302585092994046
#define LN2 0.6931471805599453
#define LOG10_2 0.30102999566398120
#define LOG2_10 3.3219280948873623
#define LOG2_PATM_R 3.60722334318630807
// the same and log2(1e-300) in Q52
#define FX_LOG2_PATM_R 16245489704216012LL
#define FX_LOG2_1EM300 (-4488190239085892024LL)

#define ST_OK 0
#define ST_MAX_STEPS 1
#define ST_H_UNDERFLOW 2
#define ST_NONFINITE 3
#define ST_SKIPPED 4
#define ST_TAPE_FULL 5

#define NEQ NS
#define NB ((NEQ + WL - 1) / WL)  // WL-row chunks of a state vector held by the first warp
#define BATH (NS - 1)

#define SUBWARP (TEAM > 1 && TEAM < 32)
#if TEAM == 1
#define SS TPB
#define NTEAM TPB
#elif TEAM <= 32
#define SS 1
#define NTEAM (TPB / TEAM)
#else
#define SS 1
#define NTEAM 1
#endif
// lanes of the team's first warp (the warp-level parts: pivot scale, stage solves) and the
// first butterfly offset of a team reduction
#define WL (TEAM < 32 ? TEAM : 32)
#define XOR0 (WL / 2)

// per-cell shared-memory slots (units of SS doubles), sized so that eight 53-species cells fit
// in one SM's shared memory:
// * f at a stage argument overwrites the argument (OFF_F = OFF_YT): the argument is dead once
//   the concentrations and thermo are formed from it;
// * what only the Jacobian assembly uses aliases YT and the stage vectors, which are dead while the
//   Jacobian is formed (it is the first thing a step attempt computes): d omega/dT in YT, B_k in the
//   last stage slot, the rate constants of a chunk of reactions (OFF_KF) from U1 on, and, after the
//   reactions, f(y) in U1 and AL in U2; the chain rule writes JT over DOMT and BE over BK in place;
// * the LU keeps 1/U_kk on the diagonal of A, and the row permutation is packed two ints per
//   slot (the single-lane layout also keeps the pivot sequence).
#define OFF_A 0
#define OFF_Y (OFF_A + NEQ * NEQ)
#define OFF_YT (OFF_Y + NEQ)
#define OFF_F OFF_YT
#define OFF_U1 (OFF_YT + NEQ)
#define OFF_U2 (OFF_U1 + NEQ)
#define OFF_U3 (OFF_U2 + NEQ)
#define OFF_U4 (OFF_U3 + NEQ)
// at least three stage slots (the Jacobian assembly uses the first two and the last)
#define NSTG (RS > 3 ? RS : 3)
#if NEED_F0
#define OFF_F0 (OFF_U1 + NSTG * NEQ)  // f(y) kept for a later stage whose argument is y itself
#define OFF_C (OFF_F0 + NEQ)
#else
#define OFF_C (OFF_U1 + NSTG * NEQ)
#endif
#define OFF_CP (OFF_C + NS)
#define OFF_HRT (OFF_CP + NS)
#define OFF_G (OFF_HRT + NS)  // log2 exp(s/R - h/RT): Q52 integers, doubles outside fx_range
#define OFF_OM (OFF_G + NS)
#define OFF_DOMT OFF_YT
#define OFF_BK (OFF_U1 + (NSTG - 1) * NEQ)
#define OFF_AL OFF_U2
#define OFF_JT OFF_DOMT
#define OFF_BE OFF_BK
#define PACKED_INTS(n) (((n) + 1) / 2)
#if TEAM == 1
#define OFF_PIV (OFF_OM + NS)
#define OFF_PERM (OFF_PIV + PACKED_INTS(NEQ))
#else
#define OFF_PERM (OFF_OM + NS)
#endif
// net rates of a chunk of CHUNK reactions, and their rate constants (k_f, then k_r): where they fit
// among the dead stage slots, else behind the net rates
#define OFF_Q (OFF_PERM + PACKED_INTS(NEQ))
#if TEAM == 1
#define OFF_RED OFF_Q
#elif 2 * CHUNK <= (NSTG - 1) * NEQ
#define OFF_KF OFF_U1
#define OFF_RED (OFF_Q + CHUNK)
#else
#define OFF_KF (OFF_Q + CHUNK)
#define OFF_RED (OFF_Q + 3 * CHUNK)
#endif
#define SLOTS (OFF_RED + 24)
// lanes that share a row (column) of the matrix in the Jacobian's row and column sums, and the row
// count rounded up so that whole warps take part in their shuffles
#if TEAM > 1 && TEAM >= 4 * NS
#define RSPLIT 4
#elif TEAM > 1 && TEAM >= 2 * NS
#define RSPLIT 2
#else
#define RSPLIT 1
#endif
// the blocked LU: a row (and a column) of the matrix per lane, and room for its exchanges in the
// five thermo slots; narrower teams take the column-by-column form, and so do systems of up to 32
// species (13 species: 19.8 K clocks against 27.8 K blocked, 53 species: 190 K against 149 K)
#define LU_MIN 33
#if TEAM >= 32 && NEQ <= TEAM && NEQ >= LU_MIN && 22 * ((NEQ + 31) / 32 + 1) + 16 <= 5 * NS
#define LU_BLOCKED 1
#else
#define LU_BLOCKED 0
#endif
// the blocked stage solves: RSPLIT lanes per row of the matrix
#if TEAM >= 32 && NEQ <= TEAM
#define SOLVE_BLK 1
#else
#define SOLVE_BLK 0
#endif
#define NS_PAD ((NS + TEAM / RSPLIT - 1) / (TEAM / RSPLIT) * (TEAM / RSPLIT))
// distance between consecutive teams' slots: for sub-warp teams padded to TEAM (mod 16) doubles,
// so that the teams of a half-warp reading the same offset of their arrays use disjoint banks
#if SUBWARP
#define TSTRIDE (SLOTS + ((TEAM - SLOTS % 16 + 16) % 16))
#else
#define TSTRIDE SLOTS
#endif
#define UOFF(i) (OFF_U1 + (i) * NEQ)

// Per-cell cache of the W-method's factorised iteration matrix (chem_int_opts.jac_cache, global
// memory, one contiguous block per cell whatever the launch configuration): the N x N factors with
// 1/U_kk on the diagonal, the composed row permutation and the pivot sequence (packed ints), the
// step size h_W they were built for (0: empty) and their age in accepted steps.  A new factorisation
// (Jacobian at the attempt's state) is made when h_W differs from the attempt's step size or
// the age reaches WAGE_MAX.
#define WC_PERM (NEQ * NEQ)
#define WC_PIV (WC_PERM + PACKED_INTS(NEQ))
#define WC_H (WC_PIV + PACKED_INTS(NEQ))
#define WC_AGE (WC_H + 1)
#define WC_STRIDE (WC_AGE + 1)
#define WAGE_MAX 32

// ------------------------------------------------------------------------------ team plumbing

// mask of the calling lane's team within its warp (all lanes for TEAM >= 32)
__device__ __forceinline__ unsigned team_mask() {
#if SUBWARP
  return ((1u << TEAM) - 1u) << ((threadIdx.x & 31) & ~(TEAM - 1));
#else
  return 0xffffffffu;
#endif
}

__device__ __forceinline__ void tsync() {
#if SUBWARP
  __syncwarp(team_mask());
#elif TEAM == 32
  __syncwarp();
#elif TEAM > 32
  __syncthreads();
#endif
}

struct Team {
  double* base;  // element i of array at slot offset o: base[(o + i) * SS]
  int tl;        // lane within the team
  __device__ __forceinline__ double& at(int o, int i) const { return base[(o + i) * SS]; }
  __device__ __forceinline__ double& A(int i, int j) const { return base[(OFF_A + i * NEQ + j) * SS]; }
#if TEAM == 1
  __device__ __forceinline__ int& piv(int i) const {
    return reinterpret_cast<int*>(&base[(OFF_PIV + (i >> 1)) * SS])[i & 1];
  }
#endif
  __device__ __forceinline__ int& perm(int i) const {
    return reinterpret_cast<int*>(&base[(OFF_PERM + (i >> 1)) * SS])[i & 1];
  }
  // 1/U_kk of the factorised matrix, kept on its diagonal
  __device__ __forceinline__ double& invd(int k) const { return A(k, k); }
};

extern __shared__ double smem[];

__device__ __forceinline__ Team make_team() {
  Team tm;
#if TEAM == 1
  tm.base = smem + threadIdx.x;
  tm.tl = 0;
#elif TEAM <= 32
  tm.base = smem + (threadIdx.x / TEAM) * TSTRIDE;
  tm.tl = threadIdx.x & (TEAM - 1);
#else
  tm.base = smem;
  tm.tl = threadIdx.x;
#endif
  return tm;
}

// The parts of a step attempt are functions of their own, called out of line: inlined into every place
// that uses them the integrator was 480 to 780 KB of instructions, far beyond the SM's instruction
// caches, and spent most of its time fetching them.  They find the team's shared memory
// themselves (a pointer argument would lose its address space).
#define OUTLINE __device__ __noinline__

#if TEAM > 32
// sum of the team's warp partials, in every lane (shuffles: log2 of the warp count FP64 adds per
// warp, where a loop over the partials takes one each)
__device__ __forceinline__ double warp_partials(const double* red) {
  double v = red[threadIdx.x & (TEAM / 32 - 1)];
#pragma unroll
  for (int o = TEAM / 64; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
#endif

// sum over the team; every lane gets the same bits (butterfly with commutative adds)
__device__ __forceinline__ double team_sum(const Team& tm, double v) {
#if TEAM == 1
  return v;
#else
  const unsigned msk = team_mask();
#pragma unroll
  for (int o = XOR0; o > 0; o >>= 1) v += __shfl_xor_sync(msk, v, o);
#if TEAM > 32
  double* red = &tm.base[OFF_RED];
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = warp_partials(red);
  __syncthreads();
#endif
  return v;
#endif
}

// maximum over the team (same reduction tree as team_sum)
__device__ __forceinline__ double team_max(const Team& tm, double v) {
#if TEAM == 1
  return v;
#else
  const unsigned msk = team_mask();
#pragma unroll
  for (int o = XOR0; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(msk, v, o));
#if TEAM > 32
  double* red = &tm.base[OFF_RED];
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = red[0];
  for (int w = 1; w < TEAM / 32; ++w) v = fmax(v, red[w]);
  __syncthreads();
#endif
  return v;
#endif
}

// two sums over the team in one reduction
__device__ __forceinline__ void team_sum2(const Team& tm, double& a, double& b) {
#if TEAM > 1
  const unsigned msk = team_mask();
#pragma unroll
  for (int o = XOR0; o > 0; o >>= 1) {
    a += __shfl_xor_sync(msk, a, o);
    b += __shfl_xor_sync(msk, b, o);
  }
#if TEAM > 32
  double* red = &tm.base[OFF_RED];
  __syncthreads();
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = a;
    red[TEAM / 32 + (threadIdx.x >> 5)] = b;
  }
  __syncthreads();
  a = warp_partials(red);
  b = warp_partials(red + TEAM / 32);
  __syncthreads();
#endif
#endif
}

// any-lane flag over the team
__device__ __forceinline__ bool team_any(const Team& tm, bool f) {
#if TEAM == 1
  return f;
#elif TEAM <= 32
  return __any_sync(team_mask(), f);
#else
  return __syncthreads_or(f) != 0;
#endif
}

template <class T>
__device__ __forceinline__ void scatter_add(double* p, double v) {
#if TEAM == 1
  *p += v;
#else
  atomicAdd(p, v);
#endif
}

// sum over the RSPLIT adjacent lanes of a row (they are of one team, whose lanes alone take part: the
// other teams of a warp are at their own cells)
__device__ __forceinline__ double rsplit_sum(double v) {
#pragma unroll
  for (int o = RSPLIT / 2; o > 0; o >>= 1) v += __shfl_xor_sync(team_mask(), v, o);
  return v;
}

// |x| as an order-preserving integer (integer pipe instead of the FP64 pipe)
__device__ __forceinline__ long long abs_key(double x) {
  return __double_as_longlong(x) & 0x7fffffffffffffffLL;
}

// ------------------------------------------------------------------------------ thermo + C

// Concentrations, thermo per species and mixture sums for state y (slot OFF_Y or OFF_YT): writes C,
// cp, h/RT, log2 exp(s/R - h/RT) and (WJ) the sum of n dcp/dT.
struct CellScalars {
  double T, invT, V, cpm, dcpm;  // cpm = sum n_k cp_k / R, dcpm = sum n_k dcp_k/dT / R
  double l2T;                    // log2 T
  fx_i64 l2Tq, iTq;              // log2 T in Q59 and 1/T in Q71 (fx only)
  bool fx;                       // logarithms of the rate constants in fixed point
};

// Where the fixed-point logarithms hold: 1/T < 2^-8 fits Q71 and log2 T < 13 fits Q59.  MECH_FX says
// that the mechanism's own numbers keep every logarithm below 1900 (of 2048) over this range;
// temperatures outside of it (or NaN) take the FP64 functions.
__device__ __forceinline__ bool fx_range(double T) { return MECH_FX && T > 256.0 && T < 8192.0; }

// mass closure: n_bath = (1 - sum_k W_k n_k) / W_bath; n_tot = sum of all moles; V = n_tot R T/P,
// 1/V = (P/RT) / n_tot
__device__ __forceinline__ void closure_scalars(const Team& tm, double T, double invT, double P, double wsum,
                                                double nsum, double& nb, double& V, double& invV) {
  nb = (1.0 - wsum) * mk_invW[BATH];
  const double nt = nsum + nb;
#if TEAM == 1
  const double rn = fx_rcp(nt), rP = fx_rcp(P);
#else
  // two lanes take the two reciprocals at once
  const double r = fx_rcp((tm.tl & 1) ? P : nt);
  const unsigned msk = team_mask();
  const double rn = __shfl_sync(msk, r, 0, WL), rP = __shfl_sync(msk, r, 1, WL);
#endif
  V = nt * (R_U * T) * rP;
  invV = rn * (P * invT * INV_R_U);
}

__device__ __noinline__ double log2_slow(double x) { return log2(x); }

// WJ: with what the Jacobian needs
__device__ __forceinline__ void thermo_conc(const Team& tm, int oy, double P, CellScalars& cs, const bool WJ) {
  const double T = tm.at(oy, 0);
  cs.T = T;
  cs.fx = fx_range(T);
  if (cs.fx) {
    const int e = fx_exponent(T);  // 8 .. 12
    const fx_u64 x = fx_rcp_mant(fx_mant(T));
    cs.iTq = (fx_i64)(x >> (e - 8));
    cs.invT = fx_as_double(((fx_u64)(1021 - e) << 52) + ((x + 0x200) >> 10));
    cs.l2Tq = ((fx_i64)e << 59) + (fx_log2_mant(fx_mant(T)) >> 3);
    cs.l2T = fx_to_double(cs.l2Tq, 59);
  } else {
    cs.invT = fx_rcp_slow(T);
    cs.l2T = log2_slow(T);
  }
  const double invT = cs.invT, l2T = cs.l2T;
  double nb, V, invV;
  // the closure's sums: by the last warp alone (it holds the fewest species), while the others
  // begin with the thermo polynomials
#if TEAM > 32
  if (tm.tl >= TEAM - 32) {
    double wsum = 0.0, nsum = 0.0;
    for (int k = tm.tl - (TEAM - 32); k < NS - 1; k += 32) {
      const double n = tm.at(oy, 1 + k);
      wsum += mk_W[k] * n;
      nsum += n;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
      nsum += __shfl_xor_sync(0xffffffffu, nsum, o);
    }
    closure_scalars(tm, T, invT, P, wsum, nsum, nb, V, invV);
    if (tm.tl == TEAM - 1) {
      tm.base[OFF_RED + 18] = nb;
      tm.base[OFF_RED + 19] = V;
      tm.base[OFF_RED + 20] = invV;
    }
  }
#else
  {
    double wsum = 0.0, nsum = 0.0;
    for (int k = tm.tl; k < NS - 1; k += TEAM) {
      const double n = tm.at(oy, 1 + k);
      wsum += mk_W[k] * n;
      nsum += n;
    }
    team_sum2(tm, wsum, nsum);
    closure_scalars(tm, T, invT, P, wsum, nsum, nb, V, invV);
  }
#endif
  double cpm = 0.0, dcpm = 0.0, cpb = 0.0, dcpb = 0.0;
  for (int k = tm.tl; k < NS; k += TEAM) {
    const double n = k < NS - 1 ? tm.at(oy, 1 + k) : 0.0;
    const int r = T < mk_Tmid[k] ? 0 : 1;
    const double* c = mk_cp[k][r];
    const double* hh = mk_h[k][r];
    const double* g = mk_g[k][r];
    const double cp = c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4])));
    const double hRT = hh[0] + T * (hh[1] + T * (hh[2] + T * (hh[3] + T * hh[4]))) + hh[5] * invT;
    // log2 exp(s/R - h/RT): the large terms a1 log2 T and -a6/(T ln2) in fixed point, exact to 2^-52
    const double lg = g[0] + T * (g[1] + T * (g[2] + T * (g[3] + T * g[4])));
    if (cs.fx) {
      const longlong2 gq = mk_gq[k][r];
      const fx_i64 G = fx_from_double(lg, 52) + fx_mulhi_s(gq.x, cs.l2Tq) + fx_mulhi_s(gq.y, cs.iTq);
      tm.at(OFF_G, k) = fx_as_double((fx_u64)G);
    } else {
      tm.at(OFF_G, k) = lg + c[0] * l2T - hh[5] * invT * (1.0 / LN2);
    }
    tm.at(OFF_CP, k) = cp;
    tm.at(OFF_HRT, k) = hRT;
    cpm += n * cp;
    if (k == BATH) cpb = cp;
    if (WJ) {
      const double* d = mk_dcp[k][r];
      const double dcp = d[0] + T * (d[1] + T * (d[2] + T * d[3]));
      dcpm += n * dcp;
      if (k == BATH) dcpb = dcp;
    }
  }
#if TEAM > 32
  __syncthreads();
  nb = tm.base[OFF_RED + 18];
  V = tm.base[OFF_RED + 19];
  invV = tm.base[OFF_RED + 20];
#endif
  cpm += nb * cpb;  // the bath's lane
  if (WJ) dcpm += nb * dcpb;
  for (int k = tm.tl; k < NS; k += TEAM) tm.at(OFF_C, k) = (k < NS - 1 ? tm.at(oy, 1 + k) : nb) * invV;
  cs.V = V;
  if (WJ) {
    team_sum2(tm, cpm, dcpm);
    cs.dcpm = dcpm;
  } else {
    cpm = team_sum(tm, cpm);
  }
  cs.cpm = cpm;
  tsync();
}

// ------------------------------------------------------------------------------ reactions

// -x by flipping the sign bit (integer pipe)
__device__ __forceinline__ double dneg(double x) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ULL);
}
// nu * x for an integer stoichiometric coefficient nu: no FP64 instruction when |nu| = 1, the
// common case
__device__ __forceinline__ double nu_times(int nu, double x) {
  if (nu == 1) return x;
  if (nu == -1) return dneg(x);
  return (double)nu * x;
}

// species index -> row/column of the state matrix: species 0..NS-2 -> 1..NS-1, bath -> 0
__device__ __forceinline__ int smap(int k) { return k == BATH ? 0 : k + 1; }

// Rate constants of one reaction and their derivatives: k_f and k_r (without the [M] factor of a
// THIRD reaction), d ln k_f / dT at constant C, d ln k_f / d[M], d ln K_c / dT is the caller's.
struct Rate {
  double kf, kr, dlT, dlM;
};

// FP64 form, for temperatures, ln A values or falloff blends outside the fixed-point range; lKc is
// log2 K_c.  Kept out of line: the normal path never comes here.
__device__ __noinline__ void rate_fp(int r, int kind, double T, double invT, double l2T, double lA, double M,
                                     double lKc, const bool WJ, Rate* out) {
  const double lnT = l2T * LN2;
  const double kinf = exp(lA + mk_b[r] * lnT - mk_th[r] * invT);
  double kf = kinf;
  double dlkf_dT = 0.0, dlkf_dM = 0.0;
  if (WJ) dlkf_dT = (mk_b[r] + mk_th[r] * invT) * invT;
  if (kind >= LIND) {
    const double k0 = exp(mk_lnA0[r] + mk_b0[r] * lnT - mk_th0[r] * invT);
    double Pr = k0 * M / kinf;
    bool floored = false;
    if (Pr < 1e-300) { Pr = 1e-300; floored = true; }
    double F = 1.0, dlF_dlPr = 0.0, dlF_dT = 0.0;
    if (kind == TROE) {
      const double a = mk_troe[r][0];
      const double e3 = exp(-T * mk_troe[r][1]);
      const double e1 = exp(-T * mk_troe[r][2]);
      const double T2 = mk_troe[r][3];
      const double e2 = T2 > 0.0 ? exp(-T2 * invT) : 0.0;
      const double Fc = (1.0 - a) * e3 + a * e1 + e2;
      const double lFc = log10(Fc);
      const double n = 0.75 - 1.27 * lFc;
      const double x = log10(Pr) + (-0.4 - 0.67 * lFc);
      const double id = 1.0 / (n - 0.14 * x);
      const double f1 = x * id;
      const double den = 1.0 / (1.0 + f1 * f1);
      F = exp(lFc * den * LN10);
      if (WJ) {
        const double g2 = 2.0 * lFc * f1 * den * den;  // -d log10F / d f1
        if (!floored) dlF_dlPr = -g2 * n * id * id;
        const double dFc = -(1.0 - a) * mk_troe[r][1] * e3 - a * mk_troe[r][2] * e1 +
                           (T2 > 0.0 ? T2 * invT * invT * e2 : 0.0);
        const double df1_dlFc = (-0.67 * n + 1.27 * x) * id * id;
        dlF_dT = (den - g2 * df1_dlFc) * dFc / Fc;
      }
    }
    kf = kinf * (Pr / (1.0 + Pr)) * F;
    if (WJ) {
      const double g = floored ? 0.0 : 1.0 / (1.0 + Pr) + dlF_dlPr;
      const double dlk0 = (mk_b0[r] + mk_th0[r] * invT) * invT;
      dlkf_dM = g / M;
      dlkf_dT = dlkf_dT + g * (dlk0 - dlkf_dT) + dlF_dT;
    }
  }
  out->kf = kf;
  out->kr = kf * exp2(-lKc);
  out->dlT = dlkf_dT;
  out->dlM = dlkf_dM;
}

// Falloff in fixed point: the logarithm of k (less that of 1 / (1 + Pr), returned as g1) from that of
// k_inf.
struct Falloff {
  fx_i64 lk;
  double g1, dlT, dlM;
  bool ok;
};
template <bool WJ>
__device__ __forceinline__ Falloff falloff_fx(int r, int kind, double T, double invT, fx_i64 l2Tq, fx_i64 iTq, double M,
                                           fx_i64 lk) {
  Falloff o;
  o.ok = false;
  // log2 Pr = log2 k0 + log2 [M] - log2 k_inf, floored at 1e-300
  const longlong2 k2 = mk_kfx0[r][0];
  fx_i64 lPr = FX_LOG2_1EM300;
  bool floored = true;
  if (fx_normal_pos(M)) {
    const fx_i64 l = k2.x + fx_mulhi_s(k2.y, l2Tq) - fx_mulhi_s(mk_kfx0[r][1].x, iTq) + fx_log2(M) - lk;
    if (l >= FX_LOG2_1EM300) { lPr = l; floored = false; }
  }
  o.g1 = fx_rcp(1.0 + fx_exp2(lPr));  // 1 / (1 + Pr)
  o.lk = lk + lPr;
  double dlF_dlPr = 0.0, dlF_dT = 0.0;
  if (kind == TROE) {
    const double a = mk_troe[r][0];
    const double* t = mk_troe_l2[r];  // log2(e) / T***, log2(e) / T*, log2(e) T**
    const double e3 = fx_exp2(-fx_from_double(T * t[0], 52));
    const double e1 = fx_exp2(-fx_from_double(T * t[1], 52));
    double Fc = (1.0 - a) * e3 + a * e1;
    double e2 = 0.0;
    if (t[2] > 0.0) {
      e2 = fx_exp2(-fx_from_double(t[2] * invT, 52));
      Fc += e2;
    }
    if (!fx_normal_pos(Fc)) return o;
    const double lFc = fx_log2_d(Fc) * LOG10_2;
    const double n = 0.75 - 1.27 * lFc;
    const double x = fx_to_double(lPr, 52) * LOG10_2 + (-0.4 - 0.67 * lFc);
    const double id = fx_rcp(n - 0.14 * x);
    const double f1 = x * id;
    const double den = fx_rcp(1.0 + f1 * f1);
    const double lF = lFc * den;
    if (!(fabs(lF) < 100.0)) return o;
    o.lk += fx_from_double(lF * LOG2_10, 52);
    if (WJ) {
      const double g2 = 2.0 * lF * f1 * den;  // -d log10F / d f1
      const double id2 = id * id;
      if (!floored) dlF_dlPr = -g2 * n * id2;
      double dFc = -(1.0 - a) * mk_troe[r][1] * e3 - a * mk_troe[r][2] * e1;
      if (t[2] > 0.0) dFc += mk_troe[r][3] * invT * invT * e2;
      const double df1_dlFc = (-0.67 * n + 1.27 * x) * id2;
      dlF_dT = (den - g2 * df1_dlFc) * dFc * fx_rcp(Fc);
    }
  }
  if (WJ) {
    const double dlk = (mk_b[r] + mk_th[r] * invT) * invT;
    const double g = floored ? 0.0 : o.g1 + dlF_dlPr;
    const double dlk0 = (mk_b0[r] + mk_th0[r] * invT) * invT;
    o.dlM = floored ? 0.0 : g * fx_rcp(M);
    o.dlT = dlk + g * (dlk0 - dlk) + dlF_dT;
  }
  o.ok = true;
  return o;
}

// Fixed-point form: log2 k in Q52 as ln A / ln2 + b log2 T - (theta / ln2) / T, the falloff blend and
// the equilibrium constant added as logarithms, one fx_exp2 for k_f and one for k_r.  An FP64
// exp() per reaction and the products of species' exponentials for k_r took 300 + 80 clocks of an
// SM per warp, the two integer exponentials take 60.  With the gathers below the source of 50,000
// 53-species cells went from 2.91 to 1.38 ms, 37 M cells/s; what bounds it now: the falloff rounds'
// chain (some 8,000 clocks of a Troe reaction, on one warp) and table loads from L2.  Returns
// false where the values leave the fixed-point range.
__device__ __forceinline__ bool rate_fx(int r, int kind, const CellScalars& cs, const longlong2 k1, fx_i64 th,
                                        const double* __restrict__ lA_ext, double M, fx_i64 lKc, const bool WJ,
                                        Rate& out) {
  fx_i64 lk = k1.x;
  if (lA_ext) {
    const double lA = *lA_ext;
    if (!(fabs(lA) < 500.0)) return false;
    lk = fx_mulhi_s(fx_from_double(lA, 54), 0x5c551d94ae0bf85eLL);  // Q54 x Q62: log2 A in Q52
    const fx_i64 d = (lk >> 1) - (k1.x >> 1);  // what the mechanism's own numbers leave room for (Q51)
    if (d > FX_LNA_MARGIN || d < -FX_LNA_MARGIN) return false;
  }
  lk += fx_mulhi_s(k1.y, cs.l2Tq) - fx_mulhi_s(th, cs.iTq);
  double g1 = 1.0;
  out.dlM = 0.0;
  if (kind >= LIND) {
    const Falloff o = WJ ? falloff_fx<true>(r, kind, cs.T, cs.invT, cs.l2Tq, cs.iTq, M, lk)
                         : falloff_fx<false>(r, kind, cs.T, cs.invT, cs.l2Tq, cs.iTq, M, lk);
    if (!o.ok) return false;
    lk = o.lk;
    g1 = o.g1;
    out.dlT = o.dlT;
    out.dlM = o.dlM;
  } else if (WJ) {
    out.dlT = (mk_b[r] + mk_th[r] * cs.invT) * cs.invT;
  }
  out.kf = fx_exp2(lk);
  out.kr = fx_exp2(lk - lKc);
  if (kind >= LIND) {
    out.kf *= g1;
    out.kr *= g1;
  }
  return true;
}

#if TEAM > 1
// dst[k] += sum_r nu_kr q_r over a chunk's reactions (their values in OFF_Q), without shared-memory
// atomics (a compare-and-swap loop per FP64 add: 140 clocks, and as much again for every lane that
// hits the same species).  A lane sums a run of up to seven entries of one species (a coefficient n
// stands n times); the runs of a species lie in neighbouring lanes and are added by shuffles, and
// the first lane stores.  A run is one 16-byte record, loaded before the barrier it waits at (the
// lists come from L2: gathered entry by entry they took longer than the atomics): species (8 bits), add the value of the lane
// 1, 2, 4 further (bits 8..10), store (11), by an atomic (12: more than eight runs), then seven
// entries of position (9 bits) and sign (bit 15); bit 14: none.
__device__ __forceinline__ void gather_run(const Team& tm, const uint4 g, int dst) {
  const unsigned e[7] = {g.x >> 16, g.y & 0xffff, g.y >> 16, g.z & 0xffff, g.z >> 16, g.w & 0xffff, g.w >> 16};
  double q[7];
#pragma unroll
  for (int i = 0; i < 7; ++i) q[i] = tm.at(OFF_Q, e[i] & 0x1ff);
#pragma unroll
  for (int i = 0; i < 7; ++i) {
    q[i] = (e[i] & 0x8000u) ? dneg(q[i]) : q[i];
    q[i] = (e[i] & 0x4000u) ? 0.0 : q[i];
  }
  // (an FP64 add costs its pipe time for one lane or all: skipped where no lane of the warp has one;
  // teams of four and eight lanes add without asking, since a warp takes one team's vote at a time:
  // 65,536 13-species cells at 8 lanes 12.1 -> 11.3 ms, at 16 lanes 12.8 with the votes, 13.8 without)
  const unsigned msk = team_mask();
  double v = q[0] + q[1];
#pragma unroll
  for (int i = 2; i < 7; ++i)
    if (TEAM < 16 || __any_sync(msk, !(e[i] & 0x4000u))) v += q[i];
#pragma unroll
  for (int o = 1; o < 8 && o < WL; o <<= 1) {
    const bool add = (g.x & (256u << (o >> 1))) != 0;
    if (TEAM < 16 || __any_sync(msk, add)) {
      const double w = __shfl_down_sync(msk, v, o, WL);
      if (add) v += w;
    }
  }
  double* p = &tm.at(dst, g.x & 255u);
  if (g.x & 0x1000u) atomicAdd(p, v);
  else if (g.x & 0x800u) *p += v;
}
#if TEAM < 16
__device__ __forceinline__
#else
OUTLINE
#endif
void gather_species(int ch, const uint4 first, int dst) {
  const Team tm = make_team();
  const int n = mk_osegoff[ch + 1] - mk_osegoff[ch];  // a multiple of TEAM
  uint4 g = first;
#pragma unroll 1
  for (int sg = tm.tl;;) {
    gather_run(tm, g, dst);
    sg += TEAM;
    if (sg >= n) break;
    g = mk_oseg[mk_osegoff[ch] + sg];
  }
}

#if GATHER_J
// A[row][col] += sum of +-k x concentration over the chunk's contributions (rate constants in
// OFF_KF): one FMA each, every entry owned by one lane.  Four contributions come in one 16-byte
// load, issued a group ahead: entry (14 bits), position of k (9), species of the factor (7; 126:
// none, 127: factor one), same entry as the previous contribution (1), negative (1).
__device__ __forceinline__ void gather_jacobian(const Team& tm, int ch) {
  const uint4* ent = mk_jent + (long long)mk_joff[ch] * TEAM + tm.tl;
  const int n = mk_joff[ch + 1] - mk_joff[ch];
  double last = 0.0;
  uint4 nx = n > 0 ? ent[0] : make_uint4(0, 0, 0, 0);
  for (int t = 0; t < n; ++t) {
    const unsigned e[4] = {nx.x, nx.y, nx.z, nx.w};
    if (t + 1 < n) nx = ent[(t + 1) * TEAM];
    double a[4], k[4], c[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int sp = (e[i] >> 23) & 127;
      a[i] = tm.at(OFF_A, e[i] & 0x3fff);
      k[i] = tm.at(OFF_KF, (e[i] >> 14) & 511);
      c[i] = sp >= 126 ? 1.0 : tm.at(OFF_C, sp);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double kk = (e[i] >> 31) ? dneg(k[i]) : k[i];
      const double v = fma(kk, c[i], (e[i] & 0x40000000u) ? last : a[i]);
      last = v;
      if (((e[i] >> 23) & 127) != 126) tm.at(OFF_A, e[i] & 0x3fff) = v;
    }
  }
}
#endif
#endif

// Net production rates omega (slot OFF_OM, zeroed by the caller) and, with WJ, the reaction
// part of the Jacobian: A[smap(k)][smap(j)] += d omega_k / d C_j (without the default-
// efficiency third-body part, which is collected per species in OFF_BK), d omega_k/dT at
// constant C in OFF_DOMT.  The caller zeroes A, OFF_DOMT and OFF_BK.
// A reaction's indices and coefficients come in one 16-byte record: six species (16 bits each),
// then nre, npr, kind (2 bits each), dnu + 16 (5 bits, at bit 8), the coefficients (2 bits each).
// Teams of several lanes take CHUNK reactions at a time: each lane leaves its reactions' net rates,
// rate constants and d q/dT in shared memory, then the team gathers them by species and by
// Jacobian entry.  What few reactions have (third-body parts, sides of third order) and a single
// lane's sums are added in place.
__device__ __forceinline__ void reaction_loop(const Team& tm, const CellScalars& cs, double P,
                                              const double* __restrict__ lnA_ext, const bool WJ) {
  const double T = cs.T, invT = cs.invT;
  const double Ctot = P * invT * INV_R_U;    // sum_k C_k = P / (R T)
#if TEAM == 1
#pragma unroll 1
  for (int r = 0; r < NR; ++r) {
#else
#pragma unroll 1
  for (int ch = 0; ch < NCHUNK; ++ch) {
    const uint4 run = mk_oseg[mk_osegoff[ch] + tm.tl];
    double dqT[(CHUNK + TEAM - 1) / TEAM];
#pragma unroll
    for (int rd = 0; rd < (CHUNK + TEAM - 1) / TEAM; ++rd) {
      const int j = rd * TEAM + tm.tl, r = ch * CHUNK + j;
      if (j < CHUNK && r < NR) {
#endif
    // everything the reaction needs from the tables first: they come from L2 mostly
    const int4 rec = mk_rec[r];
    const longlong2 kf1 = mk_kfx[r][0], kf2 = mk_kfx[r][1];
    const int fl = rec.w, kind = (fl >> 4) & 3, dnu = ((fl >> 8) & 31) - 16;
    // species and coefficient (0: none) of slot i: reactants 0..2, products 3..5
    auto sp = [&](int i) -> int {
      const unsigned x = i < 2 ? rec.x : (i < 4 ? rec.y : rec.z);
      return (i & 1) ? x >> 16 : x & 0xffff;
    };
    auto nu = [&](int i) -> int { return (fl >> (13 + 2 * i)) & 3; };
    const double* lAe = lnA_ext ? &lnA_ext[mk_rorig[r]] : nullptr;
    const int eff0 = (int)kf2.y, eff1 = (int)(kf2.y >> 32);
    double M = 0.0;
    if (kind != ELEM) {
      M = Ctot;
#pragma unroll 1
      for (int e = eff0; e < eff1; ++e) M += mk_effval[e] * tm.at(OFF_C, mk_effsp[e]);
    }
    // log2 K_c = sum_k nu_k log2 exp(s/R - h/RT) + dnu log2(P_atm / R T)
    Rate q;
    bool ok = false;
    if (cs.fx) {
      fx_i64 lKc = dnu * (FX_LOG2_PATM_R - (cs.l2Tq >> 7));
#pragma unroll
      for (int i = 0; i < 6; ++i)
        if (nu(i)) lKc += (i < 3 ? -nu(i) : nu(i)) * (fx_i64)fx_bits(tm.at(OFF_G, sp(i)));
      ok = rate_fx(r, kind, cs, kf1, kf2.x, lAe, M, lKc, WJ, q);
    }
    if (!ok) {
      double lKc = dnu * (LOG2_PATM_R - cs.l2T);
#pragma unroll 1
      for (int i = 0; i < 6; ++i)
        if (nu(i)) {
          const double g = tm.at(OFF_G, sp(i));
          lKc += (i < 3 ? -nu(i) : nu(i)) * (cs.fx ? fx_to_double((fx_i64)fx_bits(g), 52) : g);
        }
      Rate qs;  // (its address is taken: kept apart from the registers of the normal path)
      rate_fp(r, kind, T, invT, cs.l2T, lAe ? *lAe : mk_lnA[r], M, lKc, WJ, &qs);
      q = qs;
    }
    double fwd = q.kf, rev = q.kr;
    double dlKc = 0.0;  // T d ln K_c/dT = sum nu'' h/RT - sum nu' h/RT - dnu
    if (WJ) dlKc = -mk_dnuf[r];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      const int n = nu(i);
      if (n) {
        const int k = sp(i);
        const double c = tm.at(OFF_C, k);
        double& x = i < 3 ? fwd : rev;
        x *= c;
        if (WJ) {
          const double h = tm.at(OFF_HRT, k);
          dlKc += i < 3 ? dneg(h) : h;
        }
        if (n > 1) {
#pragma unroll 1
          for (int v = 1; v < n; ++v) {
            x *= c;
            if (WJ) {
              const double h = tm.at(OFF_HRT, k);
              dlKc += i < 3 ? dneg(h) : h;
            }
          }
        }
      }
    }
    const double qnet = fwd - rev;
    const double qr = kind == THIRD ? M * qnet : qnet;
#if TEAM == 1
#pragma unroll 1
    for (int i = 0; i < 6; ++i)
      if (nu(i)) tm.at(OFF_OM, sp(i)) += nu_times(i < 3 ? -nu(i) : nu(i), qr);
#else
    tm.at(OFF_Q, j) = qr;
#endif
    if (WJ) {
      double dqdT = qnet * q.dlT + rev * (dlKc * invT);
      if (kind == THIRD) {
        dqdT *= M;
        q.kf *= M;
        q.kr *= M;
      }
#if TEAM > 1
      dqT[rd] = dqdT;
      tm.at(OFF_KF, j) = q.kf;
      tm.at(OFF_KF, CHUNK + j) = q.kr;
#endif
      if (kind != ELEM) {
        // dq/d[M]: the [M] factor of THIRD reactions, the falloff blend of LIND/TROE
        const double beta = kind == THIRD ? qnet : qnet * q.dlM;
#pragma unroll 1
        for (int i = 0; i < 6; ++i)
          if (nu(i)) {
            const double nb = nu_times(i < 3 ? -nu(i) : nu(i), beta);
            scatter_add<double>(&tm.at(OFF_BK, sp(i)), nb);
#pragma unroll 1
            for (int e = eff0; e < eff1; ++e)
              scatter_add<double>(&tm.A(smap(sp(i)), smap(mk_effsp[e])), nb * mk_effval[e]);
          }
      }
#if TEAM == 1 || !GATHER_J || HAS_GENERAL
      if (TEAM == 1 || !GATHER_J || (fl & 0x80)) {
        // dq/dC_d of the mass-action products, into the rows of every species of the reaction
#pragma unroll 1
        for (int d = 0; d < 6; ++d)
          if (nu(d)) {
            double p = nu_times(d < 3 ? nu(d) : -nu(d), d < 3 ? q.kf : q.kr);
#pragma unroll 1
            for (int i2 = d < 3 ? 0 : 3; i2 < (d < 3 ? 3 : 6); ++i2) {
              const int e = i2 == d ? nu(d) - 1 : nu(i2);
#pragma unroll 1
              for (int v = 0; v < e; ++v) p *= tm.at(OFF_C, sp(i2));
            }
#pragma unroll 1
            for (int i = 0; i < 6; ++i)
              if (nu(i)) scatter_add<double>(&tm.A(smap(sp(i)), smap(sp(d))), nu_times(i < 3 ? -nu(i) : nu(i), p));
          }
      }
#endif
#if TEAM == 1
#pragma unroll 1
      for (int i = 0; i < 6; ++i)
        if (nu(i)) tm.at(OFF_DOMT, sp(i)) += nu_times(i < 3 ? -nu(i) : nu(i), dqdT);
#endif
    }
#if TEAM > 1
      }
    }
    tsync();
    gather_species(ch, run, OFF_OM);
    if (WJ) {
#if GATHER_J
      gather_jacobian(tm, ch);
#endif
      tsync();
#pragma unroll
      for (int rd = 0; rd < (CHUNK + TEAM - 1) / TEAM; ++rd)
        if (rd * TEAM + tm.tl < CHUNK) tm.at(OFF_Q, rd * TEAM + tm.tl) = dqT[rd];
      tsync();
      gather_species(ch, run, OFF_DOMT);
    }
    tsync();
#endif
  }
#if TEAM == 1
  tsync();
#endif
}

// f from omega: f[0] = dT/dt = -T sum_k (h_k/RT) V omega_k / sum_k n_k cp_k/R,
// f[1+k] = V omega_k.  Returns dT/dt.
__device__ __forceinline__ double source_from_omega(const Team& tm, const CellScalars& cs, int of) {
  double hs = 0.0;
  for (int k = tm.tl; k < NS; k += TEAM) {
    const double om = tm.at(OFF_OM, k);
    hs += tm.at(OFF_HRT, k) * om;
    if (k < NS - 1) tm.at(of, 1 + k) = cs.V * om;
  }
  hs = team_sum(tm, hs);
  const double fT = -cs.T * cs.V * hs * fx_rcp(cs.cpm);
  if (tm.tl == 0) tm.at(of, 0) = fT;
  tsync();
  return fT;
}

__device__ __forceinline__ void zero_rates(const Team& tm, bool with_j) {
  for (int k = tm.tl; k < NS; k += TEAM) {
    tm.at(OFF_OM, k) = 0.0;
    if (with_j) { tm.at(OFF_DOMT, k) = 0.0; tm.at(OFF_BK, k) = 0.0; }
  }
  if (with_j)
    for (int e = tm.tl; e < NEQ * NEQ; e += TEAM) tm.at(OFF_A, e) = 0.0;
  tsync();
}

// f(y) into slot `of` for the state at slot `oy` and, for sgn != 0, the state Jacobian into A: J for
// sgn = 1 (shift = 0), and M = I shift - J with shift = 1/(gamma h) for sgn = -1.
template <int sgn>
OUTLINE void evaluate(int oy, int of, double P, const double* lnA_ext, double shift) {
  const Team tm = make_team();
  CellScalars cs;
  thermo_conc(tm, oy, P, cs, sgn != 0);
  zero_rates(tm, sgn != 0);
  reaction_loop(tm, cs, P, lnA_ext, sgn != 0);
  const double fT = source_from_omega(tm, cs, of);
  if (sgn == 0) return;
  const long long flip = sgn < 0 ? (long long)0x8000000000000000ULL : 0;
  auto signed_by = [&](double x) { return __longlong_as_double(__double_as_longlong(x) ^ flip); };
  const double T = cs.T, V = cs.V, invT = cs.invT;
  const double Ctot = P * invT * INV_R_U;
  const double RTP = R_U * T * fx_rcp(P);  // R T / P
  // per species row k (B_k = default-efficiency third-body part, added to every column):
  //   D_k = omega_k - sum_m (d omega_k/dC_m) C_m,
  //   d f_k/d n_j = d omega_k/dC_j - w_j d omega_k/dC_bath + (RT/P)(1 - w_j) D_k
  //               = A_kj + P1_k - w_j P2_k with P1 = B_k + (RT/P) D_k, P2 = A_kb + B_k + (RT/P) D_k,
  //   d f_k / dT = V (D_k / T + d omega_k/dT).
  // RSPLIT lanes share a row's dot product (and a column's below): the dependent FMAs of a lane set
  // the time of these passes
  for (int kk = tm.tl / RSPLIT; kk < NS_PAD; kk += TEAM / RSPLIT) {
    const int k = kk < NS ? kk : NS - 1;
    const int row = smap(k);
    double d0 = 0.0, d1 = 0.0;
    int j = tm.tl % RSPLIT;
    for (; j + RSPLIT < NS; j += 2 * RSPLIT) {
      d0 += tm.A(row, smap(j)) * tm.at(OFF_C, j);
      d1 += tm.A(row, smap(j + RSPLIT)) * tm.at(OFF_C, j + RSPLIT);
    }
    if (j < NS) d0 += tm.A(row, smap(j)) * tm.at(OFF_C, j);
    const double dot = rsplit_sum(d0 + d1);
    if (kk < NS && tm.tl % RSPLIT == 0) {
      const double Bk = tm.at(OFF_BK, k);
      const double D = tm.at(OFF_OM, k) - dot - Bk * Ctot;
      const double be = Bk + RTP * D;
      tm.at(OFF_AL, k) = tm.A(row, 0) + be;
      tm.at(OFF_BE, k) = be;
      tm.at(OFF_JT, k) = V * (D * invT + tm.at(OFF_DOMT, k));
    }
  }
  tsync();
  // species rows, w_j = W_j / W_bath (the diagonal shift of M comes last)
#if TEAM == 1
  for (int i = 1; i < NEQ; ++i) {
    const double al = tm.at(OFF_AL, i - 1), be = tm.at(OFF_BE, i - 1);
    for (int l = 1; l < NEQ; ++l) {
      const double w = mk_wratio[l - 1];
      tm.A(i, l) = signed_by(fma(-w, al, tm.A(i, l) + be));
    }
    tm.A(i, 0) = signed_by(tm.at(OFF_JT, i - 1));
  }
#else
  {
    int i = 1 + tm.tl / NEQ, l = tm.tl % NEQ;
    for (int e = tm.tl; e < (NEQ - 1) * NEQ; e += TEAM) {
      const int k = i - 1;
      if (l == 0) {
        tm.A(i, 0) = signed_by(tm.at(OFF_JT, k));
      } else {
        const double w = mk_wratio[l - 1], al = tm.at(OFF_AL, k), a = tm.A(i, l) + tm.at(OFF_BE, k);
        tm.A(i, l) = signed_by(fma(-w, al, a));
      }
      i += TEAM / NEQ;
      l += TEAM % NEQ;
      if (l >= NEQ) { l -= NEQ; ++i; }
    }
  }
#endif
  tsync();
  // temperature row: f_T = -Q / cpm with Q = T sum_k (h_k/RT) f'_k over all species (f'_k =
  // V omega_k, bath included); dQ/dn_j = T sum_k (h_k/RT) J_kj, dQ/dT = sum_k cp_k f'_k +
  // T sum_k (h_k/RT) J_kT; d cpm/dn_j = cp_j - w_j cp_bath, d cpm/dT = sum_k n_k dcp_k/dT.
  const double hb = tm.at(OFF_HRT, BATH), alb = tm.at(OFF_AL, BATH), beb = tm.at(OFF_BE, BATH);
  const double icpm = fx_rcp(cs.cpm);
  double cpf = 0.0;  // sum_k cp_k omega_k, a team reduction rather than one lane's loop
  for (int k = tm.tl; k < NS; k += TEAM) cpf += tm.at(OFF_CP, k) * tm.at(OFF_OM, k);
  cpf = team_sum(tm, cpf);
  for (int ll = tm.tl / RSPLIT; ll < NS_PAD; ll += TEAM / RSPLIT) {
    const int l = ll < NEQ ? ll : NEQ - 1;
    double s0 = 0.0, s1 = 0.0;
    int i = 1 + tm.tl % RSPLIT;
    for (; i + RSPLIT < NEQ; i += 2 * RSPLIT) {
      s0 += tm.at(OFF_HRT, i - 1) * tm.A(i, l);
      s1 += tm.at(OFF_HRT, i - 1 + RSPLIT) * tm.A(i + RSPLIT, l);
    }
    if (i < NEQ) s0 += tm.at(OFF_HRT, i - 1) * tm.A(i, l);
    double s = rsplit_sum(s0 + s1);
    s = signed_by(s);  // the rows above carry the sign
    if (ll < NEQ && tm.tl % RSPLIT == 0) {
      double val;
      if (l == 0) {
        s += hb * tm.at(OFF_JT, BATH);
        const double dQdT = cpf * V + T * s;
        val = -(dQdT + fT * cs.dcpm) * icpm;
      } else {
        const double w = mk_wratio[l - 1];
        const double Jb = tm.A(0, l) - w * alb + beb;  // bath row, before it is overwritten
        s += hb * Jb;
        const double dcpm = tm.at(OFF_CP, l - 1) - w * tm.at(OFF_CP, BATH);
        val = -(T * s + fT * dcpm) * icpm;
      }
      tm.A(0, l) = signed_by(val);
    }
  }
  tsync();
  if (sgn < 0) {
    for (int i = tm.tl; i < NEQ; i += TEAM) tm.A(i, i) += shift;
    tsync();
  }
}

__device__ __forceinline__ void eval_f(int oy, int of, double P, const double* lnA_ext) {
  evaluate<0>(oy, of, P, lnA_ext, 0.0);
}
template <int SGN>
__device__ __forceinline__ void eval_f_jac(int oy, int of, double P, const double* lnA_ext, double shift) {
  evaluate<SGN>(oy, of, P, lnA_ext, shift);
}

// ------------------------------------------------------------------------------ LU + solves

#if LU_BLOCKED
// ---- blocked LU: panels of eight columns in FP64, the trailing update on the tensor cores.
//
// The rank-8 update C -= L U (L m x 8, U 8 x m) is 8 m^2 FP64 FMAs: nearly all of the
// factorisation's work, and the FP64 pipe gives a warp one per 64 clocks.  Here it is computed as
// an integer product, the splitting of operands into short digits whose products are summed without error
// (Ozaki, Ogita, Oishi & Rump 2012, Numerical Algorithms 59): every row of L and column of U is
// scaled by a power of two, cut off 61 bits below its largest entry
// and split into LU_SL signed digits of nine bits, which fp16 holds exactly; mma.sync accumulates the
// digit products of equal weight in FP32 without rounding (at most 56 products of 2^16, offset by
// 1.5 2^23 so that the sums can be read off the bit patterns); the sums are put together in a 64-bit
// integer, rounded once to a double and subtracted from C: one FP64 add in place of eight FMAs, and
// one rounding in place of eight.  What is left out (the cut, and digit products of weight 7 and more) comes
// to 2^-60 typically and 2^-55 at most of the largest scaled entry of the row times that of the
// column: where one product of the eight has both, an eighth to a hundredth of what eight FP64
// roundings leave; an element whose products all pair a large entry with one 2^-20 of its row's or
// column's largest keeps about 41 bits, fewer than FP64 would.
// To keep the scaling from losing small products, U's rows are first brought to a common
// magnitude and L's columns scaled inversely (rates of very different species meet in a panel).
// The solutions' errors in the solver's weighted norm, against 160-bit arithmetic on 53- and
// 111-species iteration matrices (steps of 1e-9 to 1e-6 s), are those of the FP64 update; so are those of
// integrations that weigh trace species like the others (atol 1e-22 at rtol 1e-6, 1e-20 at 1e-8: the
// median errors of 128 53-species and 64 111-species cells within 25% of the FP64 update's, either way).
// Clocks per factorisation, column by column (with one column of look-ahead at 111 species) and in
// this form: 53 species 190 K -> 149 K, 111 species 424 K -> 342 K, with the panel look-ahead 315 K; at
// 13 species 20 K -> 28 K, hence LU_MIN.  What bounds it: the panel's chain (1,170 clocks a column,
// 290 of them FP64) and, in the update, the FP64 subtractions and the recombination's integer
// instructions (about 250 per tile of 16 x 8).
#define LU_SL 7
#define LU_NB 8
#define LU_NW ((NEQ + 31) / 32)  // warps of the panel factorisation, one row per lane
// scratch in the thermo slots (dead during the factorisation): two sets of candidate rows
// (eight values, 1/pivot, key and position), one per warp and the panel's top row, then, for two
// panels in turn, eight pivot rows and the magnitudes of U's eight rows
#define LUS_ROW(set, w) (OFF_C + ((set) * (LU_NW + 1) + (w)) * 11)
#define LUS_INT(k0) (OFF_C + 2 * (LU_NW + 1) * 11 + ((k0) / LU_NB & 1) * 8)

__device__ __forceinline__ void lu_bar() {
#if LU_NW == 1
  __syncwarp();
#elif LU_NW * 32 == TEAM
  __syncthreads();
#else
  asm volatile("bar.sync 1, %0;" ::"r"(LU_NW * 32) : "memory");
#endif
}

// Columns k0..k0+kb-1, rows k0..N-1, by LU_NW warps with a row per lane in registers: per column a
// warp argmax (three reductions), one exchange of the warps' candidates through shared memory (the
// candidate's whole row and its reciprocal with it), and the rank-1 update of the panel.
__device__ __forceinline__ void lu_panel8(const Team& tm, int k0) {
  const int kb = NEQ - k0 < LU_NB ? NEQ - k0 : LU_NB;
  const int m = NEQ - k0, w = tm.tl >> 5;
  const bool in = tm.tl < m;
  double v[LU_NB];
#pragma unroll
  for (int c = 0; c < LU_NB; ++c) v[c] = in && c < kb ? tm.A(k0 + tm.tl, k0 + c) : 0.0;
  int* ints = reinterpret_cast<int*>(&tm.base[LUS_INT(k0)]);
  if (tm.tl < LU_NB) ints[LU_NB + tm.tl] = 0;
#pragma unroll
  for (int j = 0; j < LU_NB; ++j) {
    if (j < kb) {
      const bool cand = in && tm.tl >= j;
      // every lane's reciprocal, while the reductions wait; the chosen lane redoes an exceptional one
      double inv = fx_rcp_normal(v[j]);
      const unsigned long long key = (unsigned long long)abs_key(v[j]);
      const unsigned hi = cand ? (unsigned)(key >> 32) : 0u, lo = cand ? (unsigned)key : 0u;
      const unsigned mhi = __reduce_max_sync(0xffffffffu, hi);
      const unsigned mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? lo : 0u);
      const unsigned pos = __reduce_min_sync(0xffffffffu, cand && hi == mhi && lo == mlo ? (unsigned)tm.tl : 0xffffu);
      double* mine = &tm.base[LUS_ROW(j & 1, w)];
      if ((unsigned)tm.tl == pos) {
#pragma unroll
        for (int c = 0; c < LU_NB; ++c) mine[c] = v[c];
        if (!fx_rcp_ok(v[j])) inv = fx_rcp_slow(v[j]);
        mine[8] = inv;
      }
      if ((tm.tl & 31) == 0) {
        mine[9] = __longlong_as_double(((long long)mhi << 32) | mlo);
        mine[10] = __longlong_as_double((long long)pos);
      }
      double* top = &tm.base[LUS_ROW(j & 1, LU_NW)];
      if (tm.tl == j) {
#pragma unroll
        for (int c = 0; c < LU_NB; ++c) top[c] = v[c];
      }
      lu_bar();
      // the winner: the largest key, the lowest position on ties (warps hold ascending positions; a
      // warp without a candidate has position 0xffff)
      const double* best = &tm.base[LUS_ROW(j & 1, 0)];
      long long ck[LU_NW];
      unsigned cp[LU_NW];
#pragma unroll
      for (int x = 0; x < LU_NW; ++x) {
        ck[x] = __double_as_longlong(best[x * 11 + 9]);
        cp[x] = (unsigned)__double_as_longlong(best[x * 11 + 10]);
      }
      long long bk = cp[0] != 0xffffu ? ck[0] : -1;
      unsigned p = cp[0];
      int bw = 0;
#pragma unroll
      for (int x = 1; x < LU_NW; ++x)
        if (cp[x] != 0xffffu && ck[x] > bk) { bk = ck[x]; p = cp[x]; bw = x * 11; }
      best += bw;
      if ((unsigned)tm.tl == p && p != (unsigned)j) {
#pragma unroll
        for (int c = 0; c < LU_NB; ++c) v[c] = top[c];
      }
      const double pinv = best[8];
      if (tm.tl == j) {
#pragma unroll
        for (int c = 0; c < LU_NB; ++c) v[c] = best[c];
        v[j] = pinv;  // 1/U_kk on the diagonal
        ints[j] = k0 + (int)p;
      }
      if (in && tm.tl > j) {
        const double l = v[j] * pinv;
        v[j] = l;
#pragma unroll
        for (int c = j + 1; c < LU_NB; ++c) v[c] = fma(-l, best[c], v[c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < LU_NB; ++c)
    if (in && c < kb) tm.A(k0 + tm.tl, k0 + c) = v[c];
}

// magnitude of x as a biased exponent (0: zero or denormal, taken as zero below)
__device__ __forceinline__ int lu_mag(double x) { return (int)(fx_bits(x) >> 52) & 2047; }

// x 2^s as the 61-bit integer X = x 2^s / 2^(top - 1022) 2^61 (cut off, not rounded), where mag <= top are the biased exponents of
// |x 2^s| and of the largest number of its row or column; the constant makes every nine-bit digit
// of the sum an unsigned one, 256 above the signed digit it stands for
__device__ __forceinline__ fx_u64 lu_digits(double x, int mag, int top) {
  const fx_u64 b = fx_bits(x);
  const fx_i64 m = mag < -4000 ? 0 : (fx_i64)fx_mant(x);
  const int d = top - mag - 8;  // >= -8
  fx_i64 v = d <= 0 ? m << -d : m >> (d < 63 ? d : 63);
  if ((fx_i64)b < 0) v = -v;
  return (fx_u64)v + 256ULL * 0x0040201008040201ULL;
}
// digit pairs of two elements as half2 registers, most significant first
__device__ __forceinline__ void lu_halves(fx_u64 y0, fx_u64 y1, unsigned* h) {
#pragma unroll
  for (int s = 0; s < LU_SL; ++s) {
    const int sh = 9 * (LU_SL - 1 - s);
    const unsigned a = (unsigned)(y0 >> sh) & 511u, b = (unsigned)(y1 >> sh) & 511u;
    const unsigned x = 0x64006400u | a | (b << 16);  // 1024 + digit + 256
    asm("sub.f16x2 %0, %1, %2;" : "=r"(h[s]) : "r"(x), "r"(0x65006500u));  // - 1280
  }
}
__device__ __forceinline__ void lu_mma16(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                         unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void lu_mma8(float* c, unsigned a0, unsigned a1, unsigned b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

// The product T 2^(e - 1085) of the scaled sums as a double, T = sum_t a_t 2^(9 (5 - t)); a_t are the
// accumulators' bit patterns (0x4b400000 + the sum).  With e the sum of the two tops less 1018 this is the
// product of the numbers whose digits were multiplied.
__device__ __forceinline__ double lu_value(const unsigned* a, int e) {
  const unsigned k = 0x4b400000u;
  const int p01 = (int)(a[0] * 512u + a[1] - k * 513u), p23 = (int)(a[2] * 512u + a[3] - k * 513u);
  const int p45 = (int)(a[4] * 512u + a[5] - k * 513u), p6 = (int)(a[6] - k + 256u) >> 9;
  const fx_i64 T = ((fx_i64)p01 << 36) + ((fx_i64)p23 << 18) + ((fx_i64)p45 + p6);
  const fx_u64 sg = (fx_u64)T & 0x8000000000000000ULL;
  const fx_u64 u = T < 0 ? 0 - (fx_u64)T : (fx_u64)T;
  const int z = fx_clz(u);
  const fx_u64 r = (((u << z) >> 1) + 0x200) >> 10;
  const int ef = e - z;  // biased exponent - 1
  if (ef <= 0 || u == 0) return 0.0;
  return fx_as_double(sg | (ef >= 2045 ? 0x7ff0000000000000ULL : ((fx_u64)ef << 52) + r));
}

// A[k1.., k1..] -= A[k1.., k0..k0+7] A[k0..k0+7, k1..] for the column tiles c0..c1-1 (of eight columns), by
// warp w of nw: tiles of 16 x 8 are dealt to the warps in runs along a strip of rows (its digits stay
// in registers).
__device__ __forceinline__ void lu_update8(const Team& tm, int k0, int w, int nw, int c0, int c1) {
  const int k1 = k0 + LU_NB, m = NEQ - k1;
  const int nt = c1 - c0, tot = (m + 15) / 16 * nt;
  const int ln = tm.tl & 31, g = ln >> 2, t = ln & 3;
  const int* rho = reinterpret_cast<const int*>(&tm.base[LUS_INT(k0)]) + LU_NB;
  const int rho0 = rho[2 * t], rho1 = rho[2 * t + 1];
  int strip = -1, topl0 = 0, topl1 = 0;
  unsigned la[LU_SL], lb[LU_SL];
  const int q1 = (w + 1) * tot / nw;
#pragma unroll 1
  for (int q = w * tot / nw; q < q1; ++q) {
    const int s = q / nt, j0 = k1 + (c0 + q - s * nt) * 8;
    const int r0 = k1 + s * 16 + g, r1 = r0 + 8;
    if (s != strip) {
      strip = s;
      double x[4];
      int mg[4];
      x[0] = r0 < NEQ ? tm.A(r0, k0 + 2 * t) : 0.0;
      x[1] = r0 < NEQ ? tm.A(r0, k0 + 2 * t + 1) : 0.0;
      x[2] = r1 < NEQ ? tm.A(r1, k0 + 2 * t) : 0.0;
      x[3] = r1 < NEQ ? tm.A(r1, k0 + 2 * t + 1) : 0.0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        mg[i] = lu_mag(x[i]);
        mg[i] = mg[i] == 0 ? -8000 : mg[i] + (i & 1 ? rho1 : rho0);
      }
      topl0 = max(mg[0], mg[1]);
      topl1 = max(mg[2], mg[3]);
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        topl0 = max(topl0, __shfl_xor_sync(0xffffffffu, topl0, o));
        topl1 = max(topl1, __shfl_xor_sync(0xffffffffu, topl1, o));
      }
      lu_halves(lu_digits(x[0], mg[0], topl0), lu_digits(x[1], mg[1], topl0), la);
      lu_halves(lu_digits(x[2], mg[2], topl1), lu_digits(x[3], mg[3], topl1), lb);
    }
    unsigned ub[LU_SL];
    int topu;
    {
      const int j = j0 + g;
      const double x0 = j < NEQ ? tm.A(k0 + 2 * t, j) : 0.0, x1 = j < NEQ ? tm.A(k0 + 2 * t + 1, j) : 0.0;
      int m0 = lu_mag(x0), m1 = lu_mag(x1);
      m0 = m0 == 0 ? -8000 : m0 - rho0;
      m1 = m1 == 0 ? -8000 : m1 - rho1;
      topu = max(m0, m1);
      topu = max(topu, __shfl_xor_sync(0xffffffffu, topu, 1));
      topu = max(topu, __shfl_xor_sync(0xffffffffu, topu, 2));
      lu_halves(lu_digits(x0, m0, topu), lu_digits(x1, m1, topu), ub);
    }
    float acc[LU_SL][4];
#pragma unroll
    for (int l = 0; l < LU_SL; ++l) {
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[l][i] = 12582912.0f;  // 1.5 2^23
#pragma unroll
      for (int i = 0; i + 1 <= l; i += 2) lu_mma16(acc[l], la[i], lb[i], la[i + 1], lb[i + 1], ub[l - i], ub[l - i - 1]);
      if ((l & 1) == 0) lu_mma8(acc[l], la[l], lb[l], ub[0]);
    }
    // the tops of the thread's two output columns 2t, 2t+1 (held by the lanes of those columns)
    const int tu0 = __shfl_sync(0xffffffffu, topu, 8 * t), tu1 = __shfl_sync(0xffffffffu, topu, 8 * t + 4);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = i < 2 ? r0 : r1, j = j0 + 2 * t + (i & 1);
      unsigned a[LU_SL];
#pragma unroll
      for (int l = 0; l < LU_SL; ++l) a[l] = __float_as_uint(acc[l][i]);
      if (r < NEQ && j < NEQ) tm.A(r, j) -= lu_value(a, (i < 2 ? topl0 : topl1) + (i & 1 ? tu1 : tu0) - 1018);
    }
  }
}
#endif

// In-place LU with partial pivoting of A (N x N): largest |a| in the column, lowest row on
// ties.  1/U_kk replaces U_kk on the diagonal, the composed row permutation (row i of P A is row
// perm[i] of A) goes to OFF_PERM, and the single-lane layout also keeps the pivot sequence.
OUTLINE void lu_factor() {
  const Team tm = make_team();
#if TEAM == 1
  for (int k = 0; k < NEQ; ++k) {
    int p = k;
    long long best = abs_key(tm.A(k, k));
    for (int i = k + 1; i < NEQ; ++i) {
      const long long v = abs_key(tm.A(i, k));
      if (v > best) { best = v; p = i; }
    }
    tm.piv(k) = p;
    if (p != k)
      for (int j = 0; j < NEQ; ++j) { const double t = tm.A(k, j); tm.A(k, j) = tm.A(p, j); tm.A(p, j) = t; }
    const double inv = fx_rcp(tm.A(k, k));
    tm.invd(k) = inv;
    for (int i = k + 1; i < NEQ; ++i) {
      const double l = tm.A(i, k) * inv;
      tm.A(i, k) = l;
      for (int j = k + 1; j < NEQ; ++j) tm.A(i, j) -= l * tm.A(k, j);
    }
  }
  for (int i = 0; i < NEQ; ++i) tm.perm(i) = i;
  for (int k = 0; k < NEQ; ++k) { const int p = tm.piv(k); if (p != k) { const int t = tm.perm(k); tm.perm(k) = tm.perm(p); tm.perm(p) = t; } }
#elif LU_BLOCKED
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.perm(i) = i;
  tsync();
  // Per panel: its row exchanges and U12 in the other columns, then its update of the trailing matrix
  // and the next panel.  Teams with more warps than a panel needs take the two together: the panel's
  // warps update its eight columns and factor them while the others update the rest.
#pragma unroll 1
  for (int k0 = -LU_NB;; k0 += LU_NB) {
    if (k0 >= 0) {
      // the panel's row exchanges in the other columns, a lane each, and right of the panel the
      // triangular solve U12 = L11^-1 A12
      const int kb = NEQ - k0 < LU_NB ? NEQ - k0 : LU_NB;
      int* ints = reinterpret_cast<int*>(&tm.base[LUS_INT(k0)]);
      const int c = tm.tl;
      if (c == TEAM - 1) {  // the composed permutation
#pragma unroll 1
        for (int i = 0; i < kb; ++i) {
          const int p = ints[i], t = tm.perm(k0 + i);
          tm.perm(k0 + i) = tm.perm(p);
          tm.perm(p) = t;
        }
      }
      double u[LU_NB];
#pragma unroll
      for (int i = 0; i < LU_NB; ++i) u[i] = 0.0;
      if (c < k0 || (c >= k0 + kb && c < NEQ)) {
#pragma unroll 1
        for (int i = 0; i < kb; ++i) {
          const int p = ints[i];
          if (p != k0 + i) {
            const double a = tm.A(k0 + i, c), b = tm.A(p, c);
            tm.A(k0 + i, c) = b;
            tm.A(p, c) = a;
          }
        }
        if (c >= k0 + LU_NB) {
#pragma unroll
          for (int i = 0; i < LU_NB; ++i) u[i] = tm.A(k0 + i, c);
#pragma unroll
          for (int i = 1; i < LU_NB; ++i) {
#pragma unroll
            for (int k = 0; k < i; ++k) u[i] = fma(-tm.A(k0 + i, k0 + k), u[k], u[i]);
          }
#pragma unroll
          for (int i = 1; i < LU_NB; ++i) tm.A(k0 + i, c) = u[i];
        }
      }
      if (k0 + LU_NB >= NEQ) break;
      // the magnitudes of U's rows, which balance the update's scales
#pragma unroll
      for (int i = 0; i < LU_NB; ++i) {
        const int mx = __reduce_max_sync(0xffffffffu, lu_mag(u[i]));
        if ((tm.tl & 31) == 0 && mx > 0) atomicMax(&ints[LU_NB + i], mx);
      }
      tsync();
    }
    const int w = TEAM > 32 ? tm.tl >> 5 : 0;
    const bool mine = w < LU_NW;  // a warp of the panel
    const int ahead = TEAM > LU_NW * 32 ? LU_NW : 0;
    if (k0 >= 0) {
      const int all = (NEQ - k0 - LU_NB + 7) / 8;
      lu_update8(tm, k0, ahead && !mine ? w - ahead : w, ahead ? (mine ? ahead : TEAM / 32 - ahead) : TEAM / 32,
                 ahead && !mine ? 1 : 0, ahead && mine ? 1 : all);
    }
    if (!ahead) tsync();
    if (mine) {
      if (ahead) lu_bar();
      lu_panel8(tm, k0 + LU_NB);
    }
    tsync();
  }
  tsync();
#else
  // the composed permutation is built as the pivots are chosen (lane 0, after the row swap's
  // barrier), so no serial pass over the pivots is needed afterwards
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.perm(i) = i;
  for (int k = 0; k < NEQ; ++k) {
    // pivot search: (|a| key desc, row asc)
    long long best = -1;
    int p = NEQ;
    for (int i = k + tm.tl; i < NEQ; i += TEAM) {
      const long long v = abs_key(tm.A(i, k));
      if (v > best) { best = v; p = i; }
    }
    const unsigned msk = team_mask();
#pragma unroll
    for (int o = XOR0; o > 0; o >>= 1) {
      const long long vb = __shfl_xor_sync(msk, best, o);
      const int pb = __shfl_xor_sync(msk, p, o);
      if (vb > best || (vb == best && pb < p)) { best = vb; p = pb; }
    }
#if TEAM > 32
    {
      long long* rv = reinterpret_cast<long long*>(&tm.base[OFF_RED]);
      int* ri = reinterpret_cast<int*>(&tm.base[OFF_RED + 8]);
      if ((threadIdx.x & 31) == 0) { rv[threadIdx.x >> 5] = best; ri[threadIdx.x >> 5] = p; }
      __syncthreads();
      best = rv[0];
      p = ri[0];
      for (int w = 1; w < TEAM / 32; ++w)
        if (rv[w] > best || (rv[w] == best && ri[w] < p)) { best = rv[w]; p = ri[w]; }
      __syncthreads();
    }
#endif
    if (p != k)
      for (int j = tm.tl; j < NEQ; j += TEAM) { const double t = tm.A(k, j); tm.A(k, j) = tm.A(p, j); tm.A(p, j) = t; }
    tsync();
    // 1/pivot and the column scale by the first warp only: a warp-level FP64 instruction costs the
    // same pipe time whatever its lane count, so the other warps must not repeat the division
    if (tm.tl < 32) {
      const double inv = fx_rcp(tm.A(k, k));
      __syncwarp(msk);  // every lane has read U_kk before lane 0 replaces it by its inverse
      if (tm.tl == 0) {
        tm.invd(k) = inv;
        if (p != k) { const int t = tm.perm(k); tm.perm(k) = tm.perm(p); tm.perm(p) = t; }
      }
      for (int i = k + 1 + tm.tl; i < NEQ; i += WL) tm.A(i, k) *= inv;
    }
    tsync();
    const int m = NEQ - k - 1;
    if (m > 0) {
      const int tot = m * m;
      const int qd = TEAM / m, rm = TEAM - qd * m;
      int i = tm.tl / m, j = tm.tl - (tm.tl / m) * m;
      for (int e = tm.tl; e < tot; e += TEAM) {
        tm.A(k + 1 + i, k + 1 + j) -= tm.A(k + 1 + i, k) * tm.A(k, k + 1 + j);
        i += qd;
        j += rm;
        if (j >= m) { j -= m; ++i; }
      }
    }
    tsync();
  }
#endif
}

#if SOLVE_BLK
// ---- stage solves in blocks of eight rows with inverted diagonal blocks.
//
// A substitution step per column (broadcast, multiply, update) costs 200 to 300 clocks of latency, 222
// times per solve at 111 species.  With the 8 x 8 triangles on the diagonal inverted once per
// factorisation (36 FP64 instructions, all triangles at once), a block takes one 8 x 8 product (two
// products a lane and two shuffles), one barrier and eight columns' worth of independent FMAs spread
// over RSPLIT lanes per row: clocks per attempt in the four solves 121 K -> 70 K (53 species, few
// cells), 230 K -> 136 K (111 species), of which the inversion takes 6 to 9 K.  Against 160-bit arithmetic the solutions' errors are no larger than
// those of the plain substitution (geometric mean of their ratio 0.72 on 53- and 111-species
// iteration matrices).
#define NBK ((NEQ + 7) / 8)
#define SLW ((NEQ * RSPLIT + 31) / 32)  // warps that hold rows

__device__ __forceinline__ void solve_bar() {
#if SLW == 1
  __syncwarp();
#elif SLW * 32 == TEAM
  __syncthreads();
#else
  asm volatile("bar.sync 1, %0;" ::"r"(SLW * 32) : "memory");
#endif
}

// The 8 x 8 diagonal blocks of L (unit lower) and U (1/U_kk on its diagonal) replaced by their
// inverses.  Eight lanes take a triangle, one column each; U's is read back to front so that both
// kinds are the same forward substitution.
OUTLINE void lu_invert() {
  const Team tm = make_team();
#pragma unroll 1
  for (int u0 = 0; u0 < 16 * NBK; u0 += TEAM) {
    const int u = u0 + tm.tl, b = (u >> 4) * 8, c = u & 7;
    const bool up = (u & 8) != 0;
    const int m = NEQ - b < 8 ? NEQ - b : 8;  // (negative beyond the last block)
    const int o = up ? b + m - 1 : b, st = up ? -1 : 1;
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      double v = 0.0, d = 1.0;
      if (i < m) {
        if (up) d = tm.A(o + i * st, o + i * st);
#pragma unroll
        for (int k = 0; k < i; ++k) v = fma(-tm.A(o + i * st, o + k * st), x[k], v);
      }
      x[i] = i == c ? d : v * d;
    }
    __syncwarp();  // the triangle is read before it is overwritten
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < m && (up ? i >= c : i > c)) tm.A(o + i * st, o + c * st) = x[i];
  }
  tsync();
}

// Solve M x = b (TR: M^T x = b) in place on the vector at slot ob, with P M = L U: L then U, or U^T then
// L^T and the permutation last.  Row i belongs to RSPLIT neighbouring lanes; the warp that holds a
// block's rows multiplies them by the block's inverse (four lanes per row) and publishes them in the
// vector's slots.
template <bool TR>
OUTLINE void lu_solve_blk(int ob) {
  const Team tm = make_team();
  if (tm.tl < SLW * 32) {
    const int ln = tm.tl & 31, w = TEAM > 32 ? tm.tl >> 5 : 0;
    const int row = tm.tl / RSPLIT, h = tm.tl % RSPLIT;
    const int j = ln >> 2, q = ln & 3;
    double r = row < NEQ ? tm.at(ob, TR ? row : tm.perm(row)) : 0.0;
    solve_bar();  // every entry of b is read before the slots receive x
#pragma unroll 1
    for (int s = 0; s < 2 * NBK; ++s) {
      const bool fwd = s < NBK;
      const int b = 8 * (fwd ? s : 2 * NBK - 1 - s);
      if (w == ((b * RSPLIT) >> 5)) {
        const int l0 = (b * RSPLIT) & 31;
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int k = 2 * q + i;
          const double rk = __shfl_sync(0xffffffffu, r, l0 + k * RSPLIT);
          // entry (j, k) of the block's inverse: unit lower for the first sweep of M and the mirror
          // image of that for M^T
          const bool in = b + (j > k ? j : k) < NEQ;
          const bool unit = fwd != TR;
          double a = 0.0;
          if (in && (fwd ? (unit ? k < j : k <= j) : (unit ? k > j : k >= j)))
            a = TR ? tm.A(b + k, b + j) : tm.A(b + j, b + k);
          if (unit && j == k) a = 1.0;
          v = fma(a, rk, v);
        }
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        if (q == 0 && b + j < NEQ) tm.at(ob, b + j) = v;
        const double own = __shfl_sync(0xffffffffu, v, ((row - b) & 7) * 4);
        if (row >= b && row < b + 8) r = own;
      }
      solve_bar();
      const bool upd = fwd ? (row >= b + 8 && row < NEQ) : row < b;
      double p = h == 0 ? r : 0.0;
      if (upd) {
#pragma unroll
        for (int i = 0; i < 8 / RSPLIT; ++i) {
          const int k = b + h + i * RSPLIT;
          if (k < NEQ) p = fma(-(TR ? tm.A(k, row) : tm.A(row, k)), tm.at(ob, k), p);
        }
      }
      p = rsplit_sum(p);
      if (upd) r = p;
    }
    if (TR) {
      solve_bar();
      if (row < NEQ && h == 0) tm.at(ob, tm.perm(row)) = r;
    }
  }
  tsync();
}
#endif

// Solve (LU) x = b in place on the vector at slot ob by one warp (teams narrower than the matrix).
OUTLINE void lu_solve(int ob) {
  const Team tm = make_team();
#if TEAM == 1
  for (int k = 0; k < NEQ; ++k) {
    const int p = tm.piv(k);
    if (p != k) { const double t = tm.at(ob, k); tm.at(ob, k) = tm.at(ob, p); tm.at(ob, p) = t; }
  }
  for (int i = 0; i < NEQ; ++i) {
    double s = tm.at(ob, i);
    for (int j = 0; j < i; ++j) s -= tm.A(i, j) * tm.at(ob, j);
    tm.at(ob, i) = s;
  }
  for (int i = NEQ - 1; i >= 0; --i) {
    double s = tm.at(ob, i);
    for (int j = i + 1; j < NEQ; ++j) s -= tm.A(i, j) * tm.at(ob, j);
    tm.at(ob, i) = s * tm.invd(i);
  }
#else
  // One warp, the vector in registers: lane l holds rows l, l + 32, ... (NB chunks).  Each
  // substitution step broadcasts the finished x_k with a shuffle and updates the rows it feeds,
  // so the dependent chain per step is a shuffle and an FMA, with no shared-memory round trip
  // and no barrier; the matrix loads do not depend on x and are issued ahead.  The update order
  // per row (k increasing forward, decreasing backward) is that of the column-oriented sweep.
  if (tm.tl < 32) {
    const int ln = tm.tl & (WL - 1);
    const unsigned msk = team_mask();
    double xr[NB];
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      const int i = ln + WL * c;
      xr[c] = i < NEQ ? tm.at(ob, tm.perm(i)) : 0.0;  // P b
    }
    // L (unit lower) forward
#pragma unroll
    for (int kb = 0; kb < NB; ++kb) {
#pragma unroll
      for (int kk = 0; kk < WL; ++kk) {
        const int k = kb * WL + kk;
        if (k < NEQ - 1) {
          const double xk = __shfl_sync(msk, xr[kb], kk, WL);
#pragma unroll
          for (int c = kb; c < NB; ++c) {
            const int i = ln + WL * c;
            if ((c > kb || ln > kk) && i < NEQ) xr[c] = fma(-tm.A(i, k), xk, xr[c]);
          }
        }
      }
    }
    // U backward, 1/U_kk from the factorisation
#pragma unroll
    for (int kb = NB - 1; kb >= 0; --kb) {
#pragma unroll
      for (int kk = WL - 1; kk >= 0; --kk) {
        const int k = kb * WL + kk;
        if (k < NEQ) {
          const double xk = __shfl_sync(msk, xr[kb], kk, WL) * tm.invd(k);
          if (ln == kk) xr[kb] = xk;
#pragma unroll
          for (int c = 0; c <= kb; ++c) {
            const int i = ln + WL * c;
            if (c < kb || ln < kk) xr[c] = fma(-tm.A(i, k), xk, xr[c]);
          }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      const int i = ln + WL * c;
      if (i < NEQ) tm.at(ob, i) = xr[c];
    }
  }
  tsync();
#endif
}

#if TEAM > 1
// Column-oriented solve by the team's first warp through shared memory (the adjoint kernels use it: it needs
// no registers for the vector, and the adjoint kernels run at their register cap).
OUTLINE void lu_solve_col(int ob) {
  const Team tm = make_team();
  if (tm.tl < 32) {
    const int ln = tm.tl & (WL - 1);
    const unsigned msk = team_mask();
    {  // P b through the composed permutation
      double g[NB];
#pragma unroll
      for (int c = 0; c < NB; ++c) {
        const int i = ln + WL * c;
        g[c] = i < NEQ ? tm.at(ob, tm.perm(i)) : 0.0;
      }
      __syncwarp(msk);
#pragma unroll
      for (int c = 0; c < NB; ++c) {
        const int i = ln + WL * c;
        if (i < NEQ) tm.at(ob, i) = g[c];
      }
    }
    __syncwarp(msk);
    for (int k = 0; k < NEQ - 1; ++k) {
      const double xk = tm.at(ob, k);
      for (int i = k + 1 + ln; i < NEQ; i += WL) tm.at(ob, i) -= tm.A(i, k) * xk;
      __syncwarp(msk);
    }
    for (int k = NEQ - 1; k >= 0; --k) {
      const double xk = tm.at(ob, k) * tm.invd(k);
      __syncwarp(msk);
      if (ln == (k & (WL - 1))) tm.at(ob, k) = xk;
      for (int i = ln; i < k; i += WL) tm.at(ob, i) -= tm.A(i, k) * xk;
      __syncwarp(msk);
    }
  }
  tsync();
}

#endif

// ------------------------------------------------------------------------------ ROS4 step

// One attempt of the s-stage Rosenbrock method of the generated header (Sec. 2.3, transformed
// form): coefficients rk_a, rk_c, rk_m, rk_e, gamma RGAM, RS stages; rk_newf[i] says whether stage
// i needs f at a new argument (1), reuses the previous stage's f (0: equal argument), or uses
// f(y) (2: the argument is y).  Size hh from y (OFF_Y): y_new into OFF_YT; returns the square of
// the weighted RMS error (infinity if anything is non-finite).
// REG_SOLVE selects, where the blocked solves do not apply, the register-resident stage solves, used
// for state vectors of more than 64 entries; the adjoint's replay takes the column-oriented ones
// (same arithmetic in the same order) to stay within its register budget.
template <bool REG_SOLVE>
__device__ __forceinline__ void stage_solve(int ob) {
#if SOLVE_BLK
  lu_solve_blk<false>(ob);
#elif TEAM > 1
  if (REG_SOLVE) lu_solve(ob);
  else lu_solve_col(ob);
#else
  lu_solve(ob);
#endif
}

template <bool REG_SOLVE = (NB >= 3)>
__device__ double ros4_attempt(const Team& tm, double P, double hh, double rtol, double atol,
                              const double* lnA_ext, double* rho = nullptr, double* wc = nullptr) {
#if ERK
  // explicit Runge-Kutta (RKF45) in increment form: u_i = hh f(y + sum_{j<i} a_ij u_j); no
  // Jacobian, no factorisation
#pragma unroll
  for (int st = 0; st < RS; ++st) {
    if (st > 0) {
      for (int i = tm.tl; i < NEQ; i += TEAM) {
        double v = tm.at(OFF_Y, i);
        for (int j = 0; j < st; ++j)
          if (rk_a[st * RS + j] != 0.0) v += rk_a[st * RS + j] * tm.at(UOFF(j), i);
        tm.at(OFF_YT, i) = v;
      }
      tsync();
    }
    eval_f(st == 0 ? OFF_Y : OFF_YT, OFF_F, P, lnA_ext);
    const int ou = UOFF(st);
    for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(ou, i) = hh * tm.at(OFF_F, i);
    tsync();
  }
#else
  // stage 1: f0 into U1, M = I/(gamma h) - J (with a W-method cache: the cached factorisation
  // of I/(gamma h) - W when it was made for this step size and is young enough)
  const bool reuse = wc && wc[WC_H] == hh && wc[WC_AGE] < WAGE_MAX;
  if (reuse) {
    eval_f(OFF_Y, OFF_U1, P, lnA_ext);
    for (int e = tm.tl; e < NEQ * NEQ; e += TEAM) tm.at(OFF_A, e) = wc[e];
    for (int e = tm.tl; e < PACKED_INTS(NEQ); e += TEAM) {
      tm.at(OFF_PERM, e) = wc[WC_PERM + e];
#if TEAM == 1
      tm.at(OFF_PIV, e) = wc[WC_PIV + e];
#endif
    }
    tsync();
  } else {
    eval_f_jac<-1>(OFF_Y, OFF_U1, P, lnA_ext, fx_rcp(RGAM * hh));
  }
  if (rho && !reuse) {
    // stiffness estimate: Gershgorin bound of the Jacobian scaled by the error weights,
    // max_i sum_j |J_ij| w_j / w_i with w = atol + rtol |y| (J_ij = -A_ij off the diagonal,
    // shift - A_ii on it)
    const double shift = fx_rcp(RGAM * hh);
    double mx = 0.0;
    for (int i = tm.tl; i < NEQ; i += TEAM) {
      double sum = 0.0;
      for (int j = 0; j < NEQ; ++j) {
        const double a = tm.A(i, j);
        sum += fabs(i == j ? shift - a : a) * (atol + rtol * fabs(tm.at(OFF_Y, j)));
      }
      const double r = sum / (atol + rtol * fabs(tm.at(OFF_Y, i)));
      mx = r > mx ? r : mx;
    }
    *rho = team_max(tm, mx);
  }
#if NEED_F0
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(OFF_F0, i) = tm.at(OFF_U1, i);
  tsync();
#endif
  if (!reuse) {
    lu_factor();
    if (wc) {  // keep the factorisation for later attempts of this size
      for (int e = tm.tl; e < NEQ * NEQ; e += TEAM) wc[e] = tm.at(OFF_A, e);
      for (int e = tm.tl; e < PACKED_INTS(NEQ); e += TEAM) {
        wc[WC_PERM + e] = tm.at(OFF_PERM, e);
#if TEAM == 1
        wc[WC_PIV + e] = tm.at(OFF_PIV, e);
#endif
      }
      if (tm.tl == 0) { wc[WC_H] = hh; wc[WC_AGE] = 0.0; }
      tsync();  // copied by every lane before lu_invert overwrites the diagonal blocks
    }
  }
#if SOLVE_BLK
  lu_invert();  // (the cache keeps plain factors, which every launch configuration can read)
#endif
  stage_solve<REG_SOLVE>(OFF_U1);
  const double ih = fx_rcp(hh);
#pragma unroll
  for (int st = 1; st < RS; ++st) {
    if (rk_newf[st] == 1) {
      for (int i = tm.tl; i < NEQ; i += TEAM) {
        double v = tm.at(OFF_Y, i);
        for (int j = 0; j < st; ++j)
          if (rk_a[st * RS + j] != 0.0) v += rk_a[st * RS + j] * tm.at(UOFF(j), i);
        tm.at(OFF_YT, i) = v;
      }
      tsync();
      eval_f(OFF_YT, OFF_F, P, lnA_ext);
    }
#if NEED_F0
    const int of = rk_newf[st] == 2 ? OFF_F0 : OFF_F;
#else
    const int of = OFF_F;
#endif
    const int ou = UOFF(st);
    for (int i = tm.tl; i < NEQ; i += TEAM) {
      double v = 0.0;
      for (int j = 0; j < st; ++j)
        if (rk_c[st * RS + j] != 0.0) v += rk_c[st * RS + j] * tm.at(UOFF(j), i);
      tm.at(ou, i) = fma(ih, v, tm.at(of, i));
    }
    tsync();
    stage_solve<REG_SOLVE>(ou);
  }
#endif
  // new state, error estimate and its weighted RMS norm
  double acc = 0.0;
  bool bad = false;
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    const double y = tm.at(OFF_Y, i);
    double yn = y, e = 0.0;
#pragma unroll
    for (int j = 0; j < RS; ++j) {
      const double u = tm.at(UOFF(j), i);
      if (rk_m[j] != 0.0) yn += rk_m[j] * u;  // zero coefficients fold away at compile time
      if (rk_e[j] != 0.0) e += rk_e[j] * u;
    }
    tm.at(OFF_YT, i) = yn;
    const double ay = fabs(y), an = fabs(yn);
    const double sc = atol + rtol * (ay > an ? ay : an);
    const double z = fx_div(e, sc);
    acc += z * z;
    if (!isfinite(yn)) bad = true;
  }
  acc = team_sum(tm, acc);
  bad = team_any(tm, bad);
  tsync();
  const double err2 = acc * (1.0 / NEQ);
  return (bad || !isfinite(err2)) ? __longlong_as_double(0x7ff0000000000000LL) : err2;
}

// Controller state of one cell (team-uniform: every lane holds the same values).
struct Ctl {
  double t, h;
  int attempts, status;
  bool reject_last, done;
  bool acc;   // the last call accepted a step ...
  double hh;  // ... of this size
  bool want_rho;  // estimate the stiffness at the cell's first attempt (into rho)
  double rho;
  double* wc;     // the cell's W-method cache (global memory) or nullptr
};

// One attempt plus the controller decision (identical rules to the CPU oracle):
// fac = clamp(0.9 err^(-1/order), 0.2, 6) with err floored at 1e-10 (0.2 if non-finite); accept iff
// err <= 1; no growth right after a rejection; the last step is cut to land on dt (a step
// within 0.01% of the remainder is stretched to it); h_out is the controller's proposal after
// the last accepted step, or the proposal that the end cut shortened.
__device__ __forceinline__ void ros4_advance(const Team& tm, Ctl& c, double P, double dt, double rtol,
                                             double atol, int max_steps, double h_min,
                                             const double* lnA_ext) {
  c.acc = false;
  if (c.attempts >= max_steps) { c.status = ST_MAX_STEPS; c.done = true; return; }
  if (c.h < h_min) { c.status = ST_H_UNDERFLOW; c.done = true; return; }
  const bool last = c.t + 1.0001 * c.h >= dt;
  const double hh = last ? dt - c.t : c.h;
  const double err2 = ros4_attempt(tm, P, hh, rtol, atol, lnA_ext,
                                  (c.want_rho && c.attempts == 0) ? &c.rho : nullptr, c.wc);
  c.attempts++;
  const bool finite = isfinite(err2);
  double fac = 0.2;
  if (finite) {
    // 0.9 err^(-1/order), every lane on the integer pipe (two square roots and a division would take
    // about 1,300 clocks of FP64 latency)
    const double e = err2 > 1e-20 ? err2 : 1e-20;
    fac = 0.9 * fx_exp2(-fx_log2(e) / (2 * RORDER));
    fac = fac < 0.2 ? 0.2 : (fac > 6.0 ? 6.0 : fac);
  }
  if (finite && err2 <= 1.0) {
    for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(OFF_Y, i) = tm.at(OFF_YT, i);
    if (c.wc && tm.tl == 0) c.wc[WC_AGE] += 1.0;  // the cached factorisation ages per accepted step
    tsync();
    if (c.reject_last && fac > 1.0) fac = 1.0;
    c.reject_last = false;
    c.acc = true;
    c.hh = hh;
    const double hnext = hh * fac;
    if (last) {
      c.h = hh < c.h ? c.h : hnext;
      c.done = true;
      c.status = ST_OK;
      return;
    }
    c.t += hh;
    c.h = hnext;
  } else {
    c.reject_last = true;
    c.h = hh * fac;
  }
}

// ------------------------------------------------------------------------------ cell I/O

// y = [T, Y_k / W_k] into OFF_Y; returns false if any input is non-finite
__device__ __forceinline__ bool load_cell(const Team& tm, long long c, const double* T, const double* Y,
                                          long long ld) {
  bool bad = false;
  if (tm.tl == 0) {
    const double t = T[c];
    tm.at(OFF_Y, 0) = t;
    bad = !isfinite(t);
  }
  for (int k = tm.tl; k < NS - 1; k += TEAM) {
    const double v = Y[k * ld + c];
    tm.at(OFF_Y, 1 + k) = v * mk_invW[k];
    bad = bad || !isfinite(v);
  }
  bad = team_any(tm, bad);
  tsync();
  return !bad;
}

// T, Y back from OFF_Y; the bath-gas mass fraction from the closure
__device__ __forceinline__ void store_cell(const Team& tm, long long c, double* T, double* Y, long long ld) {
  double s = 0.0;
  for (int k = tm.tl; k < NS - 1; k += TEAM) {
    const double v = tm.at(OFF_Y, 1 + k) * mk_W[k];
    Y[k * ld + c] = v;
    s += v;
  }
  s = team_sum(tm, s);
  if (tm.tl == 0) {
    T[c] = tm.at(OFF_Y, 0);
    Y[(long long)(NS - 1) * ld + c] = 1.0 - s;
  }
}

// broadcast a team-lane-0 value
__device__ __forceinline__ long long team_bcast_ll(const Team& tm, long long v) {
#if TEAM == 1
  return v;
#elif TEAM <= 32
  return __shfl_sync(team_mask(), v, 0, TEAM);
#else
  long long* r = reinterpret_cast<long long*>(&tm.base[OFF_RED + 12]);
  if (tm.tl == 0) *r = v;
  __syncthreads();
  v = *r;
  __syncthreads();
  return v;
#endif
}

// ------------------------------------------------------------------------------ kernels

extern "C" __global__ void __launch_bounds__(TPB)
chem_eval_source_k(long long n_cells, const double* __restrict__ T, const double* __restrict__ P,
                   const double* __restrict__ n, double* __restrict__ f, long long ld,
                   const double* __restrict__ lnA_ext) {
  const Team tm = make_team();
  const long long team_id = (long long)blockIdx.x * NTEAM + (TEAM <= 32 ? threadIdx.x / TEAM : 0);
  const long long stride = (long long)gridDim.x * NTEAM;
  for (long long c = team_id; c < n_cells; c += stride) {
    if (tm.tl == 0) tm.at(OFF_Y, 0) = T[c];
    for (int k = tm.tl; k < NS - 1; k += TEAM) tm.at(OFF_Y, 1 + k) = n[k * ld + c];
    tsync();
    eval_f(OFF_Y, OFF_F, P[c], lnA_ext);
    for (int i = tm.tl; i < NEQ; i += TEAM) f[i * ld + c] = tm.at(OFF_F, i);
    tsync();
  }
}

extern "C" __global__ void __launch_bounds__(TPB)
chem_eval_jacobian_k(long long n_cells, const double* __restrict__ T, const double* __restrict__ P,
                     const double* __restrict__ n, double* __restrict__ J, long long ld,
                     const double* __restrict__ lnA_ext) {
  const Team tm = make_team();
  const long long team_id = (long long)blockIdx.x * NTEAM + (TEAM <= 32 ? threadIdx.x / TEAM : 0);
  const long long stride = (long long)gridDim.x * NTEAM;
  for (long long c = team_id; c < n_cells; c += stride) {
    if (tm.tl == 0) tm.at(OFF_Y, 0) = T[c];
    for (int k = tm.tl; k < NS - 1; k += TEAM) tm.at(OFF_Y, 1 + k) = n[k * ld + c];
    tsync();
    eval_f_jac<1>(OFF_Y, OFF_U1, P[c], lnA_ext, 0.0);  // f goes to U1: F aliases J scratch
    for (int e = tm.tl; e < NEQ * NEQ; e += TEAM) J[(long long)e * ld + c] = tm.at(OFF_A, e);
    tsync();
  }
}

// Per-cell method switching (chem_int_opts.cell_method): a launch of the alternative method's
// module (RKF45, or the W-method with its factorisation cache) runs the cells marked for it under
// their attempt budgets and keeps the input of any that fails; a launch of the Rosenbrock module
// runs the others and the failed ones and marks each cell for the next call:
//   * alternative RKF45 (AUTO_IMPLICIT): when dt * rho <= STIFF_BETA * attempts, rho the stiffness
//     estimate at the cell's first attempt (the explicit method's stability-limited steps, about
//     dt * rho / STIFF_BETA, would not outnumber the Rosenbrock attempts);
//   * alternative W-method (AUTO_IMPLICIT_W): when the cell took a single attempt and the
//     controller's next-step proposal is at least W_ENTRY_MARGIN * dt (a quiescent cell, whose
//     split steps the cached factorisation can serve; a cell whose one step only just fitted
//     would need many more steps of the second-order W-method); its cache is emptied, so the
//     W-method starts from a Jacobian at its own state;
// with budget 4 * attempts + 8; after a success of the alternative method with a attempts, it
// stays with budget 4a + 8.
#define AUTO_EXPLICIT 1
#define AUTO_IMPLICIT 2
#define AUTO_IMPLICIT_W 3
#define STIFF_BETA 3.0
#define W_ENTRY_MARGIN 2.0

// Persistent driver: each team pulls cells from the queue counter and integrates them to dt.
// With TEAM == 1 each thread refills independently (per-lane refill of retired cells); the
// loop body is one step attempt so that lanes on different cells still execute it together.
extern "C" __global__ void __launch_bounds__(TPB, MIN_BLOCKS)
chem_integrate_k(long long n_cells, double* __restrict__ T, const double* __restrict__ P,
                 double* __restrict__ Y, long long ld, double dt, double rtol, double atol,
                 double* __restrict__ h_io, int* __restrict__ status_out,
                 int* __restrict__ attempts_out, const double* __restrict__ lnA_ext,
                 int max_steps, double h_min, double T_min, unsigned long long* queue,
                 int* __restrict__ tape_nacc, double* __restrict__ tape_h, double* __restrict__ tape_ck,
                 int tape_cap, int interval, const int* __restrict__ order,
                 const unsigned int* __restrict__ order_count, int keep_failed,
                 int* __restrict__ cell_method, int auto_mode, double* __restrict__ jac_cache) {
  const Team tm = make_team();
  long long cell = -1;
  double Pc = 0.0;
  Ctl c;
  c.done = true;
  c.acc = false;
  c.want_rho = false;
  c.rho = 0.0;
  c.wc = nullptr;
  int nacc = 0;
  int ms_cell = max_steps;
  // queue positions: n_cells, or the device-held length of the cell list `order`
  const long long nq = order_count ? (long long)*order_count : n_cells;
  // bounded: every iteration either retires a cell or makes an attempt (<= max_steps per cell),
  // or consumes a queue position
  for (;;) {
    if (c.done) {
      long long nc = 0;
      if (tm.tl == 0) {
        const long long q = (long long)atomicAdd(queue, 1ULL);
        if (q >= nq) nc = n_cells;
        else if (order) nc = (order[q] >= 0 && order[q] < n_cells) ? order[q] : -1;
        else nc = q;
      }
      cell = team_bcast_ll(tm, nc);
      if (cell >= n_cells) break;
      if (cell < 0) continue;  // an invalid entry of the cell list: skipped
      Pc = P[cell];
      c.t = 0.0;
      c.h = h_io ? h_io[cell] : 0.0;
      if (!(c.h > 0.0)) c.h = dt;
      c.attempts = 0;
      c.status = ST_OK;
      c.reject_last = false;
      c.done = false;
      c.want_rho = auto_mode == AUTO_IMPLICIT;
      c.rho = 0.0;
      // the W-method's factorisation cache (not used by a Rosenbrock launch of the switching)
      c.wc = (jac_cache && auto_mode != AUTO_IMPLICIT_W) ? jac_cache + cell * (long long)WC_STRIDE : nullptr;
      // per-cell method switching: an explicit cell runs under its attempt budget
      ms_cell = max_steps;
      if (auto_mode == AUTO_EXPLICIT) {
        const int b = cell_method[cell];
        ms_cell = b > 0 && b < max_steps ? b : max_steps;
      }
      const bool ok = load_cell(tm, cell, T, Y, ld);
      nacc = 0;
      if (!ok || tm.at(OFF_Y, 0) < T_min) {
        if (tm.tl == 0) {
          if (status_out) status_out[cell] = ok ? ST_SKIPPED : ST_NONFINITE;
          if (attempts_out) attempts_out[cell] = 0;
          if (tape_nacc) tape_nacc[cell] = 0;
        }
        c.done = true;
        tsync();
        continue;
      }
      if (tape_ck)  // checkpoint 0: the initial state
        for (int i = tm.tl; i < NEQ; i += TEAM) tape_ck[(long long)i * n_cells + cell] = tm.at(OFF_Y, i);
    }
    if (tape_h && nacc >= tape_cap) {
      // the tape holds no further step: stop before attempting one, so that the stored state is
      // exactly the map the tape records (the adjoint then differentiates what was returned)
      c.status = ST_TAPE_FULL;
      c.done = true;
    } else {
      ros4_advance(tm, c, Pc, dt, rtol, atol, ms_cell, h_min, lnA_ext);
    }
    if (tape_h && c.acc && c.status != ST_TAPE_FULL) {
      // record the accepted step; checkpoint the state after every `interval` accepted steps
      if (tm.tl == 0) tape_h[(long long)nacc * n_cells + cell] = c.hh;
      ++nacc;
      if (nacc % interval == 0 && nacc < tape_cap)
        for (int i = tm.tl; i < NEQ; i += TEAM)
          tape_ck[((long long)(nacc / interval) * NEQ + i) * n_cells + cell] = tm.at(OFF_Y, i);
    }
    if (c.done) {
      if (tm.tl == 0 && tape_nacc) tape_nacc[cell] = nacc;
      // keep_failed: a cell that did not reach dt leaves its input state and step size in place
      // (a later launch integrates it again from the start)
      const bool keep = keep_failed && c.status != ST_OK;
      if (!keep) store_cell(tm, cell, T, Y, ld);
      if (tm.tl == 0) {
        if (h_io && !keep) h_io[cell] = c.h;
        if (status_out) status_out[cell] = c.status;
        if (attempts_out) attempts_out[cell] = c.attempts;
        if (auto_mode == AUTO_EXPLICIT)  // success: stay explicit, budget from this run
          cell_method[cell] = c.status == ST_OK ? 4 * c.attempts + 8 : 0;
        else if (auto_mode == AUTO_IMPLICIT)  // explicit next time if its stable steps are few
          cell_method[cell] = (c.status == ST_OK && dt * c.rho <= STIFF_BETA * c.attempts)
                                  ? 4 * c.attempts + 8 : 0;
        else if (auto_mode == AUTO_IMPLICIT_W) {  // the W-method next time if quiescent
          cell_method[cell] =
              (c.status == ST_OK && c.attempts == 1 && c.h >= W_ENTRY_MARGIN * dt) ? 12 : 0;
          if (jac_cache) jac_cache[cell * (long long)WC_STRIDE + WC_H] = 0.0;
        }
      }
      tsync();
    }
  }
}

// Cost-ordered work queue: a permutation of the cells by decreasing predicted cost (a counting
// sort over CHEM_ORDER_BINS cost buckets: histogram, descending exclusive scan, scatter).  Cells of
// equal cost are placed in no particular order.
#define ORDER_BINS 1024
extern "C" __global__ void chem_order_hist_k(long long n_cells, const int* __restrict__ cost,
                                             unsigned int* __restrict__ bins) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_cells) return;
  const int v = cost[c];
  atomicAdd(&bins[v < 0 ? 0 : (v >= ORDER_BINS ? ORDER_BINS - 1 : v)], 1u);
}

// one block of ORDER_BINS threads: starts[b] = number of cells in bins above b
extern "C" __global__ void __launch_bounds__(ORDER_BINS) chem_order_scan_k(const unsigned int* __restrict__ bins,
                                                                          unsigned int* __restrict__ starts) {
  __shared__ unsigned int sh[ORDER_BINS];
  const int t = threadIdx.x;
  sh[t] = bins[ORDER_BINS - 1 - t];  // descending order of cost
  __syncthreads();
  for (int o = 1; o < ORDER_BINS; o <<= 1) {
    const unsigned int v = t >= o ? sh[t - o] : 0u;
    __syncthreads();
    sh[t] += v;
    __syncthreads();
  }
  // inclusive scan over descending bins; exclusive start of bin b = inclusive value of its predecessor
  const int b = ORDER_BINS - 1 - t;
  starts[b] = t > 0 ? sh[t - 1] : 0u;
}

extern "C" __global__ void chem_order_scatter_k(long long n_cells, const int* __restrict__ cost,
                                                unsigned int* __restrict__ starts, int* __restrict__ order) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_cells) return;
  const int v = cost[c];
  const unsigned int pos = atomicAdd(&starts[v < 0 ? 0 : (v >= ORDER_BINS ? ORDER_BINS - 1 : v)], 1u);
  order[pos] = (int)c;
}

// Per-cell method switching: split the cells into the explicit list (cell_method > 0) and the
// implicit list; counts[0], counts[1] their lengths (zeroed by the caller).
extern "C" __global__ void chem_route_k(long long n_cells, const int* __restrict__ cell_method,
                                        int* __restrict__ list_e, int* __restrict__ list_i,
                                        unsigned int* __restrict__ counts) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_cells) return;
  if (cell_method[c] > 0) list_e[atomicAdd(&counts[0], 1u)] = (int)c;
  else list_i[atomicAdd(&counts[1], 1u)] = (int)c;
}

// After the explicit launch: its cells that ran out of budget (or step size) go to the end of the
// implicit list; the others' status is final and is copied to the caller's array.
extern "C" __global__ void chem_route_fallback_k(long long n_cells, const int* __restrict__ list_e,
                                                 unsigned int* __restrict__ counts, const int* __restrict__ st_e,
                                                 int* __restrict__ list_i, int* __restrict__ status_out) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (long long)counts[0]) return;
  const int c = list_e[q];
  if (c < 0 || c >= n_cells) return;
  const int s = st_e[c];
  if (s == ST_MAX_STEPS || s == ST_H_UNDERFLOW) list_i[atomicAdd(&counts[1], 1u)] = c;
  else if (status_out) status_out[c] = s;
}

// Plain driver, one launch per step attempt over all cells.  Per-cell controller state lives
// in the workspace: y [NEQ][n] (cell-fastest), t, h [n], packed flags/attempts/status [n].
struct PlainWs {
  double* y;
  double* t;
  double* h;
  int* flags;     // bit0 active, bit1 reject_last
  int* attempts;
  int* status;
  unsigned int* active_count;  // one counter per launch index
};

extern "C" __global__ void __launch_bounds__(TPB)
chem_plain_init_k(long long n_cells, const double* __restrict__ T, const double* __restrict__ Y,
                  long long ld, double dt, const double* __restrict__ h_in, double T_min,
                  double* wy, double* wt, double* wh, int* wflags, int* watt, int* wst) {
  const Team tm = make_team();
  const long long team_id = (long long)blockIdx.x * NTEAM + (TEAM <= 32 ? threadIdx.x / TEAM : 0);
  const long long stride = (long long)gridDim.x * NTEAM;
  for (long long c = team_id; c < n_cells; c += stride) {
    const bool ok = load_cell(tm, c, T, Y, ld);
    for (int i = tm.tl; i < NEQ; i += TEAM) wy[i * n_cells + c] = tm.at(OFF_Y, i);
    if (tm.tl == 0) {
      double h = h_in ? h_in[c] : 0.0;
      if (!(h > 0.0)) h = dt;
      wt[c] = 0.0;
      wh[c] = h;
      watt[c] = 0;
      const bool skip = ok && tm.at(OFF_Y, 0) < T_min;
      wst[c] = ok ? (skip ? ST_SKIPPED : ST_OK) : ST_NONFINITE;
      wflags[c] = (ok && !skip) ? 1 : 0;
    }
    tsync();
  }
}

// same register cap as the persistent driver, so that the two differ only in how cells are scheduled
extern "C" __global__ void __launch_bounds__(TPB, MIN_BLOCKS)
chem_plain_attempt_k(long long n_cells, double* __restrict__ T, const double* __restrict__ P,
                     double* __restrict__ Y, long long ld, double dt, double rtol, double atol,
                     double* __restrict__ h_out, int* __restrict__ status_out,
                     int* __restrict__ attempts_out, const double* __restrict__ lnA_ext,
                     int max_steps, double h_min, double* wy, double* wt, double* wh, int* wflags,
                     int* watt, int* wst, unsigned int* active_count) {
  const Team tm = make_team();
  const long long team_id = (long long)blockIdx.x * NTEAM + (TEAM <= 32 ? threadIdx.x / TEAM : 0);
  const long long stride = (long long)gridDim.x * NTEAM;
  for (long long cell = team_id; cell < n_cells; cell += stride) {
    const int fl = wflags[cell];
    if (!(fl & 1)) continue;  // team-uniform
    for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(OFF_Y, i) = wy[i * n_cells + cell];
    tsync();
    Ctl c;
    c.t = wt[cell];
    c.h = wh[cell];
    c.attempts = watt[cell];
    c.status = ST_OK;
    c.reject_last = (fl & 2) != 0;
    c.done = false;
    c.want_rho = false;
    c.wc = nullptr;
    ros4_advance(tm, c, P[cell], dt, rtol, atol, max_steps, h_min, lnA_ext);
    if (c.done) {
      store_cell(tm, cell, T, Y, ld);
      if (tm.tl == 0) {
        if (h_out) h_out[cell] = c.h;
        if (status_out) status_out[cell] = c.status;
        if (attempts_out) attempts_out[cell] = c.attempts;
        wflags[cell] = 0;
      }
    } else {
      for (int i = tm.tl; i < NEQ; i += TEAM) wy[i * n_cells + cell] = tm.at(OFF_Y, i);
      if (tm.tl == 0) {
        wt[cell] = c.t;
        wh[cell] = c.h;
        watt[cell] = c.attempts;
        wflags[cell] = 1 | (c.reject_last ? 2 : 0);
        atomicAdd(active_count, 1u);
      }
    }
    tsync();
  }
}

// Cells the plain driver never activated (non-finite or below T_min) get their status here.
extern "C" __global__ void chem_plain_finish_k(long long n_cells, int* __restrict__ status_out,
                                               int* __restrict__ attempts_out, const int* wst,
                                               const int* wflags_init_status) {
  const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_cells) return;
  const int s = wst[c];
  if (s == ST_SKIPPED || s == ST_NONFINITE) {
    if (status_out) status_out[c] = s;
    if (attempts_out) attempts_out[c] = 0;
  }
  (void)wflags_init_status;
}

// ============================================================================ discrete adjoint
// Gradients of a loss on the final state with respect to ln A of every reaction and to the
// initial state, through the ROS4 steps with the accepted step sizes frozen (Sec. 2.3 algebra,
// differentiated).  Only built for multi-lane teams (contiguous shared-memory layout), and only
// into the separately compiled adjoint module (CHEM_ADJOINT) so that forward modules compile fast.
#if TEAM >= 32 && defined(CHEM_ADJOINT) && TABLEAU_ID == 0

// forward-mode dual number: value and one directional derivative
struct DD {
  double v, d;
};
__device__ __forceinline__ DD mk(double v, double d) { DD r; r.v = v; r.d = d; return r; }
__device__ __forceinline__ DD operator+(DD a, DD b) { return mk(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ DD operator-(DD a, DD b) { return mk(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ DD operator-(DD a) { return mk(-a.v, -a.d); }
__device__ __forceinline__ DD operator*(DD a, DD b) { return mk(a.v * b.v, a.d * b.v + a.v * b.d); }
__device__ __forceinline__ DD operator/(DD a, DD b) {
  const double rb = fx_rcp(b.v);
  const double q = a.v * rb;
  return mk(q, (a.d - q * b.d) * rb);
}
__device__ __forceinline__ DD operator+(DD a, double b) { return mk(a.v + b, a.d); }
__device__ __forceinline__ DD operator+(double b, DD a) { return mk(a.v + b, a.d); }
__device__ __forceinline__ DD operator-(DD a, double b) { return mk(a.v - b, a.d); }
__device__ __forceinline__ DD operator-(double b, DD a) { return mk(b - a.v, -a.d); }
__device__ __forceinline__ DD operator*(DD a, double b) { return mk(a.v * b, a.d * b); }
__device__ __forceinline__ DD operator*(double b, DD a) { return mk(a.v * b, a.d * b); }
__device__ __forceinline__ DD operator/(DD a, double b) { const double rb = fx_rcp(b); return mk(a.v * rb, a.d * rb); }
__device__ __forceinline__ DD operator/(double b, DD a) {
  const double ra = fx_rcp(a.v);
  const double q = b * ra;
  return mk(q, -q * a.d * ra);
}
// value functions on the integer pipe (fx_*)
__device__ __forceinline__ double xexp(double a) { return fx_exp(a); }
__device__ __forceinline__ double xlog(double a) { return fx_log(a); }
__device__ __forceinline__ double xlog10(double a) { return fx_log(a) * (1.0 / LN10); }
__device__ __forceinline__ double xdiv(double a, double b) { return a * fx_rcp(b); }
__device__ __forceinline__ DD xexp(DD a) { const double e = fx_exp(a.v); return mk(e, e * a.d); }
__device__ __forceinline__ DD xlog(DD a) { return mk(fx_log(a.v), a.d * fx_rcp(a.v)); }
__device__ __forceinline__ DD xlog10(DD a) { return mk(fx_log(a.v) * (1.0 / LN10), a.d * fx_rcp(a.v) * (1.0 / LN10)); }
__device__ __forceinline__ DD xdiv(DD a, DD b) { return a / b; }
__device__ __forceinline__ DD xdiv(double a, DD b) { return a / b; }
__device__ __forceinline__ DD xdiv(DD a, double b) { return a / b; }
// a/b where b may be too small to have a reciprocal (rate constants)
__device__ __forceinline__ double xdiv_wide(double a, double b) { return fx_div(a, b); }
__device__ __forceinline__ DD xdiv_wide(DD a, DD b) {
  const double q = fx_div(a.v, b.v);
  return mk(q, fx_div(a.d - q * b.d, b.v));
}
__device__ __forceinline__ double vof(double a) { return a; }
__device__ __forceinline__ double vof(DD a) { return a.v; }
__device__ __forceinline__ double dof(double a) { return 0.0; }
__device__ __forceinline__ double dof(DD a) { return a.d; }
template <class S> struct S_is_dual { static constexpr bool value = false; };
template <> struct S_is_dual<DD> { static constexpr bool value = true; };
template <class S> __device__ __forceinline__ S szero();
template <> __device__ __forceinline__ double szero<double>() { return 0.0; }
template <> __device__ __forceinline__ DD szero<DD>() { return mk(0.0, 0.0); }
__device__ __forceinline__ void atomic_add_s(double* p, double v) { atomicAdd(p, v); }
__device__ __forceinline__ void atomic_add_s(DD* p, DD v) {
  atomicAdd(&p->v, v.v);
  atomicAdd(&p->d, v.d);
}
__device__ __forceinline__ DD shfl_xor(DD a, int o) {
  return mk(__shfl_xor_sync(0xffffffffu, a.v, o), __shfl_xor_sync(0xffffffffu, a.d, o));
}
__device__ __forceinline__ double shfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }

// adjoint slots, appended after the forward layout (units of doubles; DD arrays take 2 per entry)
#define AOFF_LAM SLOTS
#define AOFF_YB (AOFF_LAM + NEQ)
#define AOFF_UB (AOFF_YB + NEQ)
#define AOFF_W (AOFF_UB + 4 * NEQ)
#define AOFF_FB (AOFF_W + 4 * NEQ)
#define AOFF_Y2 (AOFF_FB + NEQ)
#define AOFF_Y3 (AOFF_Y2 + NEQ)
#define AOFF_V (AOFF_Y3 + NEQ)
#define AOFF_GP (AOFF_V + NEQ)
#define AOFF_TMP (AOFF_GP + NR)
#define AOFF_S (AOFF_TMP + NEQ)
// S-typed (2 doubles each) scratch of the VJP: state, gy, C, hRT, cp, ex, iex, dcp, atilde, Cbar,
// omega (11 x NS) and q (NR), plus 8 reduction slots
#define VS_Y 0
#define VS_GY (VS_Y + NEQ)
#define VS_C (VS_GY + NEQ)
#define VS_HRT (VS_C + NS)
#define VS_CP (VS_HRT + NS)
#define VS_EX (VS_CP + NS)
#define VS_IEX (VS_EX + NS)
#define VS_DCP (VS_IEX + NS)
#define VS_AT (VS_DCP + NS)
#define VS_CB (VS_AT + NS)
#define VS_OM (VS_CB + NS)
#define VS_Q (VS_OM + NS)
#define VS_RED (VS_Q + NR)
#define VS_TOTAL (VS_RED + 8 * TEAM / 32)
#define ASLOTS (AOFF_S + 2 * VS_TOTAL)

template <class S>
__device__ __forceinline__ S team_sum_s(const Team& tm, S v, S* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = v + shfl_xor(v, o);
#if TEAM > 32
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = red[0];
  for (int w = 1; w < TEAM / 32; ++w) v = v + red[w];
  __syncthreads();
#endif
  return v;
}

// Reverse-mode vector-Jacobian product of f at the state in VS_Y (type S):
//   gy = J(y)^T v  (into VS_GY)  and  gp_r += v^T d f / d lnA_r  (value part when S = double,
//   directional-derivative part when S = DD; accumulated into AOFF_GP).
// phi(y) = v^T f(y) = sum_k atilde_k omega_k with atilde_k = V v_{1+k} [k < bath]
// - v_T T V (h_k/RT) / cpm; gy = sum_k atilde_k d omega_k/dy + sum_k omega_k d atilde_k/dy.
template <class S>
OUTLINE void vjp(double P, const double* __restrict__ lnA_ext) {
  const Team tm = make_team();
  S* sb = reinterpret_cast<S*>(&tm.base[AOFF_S]);
  S* Y = sb + VS_Y;
  const double* v = &tm.base[AOFF_V];
  double* gp = &tm.base[AOFF_GP];
  const S T = Y[0];
  const S invT = xdiv(1.0, T);
  const S lnT = xlog(T);
  const S Z = szero<S>();
  S wsum = Z, nsum = Z;
  for (int k = tm.tl; k < NS - 1; k += TEAM) {
    wsum = wsum + mk_W[k] * Y[1 + k];
    nsum = nsum + Y[1 + k];
  }
  S* red = sb + VS_RED;
  wsum = team_sum_s(tm, wsum, red);
  nsum = team_sum_s(tm, nsum, red);
  const S nb = (1.0 - wsum) * mk_invW[BATH];
  const S V = (nsum + nb) * R_U * T * fx_rcp(P);
  const S invV = xdiv(1.0, V);
  S cpm = Z, dcpm = Z;
  for (int k = tm.tl; k < NS; k += TEAM) {
    const S n = k < NS - 1 ? Y[1 + k] : nb;
    sb[VS_C + k] = n * invV;
    const int r = vof(T) < mk_Tmid[k] ? 0 : 1;
    const double* c = mk_cp[k][r];
    const double* hh = mk_h[k][r];
    const double* s = mk_s[k][r];
    const double* d = mk_dcp[k][r];
    const S cp = c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4])));
    const S hRT = hh[0] + T * (hh[1] + T * (hh[2] + T * (hh[3] + T * hh[4]))) + hh[5] * invT;
    const S sR = s[0] * lnT + s[6] + T * (s[1] + T * (s[2] + T * (s[3] + T * s[4])));
    const S dcp = d[0] + T * (d[1] + T * (d[2] + T * d[3]));
    const S ex = xexp(sR - hRT);
    sb[VS_CP + k] = cp;
    sb[VS_HRT + k] = hRT;
    sb[VS_EX + k] = ex;
    sb[VS_IEX + k] = xdiv(1.0, ex);
    sb[VS_DCP + k] = dcp;
    sb[VS_CB + k] = Z;
    cpm = cpm + n * cp;
    dcpm = dcpm + n * dcp;
  }
  cpm = team_sum_s(tm, cpm, red);
  dcpm = team_sum_s(tm, dcpm, red);
  const double vT = v[0];
  const S kT = xdiv(vT * T * V, cpm);
  for (int k = tm.tl; k < NS; k += TEAM) {
    const S a0 = k < NS - 1 ? V * v[1 + k] : Z;
    sb[VS_AT + k] = a0 - kT * sb[VS_HRT + k];
  }
  tsync();
  const S Ctot = P * invT * INV_R_U;
  const S rtp = R_OVER_PATM * T;
  const S irtp = PATM_OVER_R * invT;
  S Tbar = Z, Bbar = Z;
  for (int r = tm.tl; r < NR; r += TEAM) {
    const int kind = mk_kind[r];
    const double lA = lnA_ext ? lnA_ext[mk_rorig[r]] : mk_lnA[r];
    const S kinf = xexp(lA + mk_b[r] * lnT - mk_th[r] * invT);
    S kf = kinf;
    S dlkf_dT = (mk_b[r] + mk_th[r] * invT) * invT;
    S dlkf_dM = Z;
    S M = Z;
    S one_minus_g = Z + 1.0;  // d ln kf / d ln k_inf
    if (kind != ELEM) {
      M = Ctot;
      for (int e = mk_effoff[r]; e < mk_effoff[r + 1]; ++e) M = M + mk_effval[e] * sb[VS_C + mk_effsp[e]];
    }
    if (kind >= LIND) {
      const S k0 = xexp(mk_lnA0[r] + mk_b0[r] * lnT - mk_th0[r] * invT);
      S Pr = xdiv_wide(k0 * M, kinf);
      bool floored = false;
      if (vof(Pr) < 1e-300) { Pr = Z + 1e-300; floored = true; }
      S F = Z + 1.0, dlF_dlPr = Z, dlF_dT = Z;
      if (kind == TROE) {
        const double a = mk_troe[r][0];
        const S e3 = xexp(-T * mk_troe[r][1]);
        const S e1 = xexp(-T * mk_troe[r][2]);
        const double T2 = mk_troe[r][3];
        const S e2 = T2 > 0.0 ? xexp(-T2 * invT) : Z;
        const S Fc = (1.0 - a) * e3 + a * e1 + e2;
        const S lFc = xlog10(Fc);
        const S c = -0.4 - 0.67 * lFc;
        const S n = 0.75 - 1.27 * lFc;
        const S x = xlog10(Pr) + c;
        const S d = n - 0.14 * x;
        const S id = xdiv(1.0, d);
        const S f1 = x * id;
        const S den = xdiv(1.0, 1.0 + f1 * f1);
        const S lF = lFc * den;
        F = xexp(lF * LN10);
        const S g2 = 2.0 * lFc * f1 * den * den;
        if (!floored) dlF_dlPr = -g2 * n * id * id;
        const S dFc = -(1.0 - a) * mk_troe[r][1] * e3 - a * mk_troe[r][2] * e1 +
                      (T2 > 0.0 ? T2 * invT * invT * e2 : Z);
        const S df1_dlFc = (-0.67 * n + 1.27 * x) * id * id;
        dlF_dT = (den - g2 * df1_dlFc) * xdiv(dFc, Fc);
      }
      kf = kinf * xdiv(Pr, 1.0 + Pr) * F;
      const S g = floored ? Z : xdiv(1.0, 1.0 + Pr) + dlF_dlPr;
      const S dlk0 = (mk_b0[r] + mk_th0[r] * invT) * invT;
      dlkf_dM = xdiv(g, M);
      dlkf_dT = dlkf_dT + g * (dlk0 - dlkf_dT) + dlF_dT;
      one_minus_g = 1.0 - g;
    }
    S kr = kf, fwd = kf, rev = Z + 1.0;
    const int nre = mk_nre[r], npr = mk_npr[r];
    S abar = Z;
    S dlKc = Z - mk_dnuf[r];
    for (int i = 0; i < nre; ++i) {
      const int sp = mk_rsp[r][i];
      for (int q = 0; q < mk_rnu[r][i]; ++q) { fwd = fwd * sb[VS_C + sp]; kr = kr * sb[VS_EX + sp]; }
      abar = abar - mk_rnuf[r][i] * sb[VS_AT + sp];
      dlKc = dlKc - mk_rnuf[r][i] * sb[VS_HRT + sp];
    }
    for (int i = 0; i < npr; ++i) {
      const int sp = mk_psp[r][i];
      for (int q = 0; q < mk_pnu[r][i]; ++q) { rev = rev * sb[VS_C + sp]; kr = kr * sb[VS_IEX + sp]; }
      abar = abar + mk_pnuf[r][i] * sb[VS_AT + sp];
      dlKc = dlKc + mk_pnuf[r][i] * sb[VS_HRT + sp];
    }
    const int dnu = mk_dnu[r];
    for (int q = 0; q < dnu; ++q) kr = kr * rtp;
    for (int q = 0; q < -dnu; ++q) kr = kr * irtp;
    rev = rev * kr;
    const S m = kind == THIRD ? M : Z + 1.0;
    const S qnet = fwd - rev;
    const S q = m * qnet;
    sb[VS_Q + r] = q;
    // parameter: d q / d lnA_r = q (d ln kf / d ln k_inf)
    const S gpr = abar * q * one_minus_g;
    gp[r] += S_is_dual<S>::value ? dof(gpr) : vof(gpr);
    dlKc = dlKc * invT;
    const S dqdT = m * (fwd * dlkf_dT - rev * (dlkf_dT - dlKc));
    Tbar = Tbar + abar * dqdT;
    if (kind != ELEM) {
      const S beta = kind == THIRD ? qnet : qnet * dlkf_dM;
      Bbar = Bbar + abar * beta;
      for (int e = mk_effoff[r]; e < mk_effoff[r + 1]; ++e)
        atomic_add_s(&sb[VS_CB + mk_effsp[e]], abar * beta * mk_effval[e]);
    }
    // d q / d C_j of the mass-action products
    for (int i = 0; i < nre; ++i) {
      const int nu = mk_rnu[r][i];
      S p = m * kf * mk_rnuf[r][i];
      for (int i2 = 0; i2 < nre; ++i2) {
        const int e = i2 == i ? nu - 1 : mk_rnu[r][i2];
        for (int t = 0; t < e; ++t) p = p * sb[VS_C + mk_rsp[r][i2]];
      }
      atomic_add_s(&sb[VS_CB + mk_rsp[r][i]], abar * p);
    }
    for (int i = 0; i < npr; ++i) {
      const int nu = mk_pnu[r][i];
      S p = -(m * kr * mk_pnuf[r][i]);
      for (int i2 = 0; i2 < npr; ++i2) {
        const int e = i2 == i ? nu - 1 : mk_pnu[r][i2];
        for (int t = 0; t < e; ++t) p = p * sb[VS_C + mk_psp[r][i2]];
      }
      atomic_add_s(&sb[VS_CB + mk_psp[r][i]], abar * p);
    }
  }
  Tbar = team_sum_s(tm, Tbar, red);
  Bbar = team_sum_s(tm, Bbar, red);
  tsync();
  // omega from q (fixed-order gather), and the mixture sums that use it
  S Q = Z, cpw = Z, vw = Z, Dbar = Z;
  for (int k = tm.tl; k < NS; k += TEAM) {
    S om = Z;
    for (int sg = mk_spseg_beg[k]; sg < mk_spseg_beg[k + 1]; ++sg)
      for (int e = mk_gseg_beg[sg]; e < mk_gseg_beg[sg + 1]; ++e) om = om + mk_gent_nu[e] * sb[VS_Q + mk_gent_rx[e]];
    sb[VS_OM + k] = om;
    Q = Q + sb[VS_HRT + k] * om;
    cpw = cpw + sb[VS_CP + k] * om;
    if (k < NS - 1) vw = vw + v[1 + k] * om;
    const S cb = sb[VS_CB + k] + Bbar;  // default third-body efficiency part on every C_j
    sb[VS_CB + k] = cb;
    Dbar = Dbar + cb * sb[VS_C + k];
  }
  Q = team_sum_s(tm, Q, red);
  cpw = team_sum_s(tm, cpw, red);
  vw = team_sum_s(tm, vw, red);
  Dbar = team_sum_s(tm, Dbar, red);
  tsync();
  const S Sp = vw - xdiv(vT * T * Q, cpm);  // sum_k omega_k atilde_k / V
  const S RTP = R_U * T * fx_rcp(P);
  const S icpm2 = xdiv(1.0, cpm * cpm);
  S* gy = sb + VS_GY;
  if (tm.tl == 0)
    gy[0] = Tbar - Dbar * invT + V * invT * Sp - vT * V * (xdiv(cpw, cpm) - T * Q * dcpm * icpm2);
  const S cbb = sb[VS_CB + BATH];
  const S cpb = sb[VS_CP + BATH];
  for (int j = tm.tl; j < NS - 1; j += TEAM) {
    const double w = mk_wratio[j];
    gy[1 + j] = (sb[VS_CB + j] - w * cbb) * invV - Dbar * RTP * (1.0 - w) * invV + RTP * (1.0 - w) * Sp +
                vT * T * V * Q * (sb[VS_CP + j] - w * cpb) * icpm2;
  }
  tsync();
}

#if SOLVE_BLK
__device__ __forceinline__ void adj_solve_T(int ob) { lu_solve_blk<true>(ob); }
#else
// Solve M^T x = b in place at slot ob with the LU of P M (P M = L U, so M^T = U^T L^T P):
// U^T z = b forward, L^T t = z backward, x = P^T t.  The first warp works.
OUTLINE void lu_solve_T(int ob) {
  const Team tm = make_team();
  if (tm.tl < 32) {
    const int ln = tm.tl;
    for (int i = ln; i < NEQ; i += 32) tm.at(AOFF_TMP, i) = tm.at(ob, i);
    __syncwarp();
    for (int i = 0; i < NEQ; ++i) {
      const double zi = tm.at(AOFF_TMP, i) * tm.invd(i);
      __syncwarp();
      if (ln == (i & 31)) tm.at(AOFF_TMP, i) = zi;
      for (int k = i + 1 + ln; k < NEQ; k += 32) tm.at(AOFF_TMP, k) -= tm.A(i, k) * zi;
      __syncwarp();
    }
    for (int i = NEQ - 1; i > 0; --i) {
      const double ti = tm.at(AOFF_TMP, i);
      for (int k = ln; k < i; k += 32) tm.at(AOFF_TMP, k) -= tm.A(i, k) * ti;
      __syncwarp();
    }
    for (int i = ln; i < NEQ; i += 32) tm.at(ob, tm.perm(i)) = tm.at(AOFF_TMP, i);
  }
  tsync();
}
__device__ __forceinline__ void adj_solve_T(int ob) { lu_solve_T(ob); }
#endif

// VJP at the state in slot oy (double) with weights at AOFF_V; gy added to yb scaled by the
// coefficients of up to three destinations: dst[0] += c0 gy, ...
template <class S>
__device__ __forceinline__ void set_vjp_state(const Team& tm, int oy, int odir) {
  S* sb = reinterpret_cast<S*>(&tm.base[AOFF_S]);
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    S v;
    if constexpr (S_is_dual<S>::value) v = mk(tm.at(oy, i), tm.at(odir, i));
    else v = tm.at(oy, i);
    sb[VS_Y + i] = v;
  }
  tsync();
}

__device__ __forceinline__ void add_gy(const Team& tm, bool dual, int o1, double c1, int o2, double c2, int o3, double c3) {
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    double g;
    if (dual) g = reinterpret_cast<const DD*>(&tm.base[AOFF_S])[VS_GY + i].d;
    else g = reinterpret_cast<const double*>(&tm.base[AOFF_S])[VS_GY + i];
    if (o1 >= 0) tm.at(o1, i) += c1 * g;
    if (o2 >= 0) tm.at(o2, i) += c2 * g;
    if (o3 >= 0) tm.at(o3, i) += c3 * g;
  }
  tsync();
}

// Adjoint of one frozen-h ROS4 step y_n -> y_{n+1}: on entry OFF_Y = y_n and AOFF_LAM =
// dL/dy_{n+1}; on exit AOFF_LAM = dL/dy_n, and dL/dlnA accumulated in AOFF_GP.
// Forward: M = I/(gamma h) - J(y), u_i = M^-1 r_i, r_1 = f(y), r_2 = f(Y2) + c21/h u1,
// r_3 = f(Y3) + (c31 u1 + c32 u2)/h, r_4 = f(Y3) + (c41 u1 + c42 u2 + c43 u3)/h,
// Y2 = y + a21 u1, Y3 = y + a31 u1 + a32 u2, y_{n+1} = y + sum m_i u_i.
// Reverse: ubar_i = m_i lambda, w_i = M^-T ubar_i (taken in the order 4, 3, 2, 1 as each ubar_i
// becomes final), fbar pulls back through J(Y)^T and d f / d lnA (VJP), and M's dependence on
// J(y) adds sum_i d/dy [w_i^T J(y) u_i] and d/dlnA [w_i^T J(y) u_i] (dual-number VJPs at y along
// u_i with weights w_i).
__device__ void adjoint_step(const Team& tm, double P, double h, const double* lnA_ext) {
  const int U1 = OFF_U1, U2 = OFF_U2, U3 = OFF_U3, U4 = OFF_U4;
  const int W1 = AOFF_W, W2 = AOFF_W + NEQ, W3 = AOFF_W + 2 * NEQ, W4 = AOFF_W + 3 * NEQ;
  const int B1 = AOFF_UB, B2 = AOFF_UB + NEQ, B3 = AOFF_UB + 2 * NEQ, B4 = AOFF_UB + 3 * NEQ;
  const double ih = fx_rcp(h);
  // ---- forward recompute
  eval_f_jac<-1>(OFF_Y, U1, P, lnA_ext, fx_rcp(RGAM * h));
  lu_factor();
#if SOLVE_BLK
  lu_invert();
#endif
  stage_solve<false>(U1);
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    const double v = tm.at(OFF_Y, i) + RA21 * tm.at(U1, i);
    tm.at(OFF_YT, i) = v;
    tm.at(AOFF_Y2, i) = v;
  }
  tsync();
  eval_f(OFF_YT, OFF_F, P, lnA_ext);
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(U2, i) = tm.at(OFF_F, i) + (RC21 * ih) * tm.at(U1, i);
  tsync();
  stage_solve<false>(U2);
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    const double v = tm.at(OFF_Y, i) + RA31 * tm.at(U1, i) + RA32 * tm.at(U2, i);
    tm.at(OFF_YT, i) = v;
    tm.at(AOFF_Y3, i) = v;
  }
  tsync();
  eval_f(OFF_YT, OFF_F, P, lnA_ext);
  for (int i = tm.tl; i < NEQ; i += TEAM)
    tm.at(U3, i) = tm.at(OFF_F, i) + (RC31 * ih) * tm.at(U1, i) + (RC32 * ih) * tm.at(U2, i);
  tsync();
  stage_solve<false>(U3);
  for (int i = tm.tl; i < NEQ; i += TEAM)
    tm.at(U4, i) = tm.at(OFF_F, i) + (RC41 * ih) * tm.at(U1, i) + (RC42 * ih) * tm.at(U2, i) +
                   (RC43 * ih) * tm.at(U3, i);
  tsync();
  stage_solve<false>(U4);
  // ---- reverse
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    const double l = tm.at(AOFF_LAM, i);
    tm.at(AOFF_YB, i) = l;
    tm.at(B1, i) = RM1 * l;
    tm.at(B2, i) = RM2 * l;
    tm.at(B3, i) = RM3 * l;
    tm.at(B4, i) = RM4 * l;
  }
  tsync();
  // stage 4
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(W4, i) = tm.at(B4, i);
  tsync();
  adj_solve_T(W4);
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    const double w = tm.at(W4, i);
    tm.at(AOFF_FB, i) = w;
    tm.at(B1, i) += (RC41 * ih) * w;
    tm.at(B2, i) += (RC42 * ih) * w;
    tm.at(B3, i) += (RC43 * ih) * w;
  }
  tsync();
  // stage 3
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(W3, i) = tm.at(B3, i);
  tsync();
  adj_solve_T(W3);
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    const double w = tm.at(W3, i);
    tm.at(AOFF_FB, i) += w;
    tm.at(AOFF_V, i) = tm.at(AOFF_FB, i);
    tm.at(B1, i) += (RC31 * ih) * w;
    tm.at(B2, i) += (RC32 * ih) * w;
  }
  tsync();
  set_vjp_state<double>(tm, AOFF_Y3, AOFF_Y3);
  vjp<double>(P, lnA_ext);
  add_gy(tm, false, AOFF_YB, 1.0, B1, RA31, B2, RA32);
  // stage 2
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(W2, i) = tm.at(B2, i);
  tsync();
  adj_solve_T(W2);
  for (int i = tm.tl; i < NEQ; i += TEAM) {
    const double w = tm.at(W2, i);
    tm.at(AOFF_V, i) = w;
    tm.at(B1, i) += (RC21 * ih) * w;
  }
  tsync();
  set_vjp_state<double>(tm, AOFF_Y2, AOFF_Y2);
  vjp<double>(P, lnA_ext);
  add_gy(tm, false, AOFF_YB, 1.0, B1, RA21, -1, 0.0);
  // stage 1
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(W1, i) = tm.at(B1, i);
  tsync();
  adj_solve_T(W1);
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(AOFF_V, i) = tm.at(W1, i);
  tsync();
  set_vjp_state<double>(tm, OFF_Y, OFF_Y);
  vjp<double>(P, lnA_ext);
  add_gy(tm, false, AOFF_YB, 1.0, -1, 0.0, -1, 0.0);
  // M = I/(gamma h) - J(y): second-order terms along each u_i with weights w_i
  for (int st = 0; st < 4; ++st) {
    for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(AOFF_V, i) = tm.at(AOFF_W + st * NEQ, i);
    tsync();
    set_vjp_state<DD>(tm, OFF_Y, UOFF(st));
    vjp<DD>(P, lnA_ext);
    add_gy(tm, true, AOFF_YB, 1.0, -1, 0.0, -1, 0.0);
  }
  for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(AOFF_LAM, i) = tm.at(AOFF_YB, i);
  tsync();
}

// Scratch of chem_adjoint_noalloc (the adjoint for callers that cannot allocate device memory):
// a fixed array in this module, CHEM_ADJ_SCRATCH_BYTES long, shared by every call on this
// module; the host resolves its device address once per loaded module.
static __device__ __align__(256) double chem_adj_scratch[CHEM_ADJ_SCRATCH_BYTES / 8];

__device__ __forceinline__ long long team_global_id() {
  return (long long)blockIdx.x * NTEAM + (TEAM == 32 ? (threadIdx.x >> 5) : 0);
}

// Reverse sweep over every cell's checkpointed forward: per cell, segments of `interval`
// accepted steps are recomputed from their checkpoint (states kept in this team's slice of
// `seg`), then stepped through backwards.  dL/dlnA is accumulated per team and written to
// gp_partial[team][r]; chem_adjoint_reduce_k sums the teams in a fixed order.
// (one block per SM as the register bound: the adjoint's shared memory already limits residency
// to four 64-lane or one 256-lane team per SM, so the registers go to avoiding spills)
extern "C" __global__ void __launch_bounds__(TPB, 1)
chem_adjoint_k(long long n_cells, const double* __restrict__ P, const double* __restrict__ gT,
               const double* __restrict__ gY, long long ld, double* __restrict__ gT0,
               double* __restrict__ gY0, const double* __restrict__ lnA_ext,
               const int* __restrict__ tape_nacc, const double* __restrict__ tape_h,
               const double* __restrict__ tape_ck, int interval, double* __restrict__ seg,
               double* __restrict__ gp_partial, unsigned long long* queue) {
  const Team tm = make_team();
  const long long tg = team_global_id();
  for (int r = tm.tl; r < NR; r += TEAM) tm.at(AOFF_GP, r) = 0.0;
  tsync();
  double* segc = seg + tg * (long long)interval * NEQ;
  for (;;) {
    long long nc = 0;
    if (tm.tl == 0) nc = (long long)atomicAdd(queue, 1ULL);
    const long long cell = team_bcast_ll(tm, nc);
    if (cell >= n_cells) break;
    const int nacc = tape_nacc[cell];
    const double Pc = P[cell];
    const double gb = gY[(long long)BATH * ld + cell];
    if (tm.tl == 0) tm.at(AOFF_LAM, 0) = gT[cell];
    for (int k = tm.tl; k < NS - 1; k += TEAM) tm.at(AOFF_LAM, 1 + k) = mk_W[k] * (gY[k * ld + cell] - gb);
    tsync();
    for (int sg = (nacc - 1) / interval; nacc > 0 && sg >= 0; --sg) {
      const int s0 = sg * interval;
      const int s1 = min(nacc, s0 + interval);
      for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(OFF_Y, i) = tape_ck[((long long)sg * NEQ + i) * n_cells + cell];
      tsync();
      for (int s = s0; s < s1; ++s) {
        for (int i = tm.tl; i < NEQ; i += TEAM) segc[(s - s0) * NEQ + i] = tm.at(OFF_Y, i);
        if (s + 1 < s1) {
          ros4_attempt<false>(tm, Pc, tape_h[(long long)s * n_cells + cell], 1.0, 1.0, lnA_ext);
          for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(OFF_Y, i) = tm.at(OFF_YT, i);
        }
        tsync();
      }
      for (int s = s1 - 1; s >= s0; --s) {
        for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(OFF_Y, i) = segc[(s - s0) * NEQ + i];
        tsync();
        adjoint_step(tm, Pc, tape_h[(long long)s * n_cells + cell], lnA_ext);
      }
    }
    // initial state y0 = [T0, Y0_k / W_k]; the bath mass fraction does not enter y0
    if (tm.tl == 0) {
      gT0[cell] = tm.at(AOFF_LAM, 0);
      gY0[(long long)BATH * ld + cell] = 0.0;
    }
    for (int k = tm.tl; k < NS - 1; k += TEAM) gY0[k * ld + cell] = tm.at(AOFF_LAM, 1 + k) * mk_invW[k];
    tsync();
  }
  for (int r = tm.tl; r < NR; r += TEAM) gp_partial[tg * NR + r] = tm.at(AOFF_GP, r);
}

extern "C" __global__ void chem_adjoint_reduce_k(long long n_parts, const double* __restrict__ gp_partial,
                                                 double* __restrict__ g_lnA) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= NR) return;
  double s = 0.0;
  for (long long t = 0; t < n_parts; ++t) s += gp_partial[t * NR + r];
  g_lnA[mk_rorig[r]] = s;  // mechanism order
}

// Vector-Jacobian products per cell (parity entry point of the adjoint's building block):
// gy = J(y)^T v  [NEQ x ld], gp = (d f / d lnA)^T v  [NR x ld].
extern "C" __global__ void __launch_bounds__(TPB)
chem_eval_vjp_k(long long n_cells, const double* __restrict__ T, const double* __restrict__ P,
                const double* __restrict__ n, const double* __restrict__ v, double* __restrict__ gy,
                double* __restrict__ gp, long long ld, const double* __restrict__ lnA_ext) {
  const Team tm = make_team();
  const long long stride = (long long)gridDim.x * NTEAM;
  for (long long c = team_global_id(); c < n_cells; c += stride) {
    if (tm.tl == 0) tm.at(OFF_Y, 0) = T[c];
    for (int k = tm.tl; k < NS - 1; k += TEAM) tm.at(OFF_Y, 1 + k) = n[k * ld + c];
    for (int i = tm.tl; i < NEQ; i += TEAM) tm.at(AOFF_V, i) = v[i * ld + c];
    for (int r = tm.tl; r < NR; r += TEAM) tm.at(AOFF_GP, r) = 0.0;
    tsync();
    set_vjp_state<double>(tm, OFF_Y, OFF_Y);
    vjp<double>(P[c], lnA_ext);
    const double* g = reinterpret_cast<const double*>(&tm.base[AOFF_S]) + VS_GY;
    for (int i = tm.tl; i < NEQ; i += TEAM) gy[i * ld + c] = g[i];
    for (int r = tm.tl; r < NR; r += TEAM) gp[(long long)mk_rorig[r] * ld + c] = tm.at(AOFF_GP, r);
    tsync();
  }
}

#endif  // TEAM >= 32 && CHEM_ADJOINT

extern "C" __device__ const int chem_aslots =
#if TEAM >= 32 && defined(CHEM_ADJOINT) && TABLEAU_ID == 0
    ASLOTS;
#else
    0;
#endif
