// k_lqr.cu -- the reduced unconstrained LQR (Sec. 6) and the recovery maps
// (eq. recovery-maps) on sm_103a.
//
// Riccati factors.  The paper obtains log depth from an associative LQR scan
// [ref-AS-LQR].  Here the scan elements are conditional costs V(z_a | z_b) of
// a chunk kept in square-root form, as "cost relations": constraint rows that
// hold exactly (states z_b reachable from z_a) and least-squares cost rows on
// (z_a, z_b).  Composition eliminates the shared state by equality-constrained
// least squares (wlse_elim: orthogonal and pivoted), so value functions whose
// Hessians grow without bound through stretches without control authority
// turn into constraints instead of cancelling.  Chunks compose their own
// stages, a log-depth scan over chunks gives V at every chunk boundary, and
// each chunk then runs the Riccati recursion inward in 114-bit integers, storing P_i,
// K_i, the Cholesky factor of Rbar + Bbar'P Bbar and Phi_i = Abar + Bbar K_i.
//
// Linear passes.  With those factors the remaining recursions are affine
// chains: p_i = Phi_i' (P_{i+1} c_i + p_{i+1}) + q_i + K_i' r_i backwards and
// z_{i+1} = Phi_i z_i + Bbar k_i + c_i forwards.  They run as chunked affine
// scans (k_aff_*), also used for the refinement passes on the reduced KKT
// residual and for the forward costate expansion of Sec. 7.
#include <algorithm>

#include "fx.cuh"
#include "kernels.cuh"

namespace eclqr {

__host__ int smem_lqr_up(int n, int m) {
  const int ldr = 2 * n + 1, rows = 5 * n + m, ldm = m + 2 * n + 1;
  return 2 * (2 * n) * ldr + rows * ldm + 2 * rows + 2 * (ldm + rows) + m + 16;
}
__host__ int smem_lqr_level(int n) {
  const int rows = 8 * n, ldm = 3 * n + 1;
  return rows * ldm + 2 * rows + 2 * (ldm + rows) + n + 16;
}
__host__ int smem_riccati_finish(int n, int m) { return std::max(m * (n + m + 1) + m * (n + 1) + m + 8, n * n); }
__host__ int smem_aff(int n, int m) { return 2 * (n * n + n) + n * n + 5 * n + 2 * m + 8; }
constexpr int kAffRing = 6;  // stages of k_aff_down on their way to shared memory
constexpr int kAffY = 32;    // its vectors, with room for whole segments
__host__ int smem_aff_down(int n) { return kAffRing * n * (n + 1) + 2 * kAffY + 2; }

// Cost-relation slot layout (ld 2n + 1): constraint rows at 0 (CI_ROWS of them),
// cost rows at offset 2n (2n + 1) (CI_ROWS2 of them); CI_NA / CI_NB are the
// endpoint dimensions, CI_NB = 0 marks a value function (unary, cost only).
__device__ __forceinline__ double *crel_cost(double *slot, int n) { return slot + 2 * n * (2 * n + 1); }

// ----------------------------------------------------------- chunk conditional costs
// Up-sweep over stages b-1 .. a of the conditional cost V(z_i | z_b): a cost
// relation on (z_i, z_b).  Stage i substitutes the reduced dynamics
// z_{i+1} = Abar z_i + Bbar v + cbar into the rows on (z_{i+1}, z_b), stacks the
// stage cost rows L'[z; v] + l and eliminates v (wlse_elim).
__global__ void k_lqr_up(Group g, int per_task) {
  const int t = team_task();
  if (t >= g.nslot) return;
  const ChunkInfo ci = g.chunk[t];
  const ProbInfo &P = g.prob[ci.prob];
  if (skipped_by_mask(g, ci.prob)) return;
  const int n = g.n, m = g.m, tid = team_rank();
  const int ldr = 2 * n + 1;
  double *slot = g.CS[0] + (size_t)t * g.cs_stride;
  int *cm = g.CI[0] + (size_t)t * CI_STRIDE;
  double *sm = team_smem(per_task);
  if (P.nch == 1 && (ci.c == 0 || g.fp64 == nullptr)) {
    // one chunk: k_riccati_down starts from the terminal cost itself (the FP32 sweep from its
    // square root, below), k_riccati_finish tests it
    if (tid == 0) { cm[CI_ROWS] = 0; cm[CI_NA] = 0; cm[CI_NB] = 0; cm[CI_ROWS2] = 0; }
    return;
  }
  if (ci.c == P.nch) {
    // terminal value: rows [L' | L^{-1} qbar_N], L L' = Qbar_N (eq. terminal-cost-data)
    const int sN = P.st0 + P.N;
    const double *ws = stage_ws(g, sN);
    const int nN = stage_wi(g, sN)[SI_NBAR];
    double *Hh = sm;  // bordered by qbar_N
    for (int idx = tid; idx < (nN + 1) * nN; idx += TEAM) {
      int a = idx / nN, j = idx - a * nN;
      Hh[idx] = a < nN ? ws[g.ws.Qb + a * n + j] : ws[g.ws.qb + j];
    }
    tsync();
    const int fail = wchol(Hh, nN, nN, true);
    double *cost = crel_cost(slot, n);
    for (int idx = tid; idx < nN * (nN + 1); idx += TEAM) {
      int a = idx / (nN + 1), j = idx - a * (nN + 1);
      cost[a * ldr + j] = j == nN ? Hh[nN * nN + a] : (j >= a ? Hh[j * nN + a] : 0.0);
    }
    if (tid == 0) {
      cm[CI_ROWS] = 0; cm[CI_NA] = nN; cm[CI_NB] = 0; cm[CI_ROWS2] = nN;
      if (fail) set_status(g, ci.prob, ST_NONCONVEX);
    }
    return;
  }
  const int a = ci.c * P.L, b = min(a + P.L, P.N);
  const int nbz = stage_wi(g, P.st0 + b)[SI_NBAR];
  const int rows_max = 5 * n + m, ldm_max = m + 2 * n + 1;
  double *Cons = sm, *Cost = Cons + 2 * n * ldr, *M = Cost + 2 * n * ldr, *scr = M + rows_max * ldm_max;
  // z_b' = z_b on (z_b', z_b)
  for (int idx = tid; idx < nbz * ldr; idx += TEAM) {
    int i = idx / ldr, j = idx - i * ldr;
    Cons[idx] = (j == i) ? 1.0 : ((j == nbz + i) ? -1.0 : 0.0);
  }
  tsync();
  int rc = nbz, rq = 0;
  int fail = 0;
  for (int i = b - 1; i >= a; --i) {
    const int s = P.st0 + i;
    const double *ws = stage_ws(g, s);
    const int *wi = stage_wi(g, s);
    const int nx = wi[SI_NBAR], mu = wi[SI_MBAR], n1 = stage_wi(g, s + 1)[SI_NBAR];
    const int ldm = mu + nx + nbz + 1, kh = nx + mu;
    const double *Ab = ws + g.ws.Ab, *Bb = ws + g.ws.Bb, *cb = ws + g.ws.cb, *LT = ws + g.ws.LT, *lt = ws + g.ws.lt;
    // columns v (mu) | z_i (nx) | z_b (nbz) | 1
    // rows: constraints (rc) then stage cost (kh) then old cost (rq)
    const int rtot = rc + kh + rq;
    for (int idx = tid; idx < rtot * ldm; idx += TEAM) {
      int r = idx / ldm, j = idx - r * ldm;
      double val = 0.0;
      if (r < rc || r >= rc + kh) {
        const double *row = (r < rc) ? Cons + r * ldr : Cost + (r - rc - kh) * ldr;  // [K1 (n1) | Kb (nbz) | k]
        if (j < mu) {
          for (int l = 0; l < n1; l++) val = fma(row[l], Bb[l * m + j], val);
        } else if (j < mu + nx) {
          for (int l = 0; l < n1; l++) val = fma(row[l], Ab[l * n + (j - mu)], val);
        } else if (j < mu + nx + nbz) {
          val = row[n1 + (j - mu - nx)];
        } else {
          val = row[n1 + nbz];
          for (int l = 0; l < n1; l++) val = fma(row[l], cb[l], val);
        }
      } else {
        const int q = r - rc;  // stage cost row q of L' (columns v then z, as here)
        if (j < mu + nx) val = LT[q * (n + m) + j];
        else if (j == ldm - 1) val = lt[q];
      }
      M[idx] = val;
    }
    tsync();
    LseResult lr = wlse_elim(M, ldm, rc, kh + rq, mu, nx + nbz, g.tau_rank, g.tau_inc, Cons, Cost, ldr, scr);
    rc = lr.kc;
    rq = lr.kq;
    fail |= lr.inconsistent;
  }
  for (int idx = tid; idx < rc * ldr; idx += TEAM) slot[idx] = Cons[idx];
  double *cost = crel_cost(slot, n);
  for (int idx = tid; idx < rq * ldr; idx += TEAM) cost[idx] = Cost[idx];
  if (tid == 0) {
    cm[CI_ROWS] = rc; cm[CI_NA] = stage_wi(g, P.st0 + a)[SI_NBAR]; cm[CI_NB] = nbz; cm[CI_ROWS2] = rq;
    if (fail) set_status(g, ci.prob, ST_NONCONVEX);
  }
}

// One level of the chunk suffix scan on cost relations: slot t <- slot t o slot t + d,
// eliminating the shared state (wlse_elim); a value on the right gives a value.
__global__ void k_lqr_level(Group g, int src, int d, int per_task) {
  const int t = team_task();
  if (t >= g.nslot) return;
  const ChunkInfo ci = g.chunk[t];
  const ProbInfo &P = g.prob[ci.prob];
  if (skipped_by_mask(g, ci.prob)) return;
  const int n = g.n, tid = team_rank(), ldr = 2 * n + 1;
  double *S1 = g.CS[src] + (size_t)t * g.cs_stride;
  const int *I1 = g.CI[src] + (size_t)t * CI_STRIDE;
  double *Dst = g.CS[src ^ 1] + (size_t)t * g.cs_stride;
  int *J = g.CI[src ^ 1] + (size_t)t * CI_STRIDE;
  const int rc1 = I1[CI_ROWS], na = I1[CI_NA], nm = I1[CI_NB], rq1 = I1[CI_ROWS2];
  if (ci.c + d > P.nch || nm == 0) {
    for (int idx = tid; idx < rc1 * ldr; idx += TEAM) Dst[idx] = S1[idx];
    for (int idx = tid; idx < rq1 * ldr; idx += TEAM) crel_cost(Dst, n)[idx] = crel_cost(S1, n)[idx];
    if (tid == 0) { J[CI_ROWS] = rc1; J[CI_NA] = na; J[CI_NB] = nm; J[CI_ROWS2] = rq1; }
    return;
  }
  double *S2 = g.CS[src] + (size_t)(t + d) * g.cs_stride;
  const int *I2 = g.CI[src] + (size_t)(t + d) * CI_STRIDE;
  const int rc2 = I2[CI_ROWS], nb = I2[CI_NB], rq2 = I2[CI_ROWS2];
  double *sm = team_smem(per_task);
  const int ldm = nm + na + nb + 1;
  const int rc = rc1 + rc2, rq = rq1 + rq2;
  double *M = sm, *scr = sm + (rc + rq) * ldm;
  // columns z_m | z_a | z_b | 1 ; rows: constraints of e1, e2, then costs of e1, e2
  for (int idx = tid; idx < (rc + rq) * ldm; idx += TEAM) {
    int r = idx / ldm, j = idx - r * ldm;
    bool left;
    const double *row;
    if (r < rc1) { left = true; row = S1 + r * ldr; }
    else if (r < rc) { left = false; row = S2 + (r - rc1) * ldr; }
    else if (r < rc + rq1) { left = true; row = crel_cost(S1, n) + (r - rc) * ldr; }
    else { left = false; row = crel_cost(S2, n) + (r - rc - rq1) * ldr; }
    double val = 0.0;
    if (left) {          // [z_a (na) | z_m (nm) | 1]
      if (j < nm) val = row[na + j];
      else if (j < nm + na) val = row[j - nm];
      else if (j == ldm - 1) val = row[na + nm];
    } else {             // [z_m (nm) | z_b (nb) | 1]
      if (j < nm) val = row[j];
      else if (j >= nm + na && j < nm + na + nb) val = row[nm + (j - nm - na)];
      else if (j == ldm - 1) val = row[nm + nb];
    }
    M[idx] = val;
  }
  tsync();
  LseResult lr = wlse_elim(M, ldm, rc, rq, nm, na + nb, g.tau_rank, g.tau_inc, Dst, crel_cost(Dst, n), ldr, scr);
  if (tid == 0) {
    J[CI_ROWS] = lr.kc; J[CI_NA] = na; J[CI_NB] = nb; J[CI_ROWS2] = lr.kq;
    if (lr.inconsistent) set_status(g, ci.prob, ST_NONCONVEX);
  }
}

// ----------------------------------------------------------- chunk down-sweep: Riccati
// From V_b(z) = 1/2 z'P z + p'z at the chunk end (P = C'C from the scan's cost rows, or the
// terminal cost itself), each stage forms the Hessian and gradient of cost plus value over (v, z),
//   G = H + [Bbar Abar]' P [Bbar Abar],  g = h + [Bbar Abar]' (P cbar + p),
// eliminates v by pivots on G's diagonal, and keeps P_i, p_i, the Schur complement on z.  The
// pivot rows divided by the root of their pivot are the minimiser's rows (R_vv | R_vz | o_v)
// that k_riccati_finish turns into K, k, chol(H_uu) and Phi.
//
// In FP64 this recursion loses the curvature that |P| |Abar|^2 cancels down to; carried as
// square-root rows through a Householder QR it keeps it, at n + m dependent steps per stage, each a
// reduction, a reciprocal square root and an update at 64 cycles per dependent FP64 instruction.
// Here the recursion runs in the 114-bit integers of fx.cuh.  A condition number of P up to 2^110
// is what a square root resolves in 55 bits, so the accuracy is that of the square-root form or
// better, and the work is two products with independent outputs and m short pivot steps.  Column
// exponents come from the diagonal, so entries are at most 1 in magnitude by Cauchy-Schwarz and
// the scaling of states and controls does not matter.
//
// Both hold only while the matrices stay positive semidefinite, and curvature below about 2^-106 of
// |P| |A|^2 in a direction that is no coordinate axis is rounding noise: without more, a direction
// of negative curvature gets gains of any size and the recursion grows without bound (a stretch of
// 25 stages without control that grow by 4 each: gains of 1e18 and values past the limbs' 118 bits).
// So every diagonal entry is raised by riccati_margin, more than the rounding that can make it
// indefinite, after each product and each Schur complement, and a pivot below it counts as
// noise.  Directions beyond the resolution then keep a small positive curvature, as the square
// root's rows do by their form, and the recursion forgets them as it should.  n^2 2^-106 of |P| |A|^2 is
// also the size of a square root's own rounding.
//
// What bounds it: where many problems share an SM, the fixed latency of its integer chains and the
// barriers between a stage's phases (n = 24, 14 warps an SM: 40% of the issue slots, of 46k warp
// instructions a stage 7k limb products); where few do, the latency of one stage's phases.
// Loops are kept rolled: with them unrolled the code outgrew the instruction cache and 1280
// problems of 64 stages at n = 24 took 12.8 ms instead of 8.0.  Against the FP64 QR, 64 stages of
// 1280 problems: n = 24 20.3 -> 7.8 ms, n = 16 10.2 -> 4.1, n = 8 3.38 -> 1.93; of 160 problems at
// n = 24 7.5 -> 2.9 ms (k_riccati_finish, which no longer forms P = R'R, 2.24 -> 1.0 at 1280, n = 24).
// Then pivots by one warp, the minimiser's rows in one pass, H a stage ahead, single-entry tiles and
// wider teams for few sweeps: 256 problems of 256 stages at n = 16 6.36 -> 3.45 ms, 160 problems at
// n = 32 6.15 -> 3.31, one sweep of 64 stages at n = 4 0.42 -> 0.32.
// The blocks are offsets into the task's shared memory (in elements of their type), so that every
// access compiles to a shared-memory instruction with a 32-bit address.
struct RiccatiFx {
  int oP, oW, oG, oA, oH, oI, oV, ldp, ldx;
  __host__ __device__ static int words(int n, int m) {  // 8-byte words
    const int ldx = n + m + 1, big = n > m ? n : m;
    return 2 * (n * (n + 1) + big * ldx + g_size(n, m)) + n * ldx + g_size(n, m) + (3 * ldx + m + 2) / 2 + 4;
  }
  // entries of G's and H's packed rows
  __host__ __device__ static int g_size(int n, int m) { return (n + m) * (n + m + 1) / 2 + n + m; }
  __device__ RiccatiFx(int n, int m) {
    ldp = n + 1;
    ldx = n + m + 1;
    oP = 0;
    oW = n * (n + 1);
    oG = oW + (n > m ? n : m) * ldx;
    oA = 2 * (oG + g_size(n, m));
    oH = oA + n * ldx;
    oI = 2 * (oH + g_size(n, m));
    oV = oH + g_size(n, m) + (3 * ldx + m + 2) / 2;
  }
  __device__ int4 &P(int i) const { return ((int4 *)g_smem)[oP + i]; }  // [P | p] (ld n + 1)
  __device__ int4 &W(int i) const { return ((int4 *)g_smem)[oW + i]; }  // P [Bbar Abar cbar]; the pivots' multipliers
  __device__ int4 &G(int i) const { return ((int4 *)g_smem)[oG + i]; }  // G, g: packed rows, limbs or 128-bit integers
  __device__ i128 &Gi(int i) const { return ((i128 *)g_smem)[oG + i]; }
  __device__ int2 &A(int i) const { return ((int2 *)g_smem)[oA + i]; }  // [Bbar | Abar | cbar] (n x ldx)
  __device__ double &Ad(int i) const { return g_smem[oA + i]; }         // the same as doubles
  __device__ double &H(int i) const { return g_smem[oH + i]; }          // [Rbar Mbar'; Mbar Qbar | rbar; qbar], packed
  // column exponents of A (rows weighted by P's), of G, and of P (eP(nx): that of p); the pivots'
  // shifts; a flag: a value that is not finite was met
  __device__ int &al(int i) const { return ((int *)g_smem)[oI + i]; }
  __device__ int &e(int i) const { return ((int *)g_smem)[oI + ldx + i]; }
  __device__ int &eP(int i) const { return ((int *)g_smem)[oI + 2 * ldx + i]; }
  __device__ int &hp(int i) const { return ((int *)g_smem)[oI + 3 * ldx + 1 + i]; }
  // the current pivot's reciprocal, its residual and the offsets' excess bits
  __device__ long long &piv(int i) const { return ((long long *)g_smem)[oV + i]; }
  __device__ int &bad() const { return ((int *)g_smem)[oI + 3 * ldx]; }
};
// the blocks of RiccatiFx, or the FP32 sweep's (V, stacked rows, two vectors, gains and stage
// data, in floats)
__host__ int smem_riccati(int n, int m) {
  const int rows = 2 * n + m, ld = n + m + 1;
  const int f32 = n * (n + 1) + rows * ld + rows + ld + m * (n + 1) + n * (n + m + 1);
  return (std::max(RiccatiFx::words(n, m), (f32 + 1) / 2) + 9) & ~1;
}

__device__ __forceinline__ void copy_async(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void copy_async16(double *dst, const double *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int K>  // at most the K newest groups are still in flight
__device__ __forceinline__ void copy_wait_ring() { asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory"); }
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void team_sync() {
  if (blockDim.x == 32) __syncwarp();
  else __syncthreads();
}

// What a diagonal entry is raised by, in units of 2^-114 of its scale: the rounding of W (up to four units
// an entry after its scaling by 8) and of P's limbs (at most one) through n1 terms, as the norm of a matrix of kh
// rows.  Of 615 recursions at n = 2 to 16 through stretches near and beyond the resolution 355 grew without
// bound with no margin, 28 with a quarter of this one, none with half of it or all; where a square-root
// QR in FP64 still has digits of the gains, the error here is half to two thirds of its error.
__device__ __forceinline__ int riccati_margin(int n1, int kh) { return (n1 * kh >> 1) + 32; }

// (j, k), j <= k < ld, of packed upper rows
__device__ __forceinline__ int riccati_packed(int ld, int j, int k) { return j * ld - j * (j + 1) / 2 + k; }

// P and p from raw sums: the block of G from row z0 on, nz states and the offset column, with
// entry exponents e(z0 + a) + e(z0 + b) (p: e(z0 + a) + e(z0 + nz)).  Brings every diagonal entry to [2^112, 2^114),
// sets w.P and w.eP, and writes P and p in FP64 where they are given.
static __device__ __noinline__ void riccati_value(const RiccatiFx w, int nz, int z0, double *Po, int ldo, double *po) {
  const int ld = z0 + nz + 1;
  auto raw = [&](int a, int b) { return riccati_packed(ld, z0 + a, z0 + b); };
  const int tid = team_rank(), lane = tid & 31;
  if (tid < 32) {
    int pb = 0;
    const int a = lane;
    if (a < nz) {
      const i128 d = w.Gi(raw(a, a));
      // noise can leave an entry whose diagonal is not positive: its scale stays
      const int s = d > 0 ? min((kFxP - fx_bits(d)) >> 1, 52) : 0;
      w.eP(a) = w.e(z0 + a) - s;
      const i128 v = w.Gi(raw(a, nz));
      pb = v != 0 ? fx_bits(v) + s : 0;
    }
    pb = __reduce_max_sync(kFull, pb);
    if (lane == 0) w.eP(nz) = w.e(z0 + nz) + (pb ? pb - kFxP : 0);
  }
  team_sync();
  const bool bad = w.bad() != 0;
  const int items = nz * (nz + 1) / 2 + nz;
  auto store = [&](int a, int b, i128 v) {
    int s;
    const long long top = fx_lead(v, s);
    const double x = bad ? __longlong_as_double(0x7ff8000000000000ll) : fx_to(top, s + w.e(z0 + a) + w.e(z0 + b) - kFxP);
    if (b < nz) {
      Po[a * ldo + b] = x;
      Po[b * ldo + a] = x;
    } else {
      po[a] = x;
    }
  };
  // the FP64 values, which the sweep itself does not wait for, from the team's other end where its
  // last warps have no entry of their own
  const bool apart = 2 * items <= TEAM;
  int a = 0, row = 0;  // row: linear index of (a, a); nz + 1 - a entries per row
#pragma unroll 1
  for (int idx = tid; idx < items; idx += TEAM) {
    while (idx - row > nz - a) row += nz + 1 - a++;
    const int b = a + idx - row;
    const i128 v = w.Gi(raw(a, b));
    const int4 l = fx_split4(fx_shift(v, w.e(z0 + a) + w.e(z0 + b) - w.eP(a) - w.eP(b)));
    w.P(a * w.ldp + b) = l;
    if (b < nz) w.P(b * w.ldp + a) = l;
    if (Po && !apart) store(a, b, v);
  }
  if (Po && apart) {
    const int idx = TEAM - 1 - tid;
    if (idx < items) {
      a = row = 0;
      while (idx - row > nz - a) row += nz + 1 - a++;
      store(a, a + idx - row, w.Gi(raw(a, a + idx - row)));
    }
  }
  team_sync();
}

// Starts the copy of a stage's [Bbar | Abar | cbar] (n1 rows) into w.Ad.
static __device__ __forceinline__ void riccati_fetch(const Group &g, const RiccatiFx w, const double *ws, int n1, int nx,
                                                     int mu) {
  const int kh = nx + mu, ld = kh + 1;
  const double *Ab = ws + g.ws.Ab, *Bb = ws + g.ws.Bb, *cb = ws + g.ws.cb;
  const float rld = rcp_seed((float)ld);
#pragma unroll 1
  for (int idx = team_rank(); idx < n1 * ld; idx += TEAM) {
    const int l = (int)(((float)idx + 0.5f) * rld), j = idx - l * ld;
    copy_async(&w.Ad(l * w.ldx + j), j < mu ? Bb + l * g.m + j : (j < kh ? Ab + l * g.n + (j - mu) : cb + l));
  }
}

// Starts the copy of a stage's H and h in the order (v, z, 1), packed rows, into w.H: the lower triangles
// of Rbar and Qbar, those that k_elim's Cholesky found positive definite (the upper ones differ by rounding,
// and where a Hessian is singular to rounding that is the sign of its smallest eigenvalue).
static __device__ __forceinline__ void riccati_fetch_h(const Group &g, const RiccatiFx w, const double *ws, int nx, int mu) {
  const int n = g.n, m = g.m, kh = nx + mu, ld = kh + 1;
  const double *Qb = ws + g.ws.Qb, *Mb = ws + g.ws.Mb, *Rb = ws + g.ws.Rb, *qb = ws + g.ws.qb, *rb = ws + g.ws.rb;
  int j = 0, row = 0;
#pragma unroll 1
  for (int idx = team_rank(); idx < kh * (kh + 1) / 2 + kh; idx += TEAM) {
    while (idx - row >= ld - j) row += ld - j++;
    const int k = j + idx - row;
    const double *src;
    if (k == kh) src = j < mu ? rb + j : qb + (j - mu);
    else if (k < mu) src = Rb + k * m + j;
    else src = j < mu ? Mb + (k - mu) * m + j : Qb + (k - mu) * n + (j - mu);
    copy_async(&w.H(idx), src);
  }
}

// W = P [Bbar | Abar | cbar] + [0 | 0 | p] in units of 2^-111: T x T entries per item
template <int T>
static __device__ __forceinline__ void riccati_w(const RiccatiFx w, int n1, int kh) {
  const int ld = kh + 1, ldx = w.ldx, ldp = w.ldp, cols = (ld + T - 1) / T;
  const float rcols = rcp_seed((float)cols);
#pragma unroll 1
  for (int it = team_rank(); it < cols * ((n1 + T - 1) / T); it += TEAM) {
    const int rp = (int)(((float)it + 0.5f) * rcols), c = T * (it - rp * cols), r = T * rp;
    const int r1 = min(r + T - 1, n1 - 1), c1 = min(c + T - 1, kh);
    FxAcc acc[T * T];
#pragma unroll
    for (int q = 0; q < T * T; q++) acc[q].zero();
    int i0 = r * ldp, i1 = r1 * ldp, j0 = c, j1 = c1;
#pragma unroll 2
    for (int l = 0; l < n1; l++, i0++, i1++, j0 += ldx, j1 += ldx) {
      const int4 x0 = w.P(i0);
      const int2 a0 = w.A(j0);
      acc[0].mad(x0, a0);
      if (T == 2) {
        const int4 x1 = w.P(i1);
        const int2 a1 = w.A(j1);
        acc[1 % (T * T)].mad(x0, a1);
        acc[2 % (T * T)].mad(x1, a0);
        acc[3 % (T * T)].mad(x1, a1);
      }
    }
#pragma unroll
    for (int q = 0; q < T * T; q++) {
      const int rr = q < T ? r : r1, cc = T == 2 && (q & 1) ? c1 : c;
      i128 v = acc[q].template value<60>();
      if (cc == kh) v += fx_shift(fx_join4(w.P(rr * ldp + n1)), w.eP(n1) - w.al(kh) - 3);
      w.W(rr * ldx + cc) = fx_split4(v);
    }
  }
}

// raw G = [Bbar Abar]' W in units of 2^-114: T x T entries (j, k), j <= k, per item
template <int T>
static __device__ __forceinline__ void riccati_g(const RiccatiFx w, int n1, int kh) {
  const int ld = kh + 1, ldx = w.ldx, cols = (ld + T - 1) / T;
  int jt = 0, start = 0;  // block row jt: block columns jt .. cols - 1
#pragma unroll 1
  for (int it = team_rank();; it += TEAM) {
    while (T * jt < kh && it - start >= cols - jt) start += cols - jt++;
    if (T * jt >= kh) break;
    const int j = T * jt, j1 = min(j + T - 1, kh - 1), k = j + T * (it - start), k1 = min(k + T - 1, kh);
    FxAcc acc[T * T];
#pragma unroll
    for (int q = 0; q < T * T; q++) acc[q].zero();
    int ia = j, ib = j1, ka = k, kb = k1;
#pragma unroll 2
    for (int l = 0; l < n1; l++, ia += ldx, ib += ldx, ka += ldx, kb += ldx) {
      const int4 x0 = w.W(ka);
      const int2 a0 = w.A(ia);
      acc[0].mad(x0, a0);
      if (T == 2) {
        const int4 x1 = w.W(kb);
        const int2 a1 = w.A(ib);
        acc[1 % (T * T)].mad(x1, a0);
        acc[2 % (T * T)].mad(x0, a1);
        acc[3 % (T * T)].mad(x1, a1);
      }
    }
#pragma unroll
    for (int q = 0; q < T * T; q++) {
      const int jj = q < T ? j : j1, kk = T == 2 && (q & 1) ? k1 : k;
      if (jj <= kk) w.Gi(riccati_packed(ld, jj, kk)) = acc[q].template value<54>() + (jj == kk ? riccati_margin(n1, kh) : 0);
    }
  }
}

// One stage: from w.P, w.eP (n1 states) and the fetched w.Ad and w.H to the value of the stage's nx
// states.  Rv: the minimiser's rows (ld n + m + 1); Po, po: P_i and p_i; null where the stage is not
// stored.  fetch() and fetch_h() start the copies of the next stage's w.Ad and w.H.
template <typename Fetch, typename FetchH>
static __device__ __forceinline__ void riccati_stage(const Group &g, const RiccatiFx w, int n1, int nx, int mu,
                                                     double *Rv, double *Po, double *po, Fetch fetch, FetchH fetch_h) {
  const int n = g.n, m = g.m, tid = team_rank();
  const int kh = nx + mu, ld = kh + 1, ldx = w.ldx;
  auto packed = [&](int j, int k) { return riccati_packed(ld, j, k); };
  // [Bbar | Abar | cbar] and its column exponents, the rows weighted by P's exponents
#pragma unroll 1
  for (int j = tid; j < ld; j += TEAM) w.al(j) = j == kh ? w.eP(n1) : kFxNone;
  copy_wait();
  team_sync();
  const float rld = rcp_seed((float)ld);
#pragma unroll 1
  for (int idx = tid; idx < n1 * ld; idx += TEAM) {
    const int l = (int)(((float)idx + 0.5f) * rld), j = idx - l * ld;
    const double x = w.Ad(l * ldx + j);
    const int ex = fx_expo(x);
    if (ex != kFxNone) atomicMax(&w.al(j), ex + w.eP(l));
    if (fx_nonfinite(x)) w.bad() = 1;
  }
  team_sync();
#pragma unroll 1
  for (int idx = tid; idx < n1 * ld; idx += TEAM) {
    const int l = (int)(((float)idx + 0.5f) * rld), j = idx - l * ld;
    w.A(l * ldx + j) = fx_split(fx_from(w.Ad(l * ldx + j), w.al(j) - w.eP(l)));
  }
  team_sync();
  // The tiles: 2 x 2 entries per item share their operands, single entries spread over four times the
  // lanes.  Single entries while the team takes them in one pass and a half: with many sweeps per
  // SM, whose teams are small, they only add shared-memory loads (640 problems at n = 16, four
  // warps: 2.7 ms with 2 x 2 tiles, 3.2 with single entries in G alone); with few, the lanes idle
  // otherwise (one 64-stage sweep at n = 4 410 -> 353 us, 147 chunks at n = 12 178 -> 137).
  if (2 * n1 * ld > 3 * TEAM) riccati_w<2>(w, n1, kh);
  else riccati_w<1>(w, n1, kh);
  team_sync();
  if (kh * (kh + 1) + 2 * kh > 3 * TEAM) riccati_g<2>(w, n1, kh);
  else riccati_g<1>(w, n1, kh);
  team_sync();
  fetch();
  // exponents of the columns of G + H from its diagonal, of the offsets from their largest entry
  if (tid < 32) {
    int to = kFxNone;
#pragma unroll 1
    for (int j = tid; j < kh; j += 32) {
      const int jj = packed(j, j), jo = packed(j, kh);
      const i128 d = w.Gi(jj), o = w.Gi(jo);
      const int t = max(d != 0 ? fx_bits(d) - kFxP + 2 * w.al(j) : kFxNone, fx_expo(w.H(jj)));
      const int e = t > kFxNone / 2 ? (t + 2) >> 1 : 0;
      w.e(j) = e;
      to = max(to, (o != 0 ? fx_bits(o) - kFxP + w.al(j) + w.al(kh) : kFxNone) - e);
      to = max(to, fx_expo(w.H(jo)) - e);
    }
    to = __reduce_max_sync(kFull, to);
    if (tid == 0) w.e(kh) = to > kFxNone / 2 ? to + 1 : 0;
  }
  team_sync();
  {
    int j = 0, row = 0;
#pragma unroll 1
    for (int idx = tid; idx < kh * (kh + 1) / 2 + kh; idx += TEAM) {
      while (idx - row >= ld - j) row += ld - j++;
      const int k = j + idx - row;
      const double h = w.H(idx);
      if (fx_nonfinite(h)) w.bad() = 1;
      const int ejk = w.e(j) + w.e(k);
      const i128 v = fx_shift(w.Gi(idx), w.al(j) + w.al(k) - ejk) + fx_from4(h, ejk);
      // the z block stays whole integers, which the last product is subtracted from
      if (j < mu) w.G(idx) = fx_split4(v);
      else w.Gi(idx) = v;
    }
  }
  team_sync();
  fetch_h();
  // pivots on v: y_j = G_kj 2^h, l_j = y_j / (d 2^(2h)) (units of 2^-112, in
  // w.W), G_ij -= l_i y_j for rows i < mu
#pragma unroll 1
  for (int k = 0; k < mu; k++) {
    const int gk = packed(k, 0);
    if (tid < 32) {  // one long chain of scalars: the other warps wait for it instead of repeating it
      i128 d = fx_join4(w.G(gk + k));
      const bool noise = d <= riccati_margin(n1, kh);
      if (noise) d = (i128)1 << (kFxP - 53);  // rounding noise of a singular pivot
      const int h = (kFxP - fx_bits(d)) >> 1;
      const i128 dp = d << (2 * h);
      const unsigned long long g0 = (unsigned long long)fx_rcp((unsigned long long)(dp >> 50));
      // 2^114 - (dp g0 >> 55), below 2^63: the low 64 bits are all of it
      const unsigned long long lo = (unsigned long long)dp, t = (__umul64hi(lo, g0) << 9) | ((lo * g0) >> 55);
      // the offsets' column has no bound by the diagonal: where the shift would pass 2^114, its
      // exponent is raised first.  Then y / sqrt(d 2^(2h)) of the offsets is at most 2^58 for each pivot,
      // and a later row, whose y / sqrt(d 2^(2h)) over the pivots have squares that sum to its diagonal,
      // at most 2^114, collects at most sqrt(15) 2^115: below the limbs' 2^118.  (From 2^116 it could pass them.)
      const int over = fx_bits(fx_join4(w.G(gk + kh))) + h - kFxP;
      if (tid == 0) {
        if (noise) w.G(gk + k) = fx_split4(d);
        w.hp(k) = h;
        w.piv(0) = (long long)g0;
        w.piv(1) = (long long)(0ull - (((unsigned long long)(dp >> 64) * g0) << 9) - t);
        w.piv(2) = over;
      }
    }
    team_sync();
    const int h = w.hp(k), over = (int)w.piv(2);
    const int2 g2 = fx_split(w.piv(0));
    const long long r = w.piv(1);
    if (over > 0) {
#pragma unroll 1
      for (int i = tid; i < kh; i += TEAM) {
        const int x = packed(i, kh);
        if (i < mu) w.G(x) = fx_split4(fx_shift(fx_join4(w.G(x)), -over));
        else w.Gi(x) = fx_shift(w.Gi(x), -over);
      }
      if (tid == 0) w.e(kh) += over;
      team_sync();
    }
    FxAcc acc;
#pragma unroll 1
    for (int j = k + tid; j < ld; j += TEAM) {
      const i128 y = fx_join4(w.G(gk + j)) << h;
      const int4 y4 = fx_split4(y);
      w.G(gk + j) = y4;
      acc.zero();
      acc.mad(y4, g2);
      const i128 t = acc.value<57>();
      // the offsets' (j = kh) can wrap: their multiplier has no reader
      w.W(k * ldx + j) = fx_split4(t + __mul64hi((long long)((unsigned long long)(t >> 57) << 6), r << 1));
    }
    team_sync();
    // rows k + 1 .. mu - 1
    int i = k + 1, row = 0;
#pragma unroll 1
    for (int idx = tid;; idx += TEAM) {
      while (i < mu && idx - row >= ld - i) row += ld - i++;
      if (i >= mu) break;
      const int j = i + idx - row;
      FxAcc4 a4;
      a4.zero();
      a4.mad(w.W(k * ldx + i), w.G(gk + j));
      const int x = packed(i, j);
      w.G(x) = fx_split4(fx_join4(w.G(x)) - a4.value());
    }
    team_sync();
  }
  // Schur complement on z
  {
    int a = 0, row = 0;
#pragma unroll 1
    for (int idx = tid; idx < nx * (nx + 1) / 2 + nx; idx += TEAM) {
      while (idx - row > nx - a) row += nx + 1 - a++;
      const int b = a + idx - row;
      FxAcc4 acc;
      acc.zero();
#pragma unroll 1
      for (int k = 0; k < mu; k++) acc.mad(w.W(k * ldx + mu + a), w.G(packed(k, mu + b)));
      w.Gi(packed(mu + a, mu + b)) -= acc.value() - (a == b ? riccati_margin(n1, kh) : 0);
    }
  }
  // the minimiser's rows y_j / sqrt(d 2^(2h))
  const bool bad = w.bad() != 0;
  if (Rv) {
    // every row at once, from the packed rows 0 .. mu - 1, from the team's other end: its last warps
    // have fewer entries of the Schur complement, or none
    int k = 0, row = 0;
#pragma unroll 1
    for (int idx = TEAM - 1 - tid; idx < packed(mu, mu); idx += TEAM) {
      while (idx - row >= ld - k) row += ld - k++;
      const int j = k + idx - row;
      const unsigned long long rs = fx_rsqrt((unsigned long long)((fx_join4(w.G(row)) << w.hp(k)) >> 50));
      int s;
      const long long top = fx_lead(fx_join4(w.G(idx)), s);
      // (4 d)^(-1/2) 2^62, so the value is 2 2^(s - 114 + 2) of the product's upper half
      const double x = fx_to(__mul64hi(top, (long long)rs), s + 3 - kFxP + w.e(j));
      Rv[k * (n + m + 1) + j] = bad ? __longlong_as_double(0x7ff8000000000000ll) : x;
    }
  }
  team_sync();
  riccati_value(w, nx, mu, Po, n, po);
}

static __device__ void riccati_task(const Group &g, int fin, int t, int per_task);
__global__ void k_riccati_down(Group g, int fin, int per_task, int *queue) {
  for_tasks(g.nslot, queue, [&](int t) { riccati_task(g, fin, t, per_task); });
}

static __device__ void riccati_task(const Group &g, int fin, int t, int per_task) {
  if (t >= g.nslot) return;
  const ChunkInfo ci = g.chunk[t];
  const ProbInfo &P = g.prob[ci.prob];
  if (skipped_by_mask(g, ci.prob)) return;
  if (g.fp64 != nullptr && g.fp64[P.id] == 0) return;  // mixed precision: k_riccati_down_f32 sweeps it
  if (ci.c >= P.nch) return;
  const int n = g.n, tid = team_rank();
  const int a = ci.c * P.L, b = min(a + P.L, P.N);
  // every chunk but the last re-sweeps the next chunk's stages from the same scan value, so that the
  // value function it starts from is, bit for bit, the one the next chunk computes at their boundary
  const bool resweep = ci.c + 1 < P.nch;
  const int start = resweep ? min(b + P.L, P.N) : b;
  const RiccatiFx w(n, g.m);
  // V_b
  if (tid == 0) w.bad() = 0;
  if (start == P.N) {  // the terminal cost
    double *ws = stage_ws(g, P.st0 + P.N);
    const double *Qb = ws + g.ws.Qb, *qb = ws + g.ws.qb;
    const int nz = stage_wi(g, P.st0 + P.N)[SI_NBAR];
#pragma unroll 1
    for (int j = tid; j < nz; j += TEAM) {
      const int t2 = fx_expo(Qb[j * n + j]);
      w.e(j) = t2 > kFxNone / 2 ? (t2 + 1) >> 1 : 0;
    }
    __syncthreads();
    if (tid < 32) {
      int mx = tid < nz ? fx_expo(qb[tid]) - w.e(tid) : kFxNone;
      mx = __reduce_max_sync(kFull, mx);
      if (tid == 0) w.e(nz) = mx > kFxNone / 2 ? mx : 0;
    }
    __syncthreads();
#pragma unroll 1
    for (int idx = tid; idx < nz * (nz + 1); idx += TEAM) {
      const int j = idx / (nz + 1), k = idx - j * (nz + 1);
      if (k < j) continue;
      const double x = k < nz ? Qb[k * n + j] : qb[j];  // the triangle that the convexity test reads
      if (fx_nonfinite(x)) w.bad() = 1;
      w.Gi(riccati_packed(nz + 1, j, k)) = fx_from4(x, w.e(j) + w.e(k));
    }
    __syncthreads();
    riccati_value(w, nz, 0, b == P.N ? ws + g.ws.P : nullptr, n,
                  ws + g.ws.p);
  } else {  // P = C'C, p = C'c from the scan's cost rows, scaled by column and (at most 0, in al) by row
    const int slot = t + 2, ldr = 2 * n + 1;
    const double *src = crel_cost(g.CS[fin] + (size_t)slot * g.cs_stride, n);
    const int nz = g.CI[fin][(size_t)slot * CI_STRIDE + CI_NA], rv = g.CI[fin][(size_t)slot * CI_STRIDE + CI_ROWS2];
#pragma unroll 1
    for (int j = tid; j <= nz; j += TEAM) {
      int mx = kFxNone;
#pragma unroll 1
      for (int r = 0; r < rv; r++) mx = max(mx, fx_expo(src[r * ldr + j]));
      w.e(j) = mx > kFxNone / 2 ? mx : 0;
    }
    __syncthreads();
#pragma unroll 1
    for (int r = tid; r < rv; r += TEAM) {
      int mx = kFxNone;
#pragma unroll 1
      for (int j = 0; j <= nz; j++) mx = max(mx, fx_expo(src[r * ldr + j]) - w.e(j));
      w.al(r) = mx > kFxNone / 2 ? mx : 0;
#pragma unroll 1
      for (int j = 0; j <= nz; j++) {
        w.A(r * w.ldx + j) = fx_split(fx_from(src[r * ldr + j], w.al(r) + w.e(j)));
        if (fx_nonfinite(src[r * ldr + j])) w.bad() = 1;
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int idx = tid; idx < nz * (nz + 1); idx += TEAM) {
      const int j = idx / (nz + 1), k = idx - j * (nz + 1);
      if (k < j) continue;
      i128 s = j == k ? rv * nz : 0;  // the rounding of rv shifted terms, as a matrix norm
#pragma unroll 1
      for (int r = 0; r < rv; r++) {
        const int2 x = w.A(r * w.ldx + j), y = w.A(r * w.ldx + k);
        const i128 v = ((i128)fx_mad(x.x, y.x, 0) << (2 * kFxB)) + ((i128)fx_mad(x.x, y.y, fx_mad(x.y, y.x, 0)) << kFxB) +
                       fx_mad(x.y, y.y, 0);
        s += fx_shift(v, 2 * w.al(r));
      }
      w.Gi(riccati_packed(nz + 1, j, k)) = s;
    }
    __syncthreads();
    riccati_value(w, nz, 0, nullptr, n, nullptr);
  }
  int n1 = stage_wi(g, P.st0 + start)[SI_NBAR], nx = 0, mu = 0;
  if (start > a) {
    const int s = P.st0 + start - 1;
    nx = stage_wi(g, s)[SI_NBAR];
    mu = stage_wi(g, s)[SI_MBAR];
    riccati_fetch(g, w, stage_ws(g, s), n1, nx, mu);
    riccati_fetch_h(g, w, stage_ws(g, s), nx, mu);
  }
#pragma unroll 1
  for (int i = start - 1; i >= a; --i) {
    const bool store = i < b;  // the next chunk's stages are stored by that chunk
    const int s = P.st0 + i;
    double *ws = stage_ws(g, s);
    int nx2 = 0, mu2 = 0;
    if (i > a) {
      nx2 = stage_wi(g, s - 1)[SI_NBAR];
      mu2 = stage_wi(g, s - 1)[SI_MBAR];
    }
    riccati_stage(g, w, n1, nx, mu, store ? ws + g.ws.Rv : nullptr, store ? ws + g.ws.P : nullptr, ws + g.ws.p,
                  [&] {
                    if (i > a) riccati_fetch(g, w, stage_ws(g, s - 1), nx, nx2, mu2);
                  },
                  [&] {
                    if (i > a) riccati_fetch_h(g, w, stage_ws(g, s - 1), nx2, mu2);
                  });
    n1 = nx;
    nx = nx2;
    mu = mu2;
  }
}

// ----------------------------------------------------------- Riccati factors, every stage at once
// For each stage i < N that the sweep stored (FP64 sweeps only): from the
// minimiser's rows, R_vv [K | k] = -[R_vz | o_v] by back substitution, the
// Cholesky factor of H_uu = R_vv'R_vv (R_vv' with rows signed to a positive
// diagonal) and Phi = Abar + Bbar K (the closed-loop map of the affine chains).
__global__ void k_riccati_finish(Group g, int per_task) {
  for_stages(g, [&](const int s) {
    const StageInfo S = g.st[s];
    const ProbInfo &P = g.prob[S.prob];
    if (skipped_by_mask(g, S.prob)) return;
    const int n = g.n, m = g.m, tid = team_rank();
    double *ws = stage_ws(g, s);
    const int *wi = stage_wi(g, s);
    if (S.i >= P.N) {
      // one chunk: the terminal cost has to be convex (otherwise tested by k_lqr_up)
      if (P.nch > 1 || g.fp64 != nullptr) return;
      const int nN = wi[SI_NBAR];
      double *Hh = team_smem(per_task);
      for (int idx = tid; idx < nN * nN; idx += TEAM) Hh[idx] = ws[g.ws.Qb + idx / nN * n + idx % nN];
      tsync();
      if (wchol(Hh, nN, nN, false) && tid == 0) set_status(g, S.prob, ST_NONCONVEX);
      return;
    }
    if (g.fp64 != nullptr && g.fp64[P.id] == 0) return;  // k_riccati_down_f32 stored this problem's factors
    const int nx = wi[SI_NBAR], mu = wi[SI_MBAR], n1 = stage_wi(g, s + 1)[SI_NBAR];
    const int ldr = n + m + 1;
    double *sm = team_smem(per_task);
    double *R = sm, *Kt = R + m * ldr;
    const double *Rv = ws + g.ws.Rv, *Ab = ws + g.ws.Ab, *Bb = ws + g.ws.Bb;
    for (int idx = tid; idx < mu * (nx + mu + 1); idx += TEAM) {
      int r = idx / (nx + mu + 1), j = idx - r * (nx + mu + 1);
      R[r * ldr + j] = Rv[r * ldr + j];
    }
    tsync();
    // K, k:  R_vv [K | k] = -[R_vz | o_v]; the diagonal's reciprocals up front
    double *inv = Kt + m * (n + 1);
    for (int r = tid; r < mu; r += TEAM) inv[r] = 1.0 / R[r * ldr + r];
    tsync();
    for (int c = tid; c <= nx; c += TEAM) {
      for (int r = mu - 1; r >= 0; r--) {
        double s0 = -R[r * ldr + mu + c];
        for (int l = r + 1; l < mu; l++) s0 = fma(-R[r * ldr + l], Kt[l * (n + 1) + c], s0);
        Kt[r * (n + 1) + c] = s0 * inv[r];
      }
    }
    for (int idx = tid; idx < mu * mu; idx += TEAM) {
      int r = idx / mu, j = idx - r * mu;
      double sg = R[j * ldr + j] >= 0.0 ? 1.0 : -1.0;
      ws[g.ws.Lh + r * m + j] = (j <= r) ? sg * R[j * ldr + r] : 0.0;
    }
    tsync();
    for (int idx = tid; idx < mu * (nx + 1); idx += TEAM) {
      int r = idx / (nx + 1), c = idx - r * (nx + 1);
      if (c < nx) ws[g.ws.K + r * n + c] = Kt[r * (n + 1) + c]; else ws[g.ws.k + r] = Kt[r * (n + 1) + c];
    }
    for (int idx = tid; idx < n1 * nx; idx += TEAM) {
      int r = idx / nx, c = idx - r * nx;
      double s0 = Ab[r * n + c];
      for (int l = 0; l < mu; l++) s0 = fma(Bb[r * m + l], Kt[l * (n + 1) + c], s0);
      ws[g.ws.Phi + r * n + c] = s0;
    }
  });
}

// ----------------------------------------------------------- affine chain scans
// Per-stage maps by mode (d_i = dimension of the chained vector at stage i):
//   AFF_ROLL  forward  z_{i+1} = Phi_i z_i + Bbar k_i + cbar_i        -> z
//   AFF_CROLL forward  dz_{i+1} = Phi_i dz_i + Bbar k'_i + rc_i       -> dz (k' held in dv)
//   AFF_PLIN  backward p'_i = Phi_i' p'_{i+1} + rq_i + K_i' rr_i + Phi_i' P_{i+1} rc_i, the
//             refinement's linear pass for the offsets (rq, rr, rc)                  -> pp
//   AFF_NU    forward  nu_{i+1} = Pnu_i nu_i + pnu_i                  -> nu
enum { AFF_ROLL = 0, AFF_CROLL = 1, AFF_PLIN = 2, AFF_NU = 3 };

__device__ __forceinline__ int aff_dim(const Group &g, int s, int mode) {
  return (mode == AFF_NU) ? stage_wi(g, s)[SI_UR] : stage_wi(g, s)[SI_NBAR];
}
__device__ __forceinline__ bool aff_forward(int mode) { return mode != AFF_PLIN; }
__device__ __forceinline__ int aff_out(const Group &g, int mode) {
  return mode == AFF_ROLL ? g.ws.z : mode == AFF_CROLL ? g.ws.dz : mode == AFF_PLIN ? g.ws.pp : g.ws.nu;
}

// map of stage i: y_out = G y_in + gv.  Forward: in = stage i, out = stage i+1;
// backward: in = stage i+1, out = stage i.  G (dout x din, ld n) and gv into smem.
__device__ void aff_stage_map(const Group &g, int s, int mode, double *G, double *gv) {
  const int n = g.n, tid = team_rank();
  const double *ws = stage_ws(g, s), *src = ws + (mode == AFF_NU ? g.ws.Pnu : g.ws.Phi), *v = src + n * n;
  const int d0 = aff_dim(g, s, mode), d1 = aff_dim(g, s + 1, mode), dout = mode == AFF_PLIN ? d0 : d1;
  for (int idx = tid; idx < d1 * d0; idx += TEAM) {
    const int i = idx / d0, j = idx - i * d0;
    G[mode == AFF_PLIN ? j * n + i : i * n + j] = src[i * n + j];
  }
  for (int i = tid; i < dout; i += TEAM) gv[i] = v[i];
  tsync();
}

// The offsets cbar + Bbar k of every stage's map, stage-parallel, before the rollout's chain sweeps
// them (ws.gv).  k_resid and k_pcorr form those of PLIN and CROLL; NU reads pnu.
__global__ void k_aff_prep(Group g) {
  for_stages(g, [&](const int s) {
    const StageInfo S = g.st[s];
    const ProbInfo &P = g.prob[S.prob];
    if (skipped_by_mask(g, S.prob)) return;
    if (S.i >= P.N) return;
    const int m = g.m, ny = stage_wi(g, s + 1)[SI_NBAR], mu = stage_wi(g, s)[SI_MBAR];
    double *ws = stage_ws(g, s);
    const double *Bb = ws + g.ws.Bb, *kk = ws + g.ws.k, *cc = ws + g.ws.cb;
    for (int i = team_rank(); i < ny; i += TEAM) {
      double s0 = cc[i];
      for (int l = 0; l < mu; l++) s0 = fma(Bb[i * m + l], kk[l], s0);
      ws[g.ws.gv + i] = s0;
    }
  });
}

// What the chunk aggregates' kernels have to do besides aggregates: the boundary value's slot (forward:
// slot 0 of the problem holds y_0, backward: slot nch holds y_N), and an empty map where one chunk
// needs none.  Returns whether that was the task.
static __device__ bool aff_up_ends(const Group &g, const ChunkInfo ci, const ProbInfo &P, int mode, bool fwd) {
  const int n = g.n, tid = team_rank();
  if (ci.c == P.nch) {
    const int s = fwd ? P.st0 : P.st0 + P.N;
    const int slot = fwd ? P.ch0 : P.ch0 + P.nch;
    const int dim = aff_dim(g, s, mode);
    double *gv = g.CS[0] + (size_t)slot * g.cs_stride + n * n;
    const double *src = stage_ws(g, s);
    for (int i = tid; i < dim; i += TEAM) {
      double v;
      if (mode == AFF_ROLL) v = src[g.ws.z + i];
      else if (mode == AFF_CROLL) v = 0.0;
      else if (mode == AFF_PLIN) v = src[g.ws.rq + i];  // p'_N = rq_N
      else v = src[g.ws.nu + i];
      gv[i] = v;
    }
    if (tid == 0) {
      int *cm = g.CI[0] + (size_t)slot * CI_STRIDE;
      cm[CI_ROWS] = 1; cm[CI_NA] = dim; cm[CI_NB] = 0;
    }
    return true;
  }
  if (P.nch > 1) return false;
  // one chunk: k_aff_down starts from the boundary value, so the chunk's map is not
  // composed; an empty map (no rows, no dimensions) ends the level at once
  if (tid == 0) {
    int *cm = g.CI[0] + (size_t)(fwd ? P.ch0 + ci.c + 1 : P.ch0 + ci.c) * CI_STRIDE;
    cm[CI_ROWS] = 0; cm[CI_NA] = 0; cm[CI_NB] = 0;
  }
  return true;
}

// chunk aggregates
__global__ void k_aff_up(Group g, int mode, int per_task) {
  const int t = team_task();
  if (t >= g.nslot) return;
  const ChunkInfo ci = g.chunk[t];
  const ProbInfo &P = g.prob[ci.prob];
  if (skipped_by_mask(g, ci.prob)) return;
  const int n = g.n, tid = team_rank();
  const bool fwd = aff_forward(mode);
  if (aff_up_ends(g, ci, P, mode, fwd)) return;
  const int slot = fwd ? P.ch0 + ci.c + 1 : P.ch0 + ci.c;
  const int a = ci.c * P.L, b = min(a + P.L, P.N);
  double *sm = team_smem(per_task);
  double *Gm = sm, *gm = Gm + n * n, *Gs = gm + n, *gs = Gs + n * n, *Tm = gs + n, *tmp = Tm + n * n;
  const int d0 = fwd ? aff_dim(g, P.st0 + a, mode) : aff_dim(g, P.st0 + b, mode);
  for (int idx = tid; idx < n * n; idx += TEAM) {
    int i = idx / n, j = idx - i * n;
    Gm[idx] = (i == j) ? 1.0 : 0.0;
  }
  for (int i = tid; i < n; i += TEAM) gm[i] = 0.0;
  tsync();
  int dcur = d0;  // rows of the aggregate (current output dimension)
  for (int k = 0; k < b - a; k++) {
    const int i = fwd ? a + k : b - 1 - k;
    const int s = P.st0 + i;
    aff_stage_map(g, s, mode, Gs, gs);
    const int dout = fwd ? aff_dim(g, s + 1, mode) : aff_dim(g, s, mode);
    // Tm = Gs Gm (dout x d0), tmp = Gs gm + gs
    wgemm<false, false>(dout, d0, dcur, Gs, n, Gm, n, 0, Tm, n);
    for (int r = tid; r < dout; r += TEAM) {
      double s0 = gs[r];
      for (int l = 0; l < dcur; l++) s0 = fma(Gs[r * n + l], gm[l], s0);
      tmp[r] = s0;
    }
    tsync();
    for (int idx = tid; idx < dout * d0; idx += TEAM) {
      int r = idx / d0, j = idx - r * d0;
      Gm[r * n + j] = Tm[r * n + j];
    }
    for (int r = tid; r < dout; r += TEAM) gm[r] = tmp[r];
    tsync();
    dcur = dout;
  }
  double *cs = g.CS[0] + (size_t)slot * g.cs_stride;
  for (int idx = tid; idx < n * n; idx += TEAM) cs[idx] = Gm[idx];
  if (mode == AFF_ROLL)
    for (int idx = tid; idx < n * n; idx += TEAM) g.CR[(size_t)t * g.cr_stride + idx] = Gm[idx];
  for (int i = tid; i < n; i += TEAM) cs[n * n + i] = gm[i];
  if (tid == 0) {
    int *cm = g.CI[0] + (size_t)slot * CI_STRIDE;
    cm[CI_ROWS] = 0; cm[CI_NA] = d0; cm[CI_NB] = dcur;
  }
}

// One level of a radix-4 Kogge-Stone scan over the chunk slots of an affine
// chain.  Before the level with stride d every slot holds the composition of
// the d slots ending at it; it composes that with the slots at distances d,
// 2d and 3d in the scan direction (each holding the d slots before the
// previous one), so after the levels d = 1, 4, 16, ... every slot holds its
// inclusive prefix.  A value (a boundary vector, CI_ROWS == 1) ends the
// composition.  The four-way level halves the launches of a radix-2 scan;
// the chain elements are small (n x n), so the level is launch-bound.
__global__ void k_aff_level(Group g, int src, int d, int fwd, int per_task) {
  const int t = team_task();
  if (t >= g.nslot) return;
  const ChunkInfo ci = g.chunk[t];
  const ProbInfo &P = g.prob[ci.prob];
  if (skipped_by_mask(g, ci.prob)) return;
  const int n = g.n, tid = team_rank(), sz = n * n + n;
  const int j = t - P.ch0;  // slot index 0..nch
  const double *S0 = g.CS[src] + (size_t)t * g.cs_stride;
  const int *I1 = g.CI[src] + (size_t)t * CI_STRIDE;
  double *Dst = g.CS[src ^ 1] + (size_t)t * g.cs_stride;
  int *J = g.CI[src ^ 1] + (size_t)t * CI_STRIDE;
  int rows = I1[CI_ROWS], na = I1[CI_NA], nb = I1[CI_NB];
  double *sm = team_smem(per_task);
  double *acc = sm, *oth = acc + sz, *Tm = oth + sz, *tv = Tm + n * n;
  for (int idx = tid; idx < sz; idx += TEAM) acc[idx] = S0[idx];
  tsync();
  for (int q = 1; q <= 3 && rows != 1; q++) {
    const int j2 = fwd ? j - q * d : j + q * d;
    if (j2 < 0 || j2 > P.nch) break;
    const int t2 = P.ch0 + j2;
    const double *S2 = g.CS[src] + (size_t)t2 * g.cs_stride;
    const int *I2 = g.CI[src] + (size_t)t2 * CI_STRIDE;
    const int rows2 = I2[CI_ROWS], na2 = I2[CI_NA];
    for (int idx = tid; idx < sz; idx += TEAM) oth[idx] = S2[idx];
    tsync();
    if (rows2 == 1) {
      // value: y = G v + g, dimension nb
      for (int r = tid; r < nb; r += TEAM) {
        double s0 = acc[n * n + r];
        for (int l = 0; l < na2; l++) s0 = fma(acc[r * n + l], oth[n * n + l], s0);
        tv[r] = s0;
      }
      tsync();
      for (int r = tid; r < nb; r += TEAM) acc[n * n + r] = tv[r];
      rows = 1;
      na = nb;
      nb = 0;
    } else {
      // (G G2, G g2 + g): input dimension na2, output nb
      wgemm<false, false>(nb, na2, na, acc, n, oth, n, 0, Tm, n);
      for (int r = tid; r < nb; r += TEAM) {
        double s0 = acc[n * n + r];
        for (int l = 0; l < na; l++) s0 = fma(acc[r * n + l], oth[n * n + l], s0);
        tv[r] = s0;
      }
      tsync();
      for (int idx = tid; idx < nb * na2; idx += TEAM) {
        const int r = idx / na2, c = idx - r * na2;
        acc[r * n + c] = Tm[r * n + c];
      }
      for (int r = tid; r < nb; r += TEAM) acc[n * n + r] = tv[r];
      rows = 0;
      na = na2;
    }
    tsync();
  }
  for (int idx = tid; idx < sz; idx += TEAM) Dst[idx] = acc[idx];
  if (tid == 0) { J[CI_ROWS] = rows; J[CI_NA] = na; J[CI_NB] = nb; }
}

// The chain of one chunk: y_out = G_i y_in + gv_i stage after stage, G_i = Phi_i
// (ROLL, CROLL), Phi_i' (PLIN, backward) or Pnu_i (NU), gv_i from k_aff_prep, k_resid and k_pcorr
// (pnu for NU).
//
// What bounds it: the latency of one stage.  Of that only the FP64 chain of a row (n / SEG
// multiply-adds and log2(SEG) shuffled additions of 64 cycles each) and the exchange of y are
// needed; a warp issues in order, so everything else has to leave its way.  The last warp of the CTA
// does it: it copies the blocks [G | gv] asynchronously kAffRing stages ahead into shared memory,
// stores y and looks up the dimensions.  The others hold a row over SEG lanes, read the coming
// stage's entries into registers while the FP64 instructions run, and meet it at one barrier per
// stage.  Per stage, 256 problems of 256 stages at n = 16 and 64 stages at n = 4: 0.40 and 0.32 us; 0.70
// and 0.72 with the next stage's entries read one stage ahead by the same warps, 0.63 and 0.57 with
// the ring alone.
template <int SEG, int KP>
static __device__ __forceinline__ void aff_rows(const double *ring, double *ya, double *yb, const int *sdim, int n, bool tr,
                                                int steps, int dcur) {
  const int blk = n * (n + 1), q = threadIdx.x & (SEG - 1), row = threadIdx.x / SEG;
  const int g0 = tr ? q * n + row : row * n + q, gs = tr ? SEG * n : SEG;
  double gr[KP], gv = 0.0;
  bool on = false;
  // this lane's entries of block G, din x dout (zero outside)
  auto load = [&](const double *G, int din, int dout) {
    on = row < dout;
    const double *e = G + g0;
#pragma unroll
    for (int j = 0; j < KP; j++, e += gs) gr[j] = on && q + j * SEG < din ? *e : 0.0;
    gv = on && q == 0 ? G[n * n + row] : 0.0;
  };
  __syncthreads();
  int dout = sdim[0], slot = 0;
  load(ring, dcur, dout);
  const double *G = ring;
  for (int k = 0; k < steps; k++) {
    double acc = gv;
#pragma unroll
    for (int j = 0; j < KP; j++)
      if (j * SEG < n) acc = fma(gr[j], ya[q + j * SEG], acc);
    const bool was = on;
    G += blk;
    if (++slot == kAffRing) {
      slot = 0;
      G = ring;
    }
    const int d1 = sdim[(k + 1) & 3];
    load(G, dout, d1);
    dout = d1;
#pragma unroll
    for (int s = SEG >> 1; s > 0; s >>= 1) acc += __shfl_xor_sync(kFull, acc, s);
    if (q == 0 && row < n) yb[row] = was ? acc : 0.0;
    double *t = ya; ya = yb; yb = t;
    __syncthreads();
  }
}

// The last warp of the CTA.  end: where the chain's last value goes, instead of the stages' values.
static __device__ __forceinline__ void aff_helper(const Group &g, const ProbInfo &P, int mode, int a, int b, double *ring,
                                                  double *ya, double *yb, int *sdim, double *end) {
  const int n = g.n, lane = threadIdx.x & 31, blk = n * (n + 1), steps = b - a;
  const bool fwd = aff_forward(mode);
  const int first = P.st0 + (fwd ? a : b - 1), dir = fwd ? 1 : -1;
  const ptrdiff_t step = (ptrdiff_t)dir * g.ws.stride;
  const double *src = stage_ws(g, first) + (mode == AFF_NU ? g.ws.Pnu : g.ws.Phi) + 2 * lane;
  // y_k belongs to stage a + k forwards, b - k backwards; stage b is the next chunk's unless it is the last
  double *o = stage_ws(g, P.st0 + (fwd ? a : b)) + aff_out(g, mode) + lane;
  int sent = 0;
  auto fetch = [&](int slot) {
    if (sent < steps) {
      double *dst = ring + slot * blk + 2 * lane;
#pragma unroll 4
      for (int i = 2 * lane; i < blk; i += 64, dst += 64) copy_async16(dst, src + (i - 2 * lane));
      src += step;
      sent++;
    }
    copy_commit();
  };
#pragma unroll
  for (int k = 0; k < kAffRing; k++) fetch(k);
  // output dimensions of the stages k0 .. k0 + 31, one per lane, and of the 32 after them
  auto dims = [&](int k0) {
    const int k = k0 + lane;
    return k < steps ? aff_dim(g, first + dir * k + (fwd ? 1 : 0), mode) : 0;
  };
  int dreg = dims(0), dnext = dims(32);
  if (lane < 2) sdim[lane] = dreg;
  copy_wait_ring<kAffRing - 2>();  // stages 0 and 1
  __syncthreads();
  int slot = 0;
  for (int k = 0; k < steps; k++) {
    if (!end && lane < n && (fwd || k > 0 || b == P.N)) *o = ya[lane];
    o += step;
    if (k > 0) {  // into the block of stage k - 1, whose entries went to registers before this barrier
      fetch(slot);
      if (++slot == kAffRing) slot = 0;
    }
    if (((k + 2) & 31) == 0) {
      dreg = dnext;
      dnext = dims(k + 34);
    }
    const int d = __shfl_sync(kFull, dreg, (k + 2) & 31);
    if (lane == 0) sdim[(k + 2) & 3] = d;
    copy_wait_ring<kAffRing - 3>();  // stage k + 2
    double *t = ya; ya = yb; yb = t;
    __syncthreads();
  }
  if (end) o = end + lane;
  if (lane < n && (end || !fwd || b == P.N)) *o = ya[lane];
}

// The chain over the stages [a, b) from the value sv (null: zero) of dimension d0.
static __device__ __forceinline__ void aff_sweep(const Group &g, const ProbInfo &P, int mode, int a, int b, int d0,
                                                 const double *sv, double *end) {
  const int n = g.n, steps = b - a, lanes = TEAM - 32;
  const bool tr = mode == AFF_PLIN;
  double *ring = g_smem, *ya = ring + kAffRing * n * (n + 1), *yb = ya + kAffY;
  int *sdim = (int *)(yb + kAffY);
  if (threadIdx.x >= lanes) {
    const int lane = threadIdx.x & 31;
    // y_0, and zeros beyond the dimensions of either buffer
    ya[lane] = sv && lane < d0 ? sv[lane] : 0.0;
    yb[lane] = 0.0;
    __syncwarp();
    aff_helper(g, P, mode, a, b, ring, ya, yb, sdim, end);
    return;
  }
  // a row over four lanes (two below n = 5), over fewer where the team has not as many
  if (n <= 4) aff_rows<2, 2>(ring, ya, yb, sdim, n, tr, steps, d0);
  else if (n <= 8) aff_rows<4, 2>(ring, ya, yb, sdim, n, tr, steps, d0);
  else if (4 * n > lanes && 2 * n <= lanes && n <= 16) aff_rows<2, 8>(ring, ya, yb, sdim, n, tr, steps, d0);
  else if (4 * n > lanes && 2 * n <= lanes) aff_rows<2, 16>(ring, ya, yb, sdim, n, tr, steps, d0);
  else if (4 * n > lanes) aff_rows<1, 32>(ring, ya, yb, sdim, n, tr, steps, d0);
  else if (n <= 16) aff_rows<4, 4>(ring, ya, yb, sdim, n, tr, steps, d0);
  else aff_rows<4, 8>(ring, ya, yb, sdim, n, tr, steps, d0);
}

__global__ void k_aff_down(Group g, int mode, int fin, int /*per_task*/) {
  const int t = team_task();
  if (t >= g.nslot) return;
  const ChunkInfo ci = g.chunk[t];
  const ProbInfo &P = g.prob[ci.prob];
  if (skipped_by_mask(g, ci.prob)) return;
  if (ci.c >= P.nch) return;
  const int n = g.n, a = ci.c * P.L, b = min(a + P.L, P.N);
  const bool fwd = aff_forward(mode);
  // boundary value: with one chunk the problem's own (z_0, 0, rq_N or nu_0); after the scan the
  // forward slot (ch0 + c) = y_a, the backward slot (ch0 + c + 1) = y_b
  const int slot = fwd ? P.ch0 + ci.c : P.ch0 + ci.c + 1;
  const double *end = stage_ws(g, fwd ? P.st0 : P.st0 + P.N);
  const double *sv = P.nch > 1 ? g.CS[fin] + (size_t)slot * g.cs_stride + n * n
                               : mode == AFF_CROLL ? nullptr
                                                   : end + (mode == AFF_ROLL ? g.ws.z : mode == AFF_PLIN ? g.ws.rq : g.ws.nu);
  aff_sweep(g, P, mode, a, b, aff_dim(g, P.st0 + (fwd ? a : b), mode), sv, nullptr);
}

// The chunk aggregates of the refinement's chains (CROLL, PLIN), in the place of k_aff_up: their
// matrices are the rollout's product of the same Phi's (CROLL) and its transpose (PLIN), which the
// solve's k_aff_up kept in CR, so that a chunk is one chain of its offsets from zero, n^2 a stage
// instead of n^3 (16384 stages at n = 16: 191 us a launch with the products).
__global__ void k_aff_up_again(Group g, int mode, int /*per_task*/) {
  const int t = team_task();
  if (t >= g.nslot) return;
  const ChunkInfo ci = g.chunk[t];
  const ProbInfo &P = g.prob[ci.prob];
  if (skipped_by_mask(g, ci.prob)) return;
  const bool fwd = aff_forward(mode);
  if (aff_up_ends(g, ci, P, mode, fwd)) return;
  const int n = g.n, a = ci.c * P.L, b = min(a + P.L, P.N);
  const int slot = fwd ? P.ch0 + ci.c + 1 : P.ch0 + ci.c;
  const int da = aff_dim(g, P.st0 + a, mode), db = aff_dim(g, P.st0 + b, mode);
  double *cs = g.CS[0] + (size_t)slot * g.cs_stride;
  const double *F = g.CR + (size_t)t * g.cr_stride;
  for (int idx = team_rank(); idx < n * n; idx += TEAM) {
    const int i = idx / n, j = idx - i * n;
    cs[idx] = fwd ? F[idx] : F[j * n + i];
  }
  if (team_rank() == 0) {
    int *cm = g.CI[0] + (size_t)slot * CI_STRIDE;
    cm[CI_ROWS] = 0; cm[CI_NA] = fwd ? da : db; cm[CI_NB] = fwd ? db : da;
  }
  aff_sweep(g, P, mode, a, b, 0, nullptr, cs + n * n);
}

// ----------------------------------------------------------- stage-parallel helpers of the solve
// z_0 = T_0'(s_0 - t_0) and the check H_0 s_0 + h_0 = 0 (eqs. initial-feasibility, reduced-initial)
__global__ void k_solve_init(Group g, const double *s0) {
  const int t = team_task();
  if (t >= g.nprob) return;
  const ProbInfo &P = g.prob[t];
  if (skipped_by_mask(g, t)) return;
  const int n = g.n, tid = team_rank();
  const int s = P.st0;
  double *ws = stage_ws(g, s);
  const int *wi = stage_wi(g, s);
  const int r = wi[SI_HROWS], ur = wi[SI_UR], nb = n - ur;
  const double *x0 = s0 + P.os0;
  const double *H = ws + g.ws.H, *T = ws + g.ws.UT + ur, *tt = ws + g.ws.t;
  double worst = 0.0, om = 0.0;
  for (int a = tid; a < r; a += TEAM) {
    double v = H[a * (n + 1) + n];
    om = fmax(om, fabs(v));
    for (int l = 0; l < n; l++) v = fma(H[a * (n + 1) + l], x0[l], v);
    worst = fmax(worst, fabs(v));
  }
  bool bad = false;
  for (int l = tid; l < n; l += TEAM) {
    om = fmax(om, fabs(x0[l]));
    bad = bad || !isfinite(x0[l]);
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) set_status(g, t, ST_NONFINITE);
  }
  worst = team_max(worst);
  om = fmax(1.0, team_max(om));
  if (tid == 0 && worst > g.tau_inc * om) set_status(g, t, ST_INFEASIBLE_X0);
  for (int a = tid; a < n; a += TEAM) {
    double v = 0.0;
    if (a < nb)
      for (int l = 0; l < n; l++) v = fma(T[l * n + a], x0[l] - tt[l], v);
    ws[g.ws.z + a] = v;
  }
}

// pass 0: v_i = K z + k, pi_i = P z + p.  correction passes: dv = K dz + k', dpi = P dz + p',
// then z += dz, v += dv, pi += dpi.
__global__ void k_post_roll(Group g, int corr) {
  for_stages(g, [&](const int s) {
    const StageInfo S = g.st[s];
    const ProbInfo &P = g.prob[S.prob];
    if (skipped_by_mask(g, S.prob)) return;
    const int n = g.n, m = g.m, tid = team_rank();
    double *ws = stage_ws(g, s);
    const int *wi = stage_wi(g, s);
    const int nx = wi[SI_NBAR], mu = (S.i < P.N) ? wi[SI_MBAR] : 0;
    const double *zz = ws + (corr ? g.ws.dz : g.ws.z);
    const double *kk = ws + (corr ? g.ws.dv : g.ws.k);
    const double *pp = ws + (corr ? g.ws.pp : g.ws.p);
    // one lane per row of K and of P
    for (int r = tid; r < mu + nx; r += TEAM) {
      const int a = r < mu ? r : r - mu;
      const double *row = ws + (r < mu ? g.ws.K : g.ws.P) + a * n;
      double s0 = r < mu ? kk[a] : pp[a];
      for (int l = 0; l < nx; l++) s0 = fma(row[l], zz[l], s0);
      double *o = ws + (r < mu ? g.ws.v : g.ws.pi) + a;
      *o = corr ? *o + s0 : s0;
    }
    if (!corr) {
      for (int r = mu + tid; r < m; r += TEAM) ws[g.ws.v + r] = 0.0;
      for (int r = nx + tid; r < n; r += TEAM) ws[g.ws.pi + r] = 0.0;
    } else {
      for (int r = tid; r < nx; r += TEAM) ws[g.ws.z + r] += zz[r];
    }
  });
}

// Residual of the reduced KKT system, evaluated through the original data.
// Under x_i = T z + t, u_i = Y z + Z v + y (Thm 5 substitution), with
// a = g^x + A'T_{i+1}pi_{i+1} and b = g^u + B'T_{i+1}pi_{i+1} at that point,
// the z-rows are T'a + Y'b - pi, the v-rows Z'b, and the costate rows
// cbar + Abar z + Bbar v - z_{i+1}.  Forming Qbar z + qbar instead would sum
// terms of size |Y|^2 that cancel down to pi: where the mixed rows leave D_i
// ill-conditioned |Y| is large, and that cancellation would set the accuracy
// of the costates and so of the multipliers.  The offsets that the next pass's chain (PLIN) adds to
// its maps, rq + K' rr + Phi' P_{i+1} rc (ws.gv), follow from the stage's residual at once, while it
// is in shared memory.  640 problems of 32 to 128 stages: 353 us at n = 16, 150 at n = 8 (445 and 187 with
// one lane per row and a branch per block).  Per task: 5n + 3m doubles.
__global__ void k_resid(Group g, int per_task) {
  for_stages(g, [&](const int s) {
    const StageInfo S = g.st[s];
    const ProbInfo &P = g.prob[S.prob];
    if (skipped_by_mask(g, S.prob)) return;
    const int n = g.n, m = g.m, tid = team_rank(), i = S.i;
    double *ws = stage_ws(g, s);
    const int *wi = stage_wi(g, s);
    const bool last = i == P.N;
    const double *wn = last ? ws : stage_ws(g, s + 1);
    const int nx = wi[SI_NBAR], mu = last ? 0 : wi[SI_MBAR], ny = last ? 0 : stage_wi(g, s + 1)[SI_NBAR];
    const int ur = wi[SI_UR], ur1 = last ? 0 : stage_wi(g, s + 1)[SI_UR];
    const double *z = ws + g.ws.z, *v = ws + g.ws.v, *pi = ws + g.ws.pi, *pin = wn + g.ws.pi, *zn = wn + g.ws.z;
    const double *T = ws + g.ws.UT + ur, *Tn = wn + g.ws.UT + ur1;
    const double *Y = ws + g.ws.Y, *Z = ws + g.ws.Z, *Ab = ws + g.ws.Ab, *Bb = ws + g.ws.Bb;
    double *sm = team_smem(per_task);
    double *xs = sm, *us = xs + n, *lh = us + m, *ga = lh + n, *gb = ga + n, *g2 = gb + m, *rcs = g2 + n + m;
    // T_i = I, t_i = 0 (te) or T_{i+1} = I (tne): the products with them are their other factor
    const bool te = wi[SI_TEYE] != 0, tne = !last && stage_wi(g, s + 1)[SI_TEYE] != 0;
    // An FP64 instruction costs its warp the same whatever its active lanes, so what counts is how
    // many follow one another: rows of different blocks lie side by side and run the same loop on
    // their own pointers (a branch per block would run one block after the other), long rows are two
    // items, and a few rows are split over several lanes.  p[j sp] x[j] summed onto v in order of j.
    auto dot = [](double v, const double *p, int sp, const double *x, int len) {
#pragma unroll 4
      for (int j = 0; j < len; j++) v = fma(p[(size_t)j * sp], x[j], v);
      return v;
    };
    // u_i = Y z + Z v + y
    if (!last) {
      const int parts = m <= 8 ? 4 : 2;
      split_rows(m, parts, [&](int r, int k) {
        double v0 = k == 0 ? ws[g.ws.y + r] : 0.0;
        for (int j = k; j < nx; j += parts) v0 = fma(Y[r * n + j], z[j], v0);
        for (int j = k; j < mu; j += parts) v0 = fma(Z[r * m + j], v[j], v0);
        return v0;
      }, [&](int r, double v0) { us[r] = v0; });
    }
    // x_i and T_{i+1} pi_{i+1}
    for (int r = tid; r < (last ? n : 2 * n); r += TEAM) {
      const bool rx = r < n;
      const int a = rx ? r : r - n;
      double v0 = rx ? (te ? z[a] : ws[g.ws.t + a]) : (tne ? pin[a] : 0.0);
      if (rx ? !te : !tne) v0 = dot(v0, (rx ? T : Tn) + a * n, 1, rx ? z : pin, rx ? nx : ny);
      (rx ? xs : lh)[a] = v0;
    }
    tsync();
    const double *Q = g.Q + P.oQ + (size_t)i * n * n, *q = g.qv + P.oqv + (size_t)i * n;
    const double *A = g.A + P.oA + (size_t)i * n * n, *B = g.B + P.oB + (size_t)i * n * m;
    const double *Mm = g.M + P.oM + (size_t)i * n * m, *R = g.R + P.oR + (size_t)i * m * m;
    const double *rv = g.rv + P.orv + (size_t)i * m;
    // g^x (n rows) and g^u (m); A'lh and B'lh (the same rows, into g2); the dynamics' residual (ny)
    const int rows = n + m;
    for (int r = tid; r < (last ? n : 2 * rows + ny); r += TEAM) {
      const int h = r < rows ? 0 : (r < 2 * rows ? 1 : 2), a = r - h * rows;
      const bool ra = h < 2 && a < n, rb = h < 2 && !ra;  // rows of x, of u
      const int b = rb ? a - n : a;
      const double *p1 = h == 0 ? (ra ? Q + a * n : Mm + b) : h == 1 ? (ra ? A + a : B + b) : Ab + a * n;
      const double *p2 = h == 0 ? (ra ? Mm + a * m : R + b * m) : Bb + a * m;
      double s0 = h == 0 ? (ra ? q[a] : rv[b]) : h == 1 ? 0.0 : ws[g.ws.cb + a] - zn[a];
      s0 = dot(s0, p1, h == 0 ? (ra ? 1 : m) : h == 1 ? (ra ? n : m) : 1, h == 0 ? xs : h == 1 ? lh : z, h == 2 ? nx : n);
      s0 = dot(s0, p2, 1, h == 0 ? us : v, last || h == 1 ? 0 : h == 0 ? m : mu);
      (h == 0 ? ga : h == 1 ? g2 : rcs)[a] = s0;
      if (h == 2) ws[g.ws.rc + a] = s0;
    }
    tsync();
    if (!last) {  // a = g^x + A'lh, b = g^u + B'lh
      for (int r = tid; r < rows; r += TEAM) ga[r] += g2[r];
      tsync();
    }
    // P_{i+1} rc (ny rows, into lh), rq (nx, kept in xs), rr (mu, in us)
    const double *Pn = wn + g.ws.P;
    for (int r = tid; r < ny + nx + mu; r += TEAM) {
      const int h = r < ny ? 0 : (r < ny + nx ? 1 : 2), a = h == 0 ? r : (h == 1 ? r - ny : r - ny - nx);
      double s0 = h == 1 ? (te ? ga[a] : 0.0) - pi[a] : 0.0;
      if (h == 1 && !te) s0 = dot(s0, T + a, n, ga, n);
      s0 = dot(s0, h == 0 ? Pn + a * n : (h == 1 ? Y + a : Z + a), h == 0 ? 1 : (h == 1 ? n : m), h == 0 ? rcs : gb,
               last ? 0 : (h == 0 ? ny : m));
      (h == 0 ? lh : (h == 1 ? xs : us))[a] = s0;
      if (h > 0) ws[(h == 1 ? g.ws.rq : g.ws.rr) + a] = s0;
    }
    if (last) return;
    tsync();
    const double *K = ws + g.ws.K, *Phi = ws + g.ws.Phi;
    const int parts = n <= 8 ? 4 : n <= 16 ? 2 : 1;
    split_rows(nx, parts, [&](int r, int k) {
      double v0 = k == 0 ? xs[r] : 0.0;
      for (int j = k; j < mu; j += parts) v0 = fma(K[j * n + r], us[j], v0);
      for (int j = k; j < ny; j += parts) v0 = fma(Phi[j * n + r], lh[j], v0);
      return v0;
    }, [&](int r, double v0) { ws[g.ws.gv + r] = v0; });
  });
}

// Correction controls of a refinement pass: with w = P_{i+1} rc_i + p'_{i+1},
// k'_i = -H_uu^{-1} (rr_i + Bbar' w) through the Cholesky factor of H_uu (-> dv), and the offsets
// rc + Bbar k' of the chain that follows (CROLL, ws.gv).  Short products are split over two or four
// lanes a row: 640 problems at n = 16 180 -> 137 us, at n = 8 106 -> 94.
__global__ void k_pcorr(Group g, int per_task) {
  for_stages(g, [&](const int s) {
    const StageInfo S = g.st[s];
    const ProbInfo &P = g.prob[S.prob];
    if (skipped_by_mask(g, S.prob)) return;
    if (S.i >= P.N) return;
    const int n = g.n, m = g.m, tid = team_rank();
    double *ws = stage_ws(g, s);
    const double *wn = stage_ws(g, s + 1);
    const int mu = stage_wi(g, s)[SI_MBAR], ny = stage_wi(g, s + 1)[SI_NBAR];
    double *sm = team_smem(per_task);
    double *w = sm, *hu = sm + n, *Ls = hu + m;  // Ls: chol(H_uu), mu x mu (ld m)
    const double *Pn = wn + g.ws.P, *ppn = wn + g.ws.pp, *rc = ws + g.ws.rc, *Bb = ws + g.ws.Bb;
    for (int idx = tid; idx < mu * mu; idx += TEAM) {
      const int a = idx / mu, l = idx - a * mu;
      Ls[a * m + l] = ws[g.ws.Lh + a * m + l];
    }
    const int pw = n <= 8 ? 4 : n <= 16 ? 2 : 1, ph = m <= 8 ? 4 : 2;
    split_rows(ny, pw, [&](int r, int k) {
      double s0 = k == 0 ? ppn[r] : 0.0;
      for (int l = k; l < ny; l += pw) s0 = fma(Pn[r * n + l], rc[l], s0);
      return s0;
    }, [&](int r, double s0) { w[r] = s0; });
    tsync();
    split_rows(mu, ph, [&](int r, int k) {
      double s0 = k == 0 ? ws[g.ws.rr + r] : 0.0;
      for (int l = k; l < ny; l += ph) s0 = fma(Bb[l * m + r], w[l], s0);
      return s0;
    }, [&](int r, double s0) { hu[r] = s0; });
    tsync();
    // dv = -H_uu^{-1} hu with H_uu = L L' (L = Ls, lower): forward then backward
    // substitution by the first warp, lane a holding row a (mu <= 16), column by column; the
    // diagonal's reciprocals up front, one division for all lanes instead of one per column (a
    // division is about fifteen FP64 instructions)
    if (tid < 32) {
      const int a = tid;
      double x = (a < mu) ? hu[a] : 0.0;
      const double inv = (a < mu) ? 1.0 / Ls[a * m + a] : 0.0;
      for (int l = 0; l < mu; l++) {
        if (a == l) x *= inv;
        const double xl = __shfl_sync(kFull, x, l);
        if (a > l && a < mu) x = fma(-Ls[a * m + l], xl, x);
      }
      for (int l = mu - 1; l >= 0; l--) {
        if (a == l) x *= inv;
        const double xl = __shfl_sync(kFull, x, l);
        if (a < l) x = fma(-Ls[l * m + a], xl, x);
      }
      if (a < mu) ws[g.ws.dv + a] = hu[a] = -x;
    }
    tsync();
    for (int r = tid; r < ny; r += TEAM) {
      double s0 = rc[r];
      for (int l = 0; l < mu; l++) s0 = fma(Bb[r * m + l], hu[l], s0);
      ws[g.ws.gv + r] = s0;
    }
  });
}

// x_i = T z + t, u_i = Y z + Z v + y (eq. recovery-maps)
__global__ void k_recover(Group g, double *x, double *u) {
  for_stages(g, [&](const int s) {
    const StageInfo S = g.st[s];
    const ProbInfo &P = g.prob[S.prob];
    if (skipped_by_mask(g, S.prob)) return;
    const int n = g.n, m = g.m, tid = team_rank();
    const double *ws = stage_ws(g, s);
    const int *wi = stage_wi(g, s);
    const int ur = wi[SI_UR], nb = n - ur;
    const double *T = ws + g.ws.UT + ur, *z = ws + g.ws.z;
    const bool te = wi[SI_TEYE] != 0;  // T = I, t = 0
    bool bad = false;
    for (int a = tid; a < n; a += TEAM) {
      double v = te ? z[a] : ws[g.ws.t + a];
      if (!te)
        for (int j = 0; j < nb; j++) v = fma(T[a * n + j], z[j], v);
      x[P.ox + (size_t)S.i * n + a] = v;
      bad = bad || !isfinite(v);
    }
    if (S.i < P.N) {
      const int mb = wi[SI_MBAR];
      const double *Y = ws + g.ws.Y, *Z = ws + g.ws.Z, *vv = ws + g.ws.v;
      for (int a = tid; a < m; a += TEAM) {
        double v = ws[g.ws.y + a];
        for (int j = 0; j < nb; j++) v = fma(Y[a * n + j], z[j], v);
        for (int j = 0; j < mb; j++) v = fma(Z[a * m + j], vv[j], v);
        u[P.ou + (size_t)S.i * m + a] = v;
        bad = bad || !isfinite(v);
      }
    }
    if (__syncthreads_or(bad) && tid == 0) set_status(g, S.prob, ST_NONFINITE);
  });
}

}  // namespace eclqr

namespace eclqr {
// reduced dimensions into batch-ordered arrays: nbar has N_j + 1 entries per
// problem, mbar N_j entries (the prefix of N_j + 1 minus one per earlier problem)
__global__ void k_dims(Group g, int *nbar, int *mbar) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.nstage) return;
  const StageInfo S = g.st[s];
  const ProbInfo &P = g.prob[S.prob];
  if (skipped_by_mask(g, S.prob)) return;
  const int *wi = stage_wi(g, s);
  nbar[P.ost + S.i] = wi[SI_NBAR];
  if (S.i < P.N) mbar[P.ost - P.id + S.i] = wi[SI_MBAR];
}
}  // namespace eclqr
