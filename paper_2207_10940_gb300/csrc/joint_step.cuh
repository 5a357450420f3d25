// The Gauss-Newton step of the joint problem with the non-pose unknowns
// eliminated in covariance form (Eq. 6-7).  The full system that marginalisation
// takes is assembled beside a frame's last step, at the same linearisation point,
// by a second block (step_lin_block in solve.cu).
//
// What bounds a step is the FP64 pipe: on GB300 a warp's FP64 instruction holds
// its sub-partition's pipe for 64 cycles whatever the number of active lanes
// (measured: dependent DFMA 65 cycles, two independent ones 129; an f64 mma
// m8n8k4 577, no faster per product; a 128-thread barrier 33, a shared-memory
// exchange 35).  So the step is laid out to put the fewest FP64 instructions on
// any one sub-partition along its chain, and this formulation needs far fewer
// of them than the 26-variable information form:
//
//   unknowns     x0's pose p0 and x1's pose p1 (12), y = x0's velocity, biases
//                and gravity (11), x1's velocity, biases and gravity (8).
//   x1's velocity enters the velocity rows of e_IMU only (Jacobian -I) and no
//                prior: it is free to follow, so those rows drop out and the
//                position and rotation rows keep their own covariance block S6
//                of Sigma (the marginal), fixed for the frame.
//   x1's biases  follow x0's; x1's gravity leaves one row: along the normal n
//                of its Jacobian block B, a dg0 + s with variance sigma_g^2.
//   y            under the prior (H*, b*) given p0 is Gaussian with covariance
//                P = H_yy^-1 and mean K p0 + m: P, K = -P H_yp, P b_y, and the
//                Schur complement on p0 are fixed for the frame (k_frame_begin).
//   so the 7 rows r = Jp p + Jy y + e become r' = (Jp + Jy K) p + (e + Jy m)
//   with covariance S = blockdiag(S6, sigma_g^2) + Jy P Jy^T, and the system is
//       [ -S   J' ] [ lambda ]   [ -e' ]
//       [ J'^T H  ] [   p    ] = [  b  ]
//   H, b: the prior on p0 plus the pixel terms.  The 7 multipliers are
//   eliminated before the pixel sums arrive, the 12 poses after; then
//   y = K p0 + m - P Jy^T lambda,  dv1 = e_v + J_v dx0 - S_v6 lambda.
// This is the same minimiser as Eq. 7's in exact arithmetic; the 1e8-scale IMU
// weights are never formed (their inverses are added instead).
//
// Measured against the information form (`gn_step_body`): a step on one block 102k
// -> 46k cycles (66k with the same algebra but branches between the lanes of a
// phase, index arithmetic per element and FP64 comparisons); one 640x480 camera
// 1201 -> 743 us per frame, 12 x 320x240 1449 -> 935 us, 64 x 640x480 (steps hidden
// behind other groups' pixels) 4734 -> 4547 us.
//
// Included by solve.cu, inside its namespace, after the element-wise 3x3 algebra
// and the warp-cooperative state algebra that it uses.

// Named barriers.  The ids of a step: 1 warps 0-3 and 3 warps 4-7 among themselves, 5
// warps 0-2, 6 warps 1-2; hand-offs (one side arrives and goes on, the other waits) 4
// pixel terms, 7 errors, 8 position rows, 9 poses.  A hand-off keeps an id of its own:
// the arriving warp may come back to a shared one before the waiting warps have passed
// it, and would be counted twice.
template <int ID, int N>
__device__ __forceinline__ void bar_sync() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory"); }
template <int ID, int N>
__device__ __forceinline__ void bar_arrive() { asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(N) : "memory"); }

// Pre-integration of a run of IMU pieces (and its derivatives by the biases):
// rotation R, Phi = d(R)/d(b_g) (right perturbation), V = d(v)/d(b_g),
// P = d(p)/d(b_g), Va, Pa by b_a, velocity v, position p, duration T.
constexpr int kNR = 0, kNPhi = 9, kNV = 18, kNP = 27, kNVa = 36, kNPa = 45, kNv = 54, kNp = 57, kNT = 60;
constexpr int kNode = 61;             // odd stride: consecutive nodes fall into different banks

constexpr int kLam = 7, kPose = 12, kSys = kLam + kPose;      // 19 unknowns of the sweep
constexpr int kSysEnt = kSys * (kSys + 1) / 2 + kSys;         // lower triangle + right-hand side row

// The pixel terms of the joint system.
struct PixSmem {
  double C[18][6];                    // Jacobian maps: photometric on (p0, p1), ICP on p1
  double sums[kSumsAll];
  double U[18][7];
  double P12[kPose * kPose], g12[kPose];   // lower triangle
};

struct FastSmem : PixSmem {
  double nodeA[kElimPieces][kNode];   // leaves, then every second level of the tree
  double nodeB[kElimPieces / 2][kNode];
  double X[kElimPieces / 2][18];      // V_2 - [v_2]x Phi_1 and P_2 - [p_2]x Phi_1 of each pair
  double th[kElimPieces][3], t2[kElimPieces], ser[3][kElimPieces];
  double piece[kElimPieces][8];       // as Elim::piece
  double el[kElimDoubles];            // Elim's matrices
  DState x0, x1, xbar;
  double Rref[9], rref[3];
  double one, zero;
  double dx[34];                      // the step
  // states only
  double R0[9], Q0[9], R1[9], A0[9], QR[9], QA[9], RcR1T[9], c[3], t1[3], t2c[3], rcS[3], base[3], dr[3], evb[3];
  double d[17], m[11], bp[6];         // x0 boxminus xbar; mean of y; prior vector on p0
  double eg[3], Jlg[9], Jrg[9], nv[3], mm[3], a[3], s, Gm[6], Ag[6];
  double eb[6];                       // bias errors
  // after the pre-integration
  double Jyr[3][11];                  // position rows by y
  double RW[9], APg[9], t3[3], M[9], RP[9], t4[3], u[3], er[3], ea[3], Jla[9], B13[9];
  double B14[9], B17[9], w9[3], t5[3], B9[9], B20[6], ev[3];
  double T[kLam][11];                 // Jy P
  double Jp[kLam][kPose];             // J'
  double ep[kLam];                    // e'
  double S[28];                       // S's lower triangle (without blockdiag(S6, sigma_g^2))
  // sweep
  double col[2][kSys + 1];
  double sink[128];                   // where a lane without a value to publish writes
  double z[kSys];
  double L[kSys][kSys + 2];
  double rot[24];
  double fo[21];
  double cost;
  int good, posdef[4];
};
template <int N>
struct Slots {
  static constexpr int value = N;
};

__device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; }   // i >= j

// a < b for non-negative doubles, as integers (an FP64 comparison would take the
// FP64 pipe for 64 cycles).
__device__ __forceinline__ bool pos_less(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b);
}
__device__ __forceinline__ bool finite_bits(double a) {
  return (__double2hiint(a) & 0x7ff00000) != 0x7ff00000;
}

// base + three products along strides.  Lanes that take different products of a
// phase differ in their pointers only: branches of a warp would run one after the
// other, each holding the FP64 pipe for its own instructions.
__device__ __forceinline__ double dot3(double base, const double* A, int sa, const double* B, int sb) {
  return fma(A[0], B[0], fma(A[sa], B[sb], fma(A[2 * sa], B[2 * sb], base)));
}
// the same with the third product's operands given apart
__device__ __forceinline__ double dot21(double base, const double* A, const double* B, int sb,
                                        const double* A2, const double* B2) {
  return fma(A[0], B[0], fma(A[1], B[sb], fma(*A2, *B2, base)));
}

// ---- IMU pieces --------------------------------------------------------------

// Leaves of the pieces at biases (bg, ba): R = Exp(th), Phi = -Jr(th) dt, v = a dt,
// p = a dt^2 / 2, Va = -dt I, Pa = -dt^2 / 2 I.  Warps 0-3.  The three series (or
// sines) of a piece run on three lanes, its nine matrix elements on nine; a
// thread keeps its element and strides over the pieces, so that the index
// arithmetic (divisions by 9 and 3) is done once.
__device__ void fast_leaves(FastSmem& S, int np, const double* bg, const double* ba) {
  const int t = threadIdx.x, q = t >> 4;
  if (q < 6)
    for (int k = t & 15; k < np; k += 16) {
      const double* pc = S.piece[k];
      if (q < 3) {
        S.th[k][q] = (pc[2 + q] - bg[q]) * pc[0];
      } else {
        const double v = (pc[2 + q] - ba[q - 3]) * pc[0];
        S.nodeA[k][kNv + q - 3] = v;
        S.nodeA[k][kNp + q - 3] = v * pc[1];
      }
    }
  bar_sync<1, 128>();
  if (q < 3)
    for (int k = t & 15; k < np; k += 16) {
      const double* w = S.th[k];
      const double t2 = fma(w[0], w[0], fma(w[1], w[1], w[2] * w[2]));
      double f;
      if (pos_less(t2, kSeriesT2)) { // sin t / t, (1 - cos t) / t^2, (t - sin t) / t^3
        const double c0 = q == 0 ? 1.0 : q == 1 ? 0.5 : 1.0 / 6;
        const double c1 = q == 0 ? -1.0 / 6 : q == 1 ? -1.0 / 24 : -1.0 / 120;
        const double c2 = q == 0 ? 1.0 / 120 : q == 1 ? 1.0 / 720 : 1.0 / 5040;
        const double c3 = q == 0 ? -1.0 / 5040 : q == 1 ? -1.0 / 40320 : -1.0 / 362880;
        const double c4 = q == 0 ? 1.0 / 362880 : q == 1 ? 1.0 / 3628800 : 1.0 / 39916800;
        f = fma(t2, fma(t2, fma(t2, fma(t2, c4, c3), c2), c1), c0);
      } else {
        const double th = sqrt(t2);
        double sn, cs;
        sincos(th, &sn, &cs);
        f = q == 0 ? sn / th : q == 1 ? (1.0 - cs) / t2 : (th - sn) / (t2 * th);
      }
      S.ser[q][k] = f;
      if (q == 0) S.t2[k] = t2;
    }
  bar_sync<1, 128>();
  const int k0 = t / 9, e = t - 9 * k0, r = e / 3, c = e - 3 * r;
  const int hk = r == c ? 0 : 3 - r - c;                      // [w]x element e: +-w[hk], or 0
  const bool neg = ((c - r + 3) % 3) == 1, diag = r == c;
  const double id = diag ? 1.0 : 0.0;
  if (k0 < 14)
    for (int k = k0; k < np; k += 14) {
      const double* w = S.th[k];
      const double dt = S.piece[k][0], hdt = S.piece[k][1];
      const double wk = w[hk];
      const double K = diag ? 0.0 : neg ? -wk : wk, K2 = fma(w[r], w[c], diag ? -S.t2[k] : 0.0);
      const double ea = S.ser[0][k], eb = S.ser[1][k], jb = S.ser[2][k];
      double* n = S.nodeA[k];
      n[kNR + e] = fma(eb, K2, fma(ea, K, id));
      n[kNPhi + e] = -dt * fma(jb, K2, fma(-eb, K, id));
      n[kNV + e] = 0.0;
      n[kNP + e] = 0.0;
      n[kNVa + e] = diag ? -dt : 0.0;
      n[kNPa + e] = diag ? -hdt * dt : 0.0;
      if (e == 0) n[kNT] = dt;
    }
  bar_sync<1, 128>();
}

// Composition of two runs (1 then 2):
//   R = R1 R2, Phi = R2^T Phi1 + Phi2, v = v1 + R1 v2, p = p1 + v1 T2 + R1 p2,
//   V = V1 + R1 (V2 - [v2]x Phi1), P = P1 + V1 T2 + R1 (P2 - [p2]x Phi1),
//   Va = Va1 + R1 Va2, Pa = Pa1 + Va1 T2 + R1 Pa2, T = T1 + T2
// over a binary tree of the np leaves: ceil(log2 np) levels of 6 dependent FP64
// instructions each, one output element per lane (the prefix scans and sums of
// the sequential order take 14 dependent ones per sum besides the scans).  64
// lanes take a pair's 61 elements, two pairs per pass; a lane's element is the
// same in every pass, so where its operands lie in the pair is worked out once
// (worked out per element it took three times the FP64 arithmetic: 11.9k cycles
// for 14 pieces).  Warps 0-3; returns the root.
__device__ const double* fast_tree(FastSmem& S, int np) {
  const int t = threadIdx.x;
  // first half: element xe of the pair's 18 X, pair t / 18 of 7 per pass
  const int x0 = t / 18, xe = t - 18 * x0;
  int xv1, xv2, xp1, xp2, xb;
  {
    const bool pos = xe >= 9;
    const int q = pos ? xe - 9 : xe, r = q / 3, c = q - 3 * r;
    const int r1 = r == 2 ? 0 : r + 1, r2 = r == 0 ? 2 : r - 1;
    const int v = kNode + (pos ? kNp : kNv);                  // of the second run
    xv1 = v + r1;
    xv2 = v + r2;
    xp1 = kNPhi + 3 * r1 + c;
    xp2 = kNPhi + 3 * r2 + c;
    xb = kNode + (pos ? kNP : kNV) + q;
  }
  // second half: element e of the pair, pair t / 64 of 2 per pass; operands as
  // offsets from the first run's node (the second's follows it): three products
  // A B along strides sa, sb, the base and the factor of T2 (kZero: none)
  const int e = t & 63;
  int oa, sa, ob, sb, obase, oext;
  bool inX = false;
  constexpr int kZero = -1;
  {
    const bool vec = e >= kNv;
    const int f = vec ? (e - kNv) / 3 : e / 9;                // field
    const int q = vec ? (e - kNv) - 3 * f : e - 9 * f;
    const int r = vec ? q : q / 3, c = vec ? 0 : q - 3 * r;
    const bool phi = !vec && f == 1;
    oa = phi ? kNode + r : 3 * r;                             // row r of R1, or of R2^T
    sa = phi ? 3 : 1;
    sb = vec ? 1 : 3;
    obase = (!vec && f == 0) ? kZero : phi ? kNode + e : e;
    oext = kZero;
    if (vec) {
      ob = kNode + (f == 0 ? kNv : kNp);
      if (f == 1) oext = kNv + q;
    } else if (f == 0) {
      ob = kNode + kNR + c;
    } else if (phi) {
      ob = kNPhi + c;
    } else if (f == 2 || f == 3) {
      inX = true;
      ob = (f == 2 ? 0 : 9) + c;
      if (f == 3) oext = kNV + q;
    } else {
      ob = kNode + (f == 4 ? kNVa : kNPa) + c;
      if (f == 5) oext = kNVa + q;
    }
    if (e >= kNT) {                  // T (and the spare lanes): no products
      oa = ob = sa = sb = 0;
      oext = obase = kZero;
      inX = false;
    }
  }
  double(*in)[kNode] = S.nodeA;
  double(*out)[kNode] = S.nodeB;
  for (int n = np; n > 1; n = (n + 1) >> 1) {
    const int full = n >> 1;
    if (x0 < 7)
      for (int i = x0; i < full; i += 7) {
        const double* b = in[2 * i];
        // minus row r of [v2]x Phi1: -(v_r1 Phi_r2 - v_r2 Phi_r1)
        S.X[i][xe] = fma(b[xv2], b[xp1], fma(-b[xv1], b[xp2], b[xb]));
      }
    bar_sync<1, 128>();
    for (int i = t >> 6; i < full; i += 4) {       // two pairs: the second's operands load beside the first's products
      double a[2][3], bb[2][3], base[2], ext[2], T2[2], T1[2];
      const bool two = i + 2 < full;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int p = (u && two) ? i + 2 : i;
        const double* b = in[2 * p];
        const double* B = (inX ? S.X[p] : b) + ob;
        const double* A = b + oa;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          a[u][k] = A[k * sa];
          bb[u][k] = B[k * sb];
        }
        base[u] = obase < 0 ? 0.0 : b[obase];
        ext[u] = oext < 0 ? 0.0 : b[oext];
        T1[u] = b[kNT];
        T2[u] = b[kNode + kNT];
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (u && !two) break;
        const double v = e == kNT ? T1[u] + T2[u]
                                  : fma(ext[u], T2[u], fma(a[u][0], bb[u][0], fma(a[u][1], bb[u][1], fma(a[u][2], bb[u][2], base[u]))));
        if (e < kNode) out[i + 2 * u][e] = v;
      }
    }
    if ((n & 1) && t < kNode) out[full][t] = in[n - 1][t];    // the odd run out moves up unchanged
    bar_sync<1, 128>();
    double(*s)[kNode] = in;
    in = out;
    out = s;
  }
  return in[0];
}

// First-order bias update (preint_first_order) into the node layout; warps 0-3.
// Re-integrates (and moves the linearisation point) past the thresholds.
__device__ const double* fast_first_order(const SolveParams& sp, Ctrl* c, FastSmem& S, int np) {
  const int t = threadIdx.x;
  const double* bg = S.x0.bg;
  const double* ba = S.x0.ba;
  double dbg[3], dba[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    dbg[i] = bg[i] - c->b_lin[i];
    dba[i] = ba[i] - c->b_lin[3 + i];
  }
  const double ng = sqrt(dbg[0] * dbg[0] + dbg[1] * dbg[1] + dbg[2] * dbg[2]);
  const double na = sqrt(dba[0] * dba[0] + dba[1] * dba[1] + dba[2] * dba[2]);
  if (ng == 0.0 && na == 0.0) {                  // at the linearisation point: the integration itself,
    fast_leaves(S, np, bg, ba);                  // the same bits as re-integrating every iteration
    return fast_tree(S, np);
  }
  // pre_lin: dR 9, dv 3, dp 3, Phi_g 9, V_g 9, P_g 9, V_a 9, P_a 9, T
  if (ng > sp.relin_g || na > sp.relin_a) {      // uniform over the warps
    bar_sync<1, 128>();                          // every thread has read b_lin
    fast_leaves(S, np, bg, ba);
    const double* n = fast_tree(S, np);
    if (sp.last) return n;                       // nobody uses the point any more; a reader may run beside
    if (t < 60) {
      const int src = t < 9 ? kNR + t : t < 15 ? kNv + t - 9 : kNPhi + t - 15;   // Phi, V, P, Va, Pa follow
      c->pre_lin[t] = n[src];
    } else if (t == 60) {
      c->pre_lin[60] = n[kNT];
    } else if (t >= 64 && t < 70) {
      c->b_lin[t - 64] = t < 67 ? bg[t - 64] : ba[t - 67];
    }
    return n;
  }
  const double* L = c->pre_lin;
  double* n = S.nodeA[0];
  double* th = S.fo;
  double* E = S.fo + 3;
  double* Jrm = S.fo + 12;
  if (t < 3) {
    th[t] = L[15 + 3 * t] * dbg[0] + L[16 + 3 * t] * dbg[1] + L[17 + 3 * t] * dbg[2];
  } else if (t < 9) {
    const int q = t - 3, i = q % 3;
    const double* M = q < 3 ? L + 24 : L + 33;   // V_g or P_g
    const double* N = q < 3 ? L + 42 : L + 51;   // V_a or P_a
    double v = L[(q < 3 ? 9 : 12) + i];
#pragma unroll
    for (int j = 0; j < 3; ++j) v = fma(M[3 * i + j], dbg[j], fma(N[3 * i + j], dba[j], v));
    n[(q < 3 ? kNv : kNp) + i] = v;
  } else if (t < 45) {
    n[kNV + t - 9] = L[24 + t - 9];              // V_g, P_g, V_a, P_a
  } else if (t == 45) {
    n[kNT] = L[60];
  }
  bar_sync<1, 128>();
  if (t < 9) {                                   // Exp(theta), Jr(theta): one element per lane
    const double t2 = th[0] * th[0] + th[1] * th[1] + th[2] * th[2];
    double ea, eb, jb;
    if (t2 < kSeriesT2) {
      ea = 1.0 + t2 * (-1.0 / 6 + t2 * (1.0 / 120 + t2 * (-1.0 / 5040 + t2 * (1.0 / 362880))));
      eb = 0.5 + t2 * (-1.0 / 24 + t2 * (1.0 / 720 + t2 * (-1.0 / 40320 + t2 * (1.0 / 3628800))));
      jb = 1.0 / 6 + t2 * (-1.0 / 120 + t2 * (1.0 / 5040 + t2 * (-1.0 / 362880 + t2 * (1.0 / 39916800))));
    } else {
      const double tt = sqrt(t2);
      double sn, cs;
      sincos(tt, &sn, &cs);
      ea = sn / tt;
      eb = (1.0 - cs) / t2;
      jb = (tt - sn) / (t2 * tt);
    }
    const int r = t / 3, q = t % 3;
    const double K = hat_e(th, t);
    const double K2 = th[r] * th[q] - (r == q ? t2 : 0.0);
    const double id = r == q ? 1.0 : 0.0;
    E[t] = id + ea * K + eb * K2;
    Jrm[t] = id - eb * K + jb * K2;
  }
  bar_sync<1, 128>();
  if (t < 9) n[kNR + t] = mm_e(L, E, t, false, false);
  else if (t >= 32 && t < 41) n[kNPhi + t - 32] = mm_e(Jrm, L + 15, t - 32, false, false);
  bar_sync<1, 128>();
  return n;
}

// ---- state-only terms beside the pre-integration (warps 5-7) ------------------

// Jl^-1(s w), as jlinv_e with the series cut where the next term is below 1e-16.
__device__ __forceinline__ double fast_jlinv_e(const double* w0, double s, int e) {
  const double w[3] = {s * w0[0], s * w0[1], s * w0[2]};   // sign flips, exact
  const double t2 = fma(w[0], w[0], fma(w[1], w[1], w[2] * w[2]));
  const int r = e / 3, q = e - 3 * r;
  double c;
  if (pos_less(t2, 1e-5)) {
    c = fma(t2, fma(t2, 1.0 / 30240, 1.0 / 720), 1.0 / 12);
  } else if (pos_less(t2, kSeriesT2)) {
    c = 1.0 / 12 + t2 * (1.0 / 720 + t2 * (1.0 / 30240 + t2 * (1.0 / 1209600 + t2 * (1.0 / 47900160))));
  } else {
    const double t = sqrt(t2);
    double sn, co;
    sincos(t, &sn, &co);
    c = 1.0 / t2 - (1.0 + co) / (2.0 * t * sn);
  }
  return fma(c, fma(w[r], w[q], r == q ? -t2 : 0.0), fma(-0.5, hat_e(w, e), r == q ? 1.0 : 0.0));
}

// C of the pixel terms by one warp: the photometric local Jacobian on p0,
// -[R0 0; [dr]x R0, R0] with dr = r1 - r0, and on p1, diag(R0, R0); the ICP one on p1,
// diag(R_ref, R_ref).
__device__ __forceinline__ void fill_pixel_maps(PixSmem& S, const double* R0, const double* Rref, const double* dr) {
  const int lane = threadIdx.x & 31;
  for (int idx = lane; idx < 108; idx += 32) {
    const int i = idx / 6, k = idx - 6 * i, b = i / 3, r = i - 3 * b, kb = k / 3, q = k - 3 * kb;
    double v = 0.0;
    if ((b & 1) == kb) v = b < 2 ? -R0[3 * r + q] : b < 4 ? R0[3 * r + q] : Rref[3 * r + q];
    if (!(b == 1 && kb == 0)) S.C[i][k] = v;
  }
  if (lane < 9) S.C[3 + lane / 3][lane % 3] = -hatm_e(dr, R0, lane);
}

// Rotations of the states and everything that needs them only; warp 5.
__device__ void fast_state_terms(const SolveParams& sp, FastSmem& S) {
  const int lane = threadIdx.x & 31, g3 = lane / 9, e9 = lane - 9 * g3;
  const double T = S.el[kElT];
  const double* Rc = sp.R_CS;
  if (lane < 27) (g3 == 0 ? S.R0 : g3 == 1 ? S.Q0 : S.R1)[e9] =
      quat_rot_e(g3 == 0 ? S.x0.q : g3 == 1 ? S.x0.qg : S.x1.q, e9);
  else if (lane < 30) S.c[lane - 27] = fma(S.x0.v[lane - 27], T, lane == 29 ? -0.5 * sp.g * T * T : 0.0);
  __syncwarp();
  const int r3 = e9 / 3, c3 = e9 - 3 * r3;
  if (lane < 27) {                   // A0 = R0 Rc, QR = Q0 R0, Rc^T R1^T
    const double* A = g3 == 0 ? S.R0 + 3 * r3 : g3 == 1 ? S.Q0 + 3 * r3 : Rc + r3;
    const double* B = g3 == 0 ? Rc + c3 : g3 == 1 ? S.R0 + c3 : S.R1 + 3 * c3;
    (g3 == 0 ? S.A0 : g3 == 1 ? S.QR : S.RcR1T)[e9] = dot3(0.0, A, g3 == 2 ? 3 : 1, B, g3 == 2 ? 1 : 3);
  } else if (lane < 30) {
    S.dr[lane - 27] = S.x1.r[lane - 27] - S.x0.r[lane - 27];
  }
  __syncwarp();
  if (lane < 18) {                   // QA = QR Rc, t1 = R0 rc, t2 = Q0^T c, Rc^T rc
    const int k = lane < 9 ? 0 : 1 + (lane - 9) / 3, i = (lane - 9) % 3;
    const double* A = k == 0 ? S.QR + 3 * r3 : k == 1 ? S.R0 + 3 * i : k == 2 ? S.Q0 + i : Rc + i;
    const double* B = k == 0 ? Rc + c3 : k == 2 ? S.c : sp.r_CS;
    double* out = k == 0 ? S.QA + e9 : k == 1 ? S.t1 + i : k == 2 ? S.t2c + i : S.rcS + i;
    *out = dot3(0.0, A, k < 2 ? 1 : 3, B, k == 0 ? 3 : 1);
  } else if (lane < 27) {
    S.Jyr[r3][c3] = T * S.Q0[3 * c3 + r3];                    // position by velocity: T Q0^T
  }
  __syncwarp();
  if (lane < 9) {                    // position by gravity: Q0^T [c]x, first two columns
    const double v = mhat_e(S.Q0, true, S.c, lane);
    if (lane % 3 < 2) S.Jyr[lane / 3][9 + lane % 3] = v;
  } else if (lane >= 18 && lane < 21) {
    const int i = lane - 18;
    S.base[i] = ((S.x0.r[i] + S.t1[i]) + S.t2c[i]) - S.x1.r[i];
  } else if (lane >= 21 && lane < 27) {
    const int i = lane - 21;
    S.eb[i] = i < 3 ? S.x0.bg[i] - S.x1.bg[i] : S.x0.ba[i - 3] - S.x1.ba[i - 3];
  } else if (lane >= 27 && lane < 30) {
    const int i = lane - 27;         // velocity error without its pre-integrated part
    S.evb[i] = fma(i == 2 ? -sp.g : 0.0, T, S.x0.v[i]) - S.x1.v[i];
  }
  fill_pixel_maps(S, S.R0, S.Rref, S.dr);
  __syncwarp();
}

// x1's gravity in closed form; warp 6.  e_g = log(Q0 Q1^T), its Jacobians
// A = Jl^-1 (x0) and B = -Jr^-1 (x1), two columns each; n the unit normal of B's
// range: the remaining row is a = A^T n with value s = n . e_g, and
// dg1 = -Gm (e_g + A dg0) with Gm = (B^T B)^-1 B^T.
__device__ void fast_gravity(FastSmem& S, bool gyro) {
  const int lane = threadIdx.x & 31;
  {
    const int k = lane & 3;
    const double a[4] = {S.x0.qg[0], S.x0.qg[1], S.x0.qg[2], S.x0.qg[3]};
    double o = quat_mul_k(a, S.x1.qg, k, true);
    const double w = __shfl_sync(0xffffffffu, o, lane & ~3);
    if (__double2hiint(w) < 0) o = -o;
    double s2 = k ? o * o : 0.0;
    s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 2);
    const double f = pos_less(s2, 1e-6) ? 2.0 * fma(s2, fma(s2, 3.0 / 40, 1.0 / 6), 1.0) : quat_log_factor(s2, fabs(w));
    if (lane > 0 && lane < 4) S.eg[lane - 1] = f * o;
  }
  __syncwarp();
  if (lane < 18) (lane < 9 ? S.Jlg : S.Jrg)[lane % 9] = fast_jlinv_e(S.eg, lane < 9 ? 1.0 : -1.0, lane % 9);
  __syncwarp();
  const double* B = S.Jrg;           // B = -Jrg; column m of row k at 3 k + m
  if (lane < 3) {                    // cross product of B's columns (the signs cancel)
    const int i1 = lane == 2 ? 0 : lane + 1, i2 = lane == 0 ? 2 : lane - 1;
    S.nv[lane] = fma(B[3 * i1], B[3 * i2 + 1], -(B[3 * i2] * B[3 * i1 + 1]));
  } else if (lane < 6) {             // m00, m01, m11
    const int p = lane == 5 ? 1 : 0, q = lane == 3 ? 0 : 1;
    S.mm[lane - 3] = fma(B[p], B[q], fma(B[3 + p], B[3 + q], B[6 + p] * B[6 + q]));
  } else if (lane < 12) {
    S.Ag[lane - 6] = S.Jlg[3 * ((lane - 6) >> 1) + ((lane - 6) & 1)];
  }
  __syncwarp();
  const double n2 = fma(S.nv[0], S.nv[0], fma(S.nv[1], S.nv[1], S.nv[2] * S.nv[2]));
  const double inv = rsqrt(n2);
  if (lane < 3) {
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) v = fma(S.nv[k], lane < 2 ? S.Jlg[3 * k + lane] : S.eg[k], v);
    v = gyro ? 0.0 : v * inv;
    if (lane < 2) S.a[lane] = v;
    else S.s = v, S.a[2] = 0.0;
  } else if (lane < 9) {             // Gm row m, column k; 1 / det(B^T B) = 1 / |n|^2 (Lagrange's identity)
    const int m = (lane - 3) / 3, k = (lane - 3) % 3;
    const double b0 = -B[3 * k], b1 = -B[3 * k + 1];
    const double v = m == 0 ? fma(S.mm[2], b0, -(S.mm[1] * b1)) : fma(S.mm[0], b1, -(S.mm[1] * b0));
    S.Gm[3 * m + k] = gyro ? 0.0 : v * (inv * inv);
  }
  __syncwarp();
}

// Prior at x0: d = x0 boxminus xbar, the mean m = P b_y - d_y + K d_p of y and the
// prior vector b_p' - H_pp' d_p on p0; warp 7.  d_v, d_ba, d_g are held in the
// gyro-only variant.
__device__ void fast_prior(FastSmem& S, bool gyro) {
  const int lane = threadIdx.x & 31;
  warp_state_boxminus(S.x0, S.xbar, S.d);
  const double* K = S.el + kElK;
  const double* Hp = S.el + kElHp;
  if (lane < 17) {
    const bool y = lane < 11;
    const int i = y ? lane : lane - 11;
    double v = y ? S.el[kElM0 + i] - S.d[6 + i] : S.el[kElBp + i];
#pragma unroll
    for (int k = 0; k < 6; ++k) v = fma(y ? K[6 * i + k] : -Hp[6 * i + k], S.d[k], v);
    if (y && gyro && (i < 3 || i >= 6)) v = 0.0;
    (y ? S.m : S.bp)[i] = v;
  }
  __syncwarp();
}

// ---- the pixel terms (warps 4-7) ------------------------------------------------

// P12 (lower triangle) and g12: U = w C H_loc for both terms, then U C^T.
__device__ void fast_pixel_terms(const SolveParams& sp, const Ctrl* c, PixSmem& S) {
  const int t = threadIdx.x - 128;
  if (t < kSumsAll) S.sums[t] = __ldcg(c->sums + t);
  bar_sync<3, 128>();
  if (t < 126) {
    const int i = t / 7, q = t - 7 * i;
    const bool icp = i >= 12;
    const double* s = S.sums + (icp ? 0 : kSums);
    const double w = icp ? sp.W_icp : sp.W_rgb;
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int lo = min(k, q), hi = max(k, q);
      const double h = q == 6 ? s[21 + k] : s[lo * 6 - lo * (lo - 1) / 2 + (hi - lo)];
      v = fma(S.C[i][k], h, v);
    }
    S.U[i][q] = w * v;
  }
  bar_sync<3, 128>();
  if (t < 78) {
    int i = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while (tri(i + 1, 0) <= t) ++i;
    while (tri(i, 0) > t) --i;
    const int j = t - tri(i, 0);
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) v = fma(S.U[i][k], S.C[j][k], v);
    if (j >= 6) {                    // the block-diagonal ICP map: three columns of a row
      const int b = j < 9 ? 0 : 3;
#pragma unroll
      for (int k = 0; k < 3; ++k) v = fma(S.U[i + 6][b + k], S.C[j + 6][b + k], v);
    }
    S.P12[i * kPose + j] = v;
  } else if (t >= 96 && t < 96 + kPose) {
    const int i = t - 96;
    S.g12[i] = i < 6 ? -S.U[i][6] : -(S.U[i][6] + S.U[i + 6][6]);
  }
}

// ---- the sweep ---------------------------------------------------------------------

// q <- exp(d) (x) q of two quaternions by one warp, as in warp_state_boxplus: (q0, d0) on
// lanes 0-3 and (q1, d1) on lanes 4-7 (flat: the third component of d taken as zero).
// The series of a quaternion's four components run on its four lanes (cosine on the
// first, sine on the others), cut where the next term is below 1e-17 for small steps.
__device__ __forceinline__ void fast_quat_boxplus(double* q0, const double* d0, bool flat0, double* q1,
                                                  const double* d1, bool flat1) {
  const int lane = threadIdx.x & 31, grp = (lane >> 2) & 1, k = lane & 3, base = lane & ~3;
  double* q = grp ? q1 : q0;
  const double* d = grp ? d1 : d0;
  const double dx = d[0], dy = d[1], dz = (grp ? flat1 : flat0) ? 0.0 : d[2];
  const double t2 = fma(dx, dx, fma(dy, dy, dz * dz));
  double f;
  if (__all_sync(0xffffffffu, pos_less(t2, 1e-6))) {
    f = fma(t2, fma(t2, k ? 1.0 / 3840 : 1.0 / 384, k ? -1.0 / 48 : -1.0 / 8), k ? 0.5 : 1.0);
  } else if (__all_sync(0xffffffffu, pos_less(t2, kSeriesT2))) {
    const double c4 = k ? 1.0 / 185794560 : 1.0 / 10321920, c3 = k ? -1.0 / 645120 : -1.0 / 46080;
    const double c2 = k ? 1.0 / 3840 : 1.0 / 384, c1 = k ? -1.0 / 48 : -1.0 / 8;
    f = fma(t2, fma(t2, fma(t2, fma(t2, c4, c3), c2), c1), k ? 0.5 : 1.0);
  } else {
    const double t = sqrt(t2);
    double sn, cs;
    sincos(0.5 * t, &sn, &cs);
    f = k ? (t2 > 0.0 ? sn / t : 0.5) : cs;
  }
  f *= k == 0 ? 1.0 : k == 1 ? dx : k == 2 ? dy : dz;
  double o = 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {      // component k of exp(d) (x) q, as quat_mul_k
    const double e = __shfl_sync(0xffffffffu, f, base + j);
    o = fma(((0x428E >> (4 * k + j)) & 1) ? -e : e, q[k ^ j], o);
  }
  double n2 = o * o;
  n2 += __shfl_xor_sync(0xffffffffu, n2, 1);
  n2 += __shfl_xor_sync(0xffffffffu, n2, 2);
  if (__all_sync(0xffffffffu, fabs(__double2float_rn(n2) - 1.f) < 1e-6f)) o *= fma(-0.5, n2, 1.5);
  else o *= rsqrt(n2);
  __syncwarp();
  if (lane < 8) q[k] = o;
  __syncwarp();
}

// x <- x boxplus d by one warp, as warp_state_boxplus.
__device__ __forceinline__ void fast_boxplus(DState& x, const double* d) {
  const int lane = threadIdx.x & 31;
  fast_quat_boxplus(x.q, d + 3, false, x.qg, d + 15, true);
  if (lane < 12) {
    const int g = lane / 3, i = lane - 3 * g;
    double* v = g == 0 ? x.r : g == 1 ? x.v : g == 2 ? x.bg : x.ba;
    v[i] += d[(g == 0 ? 0 : 3 + 3 * g) + i];
  }
  __syncwarp();
}

// The pixel kernel's transforms, as warp_write_transforms, from shared memory; one warp.
__device__ __forceinline__ void fast_transforms(Ctrl* c, FastSmem& S) {
  const int lane = threadIdx.x & 31, f = lane / 9, e = lane - 9 * f, r = e / 3, cc = e - 3 * r;
  if (lane < 24) {                    // R1, R0 (2 (v_r v_c + w^2 or +- w v_k) - I); r1 - r_ref, r1 - r0
    const double* q = f == 0 ? S.x1.q : S.x0.q;
    const bool rot = lane < 18, diag = r == cc, icp = lane < 21;
    const int i = (lane - 18) % 3;
    const double w = q[0], vk = diag ? w : q[4 - r - cc];
    const double x = rot ? w * ((((cc - r + 3) % 3) == 1) ? -vk : vk) : icp ? -S.rref[i] : -S.x0.r[i];
    const double h = fma(rot ? q[1 + r] : S.x1.r[i], rot ? q[1 + cc] : 1.0, x);
    S.rot[lane] = rot ? fma(2.0, h, diag ? -1.0 : 0.0) : h;
  }
  __syncwarp();
  const double* R1 = S.rot;
  const double* R0 = S.rot + 9;
  if (lane < 24) {
    const bool rot = lane < 18, icp = rot ? f == 0 : lane < 21;
    const int i = rot ? r : (lane - 18) % 3;
    const double* M = (icp ? S.Rref : R0) + i;                // column i: row i of the transpose
    const double* B = rot ? R1 + cc : S.rot + (icp ? 18 : 21);
    const double v = dot3(rot && r == cc ? -1.0 : 0.0, M, 3, B, rot ? 3 : 1);
    (icp ? c->xf_icp : c->xf_rgb)[rot ? e : 9 + i] = (float)v;
  }
}

// The step's loads from the control block, issued before anything else (the block's
// pointer comes with the launch's arguments): status, whether the frame's constants
// allow the covariance form, and the number of IMU pieces in registers, the rest to
// shared memory.
struct FastLoad {
  int status, usable, np;
};
__device__ __forceinline__ FastLoad fast_load(const Ctrl* c, FastSmem& S) {
  const int tid = threadIdx.x;
  const FastLoad r = {c->status, c->elim.ok, c->elim.np};
  const double* e = c->elim.m;
  const double* p = &c->elim.piece[0][0];
  double* q = &S.piece[0][0];
  double v[4];
  v[0] = p[tid];
  v[1] = p[tid + kSolveThreads];
  v[2] = e[tid];
  v[3] = 0.0;
  static_assert(kElimPieces * 8 == 2 * kSolveThreads && kElimDoubles - kSolveThreads == 40, "load layout");
  const double* src = tid < 20 ? reinterpret_cast<const double*>(&c->x0) + tid
                      : tid < 40 ? reinterpret_cast<const double*>(&c->x1) + tid - 20
                      : tid < 60 ? reinterpret_cast<const double*>(&c->xbar) + tid - 40
                      : tid < 69 ? c->Rref + tid - 60
                      : tid < 109 ? e + kSolveThreads + tid - 69
                      : tid < 112 ? c->rref + tid - 109 : nullptr;
  double* dst = tid < 20 ? reinterpret_cast<double*>(&S.x0) + tid
                : tid < 40 ? reinterpret_cast<double*>(&S.x1) + tid - 20
                : tid < 60 ? reinterpret_cast<double*>(&S.xbar) + tid - 40
                : tid < 69 ? S.Rref + tid - 60
                : tid < 109 ? S.el + kSolveThreads + tid - 69 : S.rref + tid - 109;
  if (src) v[3] = *src;
  q[tid] = v[0];
  q[tid + kSolveThreads] = v[1];
  S.el[tid] = v[2];
  if (src) *dst = v[3];
  return r;
}

// One Gauss-Newton step on what fast_load brought; false (for every thread, nothing
// done) when the frame's constants do not allow this form.  Whole block.
__device__ bool gn_step_fast(const SolveParams& sp, FastSmem& S, Ctrl* c, const FastLoad& fl) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool gyro = sp.track_mode == DRI_TRACK_GYRO_ONLY;
  const int np = fl.np;
  if (fl.status != 0) return true;
  if (!fl.usable) return false;
  // the sweep's entries of this thread (see there): entry e of the lower triangle
  // and the right-hand side row, longest-updated first, and where its value comes
  // from: sign (*p + *q)
  int ei[2], ej[2];
  const double *ep[2], *eq[2];
  bool eneg[2];
#pragma unroll
  for (int o = 0; o < 2; ++o) {
    const int e = tid + 128 * o;
    ei[o] = ej[o] = -1;
    ep[o] = eq[o] = &S.zero;
    eneg[o] = false;
    if (warp < 4 && e < kSysEnt) {    // column j = 18 - g holds rows j .. 19 (19: right-hand side): g + 2 entries
      int g = (int)((sqrtf(9.0f + 8.0f * e) - 3.0f) * 0.5f);
      if (g * (g + 3) / 2 > e) --g;
      if ((g + 1) * (g + 4) / 2 <= e) ++g;
      ej[o] = kSys - 1 - g;
      ei[o] = ej[o] + e - g * (g + 3) / 2;
      const int i = ei[o], j = ej[o];
      if (i < kLam) {                 // -(S + blockdiag(S6, sigma_g^2))
        ep[o] = S.S + tri(i, j);
        eneg[o] = true;
        if (i < 6) eq[o] = S.el + kElS6 + 6 * i + j;
        else if (i == j) eq[o] = S.el + kElSg;
      } else if (j < kLam) {          // J', -e'
        ep[o] = i == kSys ? S.ep + j : &S.Jp[j][i - kLam];
        eneg[o] = i == kSys;
      } else if (i == kSys) {         // the prior on p0
        if (j < kLam + 6) ep[o] = S.bp + j - kLam;
      } else if (i < kLam + 6) {
        ep[o] = S.el + kElHp + 6 * (i - kLam) + j - kLam;
      }
    }
  }
  if (tid == 0) {
    S.one = 1.0;
    S.zero = 0.0;
  }
  // J' on p1: -I for the position rows, zero where the rotation rows do not write
  if (warp == 4)
    for (int idx = lane; idx < 42; idx += 32) {
      const int i = idx / 6, k = idx - 6 * i;
      if (i < 3 || i == 6 || k < 3) S.Jp[i][6 + k] = (i < 3 && k == i && !gyro) ? -1.0 : 0.0;
    }
  __syncthreads();
  const double* root = nullptr;
  if (warp < 4) {
    if (sp.imu_mode == DRI_IMU_FIRST_ORDER) {
      root = fast_first_order(sp, c, S, np);
    } else {
      fast_leaves(S, np, S.x0.bg, S.x0.ba);
      root = fast_tree(S, np);
    }
  } else if (warp == 5) {
    fast_state_terms(sp, S);
  } else if (warp == 6) {
    fast_gravity(S, gyro);
  } else if (warp == 7) {
    fast_prior(S, gyro);
  }
  __syncthreads();
  const double* Py = S.el + kElPy;
  const double* K = S.el + kElK;
  if (warp >= 4) {                    // the pixel kernel's sums
    grid_dep_wait();
    fast_pixel_terms(sp, c, S);
    bar_arrive<4, 256>();             // P12, g12 to the sweep
    if (warp == 7) {                  // IMU cost at this linearisation: e^T W e
      bar_sync<7, 160>();             // the errors (warps 0-3)
      double v = 0.0;
      if (lane < 18) {
        auto err = [&](int i) {
          return i < 3 ? S.er[i] : i < 6 ? S.ea[i - 3] : i < 9 ? S.ev[i - 6] : i < 15 ? S.eb[i - 9] : S.eg[i - 15];
        };
        const double* W = c->Wimu + lane * 18;
        if (lane < 9) {
          for (int k = 0; k < 9; ++k) v = fma(W[k], err(k), v);
          v *= err(lane);
        } else {
          v = W[lane] * err(lane) * err(lane);
        }
      }
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) S.cost = v;
    }
  } else {
    // ---- IMU rows ----
    if (warp == 0) {
      const int f = lane / 9, e9 = lane - 9 * f, r = f == 3 ? e9 : e9 / 3, cc = f == 3 ? 0 : e9 - 3 * r;
      if (lane < 30) {                // A0 times R, Pa (position by b_a), P, p
        const double* B = root + (f == 0 ? kNR : f == 1 ? kNPa : f == 2 ? kNP : kNp) + cc;
        double* out = f == 0 ? S.RW + e9 : f == 1 ? &S.Jyr[r][6 + cc] : f == 2 ? S.APg + e9 : S.t3 + e9;
        *out = dot3(0.0, S.A0 + 3 * r, 1, B, f == 3 ? 1 : 3);
      }
      __syncwarp();
      if (lane < 21) {                // R_WS1 times Rc^T R1^T, Phi, Rc^T rc
        const int rr = f == 2 ? e9 : r;
        const double* B = f == 0 ? S.RcR1T + cc : f == 1 ? root + kNPhi + cc : S.rcS;
        double* out = f == 0 ? S.M + e9 : f == 1 ? S.RP + e9 : S.t4 + e9;
        *out = dot3(0.0, S.RW + 3 * rr, 1, B, f == 2 ? 1 : 3);
      }
      __syncwarp();
      if (lane < 15) {                // position by b_g: A0 P + [t4]x R_WS1 Phi; e_r; u = t1 + t3 - t4
        const int i = lane < 12 ? lane - 9 : lane - 12;
        const int r1 = r == 2 ? 0 : r + 1, r2 = r == 0 ? 2 : r - 1;
        const bool mat = lane < 9;
        const double x = mat ? S.APg[lane] : lane < 12 ? S.base[i] : S.t1[i];
        const double y1 = mat ? S.t4[r1] : 1.0, z1 = mat ? S.RP[3 * r2 + cc] : S.t3[i];
        const double y2 = mat ? S.t4[r2] : 1.0, z2 = mat ? S.RP[3 * r1 + cc] : S.t4[i];
        double* out = mat ? &S.Jyr[r][3 + cc] : lane < 12 ? S.er + i : S.u + i;
        *out = fma(-y2, z2, fma(y1, z1, x));
      }
      __syncwarp();
      if (gyro) {                     // the position rows carry no weight: no information
        for (int i = lane; i < 33; i += 32) S.Jyr[i / 11][i % 11] = 0.0;
        __syncwarp();
      }
      bar_arrive<8, 96>();            // the position rows to warps 1 and 2
      // e_a = log(M): the skew part v = 2 sin(t) k, t / (2 sin t) from its series in
      // sin^2 t (the angle is below 6.4 mrad in all but a frame's first iterations)
      double ea;
      {
        const int i = lane % 3, i1 = i == 2 ? 0 : i + 1, i2 = i == 0 ? 2 : i - 1;
        const double v = 0.5 * (S.M[3 * i2 + i1] - S.M[3 * i1 + i2]);
        const double v0 = __shfl_sync(0xffffffffu, v, 0), v1 = __shfl_sync(0xffffffffu, v, 1),
                     v2 = __shfl_sync(0xffffffffu, v, 2);
        const double s2 = fma(v0, v0, fma(v1, v1, v2 * v2));
        const float tr = (float)S.M[0] + (float)S.M[4] + (float)S.M[8];
        if (pos_less(s2, 4e-5) && tr > 2.f) ea = v * fma(s2, fma(s2, fma(s2, 5.0 / 112, 3.0 / 40), 1.0 / 6), 1.0);
        else ea = log_i(S.M, i);
      }
      if (lane < 3) S.ea[lane] = ea;
      __syncwarp();
      if (lane < 18) {                // Jl^-1(e_a), and -Jr^-1(e_a) into J' on p1
        const double v = fast_jlinv_e(S.ea, lane < 9 ? 1.0 : -1.0, e9);
        if (lane < 9) S.Jla[e9] = v;
        else S.Jp[3 + r][9 + cc] = -v;
      }
      __syncwarp();
      if (lane < 9) S.B13[lane] = dot3(0.0, S.Jla + 3 * r, 1, S.RP + cc, 3);
    } else if (warp == 3) {           // velocity rows, used for dv1 only
      const int f = lane / 9, e9 = lane - 9 * f, r = f < 2 ? e9 / 3 : e9 % 3, cc = f < 2 ? e9 - 3 * r : 0;
      if (lane < 24) {                // QA V, QA Va, A0 v, QA v
        const double* A = (f == 2 && e9 < 3 ? S.A0 : S.QA) + 3 * r;
        const double* B = root + (f == 0 ? kNV : f == 1 ? kNVa : kNv) + cc;
        double* out = f == 0 ? S.B14 + e9 : f == 1 ? S.B17 + e9 : e9 < 3 ? S.w9 + r : S.t5 + r;
        *out = dot3(0.0, A, 1, B, f == 2 ? 1 : 3);
      }
      __syncwarp();
      if (lane < 12) {                // -Q0 [w9]x, e_v
        const int c1 = cc == 2 ? 0 : cc + 1, c2 = cc == 0 ? 2 : cc - 1, i = lane - 9;
        const bool mat = lane < 9;
        const double x = mat ? 0.0 : S.evb[i];
        const double y1 = mat ? S.Q0[3 * r + c1] : 0.0, z1 = mat ? S.w9[c2] : 0.0;
        const double y2 = mat ? S.Q0[3 * r + c2] : 1.0, z2 = mat ? S.w9[c1] : S.t5[i];
        *(mat ? S.B9 + lane : S.ev + i) = fma(y2, z2, fma(-y1, z1, x));
      } else if (lane < 21) {
        const int q = lane - 12;
        if (q % 3 < 2) S.B20[2 * (q / 3) + q % 3] = -hat_e(S.t5, q);
      }
    }
    if (warp == 1 || warp == 2) {     // position rows: Jy P, Jp + Jy K, e + Jy m
      bar_sync<8, 96>();
      const int q = lane - 11;
      const int r = warp == 1 ? lane / 11 : lane < 11 ? 2 : lane < 29 ? q / 6 : lane - 29;
      const int cc = warp == 1 ? lane - 11 * r : lane < 11 ? lane : lane < 29 ? q - 6 * r : 0;
      const double* B = (warp == 1 || lane < 11) ? Py + cc : lane < 29 ? K + cc : S.m;
      const int sb = (warp == 1 || lane < 11) ? 11 : lane < 29 ? 6 : 1;
      if (warp == 2 || lane < 22) {
        double v = 0.0;
        if (warp == 2 && lane >= 29) v = gyro ? 0.0 : S.er[r];
        else if (warp == 2 && lane >= 11 && !gyro) v = cc < 3 ? (cc == r ? 1.0 : 0.0) : -hat_e(S.u, 3 * r + cc - 3);
#pragma unroll
        for (int k = 0; k < 11; ++k) v = fma(S.Jyr[r][k], B[k * sb], v);
        if (warp == 1 || lane < 11) S.T[r][cc] = v;
        else if (lane < 29) S.Jp[r][cc] = v;
        else S.ep[r] = v;
      }
      bar_sync<6, 64>();
      if (warp == 1 && lane < 6) {
        const int i = lane < 1 ? 0 : lane < 3 ? 1 : 2, j = lane - tri(i, 0);
        double v = 0.0;
#pragma unroll
        for (int k = 0; k < 11; ++k) v = fma(S.T[i][k], S.Jyr[j][k], v);
        S.S[tri(i, j)] = v;
      }
    }
    if (warp < 3) {
      bar_sync<5, 96>();
      // rotation rows (their only y column block is b_g: B13) and the gravity row
      if (warp == 0) {
        const int i = lane / 3, j = lane - 3 * i;
        const bool rot = lane < 9;    // S between the rotation and position rows; else the gravity row
        const double* A = rot ? S.B13 + 3 * i : S.a;
        const double* B;
        double* out;
        int sb = 1;
        double base = 0.0;
        if (rot) {
          B = &S.T[j][3];
          out = S.S + tri(3 + i, j);
        } else if (lane < 20) {
          B = Py + 9 * 11 + lane - 9;
          sb = 11;
          out = &S.T[6][lane - 9];
        } else if (lane < 23) {
          B = &S.T[lane - 20][9];
          out = S.S + tri(6, lane - 20);
        } else if (lane < 29) {
          B = K + 9 * 6 + lane - 23;
          sb = 6;
          out = &S.Jp[6][lane - 23];
        } else {
          B = S.m + 9;
          out = S.ep + 6;
          base = S.s;
        }
        const double v = dot21(base, A, B, sb, rot ? A + 2 : &S.zero, rot ? B + 2 : &S.zero);
        if (lane < 30) *out = v;
      } else {
        const int q = lane - 11;
        const int r = warp == 1 ? lane / 11 : lane < 11 ? 2 : lane < 29 ? q / 6 : lane - 29;
        const int cc = warp == 1 ? lane - 11 * r : lane < 11 ? lane : lane < 29 ? q - 6 * r : 0;
        const double* B = (warp == 1 || lane < 11) ? Py + 33 + cc : lane < 29 ? K + 18 + cc : S.m + 3;
        const int sb = (warp == 1 || lane < 11) ? 11 : lane < 29 ? 6 : 1;
        if (warp == 2 || lane < 22) {
          double v = 0.0;
          if (warp == 2 && lane >= 29) v = S.ea[r];
          else if (warp == 2 && lane >= 11 && cc >= 3) v = S.Jla[3 * r + cc - 3];
#pragma unroll
          for (int k = 0; k < 3; ++k) v = fma(S.B13[3 * r + k], B[k * sb], v);
          if (warp == 1 || lane < 11) S.T[3 + r][cc] = v;
          else if (lane < 29) S.Jp[3 + r][cc] = v;
          else S.ep[3 + r] = v;
        }
      }
      bar_sync<5, 96>();
      if (warp == 1 && lane < 10) {   // S of the rotation rows; the gravity row against them and itself
        const bool rot = lane < 6;
        const int i = lane < 1 ? 0 : lane < 3 ? 1 : 2, j = rot ? lane - tri(i, 0) : lane - 3;
        const double* A = rot ? &S.T[3 + i][3] : S.a;
        const double* B = rot ? S.B13 + 3 * j : &S.T[j][9];
        const double v = dot21(0.0, A, B, 1, rot ? A + 2 : &S.zero, rot ? B + 2 : &S.zero);
        S.S[rot ? tri(3 + i, 3 + j) : tri(6, j)] = v;
      }
    }
    bar_arrive<7, 160>();
    bar_sync<1, 128>();
    // ---- the sweep: the entries are dealt to the four warps in 32-entry chunks in
    // turn, longest-updated first, so that the entries a pivot still updates take
    // the fewest warp instructions: the second slot's 81 entries have columns 0..4
    // and are done after pivot 3 ----
    double v[2], rown[2] = {0.0, 0.0};
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const double x = *ep[o] + *eq[o];
      v[o] = eneg[o] ? -x : x;
    }
    // Pivot k (slots 0 .. O - 1): its column is published behind one barrier; the
    // products c_i c_j are taken while the reciprocal's seed is formed on the integer
    // and FP32 pipes.  No branches: a lane without a column entry writes to its sink
    // word, one whose entry is done keeps its value.
    auto pivot = [&](int k, bool neg, auto slots) {
      constexpr int O = decltype(slots)::value;
      double* cb = S.col[k & 1];
#pragma unroll
      for (int o = 0; o < O; ++o) *(ej[o] == k ? cb + ei[o] : S.sink + tid) = v[o];
      bar_sync<1, 128>();
      const double d = cb[k];
      double t[O];
#pragma unroll
      for (int o = 0; o < O; ++o) t[o] = cb[max(ei[o], 0)] * cb[max(ej[o], 0)];
      const double r = pivot_recip(neg ? -d : d);             // 1 / |d|
#pragma unroll
      for (int o = 0; o < O; ++o) {
        const double w = fma(neg ? t[o] : -t[o], r, v[o]);
        v[o] = ej[o] > k ? w : v[o];
        rown[o] = ej[o] == k ? (neg ? -r : r) : rown[o];
      }
    };
#pragma unroll 1
    for (int k = 0; k < 5; ++k) pivot(k, true, Slots<2>());
#pragma unroll 1
    for (int k = 5; k < kLam; ++k) pivot(k, true, Slots<1>());
    grid_dep_wait();
    bar_sync<4, 256>();               // the pixel terms join the pose block (slot 0's columns)
    {
      const int i = ei[0], j = ej[0];
      if (j >= kLam) v[0] += i == kSys ? S.g12[j - kLam] : S.P12[(i - kLam) * kPose + j - kLam];
    }
#pragma unroll 1
    for (int k = kLam; k < kSys; ++k) pivot(k, false, Slots<1>());
    // unit-lower L, its row 19 holding z_k / d_k; the pivots' signs
    bool posdef = true;
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      if (ei[o] > ej[o]) S.L[ej[o]][ei[o]] = v[o] * rown[o];
      if (ei[o] >= 0 && ei[o] == ej[o]) {
        const bool neg = __double2hiint(v[o]) < 0;
        posdef = posdef && finite_bits(v[o]) && v[o] != 0.0 && neg == (ei[o] < kLam);
      }
    }
    posdef = __all_sync(0xffffffffu, posdef);
    if (lane == 0) S.posdef[warp] = posdef;
    bar_sync<1, 128>();
    // The poses are known after 12 of the 19 substitutions: warp 1 moves them and writes
    // the next pixel kernel's transforms while warp 0 goes on to the other unknowns.
    double* dx = S.dx;
    if (warp == 0) {
      const double* Lr = S.L[min(lane, kSys - 1)];
      double y = Lr[kSys], l = Lr[kSys - 1];
      auto substitute = [&](int from, int to) {
#pragma unroll 1
        for (int k = from; k > to; --k) {                     // the next column's entry loads a step ahead
          const double ln = Lr[k - 1];
          y = fma(lane < k ? -l : 0.0, __shfl_sync(0xffffffffu, y, k), y);
          l = ln;
        }
      };
      substitute(kSys - 1, kLam);
      if (lane >= kLam && lane < kSys) {
        S.z[lane] = y;
        dx[lane < kLam + 6 ? lane - kLam : 4 + lane] = y;     // p0 at 0..5, p1 at 17..22
      }
      __syncwarp();
      bar_arrive<9, 64>();
      substitute(kLam, 0);
      if (lane < kLam) S.z[lane] = y;
      __syncwarp();
      // y (lanes 0-10: K p0 + m, 16-26: -T^T lambda), dv1's part without y
      // (11-13: e_v + B9 da0, 27-29: -S_v6 lambda)
      const double* lam = S.z;
      const double* p0 = S.z + kLam;
      const int h = lane & 15;
      const bool top = lane >= 16;
      double w = 0.0;
      if (h < 14) {
        const double* A = h < 11 ? (top ? &S.T[0][h] : K + 6 * h) : (top ? S.el + kElSv + 6 * (h - 11) : S.B9 + 3 * (h - 11));
        const int sa = h < 11 && top ? 11 : 1;
        const double* B = top ? lam : (h < 11 ? p0 : p0 + 3);
        const int n = h < 11 ? (top ? 7 : 6) : (top ? 6 : 3);
        w = top ? 0.0 : h < 11 ? S.m[h] : S.ev[h - 11];
#pragma unroll
        for (int k = 0; k < 7; ++k)
          if (k < n) w = fma(top ? -A[k * sa] : A[k * sa], B[k], w);
      }
      w += __shfl_down_sync(0xffffffffu, w, 16);
      if (lane < 11) dx[6 + lane] = w;
      else if (lane < 14) S.u[lane - 11] = w;                 // dv1's part
      __syncwarp();
      {
        const double* yv = dx + 6;    // v, b_g, b_a, gravity
        // lanes 0-8: dv1, row lane % 3, part lane / 3; 9-14: x1's biases follow x0's;
        // 15-17: e_g + A dg0
        const int i = lane % 3, q = lane / 3;
        const double *A = &S.zero, *B = &S.zero, *A2 = &S.zero, *B2 = &S.zero;
        int sa = 0, sb = 0;
        double base = 0.0;
        if (lane < 9) {
          A = q == 0 ? S.B14 + 3 * i : q == 1 ? S.B17 + 3 * i : S.B20 + 2 * i;
          B = q == 0 ? yv + 3 : q == 1 ? yv + 6 : yv + 9;
          A2 = q == 2 ? &S.one : A + 2;
          B2 = q == 2 ? yv + i : B + 2;
          base = q == 2 ? S.u[i] : 0.0;
          sa = sb = 1;
        } else if (lane < 15) {
          A2 = &S.one;
          B2 = yv + 3 + lane - 9;
          base = S.eb[lane - 9];
        } else if (lane < 18) {
          A = S.Ag + 2 * i;
          B = yv + 9;
          base = S.eg[i];
          sa = sb = 1;
        }
        double w = fma(A[0], B[0], fma(A[sa], B[sb], fma(*A2, *B2, base)));
        if (gyro && lane >= 12 && lane < 15) w = 0.0;
        const double w1 = __shfl_down_sync(0xffffffffu, w, 3), w2 = __shfl_down_sync(0xffffffffu, w, 6);
        const double u0 = __shfl_sync(0xffffffffu, w, 15), u1 = __shfl_sync(0xffffffffu, w, 16),
                     u2 = __shfl_sync(0xffffffffu, w, 17);
        if (lane < 3) dx[23 + lane] = gyro ? 0.0 : (w + w1) + w2;
        else if (lane >= 9 && lane < 15) dx[26 + lane - 9] = w;
        else if (lane >= 18 && lane < 20) {
          const double* G = S.Gm + 3 * (lane - 18);
          dx[32 + lane - 18] = -fma(G[0], u0, fma(G[1], u1, G[2] * u2));
        }
      }
      __syncwarp();
      const bool fin = finite_bits(dx[lane]) && finite_bits(dx[32 + (lane & 1)]);
      const bool ok = __all_sync(0xffffffffu, fin) && S.posdef[0] && S.posdef[1] && S.posdef[2] && S.posdef[3];
      if (lane == 0) S.good = ok;
      fast_quat_boxplus(S.x0.qg, dx + 15, true, S.x1.qg, dx + 32, true);
      if (lane < 18) {                // velocities and biases
        const int q = lane / 9, i = lane - 9 * q, f = i / 3;
        DState& x = q ? S.x1 : S.x0;
        (f == 0 ? x.v : f == 1 ? x.bg : x.ba)[i - 3 * f] += dx[17 * q + 6 + i];
      }
    } else if (warp == 1) {
      bar_sync<9, 64>();
      fast_quat_boxplus(S.x0.q, dx + 3, false, S.x1.q, dx + 20, false);
      if (lane < 6) (lane < 3 ? S.x0.r : S.x1.r)[lane % 3] += dx[lane < 3 ? lane : 14 + lane];
      __syncwarp();
      fast_transforms(c, S);          // of no use to anyone should the step fail
    }
  }
  __syncthreads();
  if (!S.good) {
    if (tid == 0) c->status = DRI_ELOST;
    return true;
  }
  if (warp == 0) {
    if (lane < 20) reinterpret_cast<double*>(&c->x0)[lane] = reinterpret_cast<const double*>(&S.x0)[lane];
  } else if (warp == 2) {
    if (lane < 20) reinterpret_cast<double*>(&c->x1)[lane] = reinterpret_cast<const double*>(&S.x1)[lane];
  } else if (warp >= 4 && !sp.last) { // the next iteration's linearisation point
    if (tid < 148) reinterpret_cast<double*>(&c->xl0)[tid - 128] = reinterpret_cast<const double*>(&S.x0)[tid - 128];
    else if (tid < 168) reinterpret_cast<double*>(&c->xl1)[tid - 148] = reinterpret_cast<const double*>(&S.x1)[tid - 148];
  } else if (warp >= 4) {             // what the marginalisation needs of the last iteration
    if (tid < 162) c->d[tid - 128] = S.dx[tid - 128];
    else if (tid == 162) c->lin_split = 1;
  } else if (tid == 96) {
    c->n_icp[sp.level] = (int32_t)S.sums[28];
    c->n_rgb[sp.level] = (int32_t)S.sums[kSums + 28];
    store_margin(c, sp.level);
    c->cost = sp.W_icp * S.sums[27] + sp.W_rgb * S.sums[kSums + 27] + S.cost;
    c->iterations += 1;
  }
  return true;
}

// RGB-D-only baseline (DRI_TRACK_RGBD_ONLY): one Gauss-Newton step on x1's pose with
// H_icp + lambda H_rgb (x1's blocks of the two pixel systems in W), x0 fixed; x1's
// other components unchanged.  Whole block; what needs no pixel sum is done before the
// wait for the pixel kernel, and the 6 x 6 system (27 entries with its right-hand side)
// is swept by one warp without block barriers.  Against a block-wide factorisation
// with FP64 divisions and a one-thread substitution: 18 -> 12 us per step (with its launch),
// 501x377 camera 495 -> 361 us per frame.
__device__ void gn_step_pose_only(const SolveParams& sp, FastSmem& S, Ctrl* c, const FastLoad& fl) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (fl.status != 0) return;
  // C: diag(R0, R0) (photometric, rows 0-5) and diag(R_ref, R_ref) (ICP, rows 6-11)
  if (tid < 9) S.R0[tid] = quat_rot_e(S.x0.q, tid);
  __syncwarp();
  if (warp == 0)
    for (int idx = lane; idx < 72; idx += 32) {
      const int i = idx / 6, k = idx - 6 * i, r = i % 6;
      S.C[i][k] = r / 3 == k / 3 ? (i < 6 ? S.R0 : S.Rref)[3 * (r % 3) + k % 3] : 0.0;
    }
  grid_dep_wait();                    // the pixel sums
  if (tid < kSumsAll) S.sums[tid] = __ldcg(c->sums + tid);
  __syncthreads();
  if (tid < 84) {                     // U = w C H_loc, and w C b_loc in column 6
    const int i = tid / 7, q = tid - 7 * i, b = (i % 6) / 3 * 3;
    const double* s = S.sums + (i < 6 ? kSums : 0);
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int lo = min(b + k, q), hi = max(b + k, q);
      const double h = q == 6 ? s[21 + b + k] : s[lo * 6 - lo * (lo - 1) / 2 + (hi - lo)];
      v = fma(S.C[i][b + k], h, v);
    }
    S.U[i][q] = v * (i < 6 ? sp.rgbd_lambda * sp.W_rgb : sp.W_icp);
  }
  __syncthreads();
  if (warp == 0) {
    int i = -1, j = -1;               // lower triangle by columns, then row 6: the right-hand side
    double v = 0.0;
    if (lane < 21) {
      i = (int)((sqrtf(8.f * lane + 1.f) - 1.f) * 0.5f);
      if (tri(i + 1, 0) <= lane) ++i;
      if (tri(i, 0) > lane) --i;
      j = lane - tri(i, 0);
      const int b = j / 3 * 3;
#pragma unroll
      for (int k = 0; k < 3; ++k) v = fma(S.U[i][b + k], S.C[j][b + k], fma(S.U[6 + i][b + k], S.C[6 + j][b + k], v));
    } else if (lane < 27) {
      i = 6;
      j = lane - 21;
      v = -(S.U[j][6] + S.U[6 + j][6]);
    }
    double rown = 0.0;
#pragma unroll 1
    for (int k = 0; k < 6; ++k) {
      double* cb = S.col[k & 1];
      *(j == k ? cb + i : S.sink + lane) = v;
      __syncwarp();
      const double t = cb[max(i, 0)] * cb[max(j, 0)];
      const double r = pivot_recip<true>(cb[k]);
      const double w = fma(-t, r, v);
      v = j > k ? w : v;
      rown = j == k ? r : rown;
    }
    if (i > j) S.L[j][i] = v * rown;
    bool good = !(i >= 0 && i == j) || (finite_bits(v) && v != 0.0 && __double2hiint(v) > 0);
    __syncwarp();
    const double* Lr = S.L[min(lane, 5)];
    double y = Lr[6];
#pragma unroll 1
    for (int k = 5; k > 0; --k) y = fma(lane < k ? -Lr[k] : 0.0, __shfl_sync(0xffffffffu, y, k), y);
    if (lane < 17) S.dx[lane] = lane < 6 ? y : 0.0;
    good = __all_sync(0xffffffffu, good && (lane >= 6 || finite_bits(y)));
    __syncwarp();
    if (!good) {
      if (lane == 0) c->status = DRI_ELOST;
      return;
    }
    fast_boxplus(S.x1, S.dx);
    fast_transforms(c, S);
    if (lane < 20) reinterpret_cast<double*>(&c->x1)[lane] = reinterpret_cast<const double*>(&S.x1)[lane];
    if (lane == 31) {
      const double* s = S.sums;
      c->n_icp[sp.level] = (int32_t)s[28];
      c->n_rgb[sp.level] = (int32_t)s[kSums + 28];
      store_margin(c, sp.level);
      c->cost = sp.W_icp * s[27] + sp.rgbd_lambda * sp.W_rgb * s[kSums + 27];
      c->iterations += 1;
    }
  }
}

// ---- the frame's constants (k_frame_begin) -----------------------------------------

// Entry (i, j) of a symmetric matrix after the sweep operator on index k: -1 / d on the
// pivot, a / d in its row and column, a - c_i c_j / d elsewhere; c: column k, r = 1 / d.
// Swept over an index set Y, the matrix holds -(A_YY)^-1, (A_YY)^-1 A_Y. and the Schur
// complement.
__device__ __forceinline__ double sweep_entry(int i, int j, int k, double v, const double* c, double r) {
  const double t = c[max(i, 0)] * c[max(j, 0)];
  const bool ik = i == k, jk = j == k;
  return fma(ik && jk ? -1.0 : ik || jk ? v : -t, r, ik || jk ? 0.0 : v);
}

// Fills Ctrl::elim for the frame: the sweep operator over y (components 6..16) of the
// prior's augmented matrix [H* b*] leaves -P = -H_yy^-1, P H_yp = -K, P b_y and, on the
// pose block, the Schur complement and its vector; element-parallel on its 170 entries,
// two per thread of warps 0-3.  Components that the gyro-only variant holds are left
// out (zero rows and columns).  pk, dt: the frame's np pieces; Sg: the 9 x 9 covariance
// of the (r, a, v) rows.  Warps 0-5 (4 and 5 store the pieces and the covariance
// blocks).  elim.ok stays 0 when H_yy is not safely positive definite or there are more
// pieces than the step keeps in shared memory: the frame's steps then all take the
// information form.
__device__ void prepare_elim(const SolveParams& sp, Ctrl* c, int np, const double* dt, const int* pk,
                             double T, const double* Sg, double (*col)[18], double* sink, int* bad) {
  const int tid = threadIdx.x;
  double* m = c->elim.m;
  if (tid >= 128) {
    const int t = tid - 128;
    if (np <= kElimPieces) {
      const dri_imu_sample* s = imu_samples(sp.imu);
      for (int L = t; L < 8 * np; L += 64) {
        const int k = L >> 3, q = L & 7;
        const dri_imu_sample& x = s[pk[k]];
        c->elim.piece[k][q] = q == 0 ? dt[k] : q == 1 ? 0.5 * dt[k] : q < 5 ? x.gyr[q - 2] : x.acc[q - 5];
      }
    }
    if (t < 54) {
      if (t < 36) m[kElS6 + t] = Sg[(t / 6) * 9 + t % 6];
      else m[kElSv + t - 36] = Sg[(6 + (t - 36) / 6) * 9 + (t - 36) % 6];
    } else if (t == 54) {
      m[kElSg] = sp.sigma_grav * sp.sigma_grav;
      m[kElT] = T;
    }
    return;
  }
  const bool gyro = sp.track_mode == DRI_TRACK_GYRO_ONLY;
  int ei[2], ej[2];
  double v[2], diag[2];
#pragma unroll
  for (int o = 0; o < 2; ++o) {
    const int e = tid + 128 * o;      // rows 0..16, then the row of b* (17)
    int i = -1, j = -1;
    double x = 0.0;
    if (e < 170) {
      i = e < 153 ? (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f) : 17;
      if (e < 153 && tri(i + 1, 0) <= e) ++i;
      if (e < 153 && tri(i, 0) > e) --i;
      j = e - tri(i, 0);
      x = i < 17 ? c->Hs[j * 17 + i] : c->bs[j];     // upper triangle, as assemble_state
      if (gyro && ((i < 17 && held_gyro_only(i)) || held_gyro_only(j))) x = 0.0;
    }
    ei[o] = i;
    ej[o] = j;
    v[o] = diag[o] = x;
  }
  if (tid == 0) *bad = np > kElimPieces;
  bar_sync<1, 128>();
#pragma unroll 1
  for (int k = 6; k < 17; ++k) {
    if (gyro && held_gyro_only(k)) continue;
    double* ck = col[k & 1];          // column k by symmetry
#pragma unroll
    for (int o = 0; o < 2; ++o) {
      const int i = ei[o], j = ej[o];
      *(i == k ? ck + j : j == k ? ck + i : sink + tid) = v[o];
      if (i == k && j == k && !(v[o] > 1e-12 * diag[o] && v[o] < 1e29)) *bad = 1;
    }
    bar_sync<1, 128>();
    const double r = pivot_recip<true>(ck[k]);
#pragma unroll
    for (int o = 0; o < 2; ++o) v[o] = sweep_entry(ei[o], ej[o], k, v[o], ck, r);
  }
  bar_sync<1, 128>();
#pragma unroll
  for (int o = 0; o < 2; ++o) {
    const int i = ei[o], j = ej[o];
    if (i == 17) {
      m[j < 6 ? kElBp + j : kElM0 + j - 6] = v[o];
    } else if (i >= 6 && j >= 6) {
      m[kElPy + (i - 6) * 11 + j - 6] = -v[o];
      m[kElPy + (j - 6) * 11 + i - 6] = -v[o];
    } else if (i >= 6) {
      m[kElK + (i - 6) * 6 + j] = -v[o];
    } else if (i >= 0) {
      m[kElHp + i * 6 + j] = v[o];
      m[kElHp + j * 6 + i] = v[o];
    }
  }
  if (tid == 0) {
    c->elim.np = np;
    c->elim.ok = !*bad;
  }
}
