// SPV step kernels: geometry + force sets, net force + update, Delaunay test.
//
// Sussman, arXiv 1702.02939:
//  * geometry of every cell from the circumcentres of its Delaunay triangles
//    (Sec. 2.C.1); areas, perimeters, E of Eq. 1
//  * "force sets" dE_c/dh per (cell, vertex) (Sec. 2.C.2, Eqs. A3-A5) and the
//    net force F_i = -sum_t (dh_t/dr_i)^T G_t (Eqs. A6-A7)
//  * displacement by Eq. 3 and director rotation (Sec. 2.C.3)
//  * empty-circumcircle test of the triangulation (Sec. 2.C.3)
//
// GB300 design notes: the path is bound by the FP64 pipe (about 1/74 of the
// FP32 rate), so FP64 is spent only on the physics.  The Jacobian dh/dr_i is
// used in its rank-one form J = w u^T / det (u = h - r_i, w = perp(r_k - r_j),
// det = (r_j - r_i) x (r_k - r_i)), which follows from differentiating the
// equidistance conditions |h - r_i| = |h - r_j| = |h - r_k| and equals the
// matrix of Eq. A16.  All predicates run on the FP32/integer pipes.
#include "cg_device.cuh"
#include "cg_kernels.h"
#include <algorithm>

namespace cgk {

// The doubled circumcentre h of the triangle (0, a, b), a and b in grid units,
// and its Jacobian factor s = h / det.  Squared lengths and the determinant
// exactly in 128-bit integers from the grid offsets; the numerators
// (b_y |a|^2 - a_y |b|^2, a_x |b|^2 - b_x |a|^2) in 128-bit integers too, from
// |a|^2 and |b|^2 cut to 62 significant bits by a shift common to the triangle
// (at least as accurate as FP64 products of the rounded squares), each rounded
// to double once.
// (LA, LB: the exact squared lengths.)
__device__ __forceinline__ void geom_vertex(long long AX, long long AY, unsigned __int128 LA, long long BX,
                                            long long BY, unsigned __int128 LB, double2& h, double2& s) {
  const double r = fx_rcp(i128_to_double(cross_exact(AX, AY, BX, BY)));
  // |offsets| < 2^49 and the cut squares < 2^62: the numerators fit in 113 bits
  const int S = max(u128_bits(LA > LB ? LA : LB) - 62, 0);
  const long long la = (long long)shr128(LA, S), lb = (long long)shr128(LB, S);
  h.x = i128_to_double(scaled_diff_exact(BY, la, AY, lb), S) * r;
  h.y = i128_to_double(scaled_diff_exact(AX, lb, BX, la), S) * r;
  s = make_double2(h.x * r, h.y * r);
}

__device__ __forceinline__ double power_of_two(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }
// A, P and the energy of cell i from its sums over the doubled circumcentres in
// fixed point (one unit 2^unit grid units); returns (ka, kp) for differences of
// fixed-point vertices (kFineBits finer) and of Q1.61 unit vectors.
__device__ __forceinline__ double2 geom_cell_fixed(const GeomArgs& g, int i, double sc, __int128 area,
                                                   unsigned long long per, int unit) {
  const double A = 0.125 * i128_to_double(area, 2 * unit) * sc * sc;
  const double P = 0.5 * i64_to_double((long long)per, unit) * sc;
  g.A[i] = A;
  g.P[i] = P;
  const double dA = A - g.A0, dP = fma(-g.p0[i], g.sqrtA0, P);
  if (g.energy_out) g.energy_out[i] = fma(g.KA * dA, dA, g.KP * dP * dP);
  // dA/dh = 1/2 perp(h_next - h_prev) (the 1/2, the doubling of g and the
  // grid scale fold into ka); dP/dh = e_in - e_out (unit edge vectors)
  const double ka = g.KA * dA * (0.5 * sc), kp = 2.0 * g.KP * dP;
  return make_double2(ka * power_of_two(unit - kFineBits), kp * 0x1p-61);
}
// dE/dh at a vertex from its neighbours hp, hn on the polygon and the unit
// vectors of the edges ending (e) and leaving (en) there.
__device__ __forceinline__ double2 force_set(double2 k, longlong2 hp, longlong2 hn, longlong2 e, longlong2 en) {
  const double gx = i64_to_double(hn.y - hp.y), gy = i64_to_double(hp.x - hn.x);
  const double dPx = i64_to_double(e.x - en.x), dPy = i64_to_double(e.y - en.y);
  return make_double2(fma(k.x, gx, k.y * dPx), fma(k.x, gy, k.y * dPy));
}

// One thread per cell.  Writes A, P, force sets fs[a][i] = dE_i/dh_a, and the
// per-slot Jacobian factor s[a][i] = 2 u_a / det_a (the other factor, w_a / 2,
// is rebuilt exactly from the integer positions by k_force).
//
// The geometry runs in grid units (coordinates x 2^q): relative positions come
// exactly from the int64 grid coordinates, and the powers of two cancel in the
// force (u/det scales as 2^q, w as 2^-q) or fold into one factor per cell
// (A x 2^-2q, P x 2^-q, dA/dh x 2^-q).  The circumcentres are kept doubled,
// g_a = 2 h_a = num / det: every use is homogeneous in h, so the factor 2
// (exact) folds into the per-cell constants (A x 1/4, P x 1/2, dA/dh x 1/2,
// s x 2 against w / 2).
//
// The polygon (edges, lengths, unit vectors, area, differences) is formed in
// 64-bit fixed point in a unit common to the cell, eight bits finer than a
// double holds its largest vertex: vertices down to 2^-7 of the farthest one
// lose nothing against a double, nearer ones a bit per further factor of two.
// (Force errors of cells 2^-12 and 2^-16 across among cells 1 apart, against
// FP64 arithmetic: 1.1 and 2.3 times; three bits finer only, 6 and 42 times and
// 0.2% less time.  An exact path for such cells, out of line: 17.0 -> 17.9 us
// per step at 1024 cells without one, 167.1 -> 172.0 at 262144.)
//
// FP64 instructions issue at 1/74 of the FP32 rate, and 61 per cell remain of
// 139.  One pass at 262144 cells 94.2 -> 82.9 us, at 10^6 315 -> 270; what
// bounds it now is the issue of the integer sequences (60% of the slots) at 24
// warps per SM.  The next neighbour's position is loaded ahead: 270 -> 266.
//
// Per ring slot the kernel keeps the circumcentre, then its fixed-point value
// and the unit vector of the edge ending there, for the force-set pass: the
// first kGeomSh slots in shared memory (8 KB per one-warp block, so that 24
// blocks fit on an SM), the slots of longer rings (rare) in local memory.
__global__ void __launch_bounds__(kGeomThreads, kGeomMinBlocks) k_geom(GeomArgs g) {
  __shared__ double sh_hx[kGeomSh][kGeomThreads];
  __shared__ double sh_hy[kGeomSh][kGeomThreads];
  __shared__ double sh_ex[kGeomSh][kGeomThreads];  // unit vector of the edge ending at vertex a
  __shared__ double sh_ey[kGeomSh][kGeomThreads];
  constexpr int kLo = (CG_RING > kGeomSh) ? CG_RING - kGeomSh : 1;
  double lo_hx[kLo], lo_hy[kLo], lo_ex[kLo], lo_ey[kLo];
  const int t = threadIdx.x;
  auto put = [&](double (&sh)[kGeomSh][kGeomThreads], double* lo, int a, double v) {
    if (a < kGeomSh) sh[a][t] = v;
    else lo[a - kGeomSh] = v;
  };
  auto get = [&](const double (&sh)[kGeomSh][kGeomThreads], const double* lo, int a) -> double {
    return (a < kGeomSh) ? sh[a][t] : lo[a - kGeomSh];
  };
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  for (int item = blockIdx.x * kGeomThreads + t; item < g.n; item += gridDim.x * kGeomThreads) {
    const int i = g.order ? g.order[item] : item;
    const Rep R = g.reps[g.rep[i]];
    const long long Xi = X[i], Yi = Y[i];
    const int m = g.cnt[i];
    if (m < 3 || m > CG_RING) {
      if (!g.tolerant) raise_status(g.ctl, kETOPO);
      continue;
    }
    const int* ring = g.nbr + (size_t)i * CG_RING;
    // a ring being rewritten concurrently may hold -1 entries: read the cell
    // itself there (the result is discarded and computed again)
    auto nb = [&](int a) {
      const int j = ring[a];
      return ((unsigned)j < (unsigned)g.n) ? j : i;
    };

    const int j0 = nb(0);
    const long long D0X = min_image_i(X[j0] - Xi, R.LX), D0Y = min_image_i(Y[j0] - Yi, R.LY);
    const unsigned __int128 L0 = norm2_exact(D0X, D0Y);
    unsigned __int128 LA = L0;
    long long AX = D0X, AY = D0Y;
    int top = 0;
    int jq = nb(1);  // the neighbour whose position is loaded ahead
    long long qX = X[jq], qY = Y[jq];
    for (int a = 0; a < m; ++a) {
      long long BX, BY;
      unsigned __int128 LB;
      if (a + 1 < m) {
        BX = min_image_i(qX - Xi, R.LX);
        BY = min_image_i(qY - Yi, R.LY);
        if (a + 2 < m) {
          jq = nb(a + 2);
          qX = X[jq];
          qY = Y[jq];
        }
        LB = norm2_exact(BX, BY);
      } else {
        BX = D0X; BY = D0Y; LB = L0;
      }
      double2 h, sj;
      geom_vertex(AX, AY, LA, BX, BY, LB, h, sj);
      g.s[a * N + i] = sj;
      put(sh_hx, lo_hx, a, h.x);
      put(sh_hy, lo_hy, a, h.y);
      top = max(top, exponent_of(h));
      LA = LB;
      AX = BX; AY = BY;
    }
    // the polygon in fixed point, one unit 2^unit grid units: the vertices and
    // the unit vectors of the edges ending there take the circumcentres' places
    const int unit = top - 1023 - 55;
    auto vertex = [&](int a) { return to_fixed(make_double2(get(sh_hx, lo_hx, a), get(sh_hy, lo_hy, a)), top); };
    auto keep = [&](double (&sh)[kGeomSh][kGeomThreads], double* lo, int a, long long v) {
      put(sh, lo, a, __longlong_as_double(v));
    };
    PolygonArea<kFineBits> area;
    unsigned long long per = 0;
    longlong2 H = vertex(m - 1);
    area.start(H);
    for (int a = 0; a < m; ++a) {
      const longlong2 hp = H;
      H = vertex(a);
      area.add(H);
      longlong2 e;
      unsigned long long len;
      edge_fixed(H, hp, e, len);
      per += len;
      keep(sh_hx, lo_hx, a, H.x);
      keep(sh_hy, lo_hy, a, H.y);
      keep(sh_ex, lo_ex, a, e.x);
      keep(sh_ey, lo_ey, a, e.y);
    }
    const double2 k = geom_cell_fixed(g, i, R.inv_scale, area.total(), per, unit);
    auto fixed = [&](const double (&sh)[kGeomSh][kGeomThreads], const double* lo, int a) {
      return __double_as_longlong(get(sh, lo, a));
    };
    for (int a = 0; a < m; ++a) {
      const int ap = (a == 0) ? m - 1 : a - 1;
      const int an = (a + 1 == m) ? 0 : a + 1;
      g.fs[a * N + i] = force_set(
          k, make_longlong2(fixed(sh_hx, lo_hx, ap), fixed(sh_hy, lo_hy, ap)),
          make_longlong2(fixed(sh_hx, lo_hx, an), fixed(sh_hy, lo_hy, an)),
          make_longlong2(fixed(sh_ex, lo_ex, a), fixed(sh_ey, lo_ey, a)),
          make_longlong2(fixed(sh_ex, lo_ex, an), fixed(sh_ey, lo_ey, an)));
    }
  }
}

// The pass with one thread per (cell, ring slot): a block takes 32 cells, its
// warp w the slots w, w + 8 of all of them (lane = cell, so every access is
// coalesced).  The neighbours' offsets, the circumcentres and the edges pass
// between slots through shared memory; the last warp, whose own slots are rare,
// adds the area up while the others form the edges, and the first adds up the
// perimeter and forms the cell's coefficients.
//
// The polygon itself (edges, lengths, unit vectors, area, differences) is
// formed in 64-bit fixed point, as in k_geom: 8 FP64 operations per slot remain
// of 21.
__global__ void __launch_bounds__(kSlotThreads, kGeomSlotBlocks) k_geom_slots(GeomArgs g) {
  __shared__ longlong2 s_off[CG_RING][32];  // neighbour offsets, then unit edge vectors (Q1.61)
  __shared__ double2 s_h[CG_RING][32];      // doubled circumcentres
  __shared__ longlong2 s_H[CG_RING][32];    // and in fixed point
  __shared__ unsigned long long s_len[CG_RING][32];  // length of the edge ending at the slot
  __shared__ double2 s_k[32];               // the cell's ka, kp, in the units of the differences
  __shared__ longlong2 s_area[32];
  __shared__ int s_top[32];                 // largest exponent of the cell's circumcentres
  longlong2(*s_e)[32] = s_off;
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  const int total = g.list ? *g.list_count : g.n;
  if (g.clear)
    for (int k = blockIdx.x * kSlotThreads + threadIdx.x; k < g.n_clear; k += gridDim.x * kSlotThreads) g.clear[k] = 0;
  for (int base = blockIdx.x * 32; base < total; base += gridDim.x * 32) {
    const int item = base + c;
    int i = 0, m = 0;
    if (item < total) {
      i = g.list ? g.list[item] : (g.order ? g.order[item] : item);
      m = g.cnt[i];
      if (w == 0) {
        if (g.list_bits) atomicAnd(&g.list_bits[i >> 5], ~(1u << (i & 31)));
        if ((m < 3 || m > CG_RING) && !g.tolerant) raise_status(g.ctl, kETOPO);
      }
      if (m < 3 || m > CG_RING) m = 0;
    }
    if (w == 0) s_top[c] = 0;
    const Rep& R = g.reps[g.rep[i]];
    const int* ring = g.nbr + (size_t)i * CG_RING;
    if (w < m) {
      const long long Xi = X[i], Yi = Y[i], LX = R.LX, LY = R.LY;
      for (int a = w; a < m; a += kSlotWarps) {
        // a ring being rewritten concurrently may hold -1 entries: the cell
        // itself is read there (the result is discarded and computed again)
        int j = ring[a];
        j = ((unsigned)j < (unsigned)g.n) ? j : i;
        s_off[a][c] = make_longlong2(min_image_i(X[j] - Xi, LX), min_image_i(Y[j] - Yi, LY));
      }
    }
    __syncthreads();
    int top = 0;
    for (int a = w; a < m; a += kSlotWarps) {
      const longlong2 A = s_off[a][c], B = s_off[a + 1 < m ? a + 1 : 0][c];
      double2 h, sj;
      geom_vertex(A.x, A.y, norm2_exact(A.x, A.y), B.x, B.y, norm2_exact(B.x, B.y), h, sj);
      g.s[a * N + i] = sj;
      s_h[a][c] = h;
      top = max(top, exponent_of(h));
    }
    if (top) atomicMax(&s_top[c], top);
    __syncthreads();
    top = s_top[c];
    const int unit = top - 1023 - 55;  // one fixed-point unit is 2^unit grid units
    if (w == kSlotWarps - 1) {
      PolygonArea<kFineBits> area;
      auto vertex = [&](int a) { return to_fixed(s_h[a][c], top); };
      if (m) area.start(vertex(m - 1));
      for (int a = 0; a < m; ++a) area.add(vertex(a));
      const __int128 t = area.total();
      s_area[c] = make_longlong2((long long)t, (long long)(t >> 64));
    }
    for (int a = w; a < m; a += kSlotWarps) {
      const double2 h = s_h[a][c], hp = s_h[a > 0 ? a - 1 : m - 1][c];
      const longlong2 H = to_fixed(h, top);
      longlong2 e;
      unsigned long long len;
      edge_fixed(H, to_fixed(hp, top), e, len);
      s_H[a][c] = H;
      s_e[a][c] = e;
      s_len[a][c] = len;
    }
    __syncthreads();
    if (w == 0 && m) {
      unsigned long long per = 0;
      for (int a = 0; a < m; ++a) per += s_len[a][c];
      const longlong2 t = s_area[c];
      s_k[c] = geom_cell_fixed(g, i, R.inv_scale, ((__int128)t.y << 64) | (unsigned long long)t.x, per, unit);
    }
    __syncthreads();
    const double2 k = s_k[c];
    for (int a = w; a < m; a += kSlotWarps) {
      const int ap = a > 0 ? a - 1 : m - 1, an = a + 1 < m ? a + 1 : 0;
      g.fs[a * N + i] = force_set(k, s_H[ap][c], s_H[an][c], s_e[a][c], s_e[an][c]);
    }
    __syncthreads();
  }
}

// Net force on cell i: G_t = sum over the triangle's three cells of their
// force sets, F_i = -sum_t s_t (w_t . G_t), with s_t = 2 u_t / det_t from
// k_geom and w_t / 2 = perp(r_k - r_j) / 2 rebuilt exactly from the integer
// grid offsets (an exact difference, converted on the integer pipes).  False
// (status raised) for a malformed ring.
__device__ __forceinline__ bool net_force(const ForceArgs& g, int i, double& fx_out, double& fy_out) {
  const size_t N = (size_t)g.n;
  const int m = g.cnt[i];
  if (m < 3 || m > CG_RING) {
    if (!g.tolerant) raise_status(g.ctl, kETOPO);
    return false;
  }
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  const Rep R = g.reps[g.rep[i]];
  const long long Xi = X[i], Yi = Y[i];
  const int* ring = g.nbr + (size_t)i * CG_RING;
  bool bad = false;
  // a ring being rewritten meanwhile (tolerant pass) may hold -1 entries:
  // the cell itself is read there and the result marked bad
  auto nb = [&](int a) {
    const int j = ring[a];
    const bool ok = (unsigned)j < (unsigned)g.n;
    bad |= !ok;
    return ok ? j : i;
  };
  int jfirst = nb(0);
  int pfirst = ring_pos(g.nbr, g.cnt, jfirst, i);
  int j = jfirst, pj = pfirst;
  const long long fX = min_image_i(X[jfirst] - Xi, R.LX), fY = min_image_i(Y[jfirst] - Yi, R.LY);
  long long aX = fX, aY = fY;
  double fx = 0.0, fy = 0.0;
  bad |= pfirst < 0;
  for (int a = 0; a < m; ++a) {
    int k, pk;
    long long bX, bY;
    if (a + 1 < m) {
      k = nb(a + 1);
      pk = ring_pos(g.nbr, g.cnt, k, i);
      bad |= pk < 0;
      bX = min_image_i(X[k] - Xi, R.LX);
      bY = min_image_i(Y[k] - Yi, R.LY);
    } else {
      k = jfirst;
      pk = pfirst;
      bX = fX;
      bY = fY;
    }
    // triangle (i, j, k) is slot pj-1 around j and slot pk around k
    const int mj = g.cnt[j];
    const int bj = (pj <= 0) ? (mj > 0 ? mj - 1 : 0) : pj - 1;
    const double2 f0 = g.fs[a * N + i];
    const double2 f1 = g.fs[(size_t)bj * N + j];
    const double2 f2 = g.fs[(size_t)(pk < 0 ? 0 : pk) * N + k];
    const double Gx = f0.x + f1.x + f2.x, Gy = f0.y + f1.y + f2.y;
    const double2 s = g.s[a * N + i];
    const double wx = i2d_int(bY - aY, -1), wy = i2d_int(aX - bX, -1);
    const double c = fma(wx, Gx, wy * Gy);
    fx = fma(-s.x, c, fx);
    fy = fma(-s.y, c, fy);
    j = k;
    pj = pk;
    aX = bX;
    aY = bY;
  }
  if (bad) {
    if (g.tolerant) return false;
    raise_status(g.ctl, kETOPO);
  }
  fx_out = fx;
  fy_out = fy;
  return true;
}


// The update of Eq. 3 of cell i under the force (fx, fy).
__device__ __forceinline__ void move_cell(const ForceArgs& g, int i, double fx, double fy) {
  const size_t N = (size_t)g.n;
  // Eq. 3: r <- r + dt (mu F + v0 n(theta)), rounded to the grid and wrapped
  // into the other position buffer; the director rotation
  // theta <- theta + sqrt(2 D_r dt) xi follows at the start of the next step
  // (k_dir), so the state between steps is (r, theta) of one time.
  const int cur = g.ctl->cur;
  const Rep R = g.reps[g.rep[i]];
  const double xi = g.x[(size_t)cur * N + i], yi = g.y[(size_t)cur * N + i];
  const double2 nd = g.nrm[i];  // (cos theta, sin theta), from k_dir
  double v0;
  if (g.v0_user) {  // integrate 2 with new speeds: take them over first
    v0 = g.v0_user[g.tag[i]];
    if (!isfinite(v0)) raise_status(g.ctl, kEINVAL);
    g.v0[i] = v0;
  } else {
    v0 = g.v0[i];
  }
  const double vx = g.mu * fx + v0 * nd.x, vy = g.mu * fy + v0 * nd.y;
  const double xn = fma(g.dt, vx, xi), yn = fma(g.dt, vy, yi);
  long long X, Y;
  if (isfinite(xn) && isfinite(yn)) {
    if (!R.framed) {
      X = wrap_to_grid(xn, R.Lx, R.scale, R.LX);
      Y = wrap_to_grid(yn, R.Ly, R.scale, R.LY);
    } else {
      X = move_framed(xi, g.dt, vx, R.x0, R.Lxg, R.scale, R.X0, R.LXg, R.LX);
      Y = move_framed(yi, g.dt, vy, R.y0, R.Lyg, R.scale, R.Y0, R.LYg, R.LY);
    }
  } else {
    if (g.tolerant) {  // decided again, strictly, after the repair rounds
      claim_fix(g.fix_bits, g.fix_list, &g.ctl->force_count, i);
      return;
    }
    raise_status(g.ctl, kENONFINITE);
    X = (long long)rint(xi * R.scale);
    Y = (long long)rint(yi * R.scale);
  }
  const int nxt = cur ^ 1;
  g.x[(size_t)nxt * N + i] = i2d_int(X, -R.q);
  g.y[(size_t)nxt * N + i] = i2d_int(Y, -R.q);
  g.X[(size_t)nxt * N + i] = X;
  g.Y[(size_t)nxt * N + i] = Y;
}

// Cell i's net force (integrate 0 or 1) and update of Eq. 3 (integrate 1),
// or the update alone from the stored forces of the current positions
// (integrate 2: after a change of v0).
__device__ __forceinline__ void force_cell(const ForceArgs& g, int i) {
  double fx, fy;
  if (g.integrate == 2) {
    fx = g.Fx[i];
    fy = g.Fy[i];
  } else {
    if (!net_force(g, i, fx, fy)) {
      if (g.tolerant) claim_fix(g.fix_bits, g.fix_list, &g.ctl->force_count, i);
      return;
    }
    g.Fx[i] = fx;
    g.Fy[i] = fy;
    if (!g.integrate) return;
  }
  move_cell(g, i, fx, fy);
}

// The same with one thread per (cell, ring slot), as k_geom_slots: the slots'
// triangles in parallel, their contributions added up in ring order by the
// first warp (bit-identical to force_cell), which then moves the cells.  Rings
// must not change meanwhile.
__global__ void __launch_bounds__(kSlotThreads, kForceSlotBlocks) k_force_slots(ForceArgs g) {
  __shared__ longlong2 s_off[CG_RING][32];  // neighbour offsets
  __shared__ double2 s_s[CG_RING][32];      // Jacobian factors
  __shared__ double s_c[CG_RING][32];       // w . G
  __shared__ int s_j[CG_RING][32];          // neighbours
  __shared__ int s_p[CG_RING][32];          // the cell's slot in the neighbour's ring, and the one before it
  __shared__ int s_bad[32];
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  const int total = g.list ? *g.list_count : g.n;
  for (int base = blockIdx.x * 32; base < total; base += gridDim.x * 32) {
    const int item = base + c;
    int i = 0, m = 0;
    if (item < total) {
      i = g.list ? g.list[item] : (g.order ? g.order[item] : item);
      m = g.cnt[i];
      if (w == 0) {
        if (g.list_bits) atomicAnd(&g.list_bits[i >> 5], ~(1u << (i & 31)));
        if (m < 3 || m > CG_RING) raise_status(g.ctl, kETOPO);
      }
      if (m < 3 || m > CG_RING) m = 0;
    }
    bool bad = false;
    if (w == 0) s_bad[c] = 0;
    if (w < m) {
      const Rep& R = g.reps[g.rep[i]];
      const int* ring = g.nbr + (size_t)i * CG_RING;
      const long long Xi = X[i], Yi = Y[i], LX = R.LX, LY = R.LY;
      for (int a = w; a < m; a += kSlotWarps) {
        int j = ring[a];
        const bool ok = (unsigned)j < (unsigned)g.n;
        j = ok ? j : i;
        const int mj = g.cnt[j], p = ring_pos(g.nbr, g.cnt, j, i);
        bad |= !ok || p < 0;
        // triangle (i, j, k) is the slot before i's around j and i's slot around k
        s_p[a][c] = (p < 0 ? 0 : p) | ((p <= 0 ? (mj > 0 ? mj - 1 : 0) : p - 1) << 8);
        s_j[a][c] = j;
        s_off[a][c] = make_longlong2(min_image_i(X[j] - Xi, LX), min_image_i(Y[j] - Yi, LY));
      }
    }
    __syncthreads();
    if (bad) s_bad[c] = 1;
    for (int a = w; a < m; a += kSlotWarps) {
      const int an = a + 1 < m ? a + 1 : 0;
      const double2 f0 = g.fs[a * N + i];
      const double2 f1 = g.fs[(size_t)(s_p[a][c] >> 8) * N + s_j[a][c]];
      const double2 f2 = g.fs[(size_t)(s_p[an][c] & 255) * N + s_j[an][c]];
      s_s[a][c] = g.s[a * N + i];
      const longlong2 A = s_off[a][c], B = s_off[an][c];
      const double Gx = f0.x + f1.x + f2.x, Gy = f0.y + f1.y + f2.y;
      const double wx = i2d_int(B.y - A.y, -1), wy = i2d_int(A.x - B.x, -1);
      s_c[a][c] = fma(wx, Gx, wy * Gy);
    }
    __syncthreads();
    if (w == 0 && m) {
      if (s_bad[c]) raise_status(g.ctl, kETOPO);
      double fx = 0.0, fy = 0.0;
      for (int a = 0; a < m; ++a) {
        const double2 sj = s_s[a][c];
        const double cj = s_c[a][c];
        fx = fma(-sj.x, cj, fx);
        fy = fma(-sj.y, cj, fy);
      }
      g.Fx[i] = fx;
      g.Fy[i] = fy;
      if (g.integrate) move_cell(g, i, fx, fy);
    }
    __syncthreads();
  }
}

// One thread per cell: the net force (integrate 0 or 1) and the update of
// Eq. 3 (integrate 1), or the update alone from the stored forces of the
// current positions (integrate 2: after a change of v0); with a list, the
// cells of the list (grid-stride), their list bits cleared.
__global__ void __launch_bounds__(kForceThreads) k_force(ForceArgs g) {
  const int total = g.list ? *g.list_count : g.n;
  for (int item = blockIdx.x * kForceThreads + threadIdx.x; item < total; item += gridDim.x * kForceThreads) {
    const int i = g.list ? g.list[item] : (g.order ? g.order[item] : item);
    if (g.list_bits) atomicAnd(&g.list_bits[i >> 5], ~(1u << (i & 31)));
    force_cell(g, i);
  }
}

// The fix-up list of the force pass: each rewritten ring's cell and the
// cells of its new ring (their force sets or ring positions changed).
__global__ void k_force_fix_list(ForceFixArgs g) {
  const int total = *g.dirty_count;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int d = g.dirty_list[t];
    if ((unsigned)d >= (unsigned)g.n) continue;
    claim_fix(g.fix_bits, g.fix_list, &g.ctl->force_count, d);
    const int m = min(g.cnt[d], CG_RING);
    for (int a = 0; a < m; ++a) {
      const int j = g.nbr[(size_t)d * CG_RING + a];
      if ((unsigned)j < (unsigned)g.n) claim_fix(g.fix_bits, g.fix_list, &g.ctl->force_count, j);
    }
  }
}

// Director terms of a step: with `advance`, first the rotation of the
// previous step theta <- theta + sqrt(2 D_r dt) xi; then n(theta) and the
// noise xi of this step (Philox counter (tag, step)), grid-stride over cells.
// In the step graph it runs beside the circumcircle test, the cell list and
// the repair rounds, which leave the FP64 pipe idle.
__global__ void k_dir(DirArgs g) {
  const long long step = g.ctl->step;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += gridDim.x * blockDim.x) {
    double th = g.theta[i];
    if (g.advance) {
      th = th + g.noise_amp * g.xi[i];
      g.theta[i] = th;
    }
    double sn, cs;
    dm_sincos(th, g.tab, sn, cs);
    g.nrm[i] = make_double2(cs, sn);
    g.xi[i] = director_noise(g.seed, g.tag[i], step, g.tab);
  }
}
void launch_dir(const DirArgs& a, cudaStream_t st, int blocks) {
  if (a.n <= 0) return;
  const int full = (a.n + 127) / 128;
  k_dir<<<(blocks > 0 && blocks < full) ? blocks : full, 128, 0, st>>>(a);
}

// Table of dir_math.cuh: (sin, cos)(j pi/128) from CUDA's sinpi/cospi (exact
// at multiples of pi/2), then per logarithm interval j the reciprocal of its
// centre and minus its logarithm (exactly 1 and 0 for the interval around 1).
__global__ void k_init_dir_tables(double2* tab) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < 256) {
    tab[j] = make_double2(sinpi(j / 128.0), cospi(j / 128.0));
  } else if (j >= kDirTabQ && j < kDirTabQ + 256) {
    // the same values in Q1.62 (exact: every nonzero entry is above 2^-10)
    const double sn = sinpi((j - kDirTabQ) / 128.0), cs = cospi((j - kDirTabQ) / 128.0);
    reinterpret_cast<longlong2*>(tab)[j] = make_longlong2(__double2ll_rn(sn * 0x1p62), __double2ll_rn(cs * 0x1p62));
  } else if (j < kDirTabQ) {
    const int i = j - 256;
    const double inv =
        (i == kLogOne) ? 1.0 : 1.0 / __longlong_as_double(kLogOff + ((long long)i << 44) + (1LL << 43));
    tab[j] = make_double2(inv, -log(inv));
  }
}
void launch_init_dir_tables(double2* tab, cudaStream_t st) { k_init_dir_tables<<<kDirTabEntries / 128, 128, 0, st>>>(tab); }

__global__ void k_dir_terms(int n, const double* __restrict__ theta, const int* __restrict__ tag,
                            unsigned long long seed, long long step, const double2* __restrict__ tab,
                            double* cs, double* sn, double* xi) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double s, c;
    dm_sincos(theta[i], tab, s, c);
    cs[i] = c;
    sn[i] = s;
    xi[i] = director_noise(seed, tag[i], step, tab);
  }
}
void launch_dir_terms(int n, const double* theta, const int* tag, unsigned long long seed, long long step,
                      const double2* tab, double* cs, double* sn, double* xi, cudaStream_t st) {
  if (n <= 0) return;
  const int blocks = (int)std::min<long long>((n + 127) / 128, 152LL * 16);
  k_dir_terms<<<blocks, 128, 0, st>>>(n, theta, tag, seed, step, tab, cs, sn, xi);
}

// Start of the topology phase of a step: the new positions become current,
// the step counter advances and the flagged list is emptied.
__global__ void k_begin_topology(Ctl* ctl, int flip) {
  if (flip) {
    ctl->cur ^= 1;
    ctl->step += 1;
  }
  ctl->count[0] = 0;
  ctl->count[1] = 0;
  ctl->round_count = 0;
  ctl->dirty_count = 0;
  ctl->force_count = 0;
}

__device__ __forceinline__ void flag_cell(unsigned* flags, int* list, int* count, int c) {
  const unsigned bit = 1u << (c & 31);
  const unsigned old = atomicOr(&flags[c >> 5], bit);
  if (!(old & bit)) list[atomicAdd(count, 1)] = c;
}

// Places cell i in the cell list of the step.
__device__ __forceinline__ void bin_cell_at(const TestArgs& g, const Rep& R, long long X, long long Y, int i) {
  int bx, by;
  bin_of_grid(R, X, Y, bx, by);
  bin_insert(g.bins, R.bin0 + by * R.nbx + bx, i);
}

// One ring slot of cell i: its edge (i, j_a) with i < j_a must be locally
// Delaunay (the far vertex j_{a+1} outside the circle through i, j_{a-1}, j_a)
// and its triangle (i, j_a, j_{a+1}), where i is the smallest index,
// positively oriented.  A failing quadruple or triangle flags all its cells.
__device__ __forceinline__ void test_slot(const TestArgs& g, int i, int jp, int ja, int jn, float fpx, float fpy,
                                          float fax, float fay, float fnx, float fny, long long pX, long long pY,
                                          long long aX, long long aY, long long nX, long long nY, float sc) {
  if (i >= ja) return;
  if (incircle0_sign(fpx, fpy, fax, fay, fnx, fny, pX, pY, aX, aY, nX, nY, g.tag, i, jp, ja, jn, sc) > 0) {
    flag_cell(g.flags, g.list, &g.ctl->count[0], i);
    flag_cell(g.flags, g.list, &g.ctl->count[0], jp);
    flag_cell(g.flags, g.list, &g.ctl->count[0], ja);
    flag_cell(g.flags, g.list, &g.ctl->count[0], jn);
  }
  if (i < jn && orient0_sign(fax, fay, fnx, fny, aX, aY, nX, nY) <= 0) {
    flag_cell(g.flags, g.list, &g.ctl->count[0], i);
    flag_cell(g.flags, g.list, &g.ctl->count[0], ja);
    flag_cell(g.flags, g.list, &g.ctl->count[0], jn);
  }
}

// The same from the grid, out of line: the one-thread pass comes here where
// slot_open leaves a slot open.
static __device__ __noinline__ void test_slot_exact(const TestArgs* args, const long long* __restrict__ X,
                                                    const long long* __restrict__ Y, int i, int jp, int ja, int jn) {
  const TestArgs& g = *args;
  const Rep& R = g.reps[g.rep[i]];
  const float sc = (float)R.inv_scale;
  const long long Xi = X[i], Yi = Y[i], LX = R.LX, LY = R.LY;
  const long long pX = min_image_i(X[jp] - Xi, LX), pY = min_image_i(Y[jp] - Yi, LY);
  const long long aX = min_image_i(X[ja] - Xi, LX), aY = min_image_i(Y[ja] - Yi, LY);
  const long long nX = min_image_i(X[jn] - Xi, LX), nY = min_image_i(Y[jn] - Yi, LY);
  test_slot(g, i, jp, ja, jn, i2f_scaled(pX, sc), i2f_scaled(pY, sc), i2f_scaled(aX, sc), i2f_scaled(aY, sc),
            i2f_scaled(nX, sc), i2f_scaled(nY, sc), pX, pY, aX, aY, nX, nY, sc);
}

// Whether the float offsets (real units) of j_{a-1}, j_a and j_{a+1} leave open
// that the slot is sound.
__device__ __forceinline__ bool slot_open(int i, int ja, int jn, float2 fp, float2 fa, float2 fn) {
  return i < ja && !(outside_for_sure(fp, fa, fn) && (i >= jn || left_for_sure(fa, fn)));
}

// One thread per cell: every slot of its ring.
__device__ __forceinline__ void test_cell(const TestArgs& g, int i, const long long* __restrict__ X,
                                          const long long* __restrict__ Y) {
  const Rep& R = g.reps[g.rep[i]];
  const float sc = (float)R.inv_scale;
  const long long Xi = X[i], Yi = Y[i], LX = R.LX, LY = R.LY;
  const int m = g.cnt[i];
  if (m < 3 || m > CG_RING) {
    raise_status(g.ctl, kETOPO);
    return;
  }
  const int* ring = g.nbr + (size_t)i * CG_RING;
  auto offset = [&](int j) {
    return make_float2(i2f_scaled(min_image_i(X[j] - Xi, LX), sc), i2f_scaled(min_image_i(Y[j] - Yi, LY), sc));
  };
  // sliding window over (j_{a-1}, j_a, j_{a+1}); the neighbours come kTestAhead
  // at a time, so that their gathers are in flight together
  int ja = 0, jfirst = 0;
  unsigned open = 0;  // the slots to decide in full
  float2 fp = offset(ring[m - 1]), fa = make_float2(0.0f, 0.0f), ffirst = fa;
  for (int a0 = 0; a0 < m; a0 += kTestAhead) {
    int jn[kTestAhead];
    float2 fn[kTestAhead];
#pragma unroll
    for (int q = 0; q < kTestAhead; q += 4) {
      const int4 r = *reinterpret_cast<const int4*>(ring + a0 + q);
      jn[q] = r.x; jn[q + 1] = r.y; jn[q + 2] = r.z; jn[q + 3] = r.w;
    }
#pragma unroll
    for (int q = 0; q < kTestAhead; ++q) fn[q] = offset(a0 + q < m ? jn[q] : i);
#pragma unroll
    for (int q = 0; q < kTestAhead; ++q) {
      if (a0 + q >= m) break;
      if (a0 + q == 0) {
        jfirst = jn[0];
        ffirst = fn[0];
      } else {
        if (slot_open(i, ja, jn[q], fp, fa, fn[q])) open |= 1u << (a0 + q - 1);
        fp = fa;
      }
      ja = jn[q];
      fa = fn[q];
    }
  }
  if (slot_open(i, ja, jfirst, fp, fa, ffirst)) open |= 1u << (m - 1);
  for (; open; open &= open - 1) {
    const int a = __ffs((int)open) - 1;
    test_slot_exact(&g, X, Y, i, ring[a > 0 ? a - 1 : m - 1], ring[a], ring[a + 1 < m ? a + 1 : 0]);
  }
}

// Grid-stride over cells (a smaller grid leaves room on every SM for the
// FP64 branch that runs beside the test).  Bound by the latency of the
// neighbours' gathers: four neighbours in flight and 64 registers (one at a
// time and 108 registers before) take 82 -> 54 us at 10^6 cells.  The grid
// coordinates are read again for the few slots that the float values leave
// open; carried along for all of them they cost the registers.
__global__ void __launch_bounds__(kTestThreads, 8) k_test(const __grid_constant__ TestArgs g) {
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  for (int item = blockIdx.x * kTestThreads + threadIdx.x; item < g.n; item += gridDim.x * kTestThreads)
    test_cell(g, g.order ? g.order[item] : item, X, Y);
}

// The same with one thread per (cell, ring slot), as k_geom_slots: offsets and
// their float values pass between slots through shared memory; the first warp
// places the cells in the cell list.
__global__ void __launch_bounds__(kSlotThreads, kTestSlotBlocks) k_test_slots(TestArgs g) {
  __shared__ longlong2 s_off[CG_RING][32];
  __shared__ float2 s_f[CG_RING][32];
  __shared__ int s_j[CG_RING][32];
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  for (int base = blockIdx.x * 32; base < g.n; base += gridDim.x * 32) {
    const int item = base + c;
    int i = 0, m = 0;
    float sc = 0.0f;
    if (item < g.n) {
      i = g.order ? g.order[item] : item;
      m = g.cnt[i];
      const Rep& R = g.reps[g.rep[i]];
      sc = (float)R.inv_scale;
      const long long Xi = X[i], Yi = Y[i], LX = R.LX, LY = R.LY;
      if (w == 0) {
        if (g.bins.count) bin_cell_at(g, R, Xi, Yi, i);
        if (m < 3 || m > CG_RING) raise_status(g.ctl, kETOPO);
      }
      if (m < 3 || m > CG_RING) m = 0;
      const int* ring = g.nbr + (size_t)i * CG_RING;
      for (int a = w; a < m; a += kSlotWarps) {
        const int j = ring[a];
        const long long dX = min_image_i(X[j] - Xi, LX), dY = min_image_i(Y[j] - Yi, LY);
        s_j[a][c] = j;
        s_off[a][c] = make_longlong2(dX, dY);
        s_f[a][c] = make_float2(i2f_scaled(dX, sc), i2f_scaled(dY, sc));
      }
    }
    __syncthreads();
    for (int a = w; a < m; a += kSlotWarps) {
      const int p = a > 0 ? a - 1 : m - 1, n = a + 1 < m ? a + 1 : 0;
      const int ja = s_j[a][c];
      if (i >= ja) continue;
      const float2 fp = s_f[p][c], fa = s_f[a][c], fn = s_f[n][c];
      const longlong2 op = s_off[p][c], oa = s_off[a][c], on = s_off[n][c];
      test_slot(g, i, s_j[p][c], ja, s_j[n][c], fp.x, fp.y, fa.x, fa.y, fn.x, fn.y, op.x, op.y, oa.x, oa.y, on.x,
                on.y, sc);
    }
    __syncthreads();
  }
}

// Ring-size grouping of each chunk of kOrderChunk cells (see launch_order):
// a counting sort by min(cnt, CG_RING) in shared memory.  Ranks within a
// size come from shared atomics (their order does not matter: every cell's
// results are computed independently of which thread computes them).
__global__ void __launch_bounds__(256) k_order(int n, const int* __restrict__ cnt, int* __restrict__ order) {
  __shared__ int hist[CG_RING + 1], base[CG_RING + 1];
  const int c0 = blockIdx.x * kOrderChunk;
  const int len = min(kOrderChunk, n - c0);
  if (threadIdx.x <= CG_RING) hist[threadIdx.x] = 0;
  __syncthreads();
  int msz[kOrderChunk / 256];
#pragma unroll
  for (int k = 0; k < kOrderChunk / 256; ++k) {
    const int c = k * 256 + threadIdx.x;
    int m = -1;
    if (c < len) {
      m = cnt[c0 + c];
      m = m < 0 ? 0 : (m > CG_RING ? CG_RING : m);
      atomicAdd(&hist[m], 1);
    }
    msz[k] = m;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int b = 0; b <= CG_RING; ++b) {
      base[b] = acc;
      acc += hist[b];
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kOrderChunk / 256; ++k) {
    const int c = k * 256 + threadIdx.x;
    if (msz[k] >= 0) order[c0 + atomicAdd(&base[msz[k]], 1)] = c0 + c;
  }
}

// ---------------------------------------------------------------------------
// host-side launchers
// ---------------------------------------------------------------------------
void launch_order(int n, const int* cnt, int* order, cudaStream_t st) {
  if (n <= 0) return;
  k_order<<<(n + kOrderChunk - 1) / kOrderChunk, 256, 0, st>>>(n, cnt, order);
}
void launch_geom(const GeomArgs& a, cudaStream_t st, int blocks) {
  if (a.n <= 0) return;
  // A block per 32 cells and a warp per ring slot shortens the chain that one
  // thread walks by the number of slots: it is faster while the chip is not
  // full (one pass, us, one thread per cell -> slots: 20.5 -> 10.2 at 256
  // cells, 22.5 -> 11.5 at 4096, 22.5 -> 16.4 at 16384, 34.8 -> 32.8 at 65536).
  // Beyond, the warps of the last slots idle (50 -> 55 at 131072, 82 -> 98 at
  // 262144, 266 -> 364 at 10^6).  A list (the cells whose rings a step rewrote)
  // is short.
  if (a.list || a.n <= kGeomSlotCells) {
    const int full = (a.n + 31) / 32;
    k_geom_slots<<<(blocks > 0 && blocks < full) ? blocks : full, kSlotThreads, 0, st>>>(a);
    return;
  }
  const int full = (a.n + kGeomThreads - 1) / kGeomThreads;
  k_geom<<<(blocks > 0 && blocks < full) ? blocks : full, kGeomThreads, 0, st>>>(a);
}
void launch_force(const ForceArgs& a, cudaStream_t st, int blocks) {
  if (a.n <= 0) return;
  // While all cells fit on the chip at once, a warp per slot shortens the chain
  // of gathers (one pass, us: 14.3 -> 9.4 at 256 cells, 14.3 -> 10.2 at 4096,
  // 16.4 -> 12.3 at 16384); beyond, the lanes that idle in the last slots and
  // the barriers cost more (18.4 -> 24.6 at 65536).
  if (!a.tolerant && a.integrate != 2 && (a.list || a.n <= kForceSlotCells)) {
    const int full = (a.n + 31) / 32;
    k_force_slots<<<(blocks > 0 && blocks < full) ? blocks : full, kSlotThreads, 0, st>>>(a);
    return;
  }
  const int full = (a.n + kForceThreads - 1) / kForceThreads;
  k_force<<<(blocks > 0 && blocks < full) ? blocks : full, kForceThreads, 0, st>>>(a);
}
void launch_force_fix_list(const ForceFixArgs& a, int blocks, cudaStream_t st) {
  if (a.n > 0) k_force_fix_list<<<blocks, 128, 0, st>>>(a);
}
void launch_begin_topology(Ctl* ctl, int flip, cudaStream_t st) { k_begin_topology<<<1, 1, 0, st>>>(ctl, flip); }
void launch_test(const TestArgs& a, cudaStream_t st, int blocks) {
  if (a.n <= 0) return;
  // As for the force: 17.0 -> 13.6 us at 16384 cells, 15.7 -> 14.4 at 24576
  // (cell list included in the slots' times only), 17.2 -> 19.4 at 65536.
  if (a.n <= kTestSlotCells) {
    const int full = (a.n + 31) / 32;
    k_test_slots<<<(blocks > 0 && blocks < full) ? blocks : full, kSlotThreads, 0, st>>>(a);
    return;
  }
  const int full = (a.n + kTestThreads - 1) / kTestThreads;
  k_test<<<(blocks > 0 && blocks < full) ? blocks : full, kTestThreads, 0, st>>>(a);
}

}  // namespace cgk
