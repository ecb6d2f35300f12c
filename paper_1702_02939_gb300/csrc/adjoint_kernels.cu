// Backward pass of the SPV step: Hessian-vector products and parameter
// cotangents (Sussman, arXiv 1702.02939, Eq. 3 with forces of Eqs. A6-A16).
//
// With the director noise replayed from the seed, the step map is
//   r' = r + dt (mu F(r) + v0 n(theta)),  F = -grad E,
// whose transposed Jacobian is I - dt mu H(r), H the symmetric Hessian of E.
// Reverse accumulation therefore needs H g for the running cotangent g; it is
// computed here as the forward-mode derivative of -F along g on the frozen
// topology of the step.  The tangent of every geometric quantity follows from
// the definitions:
//   circumcentre u of (0, a, b):  u.a = |a|^2/2, u.b = |b|^2/2
//       => [a; b] udot = [(a-u).adot; (b-u).bdot]
//   A = 1/2 sum u_a x u_{a+1},  P = sum |e_a|, e_a = u_a - u_{a-1}
//   edot-hat = (edot - e^ (e^.edot)) / |e|
//   force sets fs = ka/2 perp(u_next - u_prev) + kp (e^_a - e^_next)
//   net force  F_i = -sum_a s_a (w_a . G_a), s = u/det, w = perp(b - a).
// Parameter cotangents use the same tangents of A and P along g:
//   dL/dp0_i += dt mu 2 K_P sqrt(A0) Pdot_i
//   dL/dK_A  += -dt mu sum_c 2 (A_c - A0) Adot_c
//   dL/dK_P  += -dt mu sum_c 2 (P_c - P0_c) Pdot_c
//   dL/dv0_i += dt g_i . n(theta_i)
#include "cg_device.cuh"
#include "cg_kernels.h"

namespace cgk {

__device__ __forceinline__ double i2d_exact_a(long long v) {
  return __longlong_as_double(0x4338000000000000LL + v) - 0x1.8p52;
}

// A, P, the force sets and their tangents along v.  One thread per (cell, ring
// slot): a block takes 32 cells, its warp w the slots w, w + 8 of all of them
// (lane = cell).  Offsets, circumcentres, edges and their tangents pass
// between slots through shared memory; the first warp adds up the cell's sums
// while the last one forms the director's cotangent.  One thread per cell left
// each lane a chain of ~400 FP64 operations per slot (41 us at 4096 cells, one
// warp per SM); this way 14 us.  Divisions and square roots by fx_rcp and
// fx_rsqrt (within 1 ulp, no FP64 instruction).
__global__ void __launch_bounds__(kSlotThreads, kJvpSlotBlocks) k_geom_jvp(JvpArgs g) {
  __shared__ double2 s_a[CG_RING][32], s_t[CG_RING][32];  // offsets and tangents, then unit edges and theirs
  __shared__ double2 s_u[CG_RING][32], s_v[CG_RING][32];  // circumcentres and their tangents
  __shared__ double2 s_A[CG_RING][32], s_P[CG_RING][32];  // terms of A and P and their tangents
  __shared__ double2 s_k[32], s_kd[32];                   // ka, kp and their tangents
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t N = (size_t)g.n;
  const int i = blockIdx.x * 32 + c;
  const size_t off = g.flat ? 0 : (size_t)g.ctl->cur * N;
  const long long* __restrict__ X = g.X + off;
  const long long* __restrict__ Y = g.Y + off;
  int m = 0;
  double2 vi = make_double2(0.0, 0.0);
  if (i < g.n) {
    m = g.cnt[i];
    if (m < 3 || m > CG_RING) {
      if (w == 0) raise_status(g.ctl, kETOPO);
      m = 0;
    }
    vi = g.v[i];
    const Rep& R = g.reps[g.rep[i]];
    const double sc = R.inv_scale;
    const long long Xi = X[i], Yi = Y[i], LX = R.LX, LY = R.LY;
    for (int a = w; a < m; a += kSlotWarps) {
      const int j = g.nbr[(size_t)i * CG_RING + a];
      const double2 vj = g.v[j];
      s_a[a][c] = make_double2(i2d_exact_a(min_image_i(X[j] - Xi, LX)) * sc, i2d_exact_a(min_image_i(Y[j] - Yi, LY)) * sc);
      s_t[a][c] = make_double2(vj.x - vi.x, vj.y - vi.y);
    }
  }
  __syncthreads();
  for (int a = w; a < m; a += kSlotWarps) {
    const int an = a + 1 < m ? a + 1 : 0;
    const double2 A = s_a[a][c], B = s_a[an][c], Ad = s_t[a][c], Bd = s_t[an][c];
    const double la = A.x * A.x + A.y * A.y, lb = B.x * B.x + B.y * B.y;
    const double r = fx_rcp(A.x * B.y - A.y * B.x);
    const double ux = 0.5 * (B.y * la - A.y * lb) * r;
    const double uy = 0.5 * (A.x * lb - B.x * la) * r;
    const double ra = (A.x - ux) * Ad.x + (A.y - uy) * Ad.y;
    const double rb = (B.x - ux) * Bd.x + (B.y - uy) * Bd.y;
    const double udx = (B.y * ra - A.y * rb) * r;
    const double udy = (A.x * rb - B.x * ra) * r;
    const double detd = Ad.x * B.y + A.x * Bd.y - Ad.y * B.x - A.y * Bd.x;
    g.s[a * N + i] = make_double2(ux * r, uy * r);
    g.sd[a * N + i] = make_double2(udx * r - ux * detd * r * r, udy * r - uy * detd * r * r);
    g.w[a * N + i] = make_double2(B.y - A.y, A.x - B.x);
    g.wd[a * N + i] = make_double2(Bd.y - Ad.y, Ad.x - Bd.x);
    s_u[a][c] = make_double2(ux, uy);
    s_v[a][c] = make_double2(udx, udy);
  }
  __syncthreads();
  for (int a = w; a < m; a += kSlotWarps) {
    const int ap = a > 0 ? a - 1 : m - 1;
    const double2 p = s_u[ap][c], pd = s_v[ap][c], h = s_u[a][c], hd = s_v[a][c];
    s_A[a][c] = make_double2(p.x * h.y - h.x * p.y, pd.x * h.y + p.x * hd.y - hd.x * p.y - h.x * pd.y);
    const double ex = h.x - p.x, ey = h.y - p.y, edx = hd.x - pd.x, edy = hd.y - pd.y;
    const double l2 = ex * ex + ey * ey;
    const double il = fx_rsqrt(l2);
    const double nx = ex * il, ny = ey * il;
    const double dl = nx * edx + ny * edy;
    s_P[a][c] = make_double2(l2 * il, dl);
    s_a[a][c] = make_double2(nx, ny);
    s_t[a][c] = make_double2((edx - nx * dl) * il, (edy - ny * dl) * il);
  }
  __syncthreads();
  if (w == kSlotWarps - 1 && m && g.gp0) {
    double sn, cs;
    sincos(g.theta[i], &sn, &cs);
    g.gv0[i] += g.dt * (vi.x * cs + vi.y * sn);
  }
  if (w == 0 && m) {
    double A = 0.0, Ad = 0.0, P = 0.0, Pd = 0.0;
    for (int a = 0; a < m; ++a) {
      const double2 tA = s_A[a][c], tP = s_P[a][c];
      A += tA.x;
      Ad += tA.y;
      P += tP.x;
      Pd += tP.y;
    }
    A *= 0.5;
    Ad *= 0.5;
    const double P0 = g.p0[i] * g.sqrtA0;
    double ka, kp, kad, kpd;
    if (g.coefA) {
      ka = g.coefA[i]; kp = g.coefP[i]; kad = 0.0; kpd = 0.0;
    } else {
      ka = 2.0 * g.KA * (A - g.A0); kp = 2.0 * g.KP * (P - P0);
      kad = 2.0 * g.KA * Ad; kpd = 2.0 * g.KP * Pd;
    }
    s_k[c] = make_double2(ka, kp);
    s_kd[c] = make_double2(kad, kpd);
    if (g.Adot) g.Adot[i] = Ad;
    if (g.Pdot) g.Pdot[i] = Pd;
    if (g.gp0) {  // parameter cotangents along v = g_{t+1}
      g.gp0[i] += g.dtmu * 2.0 * g.KP * g.sqrtA0 * Pd;
      g.gKA[i] += -g.dtmu * 2.0 * (A - g.A0) * Ad;
      g.gKP[i] += -g.dtmu * 2.0 * (P - P0) * Pd;
    }
  }
  __syncthreads();
  const double2 k = s_k[c], kd = s_kd[c];
  for (int a = w; a < m; a += kSlotWarps) {
    const int ap = a > 0 ? a - 1 : m - 1, an = a + 1 < m ? a + 1 : 0;
    const double2 hn = s_u[an][c], hp = s_u[ap][c], vn = s_v[an][c], vp = s_v[ap][c];
    const double gx = 0.5 * (hn.y - hp.y), gy = 0.5 * (hp.x - hn.x);
    const double gdx = 0.5 * (vn.y - vp.y), gdy = 0.5 * (vp.x - vn.x);
    const double2 e = s_a[a][c], en = s_a[an][c], ed = s_t[a][c], end = s_t[an][c];
    const double qx = e.x - en.x, qy = e.y - en.y;
    const double qdx = ed.x - end.x, qdy = ed.y - end.y;
    g.fs[a * N + i] = make_double2(k.x * gx + k.y * qx, k.x * gy + k.y * qy);
    g.fsd[a * N + i] = make_double2(kd.x * gx + k.x * gdx + kd.y * qx + k.y * qdx,
                                    kd.x * gy + k.x * gdy + kd.y * qy + k.y * qdy);
  }
}

// H g = -Fdot and the cotangent update g <- g - dt mu H g (in place: this
// kernel reads only per-slot data written by k_geom_jvp).  One thread per
// (cell, ring slot) as k_geom_jvp; the first warp adds the slots' terms up in
// ring order.
__global__ void __launch_bounds__(kSlotThreads, kJvpSlotBlocks) k_force_jvp(JvpArgs g) {
  __shared__ double2 s_s[CG_RING][32], s_sd[CG_RING][32], s_c[CG_RING][32];
  __shared__ int s_j[CG_RING][32], s_p[CG_RING][32];
  __shared__ int s_bad[32];
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t N = (size_t)g.n;
  const int i = blockIdx.x * 32 + c;
  int m = i < g.n ? g.cnt[i] : 0;
  if (m < 3 || m > CG_RING) m = 0;
  bool bad = false;
  if (w == 0) s_bad[c] = 0;
  for (int a = w; a < m; a += kSlotWarps) {
    const int j = g.nbr[(size_t)i * CG_RING + a];
    const int mj = g.cnt[j], p = ring_pos(g.nbr, g.cnt, j, i);
    bad |= p < 0;
    // triangle (i, j, k) is the slot before i's around j and i's slot around k
    s_p[a][c] = (p < 0 ? 0 : p) | ((p <= 0 ? (mj > 0 ? mj - 1 : 0) : p - 1) << 8);
    s_j[a][c] = j;
  }
  __syncthreads();
  if (bad) s_bad[c] = 1;
  for (int a = w; a < m; a += kSlotWarps) {
    const int an = a + 1 < m ? a + 1 : 0;
    const size_t o0 = a * N + i, o1 = (size_t)(s_p[a][c] >> 8) * N + s_j[a][c],
                 o2 = (size_t)(s_p[an][c] & 255) * N + s_j[an][c];
    const double2 f0 = g.fs[o0], f1 = g.fs[o1], f2 = g.fs[o2];
    const double2 e0 = g.fsd[o0], e1 = g.fsd[o1], e2 = g.fsd[o2];
    const double2 wj = g.w[o0], wd = g.wd[o0];
    s_s[a][c] = g.s[o0];
    s_sd[a][c] = g.sd[o0];
    const double Gx = f0.x + f1.x + f2.x, Gy = f0.y + f1.y + f2.y;
    const double Gdx = e0.x + e1.x + e2.x, Gdy = e0.y + e1.y + e2.y;
    s_c[a][c] = make_double2(wj.x * Gx + wj.y * Gy, wd.x * Gx + wd.y * Gy + wj.x * Gdx + wj.y * Gdy);
  }
  __syncthreads();
  if (w || !m) return;
  double Fdx = 0.0, Fdy = 0.0, Fx = 0.0, Fy = 0.0;
  for (int a = 0; a < m; ++a) {
    const double2 sj = s_s[a][c], sd = s_sd[a][c], cc = s_c[a][c];
    Fx -= sj.x * cc.x;
    Fy -= sj.y * cc.x;
    Fdx -= sd.x * cc.x + sj.x * cc.y;
    Fdy -= sd.y * cc.x + sj.y * cc.y;
  }
  if (s_bad[c]) raise_status(g.ctl, kETOPO);
  if (g.F) g.F[i] = make_double2(Fx, Fy);
  if (g.Hv) g.Hv[i] = make_double2(-Fdx, -Fdy);
  if (g.update) {
    double2 gi = g.v[i];
    gi.x += g.dtmu * Fdx;  // g - dt mu H g, H g = -Fdot
    gi.y += g.dtmu * Fdy;
    g.v[i] = gi;
  }
}

// g = (gx, gy) - F_coef : cotangent of the final positions, where F_coef is the
// "force" of the loss coefficients (minus the gradient of sum cA A + cP P).
__global__ void k_combine_final(int n, const double* gx, const double* gy, const double2* F, double2* g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) g[i] = make_double2(gx[i] - F[i].x, gy[i] - F[i].y);
}

__global__ void k_reduce2(int n, const double* a, const double* b, double* out) {
  __shared__ double sa[1024], sb[1024];
  double x = 0.0, y = 0.0;
  for (int i = threadIdx.x; i < n; i += 1024) {
    x += a[i];
    y += b[i];
  }
  sa[threadIdx.x] = x;
  sb[threadIdx.x] = y;
  __syncthreads();
  for (int o = 512; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sa[threadIdx.x] += sa[threadIdx.x + o];
      sb[threadIdx.x] += sb[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = sa[0];
    out[1] = sb[0];
  }
}

// Ring i as 16-byte words.
__device__ __forceinline__ void copy_row(int* dst, const int* src, int i) {
  const int4* q = reinterpret_cast<const int4*>(src + (size_t)i * CG_RING);
  const int4 r0 = q[0], r1 = q[1], r2 = q[2], r3 = q[3];
  int4* d = reinterpret_cast<int4*>(dst + (size_t)i * CG_RING);
  d[0] = r0;
  d[1] = r1;
  d[2] = r2;
  d[3] = r3;
}

// Snapshot of the current state (positions of the current buffer, grid
// coordinates, directors, rings, control word) to / from a flat buffer.
__global__ void k_snapshot(int n, int save, Ctl* ctl, double* x, double* y, long long* X, long long* Y, double* theta,
                           int* cnt, int* nbr, Snapshot s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const size_t N = (size_t)n;
  const int cur = save ? ctl->cur : s.ctl->cur;
  if (i < n) {
    if (save) {
      s.x[i] = x[cur * N + i]; s.y[i] = y[cur * N + i];
      s.X[i] = X[cur * N + i]; s.Y[i] = Y[cur * N + i];
      s.theta[i] = theta[i];
      s.cnt[i] = cnt[i];
      copy_row(s.nbr, nbr, i);
    } else {
      x[cur * N + i] = s.x[i]; y[cur * N + i] = s.y[i];
      X[cur * N + i] = s.X[i]; Y[cur * N + i] = s.Y[i];
      theta[i] = s.theta[i];
      cnt[i] = s.cnt[i];
      copy_row(nbr, s.nbr, i);
    }
  }
  if (i == 0) {
    if (save) *s.ctl = *ctl;
    else *ctl = *s.ctl;
  }
}

void launch_snapshot(int n, int save, Ctl* ctl, double* x, double* y, long long* X, long long* Y, double* theta,
                     int* cnt, int* nbr, const Snapshot& s, cudaStream_t st) {
  k_snapshot<<<(n + 127) / 128, 128, 0, st>>>(n, save, ctl, x, y, X, Y, theta, cnt, nbr, s);
}

void launch_geom_jvp(const JvpArgs& a, cudaStream_t st) {
  if (a.n > 0) k_geom_jvp<<<(a.n + 31) / 32, kSlotThreads, 0, st>>>(a);
}
void launch_force_jvp(const JvpArgs& a, cudaStream_t st) {
  if (a.n > 0) k_force_jvp<<<(a.n + 31) / 32, kSlotThreads, 0, st>>>(a);
}
void launch_combine_final(int n, const double* gx, const double* gy, const double2* F, double2* g, cudaStream_t st) {
  if (n > 0) k_combine_final<<<(n + 255) / 256, 256, 0, st>>>(n, gx, gy, F, g);
}
void launch_reduce2(int n, const double* a, const double* b, double* out, cudaStream_t st) {
  k_reduce2<<<1, 1024, 0, st>>>(n, a, b, out);
}

}  // namespace cgk
