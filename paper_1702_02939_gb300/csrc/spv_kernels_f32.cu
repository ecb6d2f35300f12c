// SPV step kernels in single precision: geometry + force sets, net force +
// move, and the director terms, with every floating-point operation of the
// physics in FP32 (Sussman, arXiv 1702.02939: the code builds in single or
// double precision and times both, Sec. 3 and Fig. 2).
//
// What stays exact: positions live on the dyadic grid as int64 (the move is
// accumulated and rounded to the grid in FP64), and the circumcircle test and
// repair decide every predicate exactly in integer arithmetic, so the
// triangulation of a given state is the same as in double precision.  What
// changes: A, P, the forces, n(theta) and the noise carry FP32 rounding
// (relative 2^-24 per operation).  On GB300 the FP32 pipe issues about 74
// times as many operations per clock as the FP64 pipe.
//
// Same formulas and layouts as the FP64 kernels (spv_kernels.cu), in real
// units: the per-slot arrays fs, s, w hold float2 values in the first half of
// their double2 buffers.
#include "cg_device.cuh"
#include "cg_kernels.h"

namespace cgk {

namespace {

__device__ __forceinline__ float2* as_f2(double2* p) { return reinterpret_cast<float2*>(p); }
__device__ __forceinline__ const float2* as_f2(const double2* p) { return reinterpret_cast<const float2*>(p); }

// Relative position of cell j seen from cell i: exact grid difference
// (minimum image) and its float value in real units (relative error
// <= 2u + u^2).
__device__ __forceinline__ void rel_f(const Rep& R, const long long* X, const long long* Y, long long Xi,
                                      long long Yi, int j, float sc, long long& gx, long long& gy, float& dx,
                                      float& dy) {
  gx = min_image_i(X[j] - Xi, R.LX);
  gy = min_image_i(Y[j] - Yi, R.LY);
  dx = i2f_scaled(gx, sc);
  dy = i2f_scaled(gy, sc);
}

// (a x b) in real units from the exact grid coordinates: the 128-bit
// determinant, then to float.  A float determinant of the rounded relative
// positions can vanish for two nearly coincident neighbours; this one is the
// exact value rounded once (positive for every triangle of the triangulation).
__device__ __forceinline__ float det_f(long long ax, long long ay, long long bx, long long by, float sc) {
  const __int128 d = (__int128)ax * by - (__int128)ay * bx;
  const bool neg = d < 0;
  const unsigned __int128 m = neg ? (unsigned __int128)(-d) : (unsigned __int128)d;
  const unsigned long long hi = (unsigned long long)(m >> 64), lo = (unsigned long long)m;
  // hi * 2^64 + lo with hi < 2^63; the low half enters as 2 (lo >> 1) (its last
  // bit is below the float resolution); relative error ~3u
  const float f = i2f_scaled((long long)hi, 0x1p64f * sc * sc) + i2f_scaled((long long)(lo >> 1), 2.0f * sc * sc);
  return neg ? -f : f;
}

// The circumcentre (relative to the cell) of its neighbours a and b and the
// Jacobian factor h / det; l: squared lengths of a and b.
__device__ __forceinline__ void vertex_f(long long gax, long long gay, long long gbx, long long gby, float ax, float ay,
                                         float la, float bx, float by, float lb, float sc, float2& h, float2& s) {
  const float r = 1.0f / det_f(gax, gay, gbx, gby, sc);  // 1 / ((r_j - r_i) x (r_k - r_i))
  const float hr = 0.5f * r;
  h = make_float2(fmaf(by, la, -(ay * lb)) * hr, fmaf(ax, lb, -(bx * la)) * hr);
  s = make_float2(h.x * r, h.y * r);
}

// The edge from vertex hp to h: (squared length, inverse length) and its unit
// vector; a zero-length edge has no direction.
__device__ __forceinline__ void edge_f(float2 h, float2 hp, float2& l, float2& e) {
  const float ex = h.x - hp.x, ey = h.y - hp.y;
  const float l2 = fmaf(ex, ex, ey * ey);
  const float il = l2 > 0.f ? rsqrtf(l2) : 0.f;
  l = make_float2(l2, il);
  e = make_float2(ex * il, ey * il);
}

// A, P and the energy of cell i from its accumulated sums; returns (ka, kp).
__device__ __forceinline__ float2 cell_f(const GeomArgs& g, int i, float area, float per) {
  const float A = 0.5f * area, P = per;
  g.A[i] = A;
  g.P[i] = P;
  const float dA = A - (float)g.A0, dP = P - (float)(g.p0[i] * g.sqrtA0);
  if (g.energy_out) g.energy_out[i] = (double)fmaf((float)g.KA * dA, dA, (float)g.KP * dP * dP);
  // dA/dh = 1/2 perp(h_next - h_prev); dP/dh = e_in - e_out
  return make_float2((float)g.KA * dA, 2.0f * (float)g.KP * dP);
}

}  // namespace

// One thread per cell (grid-stride; optional list of cells; tolerant mode for
// the pass beside the repair rounds), as k_geom.  Bound by the latency of the
// neighbours' gathers: the next one is loaded ahead, and with eight slots of a
// ring in shared memory (4 KB per block; the rest of a longer ring is local) 28
// blocks fit on an SM and leave L1 to the gathers (pass, us: 30.7 -> 26.9 at
// 262144 cells, 88 -> 75.7 at 10^6).
__global__ void __launch_bounds__(kGeomThreads, 28) k_geom_f32(GeomArgs g) {
  // vertex a, and the unit vector of the edge ending at it
  __shared__ float2 sh_h[kGeomSh][kGeomThreads], sh_e[kGeomSh][kGeomThreads];
  float2 long_h[CG_RING - kGeomSh], long_e[CG_RING - kGeomSh];
  const int t = threadIdx.x;
  auto put_h = [&](int a, float2 v) { if (a < kGeomSh) sh_h[a][t] = v; else long_h[a - kGeomSh] = v; };
  auto put_e = [&](int a, float2 v) { if (a < kGeomSh) sh_e[a][t] = v; else long_e[a - kGeomSh] = v; };
  auto get_h = [&](int a) { return a < kGeomSh ? sh_h[a][t] : long_h[a - kGeomSh]; };
  auto get_e = [&](int a) { return a < kGeomSh ? sh_e[a][t] : long_e[a - kGeomSh]; };
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  float2* fs = as_f2(g.fs);
  float2* sv = as_f2(g.s);
  float2* wv = as_f2(g.w);
  for (int item = blockIdx.x * kGeomThreads + t; item < g.n; item += gridDim.x * kGeomThreads) {
    const int i = g.order ? g.order[item] : item;
    const Rep R = g.reps[g.rep[i]];
    const float sc = (float)R.inv_scale;
    const long long Xi = X[i], Yi = Y[i];
    const int m = g.cnt[i];
    if (m < 3 || m > CG_RING) {
      if (!g.tolerant) raise_status(g.ctl, kETOPO);
      continue;
    }
    const int* ring = g.nbr + (size_t)i * CG_RING;
    auto nb = [&](int a) {
      const int j = ring[a];
      return ((unsigned)j < (unsigned)g.n) ? j : i;
    };
    long long g0x, g0y;
    float d0x, d0y;
    rel_f(R, X, Y, Xi, Yi, nb(0), sc, g0x, g0y, d0x, d0y);
    const float l0 = fmaf(d0x, d0x, d0y * d0y);
    float ax = d0x, ay = d0y, la = l0;
    long long gax = g0x, gay = g0y;
    int jq = nb(1);  // the neighbour whose position is loaded ahead
    long long qX = X[jq], qY = Y[jq];
    float hpx = 0.f, hpy = 0.f, h0x = 0.f, h0y = 0.f;
    float area = 0.f, per = 0.f;
    for (int a = 0; a < m; ++a) {
      float bx, by, lb;
      long long gbx, gby;
      if (a + 1 < m) {
        gbx = min_image_i(qX - Xi, R.LX);
        gby = min_image_i(qY - Yi, R.LY);
        if (a + 2 < m) {
          jq = nb(a + 2);
          qX = X[jq];
          qY = Y[jq];
        }
        bx = i2f_scaled(gbx, sc);
        by = i2f_scaled(gby, sc);
        lb = fmaf(bx, bx, by * by);
      } else {
        bx = d0x; by = d0y; lb = l0;
        gbx = g0x; gby = g0y;
      }
      float2 h, sj;
      vertex_f(gax, gay, gbx, gby, ax, ay, la, bx, by, lb, sc, h, sj);
      const float hx = h.x, hy = h.y;
      sv[a * N + i] = sj;
      wv[a * N + i] = make_float2(by - ay, ax - bx);
      put_h(a, h);
      if (a == 0) {
        h0x = hx; h0y = hy;
      } else {
        area += fmaf(hpx, hy, -(hx * hpy));
        float2 l, e;
        edge_f(h, make_float2(hpx, hpy), l, e);
        per = fmaf(l.x, l.y, per);
        put_e(a, e);
      }
      hpx = hx; hpy = hy;
      ax = bx; ay = by; la = lb;
      gax = gbx; gay = gby;
    }
    {  // closing edge h_{m-1} -> h_0 is the incoming edge of vertex 0
      area += fmaf(hpx, h0y, -(h0x * hpy));
      float2 l, e;
      edge_f(make_float2(h0x, h0y), make_float2(hpx, hpy), l, e);
      per = fmaf(l.x, l.y, per);
      sh_e[0][t] = e;
    }
    const float2 k = cell_f(g, i, area, per);
    const float ka = k.x, kp = k.y;
    for (int a = 0; a < m; ++a) {
      const int ap = (a == 0) ? m - 1 : a - 1;
      const int an = (a + 1 == m) ? 0 : a + 1;
      const float2 hn = get_h(an), hb = get_h(ap), ea = get_e(a), en = get_e(an);
      const float gx = hn.y - hb.y, gy = hb.x - hn.x;
      const float dPx = ea.x - en.x, dPy = ea.y - en.y;
      fs[a * N + i] = make_float2(fmaf(ka, gx, kp * dPx), fmaf(ka, gy, kp * dPy));
    }
  }
}

// The same pass with one thread per (cell, ring slot), as k_geom_slots.
__global__ void __launch_bounds__(kSlotThreads, kGeomF32SlotBlocks) k_geom_f32_slots(GeomArgs g) {
  __shared__ longlong2 s_off[CG_RING][32];  // neighbour offsets, exact
  __shared__ float2 s_d[CG_RING][32];       // and rounded, then unit edge vectors
  __shared__ float2 s_h[CG_RING][32];       // circumcentres
  __shared__ float2 s_l[CG_RING][32];       // edge ending at the slot: squared length, inverse length
  __shared__ float2 s_k[32];                // the cell's ka, kp
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const long long* __restrict__ X = g.X + (size_t)cur * N;
  const long long* __restrict__ Y = g.Y + (size_t)cur * N;
  float2* fs = as_f2(g.fs);
  float2* sv = as_f2(g.s);
  float2* wv = as_f2(g.w);
  const int total = g.list ? *g.list_count : g.n;
  if (g.clear)
    for (int k = blockIdx.x * kSlotThreads + threadIdx.x; k < g.n_clear; k += gridDim.x * kSlotThreads) g.clear[k] = 0;
  for (int base = blockIdx.x * 32; base < total; base += gridDim.x * 32) {
    const int item = base + c;
    int i = 0, m = 0;
    float sc = 0.f;
    if (item < total) {
      i = g.list ? g.list[item] : (g.order ? g.order[item] : item);
      m = g.cnt[i];
      if (w == 0) {
        if (g.list_bits) atomicAnd(&g.list_bits[i >> 5], ~(1u << (i & 31)));
        if ((m < 3 || m > CG_RING) && !g.tolerant) raise_status(g.ctl, kETOPO);
      }
      if (m < 3 || m > CG_RING) m = 0;
    }
    if (w < m) {
      const Rep& R = g.reps[g.rep[i]];
      sc = (float)R.inv_scale;
      const int* ring = g.nbr + (size_t)i * CG_RING;
      const long long Xi = X[i], Yi = Y[i], LX = R.LX, LY = R.LY;
      for (int a = w; a < m; a += kSlotWarps) {
        int j = ring[a];
        j = ((unsigned)j < (unsigned)g.n) ? j : i;
        const long long dX = min_image_i(X[j] - Xi, LX), dY = min_image_i(Y[j] - Yi, LY);
        s_off[a][c] = make_longlong2(dX, dY);
        s_d[a][c] = make_float2(i2f_scaled(dX, sc), i2f_scaled(dY, sc));
      }
    }
    __syncthreads();
    for (int a = w; a < m; a += kSlotWarps) {
      const int an = a + 1 < m ? a + 1 : 0;
      const longlong2 A = s_off[a][c], B = s_off[an][c];
      const float2 da = s_d[a][c], db = s_d[an][c];
      float2 h, sj;
      vertex_f(A.x, A.y, B.x, B.y, da.x, da.y, fmaf(da.x, da.x, da.y * da.y), db.x, db.y,
               fmaf(db.x, db.x, db.y * db.y), sc, h, sj);
      sv[a * N + i] = sj;
      wv[a * N + i] = make_float2(db.y - da.y, da.x - db.x);
      s_h[a][c] = h;
    }
    __syncthreads();
    for (int a = w; a < m; a += kSlotWarps) {
      float2 l, e;
      edge_f(s_h[a][c], s_h[a > 0 ? a - 1 : m - 1][c], l, e);
      s_l[a][c] = l;
      s_d[a][c] = e;
    }
    __syncthreads();
    if (w == 0 && m) {
      float area = 0.f, per = 0.f;
      for (int a = 1; a <= m; ++a) {
        const int b = a < m ? a : 0;
        const float2 hp = s_h[a - 1][c], h = s_h[b][c], l = s_l[b][c];
        area += fmaf(hp.x, h.y, -(h.x * hp.y));
        per = fmaf(l.x, l.y, per);
      }
      s_k[c] = cell_f(g, i, area, per);
    }
    __syncthreads();
    const float2 k = s_k[c];
    for (int a = w; a < m; a += kSlotWarps) {
      const int ap = a > 0 ? a - 1 : m - 1, an = a + 1 < m ? a + 1 : 0;
      const float2 hp = s_h[ap][c], hn = s_h[an][c], e = s_d[a][c], en = s_d[an][c];
      const float gx = hn.y - hp.y, gy = hp.x - hn.x;
      const float dPx = e.x - en.x, dPy = e.y - en.y;
      fs[a * N + i] = make_float2(fmaf(k.x, gx, k.y * dPx), fmaf(k.x, gy, k.y * dPy));
    }
    __syncthreads();
  }
}

// The first half of a ring's row (most rings end within it), loaded ahead of
// its use, and the slots of cell i and of the entry before it in that ring,
// packed as slot | before << 8; -1 when the ring does not list i.  Entries past
// a ring's end are -1, so the row alone tells.
struct RingHead {
  int4 a, b;
  __device__ __forceinline__ void load(const int* __restrict__ nbr, int j) {
    const int4* row = reinterpret_cast<const int4*>(nbr + (size_t)j * CG_RING);
    a = row[0];
    b = row[1];
  }
  __device__ __forceinline__ int slots(const int* __restrict__ nbr, int j, int i) const {
    int p = a.x == i ? 0 : a.y == i ? 1 : a.z == i ? 2 : a.w == i ? 3 : b.x == i ? 4 : b.y == i ? 5 : b.z == i ? 6
          : b.w == i ? 7 : -1;
    if (p > 0) return p | ((p - 1) << 8);
    int last = 2 + (a.w >= 0) + (b.x >= 0) + (b.y >= 0) + (b.z >= 0) + (b.w >= 0);
    if (b.w >= 0) {  // the ring may go on
      const int4* row = reinterpret_cast<const int4*>(nbr + (size_t)j * CG_RING);
      const int4 c = row[2], d = row[3];
      if (p < 0) {
        p = c.x == i ? 8 : c.y == i ? 9 : c.z == i ? 10 : c.w == i ? 11 : d.x == i ? 12 : d.y == i ? 13 : d.z == i ? 14
            : d.w == i ? 15 : -1;
        return p < 0 ? -1 : p | ((p - 1) << 8);
      }
      last += (c.x >= 0) + (c.y >= 0) + (c.z >= 0) + (c.w >= 0) + (d.x >= 0) + (d.y >= 0) + (d.z >= 0) + (d.w >= 0);
    }
    return p < 0 ? -1 : last << 8;
  }
};

// Net force on cell i in FP32 from the float force sets (false for a
// malformed ring: status raised, or, in the tolerant pass beside the repair
// rounds, nothing raised and the cell left to the fix-up).
__device__ __forceinline__ bool net_force_f32(const ForceArgs& g, int i, float& fx_out, float& fy_out) {
  const size_t N = (size_t)g.n;
  const float2* fs = as_f2(g.fs);
  const float2* sv = as_f2(g.s);
  const float2* wv = as_f2(g.w);
  const int m = g.cnt[i];
  if (m < 3 || m > CG_RING) {
    if (!g.tolerant) raise_status(g.ctl, kETOPO);
    return false;
  }
  const int* ring = g.nbr + (size_t)i * CG_RING;
  bool bad = false;
  auto nb = [&](int a) {  // a ring being rewritten may hold -1 entries
    const int j = ring[a];
    const bool ok = (unsigned)j < (unsigned)g.n;
    bad |= !ok;
    return ok ? j : i;
  };
  const int jfirst = nb(0);
  RingHead head;
  head.load(g.nbr, jfirst);
  const int pfirst = head.slots(g.nbr, jfirst, i);
  int j = jfirst, pj = pfirst;
  float fx = 0.f, fy = 0.f;
  bad |= pfirst < 0;
  int next = nb(1);  // the neighbour whose row is loaded ahead
  head.load(g.nbr, next);
  for (int a = 0; a < m; ++a) {
    int k, pk;
    if (a + 1 < m) {
      k = next;
      const RingHead cur_head = head;
      if (a + 2 < m) {
        next = nb(a + 2);
        head.load(g.nbr, next);
      }
      pk = cur_head.slots(g.nbr, k, i);
      bad |= pk < 0;
    } else {
      k = jfirst;
      pk = pfirst;
    }
    const float2 f0 = fs[a * N + i];
    const float2 f1 = fs[(size_t)(pj < 0 ? 0 : pj >> 8) * N + j];
    const float2 f2 = fs[(size_t)(pk < 0 ? 0 : pk & 255) * N + k];
    const float Gx = f0.x + f1.x + f2.x, Gy = f0.y + f1.y + f2.y;
    const float2 s = sv[a * N + i], w = wv[a * N + i];
    const float c = fmaf(w.x, Gx, w.y * Gy);
    fx = fmaf(-s.x, c, fx);
    fy = fmaf(-s.y, c, fy);
    j = k;
    pj = pk;
  }
  if (bad) {
    if (g.tolerant) return false;
    raise_status(g.ctl, kETOPO);
  }
  fx_out = fx;
  fy_out = fy;
  return true;
}

// The move of Eq. 3 of cell i under the force (fx, fy), accumulated in FP64 and
// rounded to the grid.
__device__ __forceinline__ void move_cell_f32(const ForceArgs& g, int i, float fx, float fy) {
  const size_t N = (size_t)g.n;
  const int cur = g.ctl->cur;
  const Rep R = g.reps[g.rep[i]];
  const double xi = g.x[(size_t)cur * N + i], yi = g.y[(size_t)cur * N + i];
  const double2 nd = g.nrm[i];  // (cos theta, sin theta), from k_dir_f32
  double v0;
  if (g.v0_user) {  // integrate 2 with new speeds: take them over first
    v0 = g.v0_user[g.tag[i]];
    if (!isfinite(v0)) raise_status(g.ctl, kEINVAL);
    g.v0[i] = v0;
  } else {
    v0 = g.v0[i];
  }
  const double vx = g.mu * (double)fx + v0 * nd.x, vy = g.mu * (double)fy + v0 * nd.y;
  const double xn = fma(g.dt, vx, xi), yn = fma(g.dt, vy, yi);
  long long Xn, Yn;
  if (isfinite(xn) && isfinite(yn)) {
    if (!R.framed) {
      Xn = wrap_to_grid(xn, R.Lx, R.scale, R.LX);
      Yn = wrap_to_grid(yn, R.Ly, R.scale, R.LY);
    } else {
      Xn = move_framed(xi, g.dt, vx, R.x0, R.Lxg, R.scale, R.X0, R.LXg, R.LX);
      Yn = move_framed(yi, g.dt, vy, R.y0, R.Lyg, R.scale, R.Y0, R.LYg, R.LY);
    }
  } else {
    if (g.tolerant) {  // decided again, strictly, after the repair rounds
      claim_fix(g.fix_bits, g.fix_list, &g.ctl->force_count, i);
      return;
    }
    raise_status(g.ctl, kENONFINITE);
    Xn = (long long)rint(xi * R.scale);
    Yn = (long long)rint(yi * R.scale);
  }
  const int nxt = cur ^ 1;
  g.x[(size_t)nxt * N + i] = i2d_exact(Xn) * R.inv_scale;
  g.y[(size_t)nxt * N + i] = i2d_exact(Yn) * R.inv_scale;
  g.X[(size_t)nxt * N + i] = Xn;
  g.Y[(size_t)nxt * N + i] = Yn;
}

// Cell i's net force and, as in k_force, the move of Eq. 3 accumulated in
// FP64 and rounded to the grid (integrate 2: the move alone from the stored
// forces, which hold the FP32 values exactly).
__device__ __forceinline__ void force_cell_f32(const ForceArgs& g, int i) {
  float fx, fy;
  if (g.integrate == 2) {
    fx = (float)g.Fx[i];
    fy = (float)g.Fy[i];
  } else {
    if (!net_force_f32(g, i, fx, fy)) {
      if (g.tolerant) claim_fix(g.fix_bits, g.fix_list, &g.ctl->force_count, i);
      return;
    }
    g.Fx[i] = fx;
    g.Fy[i] = fy;
    if (!g.integrate) return;
  }
  move_cell_f32(g, i, fx, fy);
}

// The same with one thread per (cell, ring slot), as k_force_slots.
__global__ void __launch_bounds__(kSlotThreads, kForceF32SlotBlocks) k_force_f32_slots(ForceArgs g) {
  __shared__ float2 s_s[CG_RING][32];  // Jacobian factors
  __shared__ float s_c[CG_RING][32];   // w . G
  __shared__ int s_j[CG_RING][32];     // neighbours
  __shared__ int s_p[CG_RING][32];     // the cell's slot in the neighbour's ring, and the one before it
  __shared__ int s_bad[32];
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5;
  const size_t N = (size_t)g.n;
  const float2* fs = as_f2(g.fs);
  const float2* sv = as_f2(g.s);
  const float2* wv = as_f2(g.w);
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
    for (int a = w; a < m; a += kSlotWarps) {
      int j = g.nbr[(size_t)i * CG_RING + a];
      const bool ok = (unsigned)j < (unsigned)g.n;
      j = ok ? j : i;
      const int mj = g.cnt[j], p = ring_pos(g.nbr, g.cnt, j, i);
      bad |= !ok || p < 0;
      s_p[a][c] = (p < 0 ? 0 : p) | ((p <= 0 ? (mj > 0 ? mj - 1 : 0) : p - 1) << 8);
      s_j[a][c] = j;
    }
    __syncthreads();
    if (bad) s_bad[c] = 1;
    for (int a = w; a < m; a += kSlotWarps) {
      const int an = a + 1 < m ? a + 1 : 0;
      const float2 f0 = fs[a * N + i];
      const float2 f1 = fs[(size_t)(s_p[a][c] >> 8) * N + s_j[a][c]];
      const float2 f2 = fs[(size_t)(s_p[an][c] & 255) * N + s_j[an][c]];
      const float2 wj = wv[a * N + i];
      s_s[a][c] = sv[a * N + i];
      const float Gx = f0.x + f1.x + f2.x, Gy = f0.y + f1.y + f2.y;
      s_c[a][c] = fmaf(wj.x, Gx, wj.y * Gy);
    }
    __syncthreads();
    if (w == 0 && m) {
      if (s_bad[c]) raise_status(g.ctl, kETOPO);
      float fx = 0.f, fy = 0.f;
      for (int a = 0; a < m; ++a) {
        const float2 sj = s_s[a][c];
        const float cj = s_c[a][c];
        fx = fmaf(-sj.x, cj, fx);
        fy = fmaf(-sj.y, cj, fy);
      }
      g.Fx[i] = fx;
      g.Fy[i] = fy;
      if (g.integrate) move_cell_f32(g, i, fx, fy);
    }
    __syncthreads();
  }
}

// One thread per cell, or grid-stride over a list (bits cleared), as k_force.
// Bound by the latency of its gathers: the next neighbour's row is loaded ahead
// and ten blocks per SM are asked for (pass, us: 32.8 -> 30.7 at 262144 cells,
// 92 -> 84 at 10^6).
__global__ void __launch_bounds__(kForceThreads, 10) k_force_f32(ForceArgs g) {
  const int total = g.list ? *g.list_count : g.n;
  for (int item = blockIdx.x * kForceThreads + threadIdx.x; item < total; item += gridDim.x * kForceThreads) {
    const int i = g.list ? g.list[item] : (g.order ? g.order[item] : item);
    if (g.list_bits) atomicAnd(&g.list_bits[i >> 5], ~(1u << (i & 31)));
    force_cell_f32(g, i);
  }
}

// Director terms in FP32: n(theta) of the float director, and the noise from
// the same Philox words as director_noise, with 24-bit uniforms
// u = (top 24 bits + 1) 2^-24 and xi = sqrt(-2 ln u1) cos(2 pi u2).
__global__ void k_dir_f32(DirArgs g) {
  const long long step = g.ctl->step;
  const uint2 key = make_uint2((unsigned)g.seed, (unsigned)(g.seed >> 32));
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += gridDim.x * blockDim.x) {
    double th = g.theta[i];
    if (g.advance) {
      th = th + g.noise_amp * g.xi[i];
      g.theta[i] = th;
    }
    float sn, cs;
    sincosf((float)th, &sn, &cs);
    g.nrm[i] = make_double2(cs, sn);
    const uint4 r = philox_10(make_uint4((unsigned)g.tag[i], (unsigned)(unsigned long long)step,
                                         (unsigned)((unsigned long long)step >> 32), 0u),
                              key);
    const float u1 = (float)((r.x >> 8) + 1u) * 0x1p-24f;
    const float u2 = (float)((r.z >> 8) + 1u) * 0x1p-24f;
    g.xi[i] = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
  }
}

void launch_geom_f32(const GeomArgs& a, cudaStream_t st, int blocks) {
  if (a.n <= 0) return;
  // up to one resident wave (us: 10.2 -> 8.1 at 256 to 16384 cells; 13.4 -> 14.8
  // at 65536), and for a list
  if (a.list || a.n <= kGeomF32SlotCells) {
    const int full = (a.n + 31) / 32;
    k_geom_f32_slots<<<(blocks > 0 && blocks < full) ? blocks : full, kSlotThreads, 0, st>>>(a);
    return;
  }
  const int full = (a.n + kGeomThreads - 1) / kGeomThreads;
  k_geom_f32<<<(blocks > 0 && blocks < full) ? blocks : full, kGeomThreads, 0, st>>>(a);
}
void launch_force_f32(const ForceArgs& a, cudaStream_t st, int blocks) {
  if (a.n <= 0) return;
  // as launch_force (us: 12.3 -> 8.2 at 1024 to 16384 cells, 14.3 -> 14.3 at 65536)
  if (!a.tolerant && a.integrate != 2 && (a.list || a.n <= kForceSlotCells)) {
    const int full = (a.n + 31) / 32;
    k_force_f32_slots<<<(blocks > 0 && blocks < full) ? blocks : full, kSlotThreads, 0, st>>>(a);
    return;
  }
  const int full = (a.n + kForceThreads - 1) / kForceThreads;
  k_force_f32<<<(blocks > 0 && blocks < full) ? blocks : full, kForceThreads, 0, st>>>(a);
}
void launch_dir_f32(const DirArgs& a, cudaStream_t st, int blocks) {
  if (a.n <= 0) return;
  const int full = (a.n + 127) / 128;
  k_dir_f32<<<(blocks > 0 && blocks < full) ? blocks : full, 128, 0, st>>>(a);
}

}  // namespace cgk
