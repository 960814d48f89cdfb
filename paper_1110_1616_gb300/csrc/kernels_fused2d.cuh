// Fused 2D level advance in FP32 (the mixed path): one CTA per (patch, tile),
// primitives, slopes, predicted face states, HLLD fluxes and the edge EMF kept
// in shared memory; the state is read and written once, and of the stage arrays
// only the fluxes and EMFs that the registers read go to the scratch. Included by
// kernels_impl.cuh inside AMRK_NS.
//
//   S1  W and the normal-B differences     (tile + 2 halo)
//   S2  slopes, predictor, face states, reference EMF (tile + 1 halo)
//   S3  HLLD fluxes of the x- and y-faces  (tile, + 1 across)
//   S4  E_z at the tile's corners
//   S5  update of cells, B_x, B_y
//
// The staged kernels move about 140 values a cell through L2 (five launches of
// 5 to 42 us a level step on 512^2 in 32^2 patches with a refined level, 115 us
// in all, the recovery in FP64 the longest: 2 FP64 lanes an SM); this one moves
// 16 and up to 13 for the registers, and recovers in pairs of FP32 values where
// that gives FP64's bits (with FP64 always four coarse steps take 0.93 ms):
// 34 us (four coarse steps 1.40 -> 0.69 ms with the smaller
// steps beside it), bound by instruction issue and the
// latency of its chains. Tiles are equal parts of the region (a 32^2 patch:
// four of 16^2, with its 2 extended layers four of 18^2), at most 18 wide, or
// 10 where that leaves less than a CTA per SM (the halo recomputes W on 1.5
// and the fluxes on 1.2 times a 16^2 tile's cells). Three CTAs of 256 threads an
// SM at 80 registers: 34 us; two at 118 registers 40, of 384 threads 37; 12^2
// tiles with six CTAs of 128 threads 35. The results are the staged kernels' bit
// for bit, so amrmhd_step_dt and the adjoint, which run those, make the same run.
constexpr int F2_TX = 18, F2_SMALL = 10, F2_NT = 256, F2_CTAS = 3;

struct Fused2dSmem {
  static constexpr int P = (F2_TX + 4) * (F2_TX + 4);  // W region
  static constexpr int Q = (F2_TX + 2) * (F2_TX + 2);  // predict / flux / EMF region
  union {
    struct { float w[8][P], db[2][P]; };  // S1, S2
    float f[2][7][Q];                     // S3 to S5: fluxes of the low faces, rotated
  };
  union {
    struct { float hi[2][8][Q], lo[2][8][Q]; };  // S2, S3: states at the cell's high and low x- and y-faces, rotated
    float e[Q];                                  // S4, S5: EMF of the low corners
  };
  float ref[Q];
  float dt[4];  // half-step and whole-step dt/dx
};

// i / n and i % n for 0 <= i < 2^16, n <= 2^8 (the half keeps the product off the integers)
__device__ __forceinline__ int row_of(int i, float inv) { return (int)(((float)i + 0.5f) * inv); }

// The staged kernels' recovery, which is recover() in FP64 with its results
// rounded to FP32: the velocities' quotients corrected by their remainders and
// the balance in pairs, each kept where every value within the distance from
// FP64 that it can have rounds to the same FP32 number (a quotient: 2^-44 of
// itself; the pressure: 2^-41 of the energies), else recover() itself.
__device__ __forceinline__ void recover_2d(const float* u, const float* bl, const float* br, Gm1<float> gm1, float* w) {
  const float ir = __frcp_rn(u[0]);
  float eh, el;
  ke_me(u, bl, br, ir, eh, el);
  bool ok = balance(u[4], eh, el, gm1, 0x1p-41f, w[4]);
  w[0] = u[0];
#pragma unroll
  for (int c = 1; c < 4; ++c) {
    const float v = xmul(u[c], ir), r = fmaf(-v, u[0], u[c]), d = xmul(fabsf(v), 0x1p-44f);
    w[c] = xadd(v, fmaf(r, ir, d));
    ok = ok && w[c] == xadd(v, fmaf(r, ir, -d)) && (d > 0x1p-110f || u[c] == 0.0f);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) w[5 + c] = 0.5f * (bl[c] + br[c]);
  if (!ok) {
    double uu[5], bc[3], v[8];
#pragma unroll
    for (int f = 0; f < 5; ++f) uu[f] = (double)u[f];
#pragma unroll
    for (int c = 0; c < 3; ++c) bc[c] = 0.5 * ((double)bl[c] + (double)br[c]);
    recover(uu, bc, gm1.v, v);
#pragma unroll
    for (int f = 1; f < 5; ++f) w[f] = (float)v[f];
  }
}

// the direction-D low-face state (n, t, u rotated; SIGN -1) or high-face state
template <int D> __device__ __forceinline__ void put_face(float (*s)[Fused2dSmem::Q], int q, const float* v) {
  constexpr int n = D, t = (D + 1) % 3, u = (D + 2) % 3;
  s[0][q] = v[0];
  s[1][q] = v[1 + n];
  s[2][q] = v[1 + t];
  s[3][q] = v[1 + u];
  s[4][q] = v[4];
  s[5][q] = v[5 + t];
  s[6][q] = v[5 + u];
  s[7][q] = v[5 + n];
}

__global__ void __launch_bounds__(F2_NT, F2_CTAS) k_advance2d_fused(LevelArgs a, int cap) {
  extern __shared__ __align__(16) unsigned char f2_raw[];
  Fused2dSmem& m = *reinterpret_cast<Fused2dSmem*>(f2_raw);
  const DPatch P = a.P[a.ids[blockIdx.y]];
  const int w = a.w, ex = P.n[0] + 2 * w, ey = P.n[1] + 2 * w;
  const int ntx = tile_count(ex, cap), lx = tile_len(ex, cap), ly = tile_len(ey, cap);
  const int ix = (int)blockIdx.x % ntx, iy = (int)blockIdx.x / ntx;
  if (iy >= tile_count(ey, cap)) return;
  const int x0 = 4 - w + ix * lx, y0 = 4 - w + iy * ly;
  const int tx = min(lx, 4 - w + ex - x0), ty = min(ly, 4 - w + ey - y0);
  if (tx <= 0 || ty <= 0) return;
  const int tid = threadIdx.x, sy = P.ext[0];
  const int fs = (int)P.fs;
  const float* U = (const float*)a.cur + P.off;
  float* S = (float*)a.scr + P.soff;
  if (tid < 4) {
    const double h = *a.dtp * a.dtscale;
    m.dt[tid] = (float)((tid < 2 ? 0.5 * h : h) * (tid & 1 ? a.idx[1] : a.idx[0]));
  }
  const float gamma = (float)a.gamma;
  // ---- S1
  const int wx = tx + 4, qx = tx + 2;
  {
    const Gm1<float> gm1(a.gamma - 1.0);
    const float inv = 1.0f / (float)wx;
    for (int p = tid; p < wx * (ty + 4); p += F2_NT) {
      const int py = row_of(p, inv), px = p - py * wx;
      const int L = x0 - 2 + px + sy * (y0 - 2 + py);
      float u[5], bl[3], br[3], v[8];
#pragma unroll
      for (int f = 0; f < 5; ++f) u[f] = U[f * fs + L];
      bl[0] = U[5 * fs + L];
      br[0] = U[5 * fs + L + 1];
      bl[1] = U[6 * fs + L];
      br[1] = U[6 * fs + L + sy];
      bl[2] = br[2] = U[7 * fs + L];
      recover_2d(u, bl, br, gm1, v);
#pragma unroll
      for (int f = 0; f < 8; ++f) m.w[f][p] = v[f];
      m.db[0][p] = br[0] - bl[0];
      m.db[1][p] = br[1] - bl[1];
    }
  }
  __syncthreads();
  // ---- S2
  const float invq = 1.0f / (float)qx;
  for (int q = tid; q < qx * (ty + 2); q += F2_NT) {
    const int py = row_of(q, invq), px = q - py * qx;
    const int p = (py + 1) * wx + px + 1;
    float v[8], s[2][8], wh[8], dw[8];
#pragma unroll
    for (int f = 0; f < 8; ++f) v[f] = m.w[f][p];
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const int sd = d ? wx : 1;
#pragma unroll
      for (int f = 0; f < 8; ++f)
        s[d][f] = f == BX + d ? m.db[d][p] : mm(v[f] - m.w[f][p - sd], m.w[f][p + sd] - v[f]);
    }
    const float ir = 1.0f / v[0];
    prim_terms<float, 0>(v, s[0], gamma, ir, dw);
#pragma unroll
    for (int f = 0; f < 8; ++f) wh[f] = v[f] - m.dt[0] * dw[f];
    prim_terms<float, 1>(v, s[1], gamma, ir, dw);
#pragma unroll
    for (int f = 0; f < 8; ++f) wh[f] = wh[f] - m.dt[1] * dw[f];
    m.ref[q] = wh[2] * wh[5] - wh[1] * wh[6];
    float h[8];
#pragma unroll
    for (int f = 0; f < 8; ++f) h[f] = plus_half<float>(wh[f], s[0][f]);
    put_face<0>(m.hi[0], q, h);
#pragma unroll
    for (int f = 0; f < 8; ++f) h[f] = minus_half<float>(wh[f], s[0][f]);
    put_face<0>(m.lo[0], q, h);
#pragma unroll
    for (int f = 0; f < 8; ++f) h[f] = plus_half<float>(wh[f], s[1][f]);
    put_face<1>(m.hi[1], q, h);
#pragma unroll
    for (int f = 0; f < 8; ++f) h[f] = minus_half<float>(wh[f], s[1][f]);
    put_face<1>(m.lo[1], q, h);
  }
  __syncthreads();  // W is dead from here on: its space holds the fluxes
  // ---- S3: x-faces (tx + 1) x (ty + 2), then y-faces (tx + 2) x (ty + 1), at the cell on their high side
  const int last_x = 4 + w + P.n[0], last_y = 4 + w + P.n[1];  // one past the region
  {
    const float igm1 = inv_gm1<float>(gamma, a.igm1);
    const float invf = 1.0f / (float)(tx + 1);
    const int nfx = (tx + 1) * (ty + 2), nf = nfx + qx * (ty + 1);
    for (int i = tid; i < nf; i += F2_NT) {
      const int d = i >= nfx;
      const int k = d ? i - nfx : i;
      const int row = row_of(k, d ? invq : invf);
      const int col = k - row * (d ? qx : tx + 1);
      const int py = row + d, px = col + 1 - d;
      const int q = py * qx + px, ql_ = q - (d ? qx : 1);
      float l[7], r[7], fr[7];
#pragma unroll
      for (int f = 0; f < 7; ++f) {
        l[f] = m.hi[d][f][ql_];
        r[f] = m.lo[d][f][q];
      }
      const float bn = 0.5f * (m.hi[d][7][ql_] + m.lo[d][7][q]);
      hlld_flux<float, HLLD_STAGED>(l, r, bn, gamma, igm1, fr);
#pragma unroll
      for (int f = 0; f < 7; ++f) m.f[d][f][q] = fr[f];
      if (a.keep) {
        // the tile owns the faces of its cells, and the region's last ones
        const int x = x0 - 1 + px, y = y0 - 1 + py;
        const bool own = d ? (px >= 1 && px <= tx && (py <= ty || y == last_y))
                           : (py >= 1 && py <= ty && (px <= tx || x == last_x));
        const int c = d ? y : x;
        if (own && (a.keep == 2 || c == 4 || c == 4 + (d ? P.n[1] : P.n[0]))) {
          float* F = S + (long long)(SC_F + 8 * d) * fs + x + sy * y;
          F[RHO * fs] = fr[0];
          F[(MX + d) * fs] = fr[1];
          F[(MX + d + 1) * fs] = fr[2];
          F[(d ? MX : MZ) * fs] = fr[3];
          F[EN * fs] = fr[4];
          F[BZ * fs] = d ? fr[5] : fr[6];
        }
      }
    }
  }
  __syncthreads();
  // ---- S4: the corner below and left of cell (x, y)
  {
    const float inv = 1.0f / (float)(tx + 1);
    for (int i = tid; i < (tx + 1) * (ty + 1); i += F2_NT) {
      const int py = row_of(i, inv) + 1, px = i - (py - 1) * (tx + 1) + 1;
      const int q11 = py * qx + px, q01 = q11 - 1, q10 = q11 - qx, q00 = q10 - 1;
      const float e = gs_emf<float>(-m.f[0][5][q10], -m.f[0][5][q11], m.f[1][6][q01], m.f[1][6][q11], m.ref[q00],
                                    m.ref[q10], m.ref[q01], m.ref[q11], m.f[0][0][q10], m.f[0][0][q11],
                                    m.f[1][0][q01], m.f[1][0][q11]);
      m.e[q11] = e;
      if (a.keep) {
        const int x = x0 - 1 + px, y = y0 - 1 + py;
        const bool own = (px <= tx || x == last_x) && (py <= ty || y == last_y);
        if (own && (a.keep == 2 || x == 4 || y == 4 || x == 4 + P.n[0] || y == 4 + P.n[1]))
          S[(long long)(SC_E + 2) * fs + x + sy * y] = e;
      }
    }
  }
  __syncthreads();
  // ---- S5
  {
    float* V = (float*)a.nxt + P.off;
    const float d0 = m.dt[2], d1 = m.dt[3];
    const float inv = 1.0f / (float)tx;
    for (int i = tid; i < tx * ty; i += F2_NT) {
      const int cy = row_of(i, inv), cx = i - cy * tx;
      const int x = x0 + cx, y = y0 + cy, L = x + sy * y;
      const int q = (cy + 1) * qx + cx + 1;
      const auto upd = [&](int f, int kx, int ky) {
        float v = U[f * fs + L];
        v = v - d0 * (m.f[0][kx][q + 1] - m.f[0][kx][q]);
        v = v - d1 * (m.f[1][ky][q + qx] - m.f[1][ky][q]);
        V[f * fs + L] = v;
      };
      upd(RHO, 0, 0);
      upd(MX, 1, 3);
      upd(MY, 2, 1);
      upd(MZ, 3, 2);
      upd(EN, 4, 4);
      upd(BZ, 6, 5);
      const auto bx = [&](int LL, int qq) { V[BX * fs + LL] = U[BX * fs + LL] - d1 * (m.e[qq + qx] - m.e[qq]); };
      const auto by = [&](int LL, int qq) { V[BY * fs + LL] = U[BY * fs + LL] + d0 * (m.e[qq + 1] - m.e[qq]); };
      bx(L, q);
      by(L, q);
      if (x + 1 == last_x) bx(L + 1, q + 1);
      if (y + 1 == last_y) by(L + sy, q + qx);
    }
  }
}
