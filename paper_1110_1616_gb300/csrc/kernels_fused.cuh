// Fused 3D level advance: one CTA per (patch, x-y tile, z chunk), marching
// along z with rolling plane buffers in shared memory, so that primitives,
// slopes, predicted states, HLLD fluxes and CT EMFs never leave the SM. Only
// the state is read and written in HBM. Included by kernels_impl.cuh inside
// AMRK_NS.
//
// Pipeline per iteration p (planes in patch-local storage coordinates; the
// patch's output z range is [zlo, zhi) = [4-w, n_z+4+w), a CTA's the chunk
// [zs, ze) of it: a.zlen planes from zlo + a.zlen * chunk, or all of them when
// a.zlen is 0; a chunk restarts the march 2 planes below its first output
// plane, so a split column recomputes 4 planes of primitives, 2 of predictor
// and fluxes and 1 of EMFs per extra chunk, and every output value is the
// same bit for bit whatever the split):
//   S1  W at plane p+2                   (tile + 2 halo)        -> ring of 3
//       (and the normal-B differences of the tile + 1 halo)
//   S2  slopes, predictor, the face states of the three directions and the
//       reference EMF at plane p+1 (tile + 1 halo)
//   S3  HLLD fluxes: x- and y-faces of plane p, z-faces of face plane p
//   S4  edge EMFs: E_z at plane p, E_x and E_y at edge plane p
//   S5  update of cell plane q = p-1: cells, B_x and B_y of plane q, B_z of face
//       plane q (and the top face plane zhi on the patch's last plane)
//
// What bounds it is the issue of instructions and the latency of their chains
// (16 warps an SM, see the capture in the profiles); DRAM and the FP32 pipe
// are far from their limits. So the layout serves the instruction count:
//  * a thread's positions do not depend on the plane, so every index is formed
//    once, before the march;
//  * the face states are stored, not the predicted state and its slopes, in the
//    rotated order (rho, v_n, v_t, v_u, p, B_t, B_u, B_n) of their direction:
//    S3 is one code for all faces with 16 loads at constant distances (32 loads
//    and 16 multiply-adds at computed distances before), the fluxes are stored
//    rotated too, and so S4 is one code for the three edge directions;
//  * a row is as long as the tile needs (a level's regions are cut into equal
//    tiles of at most TX x TY), so that no lane works on padding.
// 128^3 blast in 16^3 patches (autotuned): 0.482 -> 0.332 ms a launch; 256^3 in
// 32^3 patches: 3.19 -> 2.24 ms; the 64^3 + refined eighth's level 1: 0.234 ->
// 0.135 ms (beside the coarse advance; with the FP32 flux, recovery and minmod of
// mhd_device.cuh, whose results are bit for bit those before).

// Tile variants (largest x-y output tile and threads per CTA), chosen by the
// autotuning option: 0 = 16x16 / 256, 1 = 16x16 / 512, 2 = 16x8 / 256,
// 3 = 8x8 / 160, 4 = 10x10 / 256 (a 16^3 patch with its 2 extended layers is 2 x
// 2 of them). The threads are as many as make two rounds of the faces at most,
// the CTAs per SM what the shared memory allows. 128^3 blast, a launch at each
// variant's better split: 0.450, 0.332, 0.338, 0.347, 0.410 ms (8x8 with 256
// threads, whose 80 registers spilled, 0.437 when it was tried); 64 extended 16^3
// patches: 0.159, 0.147, 0.126, 0.134, 0.100 ms (16x8 tiles, there 10x7, need a second wave).
template <int V> struct FusedCfg;
template <> struct FusedCfg<0> { static constexpr int TX = 16, TY = 16, NT = 256; };
template <> struct FusedCfg<1> { static constexpr int TX = 16, TY = 16, NT = 512; };
template <> struct FusedCfg<2> { static constexpr int TX = 16, TY = 8, NT = 256; };
template <> struct FusedCfg<3> { static constexpr int TX = 8, TY = 8, NT = 160; };
template <> struct FusedCfg<4> { static constexpr int TX = 10, TY = 10, NT = 256; };

// The plane buffers of a tile of at most TX x TY cells. Rows of the W region
// (tile + 2) hold tx + 4 values, those of the Q region (tile + 1) tx + 2.
template <class T, int TX_, int TY_> struct FusedSmem {
  static constexpr int TX = TX_, TY = TY_;
  static constexpr int P = (TX + 4) * (TY + 4);  // W region
  static constexpr int Q = (TX + 2) * (TY + 2);  // predict / flux / EMF region
  T w[3][8][P];
  T hi[2][8][Q];    // state at the cell's high x- and y-face, rotated
  T hiz[2][8][Q];   // at its high z-face, 2 planes
  T lo[3][8][Q];    // at its low x-, y- and z-face
  T ref[3][3][Q];   // cell reference EMFs, 3 planes
  T f[2][3][7][Q];  // fluxes of the low faces by direction, rotated, 2 planes
  T e[2][3][Q];     // EMFs of the low edges by component, 2 planes
  T db[2][3][Q];    // normal-B face differences (slopes of B_d along d), 2 planes
};

template <class T>
__device__ __forceinline__ void hlld_face(const T* wl, const T* wr, int D, T gamma, double igm1, T* out8) {
  const int n = D, t = (D + 1) % 3, u = (D + 2) % 3;
  const T bn = T(0.5) * (wl[5 + n] + wr[5 + n]);
  const T ql[7] = {wl[0], wl[1 + n], wl[1 + t], wl[1 + u], wl[4], wl[5 + t], wl[5 + u]};
  const T qr[7] = {wr[0], wr[1 + n], wr[1 + t], wr[1 + u], wr[4], wr[5 + t], wr[5 + u]};
  T fr[7];
  hlld_flux<T, HLLD_REGISTER>(ql, qr, bn, gamma, inv_gm1<T>(gamma, igm1), fr);
  out8[RHO] = fr[0];
  out8[MX + n] = fr[1];
  out8[MX + t] = fr[2];
  out8[MX + u] = fr[3];
  out8[EN] = fr[4];
  out8[BX + t] = fr[5];
  out8[BX + u] = fr[6];
  out8[BX + n] = T(0);
}

template <class T>
__device__ __forceinline__ void load_recover(const T* U, int fs, int L, int sy, int sz, Gm1<T> gm1, T* w,
                                             T* dB = nullptr, const Floors* fl = nullptr) {
  T u[5], bl[3], br[3];
#pragma unroll
  for (int f = 0; f < 5; ++f) u[f] = U[f * fs + L];
  bl[0] = U[5 * fs + L]; br[0] = U[5 * fs + L + 1];
  bl[1] = U[6 * fs + L]; br[1] = U[6 * fs + L + sy];
  bl[2] = U[7 * fs + L]; br[2] = U[7 * fs + L + sz];
  if (fl) floor_density(u, fl->rho, fl->events);
  recover_t(u, bl, br, gm1, w);
  if (fl) floor_pressure(w, fl->p, fl->events);
  if (dB) {
#pragma unroll
    for (int d = 0; d < 3; ++d) dB[d] = br[d] - bl[d];
  }
}

// ---------------------------------------------------------------- boundary capture
// The fluxes and EMFs on the six boundary planes of a fine patch, written by the
// fused advance and read by the fine-side registers (levels > 0), instead of
// recomputing them there. Per patch at P.boff (elements of the state type): the
// 5 conserved-flux components (field-major) of every boundary face, planes in
// the order x-low, x-high, y-low, y-high, z-low, z-high, a plane of normal e
// holding n_t1 x n_t2 faces (t1 < t2 the other axes, t1 fastest); then the
// tangential EMFs of the boundary planes in the same plane order, per plane its
// two components c != e ascending, each over n_c x (n_o + 1) edges (c fastest,
// o the remaining axis).
// slot of the e-face at local (x, y, z) if it lies on a boundary plane, else -1
__device__ __forceinline__ long long bnd_face_slot(const DPatch& P, int e, int x, int y, int z) {
  const int pos[3] = {x, y, z};
  const int side = pos[e] == 4 ? 0 : (pos[e] == P.n[e] + 4 ? 1 : -1);
  if (side < 0) return -1;
  const int t1 = e == 0 ? 1 : 0, t2 = e == 2 ? 1 : 2;
  const int u = pos[t1] - 4, v = pos[t2] - 4;
  if (u < 0 || u >= P.n[t1] || v < 0 || v >= P.n[t2]) return -1;
  const long long S0 = (long long)P.n[1] * P.n[2], S1 = (long long)P.n[0] * P.n[2], S2 = (long long)P.n[0] * P.n[1];
  const long long Se = e == 0 ? S0 : (e == 1 ? S1 : S2);
  const long long base = (e == 0 ? 0 : (e == 1 ? 2 * S0 : 2 * (S0 + S1))) + side * Se;
  return base + u + (long long)P.n[t1] * v;
}
// slot of the c-edge at local (x, y, z) on the boundary plane of normal e, else -1
__device__ __forceinline__ long long bnd_edge_slot(const DPatch& P, int c, int e, int x, int y, int z) {
  const int pos[3] = {x, y, z};
  const int side = pos[e] == 4 ? 0 : (pos[e] == P.n[e] + 4 ? 1 : -1);
  if (side < 0) return -1;
  const int o = 3 - c - e;
  const int u = pos[c] - 4, v = pos[o] - 4;
  if (u < 0 || u >= P.n[c] || v < 0 || v > P.n[o]) return -1;
  long long base = 0;
#pragma unroll
  for (int ee = 0; ee < 3; ++ee)
#pragma unroll
    for (int s2 = 0; s2 < 2; ++s2)
#pragma unroll
      for (int cc = 0; cc < 3; ++cc) {
        if (cc == ee) continue;
        if (ee == e && s2 == side && cc == c) return base + u + (long long)P.n[c] * v;
        base += (long long)P.n[cc] * (P.n[3 - cc - ee] + 1);
      }
  return -1;
}
// Along one axis of an extent ex, tiles of at most T cells: the number of
// tiles, and their common length (the last one may be shorter).
__host__ __device__ __forceinline__ int tile_count(int ex, int T) { return (ex + T - 1) / T; }
__host__ __device__ __forceinline__ int tile_len(int ex, int T) {
  const int n = tile_count(ex, T);
  return (ex + n - 1) / n;
}

// One x-y tile (index `tile`, ntx tiles along x in the level's largest patch)
// of the patch at position `pslot` of a.ids, marched along z by the whole CTA
// over the z chunk `zc` (a.zlen planes each; 0: the whole column); smem_raw:
// the CTA's dynamic shared memory (a FusedSmem). MODE 0: plain; 1 (CAP): the
// level's boundary fluxes and EMFs are captured for the fine registers (patches
// with P.boff >= 0); 2 (DH): direct halo reads from the neighbour patches
// (a.nbr; a level of equal patches tiling the periodic domain, w = 0). FL: the
// recovery applies the density and pressure floors of a.fl (never with DH).
// Every thread of the CTA calls it with the same arguments.
template <class T, int VAR, int MODE, bool FL = false>
__device__ __forceinline__ void fused_tile(const LevelArgs& a, int pslot, int tile, int ntx, int zc,
                                           unsigned char* smem_raw, bool halves = false) {
  constexpr bool CAP = MODE == 1, DH = MODE == 2;
  using S = FusedSmem<T, FusedCfg<VAR>::TX, FusedCfg<VAR>::TY>;
  constexpr int TX = S::TX, TY = S::TY, NT = FusedCfg<VAR>::NT, PN = S::P, QN = S::Q;
  S& sm = *reinterpret_cast<S*>(smem_raw);
  __shared__ long long s_nb[DH ? 27 : 1];  // element offsets of the neighbour patches (DH)
  const DPatch P = a.P[a.ids[pslot]];
  if constexpr (DH) {
    if (threadIdx.x < 27) s_nb[threadIdx.x] = a.P[a.nbr[27 * pslot + threadIdx.x]].off;
    __syncthreads();
  }
  const int w = a.w;
  const int xlo = 4 - w, xhi = P.n[0] + 4 + w, ylo = 4 - w, yhi = P.n[1] + 4 + w;
  const int zlo = 4 - w, zhi = P.n[2] + 4 + w;
  // equal tiles of this patch's region (a smaller patch of the level has fewer)
  const int lx_ = tile_len(xhi - xlo, TX), ly_ = tile_len(yhi - ylo, TY);
  const int x0 = xlo + (tile % ntx) * lx_, y0 = ylo + (tile / ntx) * ly_;
  // the chunk: a.zlen planes from zlo + a.zlen zc, the whole column (a.zlen
  // 0), or with halves its lower (zc 0) or upper (zc 1) half
  const int zl = halves ? (zhi - zlo + 1) / 2 : a.zlen;
  const int zs = zlo + zc * zl, ze = zl > 0 ? min(zs + zl, zhi) : zhi;
  if (x0 >= xhi || y0 >= yhi || zs >= zhi) return;
  // a face or edge plane shared by two chunks (ze of one, zs of the next) is
  // captured by the upper chunk only
  const bool cap_ze = ze == zhi;
  const int tx = min(lx_, xhi - x0), ty = min(ly_, yhi - y0);
  const bool last_x = x0 + tx == xhi, last_y = y0 + ty == yhi;
  const int fs = (int)P.fs;  // 8 fields fit 32 bits (checked when the hierarchy is set)
  const int sy = P.ext[0], sz = P.ext[0] * P.ext[1];
  const T* U = (const T*)a.cur + P.off;
  T* V = (T*)a.nxt + P.off;
  const bool capture = CAP && P.boff >= 0;
  const Gm1<T> gm1(a.gamma - 1.0);
  const Floors* flp = FL ? &a.fl : nullptr;
  const T gamma = (T)a.gamma;
  const double dt = *a.dtp * a.dtscale;
  const T h0 = (T)(0.5 * dt * a.idx[0]), h1 = (T)(0.5 * dt * a.idx[1]), h2 = (T)(0.5 * dt * a.idx[2]);
  const T dtd[3] = {(T)(dt * a.idx[0]), (T)(dt * a.idx[1]), (T)(dt * a.idx[2])};
  const int px = tx + 4, qx = tx + 2, qy = ty + 2;  // row lengths of the W and Q regions; rows of Q
  const int tid = threadIdx.x;

  // ---- this thread's positions, the same in every plane (-1: none)
  // S1: W position tid + NT it (its index in the plane): global offset of the
  // cell in a plane, the Q position (or -1); DH: the neighbour's number
  constexpr int I1 = (PN + NT - 1) / NT;
  int g1[I1], q1[I1], k1[DH ? I1 : 1];
#pragma unroll
  for (int it = 0; it < I1; ++it) {
    const int c = tid + NT * it, yi = c / px, xi = c - px * yi;
    const bool in = c < px * (ty + 4);
    int x = x0 - 2 + xi, y = y0 - 2 + yi;
    q1[it] = in && xi >= 1 && xi < px - 1 && yi >= 1 && yi < ty + 3 ? (xi - 1) + qx * (yi - 1) : -1;
    if constexpr (DH) {
      // the cell (and its faces) in the neighbour patch that owns it: every
      // patch has the interior extent n, so a coordinate outside [4, n+4)
      // moves by n into the neighbour's interior (its own high faces at n+4
      // included); the neighbours' strides are this patch's
      int k = 13;
      if (x < 4) { x += P.n[0]; k -= 1; } else if (x >= P.n[0] + 4) { x -= P.n[0]; k += 1; }
      if (y < 4) { y += P.n[1]; k -= 3; } else if (y >= P.n[1] + 4) { y -= P.n[1]; k += 3; }
      k1[it] = k;
    }
    g1[it] = in ? x + sy * y : -1;
  }
  // S2: Q position tid + NT it: its W position
  constexpr int I2 = (QN + NT - 1) / NT;
  int w2[I2];
#pragma unroll
  for (int it = 0; it < I2; ++it) {
    const int c = tid + NT * it, yi = c / qx, xi = c - qx * yi;
    w2[it] = c < qx * qy ? (xi + 1) + px * (yi + 1) : -1;
  }
  // S3: the x-faces (tx+1) x (ty+2), the y-faces (tx+2) x (ty+1), the z-faces
  // of the Q region: index r of the right state in lo (= 8 QN D + q), the left
  // one's in hi, hiz (contiguous), the flux's in a plane of f
  constexpr int I3 = ((TX + 1) * (TY + 2) + (TX + 2) * (TY + 1) + QN + NT - 1) / NT;
  const int nfx = (tx + 1) * qy, nfy = qx * (ty + 1), nf = nfx + nfy + qx * qy;
  int l3[I3], r3[I3], f3[I3], c3[CAP ? I3 : 1];
#pragma unroll
  for (int it = 0; it < I3; ++it) {
    const int c = tid + NT * it;
    int D = 2, q = c - nfx - nfy, step = 0;
    int xi, yi;  // in the Q region
    if (c < nfx) {
      yi = c / (tx + 1);
      xi = c - (tx + 1) * yi + 1;
      D = 0;
      step = 1;
    } else if (c < nfx + nfy) {
      yi = (c - nfx) / qx;
      xi = c - nfx - qx * yi;
      yi += 1;
      D = 1;
      step = qx;
    } else {
      yi = q / qx;
      xi = q - qx * yi;
    }
    q = xi + qx * yi;
    r3[it] = c < nf ? 8 * QN * D + q : -1;
    l3[it] = 8 * QN * D + q - step;
    f3[it] = 7 * QN * D + q;
    if constexpr (CAP) {
      // boundary capture: the face's slot at its first captured plane (x- and
      // y-faces: cell plane 4, z-faces: the low face plane), -1: no boundary face
      const int x = x0 - 1 + xi, y = y0 - 1 + yi;
      c3[it] = !capture || c >= nf ? -1
                                   : (int)(D == 0 ? bnd_face_slot(P, 0, x, y, 4)
                                                  : (D == 1 ? bnd_face_slot(P, 1, x, y, 4) : bnd_face_slot(P, 2, x, y, 4)));
    }
  }
  const int cs3 = CAP ? P.n[0] * P.n[1] : 0;  // from the low to the high z-plane's slots
  // S4: the E_z edges (tx+1) x (ty+1), E_x edges tx x (ty+1), E_y edges (tx+1) x ty
  constexpr int I4 = ((TX + 1) * (TY + 1) + TX * (TY + 1) + (TX + 1) * TY + NT - 1) / NT;
  const int nez = (tx + 1) * (ty + 1), nex = tx * (ty + 1), ne = nez + nex + (tx + 1) * ty;
  int q4[I4], c4[I4], ka4[CAP ? I4 : 1], kb4[CAP ? I4 : 1];
#pragma unroll
  for (int it = 0; it < I4; ++it) {
    const int c = tid + NT * it;
    int C = 2, o = c, rl = tx + 1;
    if (c >= nez + nex) { C = 1; o = c - nez - nex; }
    else if (c >= nez) { C = 0; o = c - nez; rl = tx; }
    const int yi = o / rl, xi = o - rl * yi;
    c4[it] = C;
    q4[it] = c < ne ? (xi + 1) + qx * (yi + 1) : -1;
    if constexpr (CAP) {
      // slots at plane 4 on the boundary planes of the two normals other than C
      const int x = x0 + xi, y = y0 + yi;
      long long ka = -1, kb = -1;
      if (capture && c < ne) {
        if (C == 0) { ka = bnd_edge_slot(P, 0, 1, x, y, 4); kb = bnd_edge_slot(P, 0, 2, x, y, 4); }
        else if (C == 1) { ka = bnd_edge_slot(P, 1, 0, x, y, 4); kb = bnd_edge_slot(P, 1, 2, x, y, 4); }
        else { ka = bnd_edge_slot(P, 2, 0, x, y, 4); kb = bnd_edge_slot(P, 2, 1, x, y, 4); }
      }
      ka4[it] = (int)ka;
      kb4[it] = (int)kb;
    }
  }
  // S5: the tile's cells, and on the patch's high x (y) side the B_x (B_y)
  // faces of the column x0+tx (the row y0+ty)
  constexpr int I5 = ((TX + 1) * (TY + 1) + NT - 1) / NT;
  const int nx5 = tx + (last_x ? 1 : 0), ny5 = ty + (last_y ? 1 : 0);
  int q5[I5], g5[I5];
  bool ix5[I5], iy5[I5];
#pragma unroll
  for (int it = 0; it < I5; ++it) {
    const int c = tid + NT * it, yi = c / nx5, xi = c - nx5 * yi;
    q5[it] = c < nx5 * ny5 ? (xi + 1) + qx * (yi + 1) : -1;
    g5[it] = (x0 + xi) + sy * (y0 + yi);
    ix5[it] = xi < tx;
    iy5[it] = yi < ty;
  }

  // ---- S1: primitives of plane t
  auto stage1 = [&](int t) {
    T* W = &sm.w[(t + 3) % 3][0][0];
    T* B = &sm.db[t & 1][0][0];
    int lz = t, kz = 0;
    if constexpr (DH) {
      if (t < 4) { lz += P.n[2]; kz = -9; } else if (t >= P.n[2] + 4) { lz -= P.n[2]; kz = 9; }
    }
#pragma unroll
    for (int it = 0; it < I1; ++it) {
      if (g1[it] < 0) continue;
      T wv[8], dB[3];
      const T* src = DH ? (const T*)a.cur + s_nb[k1[DH ? it : 0] + kz] : U;
      load_recover(src, fs, g1[it] + sz * lz, sy, sz, gm1, wv, dB, flp);
      const int i = tid + NT * it;
#pragma unroll
      for (int f = 0; f < 8; ++f) W[f * PN + i] = wv[f];
      if (q1[it] >= 0) {
#pragma unroll
        for (int d = 0; d < 3; ++d) B[d * QN + q1[it]] = dB[d];
      }
    }
  };
  // ---- S2: slopes, predictor, face states and reference EMF of plane p
  auto stage2 = [&](int p) {
    const T* Wm = &sm.w[(p + 2) % 3][0][0];
    const T* W0 = &sm.w[(p + 3) % 3][0][0];
    const T* Wp = &sm.w[(p + 4) % 3][0][0];
    const T* B = &sm.db[p & 1][0][0];
    T* R = &sm.ref[(p + 3) % 3][0][0];
    T* HZ = &sm.hiz[p & 1][0][0];
#pragma unroll
    for (int it = 0; it < I2; ++it) {
      const int i = w2[it], q = tid + NT * it;
      if (i < 0) continue;
      T wc[8], s[3][8];
#pragma unroll
      for (int f = 0; f < 8; ++f) wc[f] = W0[f * PN + i];
#pragma unroll
      for (int f = 0; f < 8; ++f) {
        s[0][f] = f == BX ? B[q] : mm<T>(wc[f] - W0[f * PN + i - 1], W0[f * PN + i + 1] - wc[f]);
        s[1][f] = f == BY ? B[QN + q] : mm<T>(wc[f] - W0[f * PN + i - px], W0[f * PN + i + px] - wc[f]);
        s[2][f] = f == BZ ? B[2 * QN + q] : mm<T>(wc[f] - Wm[f * PN + i], Wp[f * PN + i] - wc[f]);
      }
      const T ir = T(1) / wc[0];
      T wh[8], dw[8];
#pragma unroll
      for (int f = 0; f < 8; ++f) wh[f] = wc[f];
      prim_terms<T, 0>(wc, s[0], gamma, ir, dw);
#pragma unroll
      for (int f = 0; f < 8; ++f) wh[f] = wh[f] - h0 * dw[f];
      prim_terms<T, 1>(wc, s[1], gamma, ir, dw);
#pragma unroll
      for (int f = 0; f < 8; ++f) wh[f] = wh[f] - h1 * dw[f];
      prim_terms<T, 2>(wc, s[2], gamma, ir, dw);
#pragma unroll
      for (int f = 0; f < 8; ++f) wh[f] = wh[f] - h2 * dw[f];
#pragma unroll
      for (int D = 0; D < 3; ++D) {
        const int n = D, t = (D + 1) % 3, u = (D + 2) % 3;
        const int o[8] = {RHO, MX + n, MX + t, MX + u, EN, BX + t, BX + u, BX + n};
        T* H = D < 2 ? &sm.hi[D < 2 ? D : 0][0][0] : HZ;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          H[k * QN + q] = plus_half<T>(wh[o[k]], s[D][o[k]]);
          sm.lo[D][k][q] = minus_half<T>(wh[o[k]], s[D][o[k]]);
        }
      }
      R[q] = wh[3] * wh[6] - wh[2] * wh[7];
      R[QN + q] = wh[1] * wh[7] - wh[3] * wh[5];
      R[2 * QN + q] = wh[2] * wh[5] - wh[1] * wh[6];
    }
  };
  // ---- S3: fluxes (x, y faces of plane p; z faces of face plane p)
  auto put_flux = [&](int it, int p, const T* fr) {
    T* fo = &sm.f[p & 1][0][0][0] + f3[it];
#pragma unroll
    for (int k = 0; k < 7; ++k) fo[k * QN] = fr[k];
    if constexpr (CAP) {
      // a boundary face of a fine patch: keep its flux for the registers
      // (x- and y-faces of the chunk's own planes, z-faces of its face
      // planes, the top one only on the column's last chunk)
      if (c3[it] >= 0) {
        const int D = r3[it] / (8 * QN);
        const bool on = D == 2 ? (p == 4 || p == P.n[2] + 4) && (p < ze || cap_ze)
                               : p >= max(zs, 4) && p < min(ze, P.n[2] + 4);
        if (on) {
          const long long F1 = bnd_faces_total(P.n);
          T* b = (T*)a.bnd + P.boff + c3[it] + (D == 2 ? (p == 4 ? 0 : cs3) : (D == 0 ? P.n[1] : P.n[0]) * (p - 4));
          // rotated back: the normal, t and u momentum fluxes
          b[0] = fr[0];
          b[(1 + D) * F1] = fr[1];
          b[(D == 2 ? 1 : 2 + D) * F1] = fr[2];
          b[(D == 0 ? 3 : D) * F1] = fr[3];
          b[4 * F1] = fr[4];
        }
      }
    }
  };
  auto stage3 = [&](int p) {
    const T* HI = &sm.hi[0][0][0];
    const T* LO = &sm.lo[0][0][0];
    const int zprev = ((p + 1) & 1) * 8 * QN;  // plane p-1's slot of hiz (right behind hi)
    auto left = [&](int it) { return HI + l3[it] + (r3[it] >= 16 * QN ? zprev : 0); };
    auto exists = [&](int it) { return r3[it] >= 0 && (r3[it] < 16 * QN || p >= zs); };
#pragma unroll
    for (int it = 0; it < I3; ++it) {
      if (!exists(it)) continue;
      const T *pl = left(it), *pr = LO + r3[it];
      T ql[7], qr[7], fr[7];
#pragma unroll
      for (int k = 0; k < 7; ++k) {
        ql[k] = pl[k * QN];
        qr[k] = pr[k * QN];
      }
      const T bn = T(0.5) * (pl[7 * QN] + pr[7 * QN]);
      hlld_flux<T>(ql, qr, bn, gamma, inv_gm1<T>(gamma, a.igm1), fr);
      put_flux(it, p, fr);
    }
  };
  // ---- S4: edge EMFs. With (a, b, C) cyclic and the fluxes rotated, the
  // a-faces' EMF is -f_a[5], the b-faces' f_b[6]; a step along z is a step to
  // the other plane's slot.
  auto stage4 = [&](int p) {
    const int cur = p & 1;
    const T* F = &sm.f[cur][0][0][0];
    const T* R = &sm.ref[(p + 3) % 3][0][0];
    T* E = &sm.e[cur][0][0];
    const int zF = cur ? 21 * QN : -21 * QN;                    // from plane p-1's fluxes to plane p's
    const int zR = (p + 3) % 3 == 0 ? -6 * QN : 3 * QN;  // the same for the references
    // the 12 values around an edge, in gs_emf's order
    auto around = [&](int it, T* v) {
      const int q = q4[it], C = c4[it];
      const int saF = C == 2 ? 1 : (C == 0 ? qx : zF), sbF = C == 2 ? qx : (C == 0 ? zF : 1);
      const int saR = C == 1 ? zR : saF, sbR = C == 0 ? zR : sbF;
      const T* Fa = F + (C == 2 ? 0 : 7 * QN * (C + 1)) + q;  // a = C + 1 (mod 3)
      const T* Fb = F + (C == 0 ? 14 * QN : 7 * QN * (C - 1)) + q;  // b = C + 2 (mod 3)
      const T* r = R + C * QN + q;
      v[0] = -Fa[5 * QN - sbF], v[1] = -Fa[5 * QN], v[2] = Fb[6 * QN - saF], v[3] = Fb[6 * QN];
      v[4] = r[-saR - sbR], v[5] = r[-sbR], v[6] = r[-saR], v[7] = r[0];
      v[8] = Fa[-sbF], v[9] = Fa[0], v[10] = Fb[-saF], v[11] = Fb[0];
    };
    auto put = [&](int it, T v) {
      const int q = q4[it], C = c4[it];
      E[C * QN + q] = v;
      if constexpr (CAP) {
        // on boundary planes of a fine patch: keep it for the registers (E_z of
        // the chunk's planes, E_x and E_y of its edge planes, the top one only
        // on the column's last chunk)
        if (ka4[it] >= 0 || kb4[it] >= 0) {
          T* b = (T*)a.bnd + P.boff + 5 * bnd_faces_total(P.n);
          const int m = p - 4;
          if (C == 2) {
            if (m >= 0 && m < P.n[2]) {
              if (ka4[it] >= 0) b[ka4[it] + m] = v;
              if (kb4[it] >= 0) b[kb4[it] + m] = v;
            }
          } else if (p < ze || cap_ze) {
            if (ka4[it] >= 0 && m >= 0 && m <= P.n[2]) b[ka4[it] + (C == 0 ? P.n[0] : P.n[1]) * m] = v;
            // from the low z-plane's component C to the high one's: both components of a plane
            if (kb4[it] >= 0 && (m == 0 || m == P.n[2]))
              b[kb4[it] + (m == 0 ? 0 : P.n[0] * (P.n[1] + 1) + P.n[1] * (P.n[0] + 1))] = v;
          }
        }
      }
    };
    auto exists = [&](int it) { return q4[it] >= 0 && (c4[it] != 2 || p < ze); };
#pragma unroll
    for (int it = 0; it < I4; ++it) {
      if (!exists(it)) continue;
      T v[12];
      around(it, v);
      put(it, gs_emf<T>(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], v[8], v[9], v[10], v[11]));
    }
  };
  // ---- S5: update of cell plane qz; the stored values are loaded a phase
  // ahead into registers when a thread has one position
  constexpr bool AHEAD = I5 == 1;
  T up[8];
  auto load_up = [&](int qz, int it) {
    const int L = g5[it] + sz * qz;
    if (ix5[it] && iy5[it]) {
#pragma unroll
      for (int f = 0; f < 8; ++f) up[f] = U[f * fs + L];
    } else if (iy5[it]) {
      up[BX] = U[BX * fs + L];
    } else if (ix5[it]) {
      up[BY] = U[BY * fs + L];
    }
  };
  auto stage5 = [&](int qz) {
    const int cur = qz & 1;
    const T* Fq = &sm.f[cur][0][0][0];
    const T* Fp = &sm.f[cur ^ 1][0][0][0];
    const T* Eq = &sm.e[cur][0][0];
    const T* Ep = &sm.e[cur ^ 1][0][0];
#pragma unroll
    for (int it = 0; it < I5; ++it) {
      const int q = q5[it];
      if (q < 0) continue;
      if constexpr (!AHEAD) load_up(qz, it);
      const int L = g5[it] + sz * qz;
      if (ix5[it] && iy5[it]) {
#pragma unroll
        for (int n = 0; n < 5; ++n) {
          // the field's place in the x, y and z fluxes (rotated momenta)
          const int kx = n, ky = n == 0 || n == 4 ? n : (n == 1 ? 3 : n - 1), kz = n == 0 || n == 4 ? n : (n == 3 ? 1 : n + 1);
          T v = up[n];
          v = v - dtd[0] * (Fq[kx * QN + q + 1] - Fq[kx * QN + q]);
          v = v - dtd[1] * (Fq[(7 + ky) * QN + q + qx] - Fq[(7 + ky) * QN + q]);
          v = v - dtd[2] * (Fp[(14 + kz) * QN + q] - Fq[(14 + kz) * QN + q]);
          V[n * fs + L] = v;
        }
        // B_z of face plane qz (and the top face plane on the last plane)
        {
          T v = up[BZ];
          v = v - dtd[0] * (Eq[QN + q + 1] - Eq[QN + q]);
          v = v + dtd[1] * (Eq[q + qx] - Eq[q]);
          V[BZ * fs + L] = v;
        }
        if (qz == zhi - 1) {
          T v = U[BZ * fs + L + sz];
          v = v - dtd[0] * (Ep[QN + q + 1] - Ep[QN + q]);
          v = v + dtd[1] * (Ep[q + qx] - Ep[q]);
          V[BZ * fs + L + sz] = v;
        }
      }
      if (iy5[it]) {  // B_x at (x, y, qz)
        T v = up[BX];
        v = v - dtd[1] * (Eq[2 * QN + q + qx] - Eq[2 * QN + q]);
        v = v + dtd[2] * (Ep[QN + q] - Eq[QN + q]);
        V[BX * fs + L] = v;
      }
      if (ix5[it]) {  // B_y at (x, y, qz)
        T v = up[BY];
        v = v - dtd[2] * (Ep[q] - Eq[q]);
        v = v + dtd[0] * (Eq[2 * QN + q + 1] - Eq[2 * QN + q]);
        V[BY * fs + L] = v;
      }
    }
  };

  // Schedule: three barriers per plane. Phase 1 pairs the fluxes of plane p
  // with the primitives of plane p+2; phase 2 the EMFs of plane p with the
  // predictor of plane p+1; phase 3 the update of plane p-1. Rings: W 3 planes
  // (S1(p+2) replaces W(p-1), which only S2(p) of the previous phase 2 read),
  // reference EMFs 3 planes (S2(p+1) writes while S4(p) reads planes p and
  // p-1), the high z-face states 2 planes (S3(p) reads plane p-1's), fluxes
  // and EMFs 2 planes.
  stage1(zs - 2);
  stage1(zs - 1);
  stage1(zs);
  __syncthreads();
  stage2(zs - 1);
  __syncthreads();
  for (int p = zs - 1; p <= ze; ++p) {
    stage3(p);
    if (p + 2 <= ze + 1) stage1(p + 2);
    __syncthreads();
    const bool upd = p - 1 >= zs && p - 1 < ze;
    if constexpr (AHEAD) {
      if (upd && q5[0] >= 0) load_up(p - 1, 0);
    }
    if (p >= zs) stage4(p);
    if (p + 1 <= ze) stage2(p + 1);
    __syncthreads();
    if (upd) stage5(p - 1);
    __syncthreads();
  }
}

// CTAs per SM the FP32 tiles are compiled for
template <int VAR> constexpr int fused_ctas_fp32() { return VAR <= 1 ? 1 : (VAR == 3 ? 3 : 2); }
template <class T, int VAR, int MODE, bool FL = false>
__global__ void __launch_bounds__(FusedCfg<VAR>::NT, sizeof(T) == 4 ? fused_ctas_fp32<VAR>() : 1)
    k_advance3d_fused(LevelArgs a, int ntx) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  int pslot = blockIdx.y, tile = blockIdx.x, zc = blockIdx.z;
  bool halves = false;
  if (a.tail > 0) {
    // one-dimensional grid over the columns (patch-major): the first ones
    // whole, the last a.tail ones as two halves each, so that the launch's last
    // partial wave holds half-length marches
    const int ntiles = ntx * tile_count(a.maxn[1] + 2 * a.w, FusedCfg<VAR>::TY);
    const int full = ntiles * a.npatch - a.tail;
    const int item = blockIdx.x;
    const int col = item < full ? item : full + (item - full) / 2;
    pslot = col / ntiles;
    tile = col % ntiles;
    zc = item < full ? 0 : (item - full) % 2;
    halves = item >= full;
  }
  fused_tile<T, VAR, MODE, FL>(a, pslot, tile, ntx, zc, smem_raw, halves);
}

// ---------------------------------------------------------------- device work queue
// The multi-level advance as persistent launches (the GPU analogue of the
// paper's threaded level advances with preference to the finer levels, Sec. 4):
// one launch per sub-step of the finest level; the resident CTAs take tasks in
// ticket order from an atomic counter over a host-ordered list. Fill tasks (a
// range of same-level copy chunks into one patch, the finest level's) come
// first, then the advance tiles, finest level first: all of the finest
// level's, then a share of every coarser level's (a coarser level's advance
// is spread over the launches of its sub-step). An advance tile waits until every fill task into its patch has
// finished (a per-patch counter against the expected count). A wait only ever
// concerns tasks of smaller tickets, which running CTAs hold and finish
// without waiting, so every wait ends; each is bounded in time all the same:
// on expiry the CTA sets ERR_QUEUE_TIMEOUT in the error word and the abort
// flag, and every CTA stops taking tasks (no wait is left in flight: the CTA
// holds no asynchronous copies while it waits).
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned int load_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

template <class T, int VAR>
__global__ void __launch_bounds__(FusedCfg<VAR>::NT, sizeof(T) == 4 ? 2 : 1)
    k_advance_queue(const __grid_constant__ QueueArgs q) {
  constexpr int NF = FusedCfg<VAR>::NT / FILL_CHUNK * FILL_CHUNK;  // threads of a fill task
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int4 s_task;
  __shared__ int s_go;
  for (;;) {
    if (threadIdx.x == 0) {
      int4 t = make_int4(-1, 0, 0, 0);
      if (!(*(volatile unsigned int*)q.err & ERR_QUEUE_TIMEOUT) && !*(volatile int*)q.abort) {
        const unsigned int k = atomicAdd(q.head, 1u);
        if (k < (unsigned int)q.ntasks) t = reinterpret_cast<const int4*>(q.tasks)[k];
      }
      s_task = t;
    }
    __syncthreads();
    const int4 t = s_task;
    if (t.x < 0) return;
    const QueueLevel& L = q.L[t.x >> 4];
    if (t.x & 1) {
      // fill task: the chunk range [t.y, t.z) of the level's same-level boxes
      int4* sch = reinterpret_cast<int4*>(smem_raw);
      T* B = (T*)L.a.cur;
      const int4* ch = reinterpret_cast<const int4*>(L.chunks);
      if (t.x & 2) fill_range<T, 5, 2, NF>(B, L.boxes, ch, t.y, t.z, sch, sch + FILL_TILE);
      else fill_range<T, 1, 4, NF>(B, L.boxes, ch, t.y, t.z, sch, sch + FILL_TILE);
      __syncthreads();
      if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(q.done + t.w, 1u);
      }
    } else {
      // advance tile: first every fill into its patch
      if (threadIdx.x == 0) {
        int go = 1;
        const unsigned int need = q.need[t.w];
        if (need) {
          const unsigned long long t0 = global_ns();
          while (load_acquire(q.done + t.w) < need) {
            if (*(volatile int*)q.abort) { go = 0; break; }
            if (global_ns() - t0 > q.wait_ns) {
              atomicOr(q.err, ERR_QUEUE_TIMEOUT);
              atomicExch(q.abort, 1);
              go = 0;
              break;
            }
            __nanosleep(128);
          }
          __threadfence();
        }
        s_go = go;
      }
      __syncthreads();
      if (s_go) fused_tile<T, VAR, 1>(L.a, t.y, t.z, L.ntx, 0, smem_raw);
    }
    __syncthreads();  // the task's shared memory is free for the next one
  }
}

// ------------------------------------------------------------------ register recompute
// Registers for the fused path, recomputed from the state the advance read:
// the same formulas as the fused kernel, evaluated at the listed faces/edges.
template <class T>
__device__ void predict_at(const T* U, const DPatch& P, int L, double dt, const double* idx, double gamma, T* wh,
                           T* sd /* 3 x 8 */, const Floors* fl) {
  const int fs = (int)P.fs;
  const int st[3] = {1, P.ext[0], P.ext[0] * P.ext[1]};
  const Gm1<T> gm1(gamma - 1.0);
  T wc[8], wm[8], wp[8];
  load_recover(U, fs, L, st[1], st[2], gm1, wc, (T*)nullptr, fl);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    load_recover(U, fs, L - st[d], st[1], st[2], gm1, wm, (T*)nullptr, fl);
    load_recover(U, fs, L + st[d], st[1], st[2], gm1, wp, (T*)nullptr, fl);
#pragma unroll
    for (int f = 0; f < 8; ++f) {
      if (f == BX + d) sd[8 * d + f] = U[(BX + d) * fs + L + st[d]] - U[(BX + d) * fs + L];
      else sd[8 * d + f] = mm(wc[f] - wm[f], wp[f] - wc[f]);
    }
  }
  const T ir = T(1) / wc[0];
  const T g = (T)gamma;
  T dw[8];
#pragma unroll
  for (int f = 0; f < 8; ++f) wh[f] = wc[f];
  const T h0 = (T)(0.5 * dt * idx[0]), h1 = (T)(0.5 * dt * idx[1]), h2 = (T)(0.5 * dt * idx[2]);
  prim_terms<T, 0>(wc, sd, g, ir, dw);
#pragma unroll
  for (int f = 0; f < 8; ++f) wh[f] = wh[f] - h0 * dw[f];
  prim_terms<T, 1>(wc, sd + 8, g, ir, dw);
#pragma unroll
  for (int f = 0; f < 8; ++f) wh[f] = wh[f] - h1 * dw[f];
  prim_terms<T, 2>(wc, sd + 16, g, ir, dw);
#pragma unroll
  for (int f = 0; f < 8; ++f) wh[f] = wh[f] - h2 * dw[f];
}

// flux through the d-face stored at L (cells L - st[d] and L), global field order
template <class T>
__device__ void face_flux_at(const T* U, const DPatch& P, int d, int L, double dt, const double* idx, double gamma,
                             double igm1, T* out8, const Floors* fl) {
  const int st[3] = {1, P.ext[0], P.ext[0] * P.ext[1]};
  T whl[8], whr[8], sl[24], sr[24], wl[8], wr[8];
  predict_at(U, P, L - st[d], dt, idx, gamma, whl, sl, fl);
  predict_at(U, P, L, dt, idx, gamma, whr, sr, fl);
#pragma unroll
  for (int f = 0; f < 8; ++f) {
    wl[f] = plus_half<T>(whl[f], sl[8 * d + f]);
    wr[f] = minus_half<T>(whr[f], sr[8 * d + f]);
  }
  hlld_face<T>(wl, wr, d, (T)gamma, igm1, out8);
}

// E_c at the c-edge stored at L (the low a,b corner of cell L), (a,b,c) cyclic
template <class T>
__device__ T edge_emf_at(const T* U, const DPatch& P, int c, int L, double dt, const double* idx, double gamma,
                         double igm1, const Floors* fl) {
  const int st[3] = {1, P.ext[0], P.ext[0] * P.ext[1]};
  const int a = (c + 1) % 3, b = (c + 2) % 3;
  const int Lc[4] = {L - st[a] - st[b], L - st[b], L - st[a], L};  // (a-1,b-1), (a,b-1), (a-1,b), (a,b)
  T wh[4][8], sd[4][24];
  for (int k = 0; k < 4; ++k) predict_at(U, P, Lc[k], dt, idx, gamma, wh[k], sd[k], fl);
  T wl[8], wr[8], fa_lo[8], fa_hi[8], fb_lo[8], fb_hi[8];
  const T g = (T)gamma;
  // a-faces at rows b-1 (cells 0 -> 1) and b (cells 2 -> 3)
#pragma unroll
  for (int f = 0; f < 8; ++f) { wl[f] = plus_half<T>(wh[0][f], sd[0][8 * a + f]); wr[f] = minus_half<T>(wh[1][f], sd[1][8 * a + f]); }
  hlld_face<T>(wl, wr, a, g, igm1, fa_lo);
#pragma unroll
  for (int f = 0; f < 8; ++f) { wl[f] = plus_half<T>(wh[2][f], sd[2][8 * a + f]); wr[f] = minus_half<T>(wh[3][f], sd[3][8 * a + f]); }
  hlld_face<T>(wl, wr, a, g, igm1, fa_hi);
  // b-faces at columns a-1 (cells 0 -> 2) and a (cells 1 -> 3)
#pragma unroll
  for (int f = 0; f < 8; ++f) { wl[f] = plus_half<T>(wh[0][f], sd[0][8 * b + f]); wr[f] = minus_half<T>(wh[2][f], sd[2][8 * b + f]); }
  hlld_face<T>(wl, wr, b, g, igm1, fb_lo);
#pragma unroll
  for (int f = 0; f < 8; ++f) { wl[f] = plus_half<T>(wh[1][f], sd[1][8 * b + f]); wr[f] = minus_half<T>(wh[3][f], sd[3][8 * b + f]); }
  hlld_face<T>(wl, wr, b, g, igm1, fb_hi);
  T r[4];
  for (int k = 0; k < 4; ++k) {
    const T* h = wh[k];
    r[k] = c == 0 ? h[3] * h[6] - h[2] * h[7] : (c == 1 ? h[1] * h[7] - h[3] * h[5] : h[2] * h[5] - h[1] * h[6]);
  }
  return gs_emf<T>(-fa_lo[BX + b], -fa_hi[BX + b], fb_lo[BX + a], fb_hi[BX + a], r[0], r[1], r[2], r[3], fa_lo[RHO],
                   fa_hi[RHO], fb_lo[RHO], fb_hi[RHO]);
}

// the floors a register recompute repeats (those of the advance it mirrors)
__device__ __forceinline__ const Floors* rc_floors(const RowArgs& a) {
  return (a.fl.rho > 0.0 || a.fl.p > 0.0) ? &a.fl : nullptr;
}

// RowArgs.fbuf = the state the level's advance read (for the coarse side the
// coarse level, for the fine side the fine level); dt = *dtp * dtscale.
template <class T>
__device__ __forceinline__ void regrc_coarse_faces_row(const RowArgs& a, long long r, double gamma, double ix, double iy,
                                      double iz) {
  if (r >= a.nrows) return;
  const int* row = a.rows + 7 * r;
  const DPatch P = a.P[row[1]];
  const double dt = *a.dtp * a.dtscale;
  const double idx[3] = {ix, iy, iz};
  T f8[8];
  face_flux_at<T>((const T*)a.fbuf + P.off, P, row[2], row[3], dt, idx, gamma, a.igm1, f8, rc_floors(a));
#pragma unroll
  for (int n = 0; n < 5; ++n) a.creg[r * 6 + n] = dt * (double)f8[n];
}

template <class T>
__device__ __forceinline__ void regrc_coarse_edges_row(const RowArgs& a, long long r, double gamma, double ix, double iy,
                                      double iz) {
  if (r >= a.nrows) return;
  const int* row = a.rows + 6 * r;
  const DPatch P = a.P[row[1]];
  const double dt = *a.dtp * a.dtscale;
  const double idx[3] = {ix, iy, iz};
  a.ecreg[r] = dt * (double)edge_emf_at<T>((const T*)a.fbuf + P.off, P, row[2], row[3], dt, idx, gamma, a.igm1, rc_floors(a));
}

template <class T>
__device__ __forceinline__ void regrc_fine_faces_row(const RowArgs& a, long long r, double gamma, double ix, double iy,
                                      double iz) {
  if (r >= a.nrows) return;
  const int* row = a.rows + 7 * r;
  const DPatch P = a.P[row[5]];
  const int d = row[2], L = row[6];
  const double dt = *a.dtp * a.dtscale;
  const double idx[3] = {ix, iy, iz};
  const double af = dt * 0.25;
  const int sx = 1, sy = P.ext[0], sz = P.ext[0] * P.ext[1];
  int o1, o2;
  if (d == 0) { o1 = sy; o2 = sz; }
  else if (d == 1) { o1 = sx; o2 = sz; }
  else { o1 = sx; o2 = sy; }
  const int off[4] = {0, o1, o2, o1 + o2};
  T f[4][8];
  const T* U = (const T*)a.fbuf + P.off;
  for (int k = 0; k < 4; ++k) face_flux_at<T>(U, P, d, L + off[k], dt, idx, gamma, a.igm1, f[k], rc_floors(a));
  double* out = a.freg + (r * 2 + (a.substep - 1)) * 6;
#pragma unroll
  for (int n = 0; n < 5; ++n)
    out[n] = af * tree4((double)f[0][n], (double)f[1][n], (double)f[2][n], (double)f[3][n]);
}

template <class T>
__device__ __forceinline__ void regrc_fine_edges_row(const RowArgs& a, long long r, double gamma, double ix, double iy,
                                      double iz) {
  if (r >= a.nrows) return;
  const int* row = a.rows + 6 * r;
  const DPatch P = a.P[row[4]];
  const int c = row[2], L = row[5];
  const double dt = *a.dtp * a.dtscale;
  const double idx[3] = {ix, iy, iz};
  const int sc = c == 0 ? 1 : (c == 1 ? P.ext[0] : P.ext[0] * P.ext[1]);
  const T* U = (const T*)a.fbuf + P.off;
  const T e0 = edge_emf_at<T>(U, P, c, L, dt, idx, gamma, a.igm1, rc_floors(a));
  const T e1 = edge_emf_at<T>(U, P, c, L + sc, dt, idx, gamma, a.igm1, rc_floors(a));
  a.efreg[r * 2 + (a.substep - 1)] = (dt * 0.5) * tree2((double)e0, (double)e1);
}

// fine-side registers from the boundary capture of the fine level's fused
// advance (the same fluxes and EMFs the recompute kernels above evaluate); a
// face or edge off the boundary planes (none by construction) is recomputed
template <class T>
__device__ __forceinline__ void regcap_fine_faces_row(const RowArgs& a, long long r, double gamma, double ix, double iy,
                                      double iz) {
  if (r >= a.nrows) return;
  const int* row = a.rows + 7 * r;
  const DPatch P = a.P[row[5]];
  const int d = row[2], L = row[6];
  const double dt = *a.dtp * a.dtscale;
  const double af = dt * 0.25;
  const int sx = 1, sy = P.ext[0], sz = P.ext[0] * P.ext[1];
  int o1, o2;
  if (d == 0) { o1 = sy; o2 = sz; }
  else if (d == 1) { o1 = sx; o2 = sz; }
  else { o1 = sx; o2 = sy; }
  const int off[4] = {0, o1, o2, o1 + o2};
  const T* b = (const T*)a.bnd + P.boff;
  const long long F = bnd_faces_total(P.n);
  T f[4][5];
  for (int k = 0; k < 4; ++k) {
    const int Lk = L + off[k];
    const int x = Lk % P.ext[0], y = (Lk / P.ext[0]) % P.ext[1], z = Lk / (P.ext[0] * P.ext[1]);
    const long long sl = P.boff >= 0 ? bnd_face_slot(P, d, x, y, z) : -1;
    if (sl >= 0) {
#pragma unroll
      for (int n = 0; n < 5; ++n) f[k][n] = b[n * F + sl];
    } else {
      const double idx[3] = {ix, iy, iz};
      T f8[8];
      face_flux_at<T>((const T*)a.fbuf + P.off, P, d, Lk, dt, idx, gamma, a.igm1, f8, rc_floors(a));
#pragma unroll
      for (int n = 0; n < 5; ++n) f[k][n] = f8[n];
    }
  }
  double* out = a.freg + (r * 2 + (a.substep - 1)) * 6;
#pragma unroll
  for (int n = 0; n < 5; ++n)
    out[n] = af * tree4((double)f[0][n], (double)f[1][n], (double)f[2][n], (double)f[3][n]);
}

template <class T>
__device__ __forceinline__ void regcap_fine_edges_row(const RowArgs& a, long long r, double gamma, double ix, double iy,
                                      double iz) {
  if (r >= a.nrows) return;
  const int* row = a.rows + 6 * r;
  const DPatch P = a.P[row[4]];
  const int c = row[2], L = row[5];
  const double dt = *a.dtp * a.dtscale;
  const int sc = c == 0 ? 1 : (c == 1 ? P.ext[0] : P.ext[0] * P.ext[1]);
  const T* b = (const T*)a.bnd + P.boff + 5 * bnd_faces_total(P.n);
  T ev[2];
  for (int k = 0; k < 2; ++k) {
    const int Lk = L + k * sc;
    const int x = Lk % P.ext[0], y = (Lk / P.ext[0]) % P.ext[1], z = Lk / (P.ext[0] * P.ext[1]);
    long long sl = -1;
    for (int e = 0; e < 3 && sl < 0 && P.boff >= 0; ++e)
      if (e != c) sl = bnd_edge_slot(P, c, e, x, y, z);
    if (sl >= 0) {
      ev[k] = b[sl];
    } else {
      const double idx[3] = {ix, iy, iz};
      ev[k] = edge_emf_at<T>((const T*)a.fbuf + P.off, P, c, Lk, dt, idx, gamma, a.igm1, rc_floors(a));
    }
  }
  a.efreg[r * 2 + (a.substep - 1)] = (dt * 0.5) * tree2((double)ev[0], (double)ev[1]);
}

// the face and the edge rows of one register side in one launch: blocks [0,
// nbf) take the face rows, the rest the edge rows (128 rows per block)
#define AMRK_REG_PAIR(NAME)                                                                          \
  template <class T>                                                                                 \
  __global__ void __launch_bounds__(128)                                                             \
      k_##NAME(RowArgs f, RowArgs e, unsigned nbf, double gamma, double ix, double iy, double iz) {  \
    if (blockIdx.x < nbf) NAME##_faces_row<T>(f, (long long)blockIdx.x * 128 + threadIdx.x, gamma, ix, iy, iz); \
    else NAME##_edges_row<T>(e, (long long)(blockIdx.x - nbf) * 128 + threadIdx.x, gamma, ix, iy, iz);  \
  }
AMRK_REG_PAIR(regrc_coarse)
AMRK_REG_PAIR(regrc_fine)
AMRK_REG_PAIR(regcap_fine)
#undef AMRK_REG_PAIR
