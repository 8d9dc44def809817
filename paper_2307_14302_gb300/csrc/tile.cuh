// tile.cuh -- tile form of the DG stage kernel for sm_103a.
//
// One warp owns a tile of 32 consecutive (Hilbert-ordered) triangles and advances it by one
// Runge-Kutta stage (Sec. 2.2, Eq. RKSSP) in three phases:
//   1. element phase A: each lane loads its triangle's record and static data, and integrates the
//      area terms of Eq. elem_weak_form (flux divergence, balance term g zeta grad(hb), friction,
//      pressure set-up) and the element rain of Eq. rain;
//   2. edge phase: every edge touching the tile is evaluated ONCE (Sec. 2.3: Roe or LLF flux at
//      p+1 Gauss points, land/ocean/river ghost states, the wet/dry closure of Sec. 2.4), about 60
//      edges per tile, one per lane and round, as the tile's plan lists them.  Both sides' records
//      come from shared memory: the tile's own records, and the records of the ~23 out-of-tile
//      neighbours staged there with cp.async while phase 1 runs.  The flux values at the Gauss points,
//      scaled by the Gauss weight and half the edge length, go into per-(element, local edge) slots in
//      shared memory, each side as seen along its own edge, with the pressure relative to that side's
//      own mean;
//   3. element phase B: each lane lifts its three edge slots into the modal right-hand side,
//      applies the diagonal inverse mass matrix (Eq. dubiner), the Shu-Osher combination, the
//      positive-depth operator M Pi_h (Sec. 2.4), stores its record and books its rain volume.
// Interior edges are oriented canonically (the lower element index is "left"), so an edge on the
// border of two tiles gives the same bits in both, and the two sides of every edge receive
// exactly opposite mass fluxes: mass is conserved to rounding of the element means.
// The three phases are one routine, tile_body, which the small-mesh kernel (steps.cuh) shares.
//
// Memory pipeline (per warp): a tile's records and its static block (geometry, plan, first vertices)
// arrive in shared memory by two TMA bulk copies (cp.async.bulk completing on an mbarrier); the next
// tile's records, and where the static buffer is doubled its static block too, are in flight while
// this tile is computed.  The modes of the tile's step-initial records are prefetched into L2 by a
// bulk prefetch at the start of the tile and read in phase 3; the out-of-tile neighbour records are
// gathered with 16-byte cp.async.  Every mbarrier wait is bounded: a wait that runs out sets
// ERR_TIMEOUT in the device error word and the kernel returns.
//
// Records are vector-major in shared memory ([RV][32], as in the tile-blocked device array), so
// the 16-byte reads of a warp, at its own slots or at any mix of neighbour slots, spread over
// the banks.  Shared memory per warp: TileLayout.
//
// The kernel takes a set of Feature bits (args.h): the generic instantiation has all of them;
// the specialised ones (tile_spec.cu) leave out the code of the features a run does not have.
#pragma once
#include "stage.cuh"

namespace dg {

constexpr int HALO = 32;    // staged out-of-tile neighbour records per tile
static_assert(HALO == TILE, "own and halo records share one vector stride in shared memory");

// The tile plan: what the neighbour codes say about a tile's edges, laid out once per mesh by
// plan_kernel (the connectivity never changes) and copied with the tile's other data.  One 32-bit
// word per edge:
//   bits 0-7    left side: source << 2 | local edge
//   bits 8-15   right side, or the boundary code (bit 16): 0 land, 1 + tidal segment,
//               1 + MAXSEG + river segment
//   bit 16      boundary edge;  bits 18-25  place of the edge's scaled normal in the geometry block;
//   bit 31      the right side is the tile's own element: the normal is negated
// sources: 0-31 own element, 32-63 staged halo record.  In-tile edges come first, then the edges to
// the first 32 neighbours in other tiles, then the boundary edges: the first round of the edge phase
// does not wait for the halo.  Tiles with more neighbours (about one in a thousand on Hilbert-ordered
// meshes) have two further batches: 32 more halo records each, and their edges.  Per tile:
// EDGE_INLINE words, the first 32 halo elements, (mixed path) the Manning coefficients, and {scenario,
// elements present, counts, further batches}; the words 64-95 and the further neighbours are in the
// overflow array.
// The plan lies between the tile's geometry and its first vertices in one block per tile (the static
// block), so that one bulk copy brings everything that does not change; a halo entry is the place of
// the neighbour's first record vector, (n / 32) RV 32 + n % 32.
// Before, every stage rebuilt this per tile from the neighbour codes (nine ballots, the population
// counts, a descriptor of two sides and a normal per edge): about 190 of 1,940 warp instructions,
// with the halo loads waiting for it.
constexpr int EDGE_INLINE = 64;
constexpr int PLAN_X = 32 + 64;  // overflow words per tile: edges 64..95, neighbours 32..95
constexpr unsigned ED_BND = 1u << 16, ED_OWN_R = 1u << 31;
template <class T>
__host__ __device__ constexpr int plan_vec() {  // 16-byte units per tile
  return (EDGE_INLINE + HALO + (sizeof(T) == 4 ? TILE : 0)) / 4 + 1;
}

template <int P, class Pol, int FT = FT_ALL>
struct TileLayout {
  using T = typename Pol::T;
  static constexpr int NG = P + 1;
  static constexpr int RV = Pol::template RV<P>;
  static constexpr int GV = Pol::GV;
  static constexpr int RVN = (sizeof(T) == 4 ? 6 + 3 * (np_of(P) - 1) + 3 : 2 * (3 * np_of(P)) + 3) / 4;  // vectors with modes
  // edge slot of one element side: Gz[NG], Gx[NG], Gy[NG] -- and the mass integral when NG is odd;
  // with an even NG the mass is the sum of the Gz, which is exactly antisymmetric across the edge
  // (the right side holds the negated values in reverse order) -- stored as pairs of T
  static constexpr bool MASSV = (NG % 2) == 1;
  static constexpr int NV = 3 * NG + (MASSV ? 1 : 0);
  static constexpr int NPR = (NV + 1) / 2;
  // first vertices of a tile (storm rain and pressure set-up only), 16-byte units
  static constexpr int XV = (FT & (FT_RAIN2 | FT_PRESS)) ? (sizeof(T) == 4 ? 16 : 32) : 0;
  // static part of a tile: geometry [32][GV], plan, first vertices
  static constexpr int PV = plan_vec<T>();
  static constexpr int S_GEO = 0;
  static constexpr int S_PLAN = S_GEO + TILE * GV;
  static constexpr int S_HALO = S_PLAN + EDGE_INLINE / 4;      // halo element indices
  static constexpr int S_MAN = S_HALO + HALO / 4;              // Manning coefficients (mixed)
  static constexpr int S_META = S_PLAN + PV - 1;
  static constexpr int S_XY = S_PLAN + PV;
  static constexpr int SV = S_XY + XV;
  static constexpr int SVM = S_XY + (sizeof(T) == 4 ? 16 : 32);  // in memory (first vertices always there)
  // per warp: two record buffers [RV][32] (the tile's block of the tile-blocked record array), the
  // static buffers, the halo records [RV][HALO], the edge slots [3][NPR][32] (pairs of T) and three
  // 8-byte mbarriers (buffers 0 and 1, single static).  Mixed p = 2 has one static buffer: the static
  // part is done with after the edge phase and the next tile's is copied in during the rest of this
  // one, which takes 2.3 KB less per warp and lets 12 warps share an SM instead of 8 (graded 300k:
  // 159 -> 143 us per step).  At p = 1 the second buffer is free (registers allow 16 warps either
  // way) and 2 % faster (hurricane 2M: 260 us per step against 265).
  static constexpr int NSTAT = (sizeof(T) == 4 && P == 2) ? 1 : 2;
  static constexpr int REC = TILE * RV;
  static constexpr int STAT = 2 * REC;
  static constexpr int HAL = STAT + NSTAT * SV;
  static constexpr int FLX = HAL + HALO * RV;
  static constexpr int BAR = FLX + 3 * NPR * 32 * 2 * (int)sizeof(T) / 16;
  static constexpr int VEC = BAR + 2;                          // 16-byte units per warp
};
template <int P, class Pol, int FT = FT_ALL>
__host__ __device__ constexpr int tile_smem_bytes(int block) {
  return 16 * TileLayout<P, Pol, FT>::VEC * (block / 32);
}

// ------------------------------------------------------------------ TMA bulk copies -----
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// global -> shared bulk copy (16-byte aligned addresses, size a multiple of 16) signalling bar
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// 16-byte load from a shared-memory address
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
// bulk prefetch of global memory into L2 (16-byte aligned, size a multiple of 16)
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// order this thread's earlier generic-proxy accesses to shared memory before later bulk copies
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// wait for the completion of phase `parity` of bar; false if it did not complete in 2^20 tries
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok = 0;
  for (int i = 0; i < (1 << 20) && !ok; ++i)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
  return ok != 0;
}

// a bulk copy that did not complete: record it in the device error word, give the warp's copies (this
// tile's and the next tile's records, the static part) one more bounded wait so that none lands in
// shared memory after the warp has left, and return
template <class Pol>
__device__ __noinline__ void tile_timeout(const StageArgs<Pol>& a, uint32_t bar, int it, bool next, bool sd, int lane) {
  if (lane == 0) atomicOr(&a.ctl->err, ERR_TIMEOUT);
  if (!sd) (void)mbar_wait(bar + 16, it & 1);
  (void)mbar_wait(bar + 8 * (it & 1), (it >> 1) & 1);
  if (next) (void)mbar_wait(bar + 8 * ((it + 1) & 1), ((it + 1) >> 1) & 1);
}

// static geometry record from shared memory (layout of load_geo); the Manning coefficient of the
// mixed path is in the tile plan
__device__ __forceinline__ void geo_from(const uint4* g, const float* man, Geo<Mixed>& G) {
  const uint4 a = g[0], b = g[1], c = g[2];
  G.lnx[0] = __uint_as_float(a.x); G.lny[0] = __uint_as_float(a.y);
  G.lnx[1] = __uint_as_float(a.z); G.lny[1] = __uint_as_float(a.w);
  G.lnx[2] = __uint_as_float(b.x); G.lny[2] = __uint_as_float(b.y);
  G.hbm = {__uint_as_float(b.z), __uint_as_float(b.w)};
  G.A = {__uint_as_float(c.x), __uint_as_float(c.y)};
  G.invA = {__uint_as_float(c.z), __uint_as_float(c.w)};
  G.man = *man;
}
__device__ __forceinline__ void geo_from(const uint4* g, const float*, Geo<Fp64>& G) {
  uint4 v[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) v[i] = g[i];
  G.lnx[0] = u2d(v[0].x, v[0].y); G.lny[0] = u2d(v[0].z, v[0].w);
  G.lnx[1] = u2d(v[1].x, v[1].y); G.lny[1] = u2d(v[1].z, v[1].w);
  G.lnx[2] = u2d(v[2].x, v[2].y); G.lny[2] = u2d(v[2].z, v[2].w);
  G.hbm = u2d(v[3].x, v[3].y);
  G.A = u2d(v[3].z, v[3].w);
  G.invA = u2d(v[4].x, v[4].y);
  G.man = u2d(v[4].z, v[4].w);
}

// ------------------------------------------------------------ scalar / packed arithmetic ---
// The area points are evaluated two at a time in packed FP32x2 (mixed path, p = 1) or one at a
// time; these overloads let one routine serve both.
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ f2 vmul(f2 a, f2 b) { return mul2(a, b); }
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ f2 vadd(f2 a, f2 b) { return add2(a, b); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ f2 vneg(f2 a) { return neg2(a); }
__device__ __forceinline__ float vmax(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double vmax(double a, double b) { return fmax(a, b); }
__device__ __forceinline__ f2 vmax(f2 a, f2 b) { return max2(a, b); }
__device__ __forceinline__ float vrcp(float a) { return frcp(a); }
__device__ __forceinline__ double vrcp(double a) { return frcp(a); }
__device__ __forceinline__ f2 vrcp(f2 a) { return rcp2(a); }
__device__ __forceinline__ float vsqrt0(float a) { return fsqrt0(a); }
__device__ __forceinline__ double vsqrt0(double a) { return fsqrt0(a); }
__device__ __forceinline__ f2 vsqrt0(f2 a) { return make_float2(fsqrt0(a.x), fsqrt0(a.y)); }
// friction coefficient tau (source -tau q): Manning g n^2 |u| / Hs^(4/3) (friction 0) or
// cf |u| / Hs (friction 1).  In FP32 as cfm 2^(lg2|q|^2 / 2 - c lg2 Hs) with c = 7/3 or 2, three
// special-function operations and no square root (|q| = 0 gives 2^-inf = 0); in FP64 from the depth
// factor hf of vdepth.
__device__ __forceinline__ float vtau(float qx, float qy, float, float, float Hs, float, float cfm, int friction) {
  const float c = friction == 0 ? 2.3333333f : 2.0f;
  return cfm * mufu_ex2(fmaf(0.5f, mufu_lg2(fmaf(qx, qx, qy * qy)), -c * mufu_lg2(Hs)));
}
__device__ __forceinline__ f2 vtau(f2 qx, f2 qy, f2 u, f2 v, f2 Hs, f2 hf, f2 cfm, int friction) {
  const f2 q2 = fma2(qx, qx, mul2(qy, qy));
  const f2 lq = make_float2(mufu_lg2(q2.x), mufu_lg2(q2.y)), lh = make_float2(mufu_lg2(Hs.x), mufu_lg2(Hs.y));
  const f2 x = fma2(p2(0.5f), lq, mul2(p2(friction == 0 ? -2.3333333f : -2.0f), lh));
  return mul2(cfm, make_float2(mufu_ex2(x.x), mufu_ex2(x.y)));
}
__device__ __forceinline__ double vtau(double, double, double u, double v, double, double hf, double cfm, int) {
  return cfm * (fsqrt0(fma(u, u, v * v)) * hf);
}
// 1/Hs and, in FP64, the friction law's depth factor
__device__ __forceinline__ float vdepth(float Hs, int, float&) { return vrcp(Hs); }
__device__ __forceinline__ f2 vdepth(f2 Hs, int, f2&) { return vrcp(Hs); }
__device__ __forceinline__ double vdepth(double Hs, int friction, double& hf) {
  double i;
  depth_inverse(Hs, friction, i, hf);
  return i;
}
template <class V>
__device__ __forceinline__ V vbc(float x);
template <>
__device__ __forceinline__ float vbc<float>(float x) { return x; }
template <>
__device__ __forceinline__ double vbc<double>(float x) { return (double)x; }
template <>
__device__ __forceinline__ f2 vbc<f2>(float x) { return make_float2(x, x); }

// a pair of constant-table entries (points q, q+1 of one mode) or one entry
template <class V, class T>
__device__ __forceinline__ V vtab(const T* row, int q);
template <>
__device__ __forceinline__ float vtab<float, float>(const float* row, int q) { return row[q]; }
template <>
__device__ __forceinline__ double vtab<double, double>(const double* row, int q) { return row[q]; }
template <>
__device__ __forceinline__ f2 vtab<f2, float>(const float* row, int q) { return make_float2(row[q], row[q + 1]); }

// ------------------------------------------------------------------------ area (p = 1) ---
// Degree-1 elements have constant basis gradients: the flux terms need only the weighted sums of
// F over the points (SF), the sources their moments against each basis function (SS).  q_x v = q_y u, so
// the two cross terms are one sum.  The degree-3 rule's points are the centroid (0), the edge midpoints
// opposite vertex k (1 + k) and the vertices (4 + k): a linear field takes its mean at the centroid,
// three sums at the vertices and one operation per midpoint (3/2 mean - 1/2 vertex k), instead of two
// products per field and point with table values.  The pairs (vertex k, midpoint k) are evaluated
// together in packed FP32x2, the centroid alone with what vanishes there left out.
template <class V>
struct AreaP1 {
  V SF[5];     // sum_q w_q (q_x, q_x u + p, q_y u, q_y, q_y v + p)
  V SS[3][2];  // sum_q w_q phi_m (s_x, s_y)
};

// values at the vertices v and at the midpoints m opposite them of the field with mean c and modes
// a, b (phi_1 = sqrt(3) (-1, 1, 0), phi_2 = (-1, -1, 2) at the vertices)
template <class T>
__device__ __forceinline__ void tri_points(T c, T a, T b, T v[3], T m[3]) {
  const T t = T(1.7320508075688772) * a, s = c - b, h = T(1.5) * c;
  v[0] = s - t;
  v[1] = s + t;
  v[2] = fma(T(2), b, c);
#pragma unroll
  for (int k = 0; k < 3; ++k) m[k] = fma(T(-0.5), v[k], h);
}
template <int K>
struct IntC {
  static constexpr int value = K;
};

// one point or pair: w and wp are its weight and weight times phi_m; CEN: the centroid (d = 0, phi_1 =
// phi_2 = 0); K: the vertex of the pair, where phi_1 vanishes at K = 2
template <bool CEN, int K, class V>
__device__ __forceinline__ void area_point_p1(AreaP1<V>& A, V d, V H, V qx, V qy, V w, const V wp[3], V H0v, V hg, V ghbx,
                                              V ghby, V cfm, int friction, V Fxs, V Fys) {
  const V Hs = vmax(H, H0v);
  V hf = vbc<V>(0.f);
  const V iH = vdepth(Hs, friction, hf);
  const V u = vmul(qx, iH), v = vmul(qy, iH);
  V tau = vbc<V>(0.f);
  if (friction <= 1) tau = vtau(qx, qy, u, v, Hs, hf, cfm, friction);
  V sx = vfma(vneg(tau), qx, Fxs), sy = vfma(vneg(tau), qy, Fys);
  V fxx, fyy;
  if (CEN) {
    fxx = vmul(qx, u);
    fyy = vmul(qy, v);
  } else {
    const V pp = vmul(vmul(hg, d), vfma(vbc<V>(2.f), H, vneg(d)));  // g/2 d (2H - d)
    sx = vfma(ghbx, d, sx);
    sy = vfma(ghby, d, sy);
    fxx = vfma(qx, u, pp);
    fyy = vfma(qy, v, pp);
  }
  A.SF[0] = vfma(w, qx, A.SF[0]);
  A.SF[1] = vfma(w, fxx, A.SF[1]);
  A.SF[2] = vfma(w, vmul(qy, u), A.SF[2]);
  A.SF[3] = vfma(w, qy, A.SF[3]);
  A.SF[4] = vfma(w, fyy, A.SF[4]);
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    if ((CEN && m > 0) || (K == 2 && m == 1)) continue;
    A.SS[m][0] = vfma(wp[m], sx, A.SS[m][0]);
    A.SS[m][1] = vfma(wp[m], sy, A.SS[m][1]);
  }
}

// Gaussian pressure set-up F = g H grad(eta_p) at a point (x, y) with depth H (graded workload)
template <class T>
__device__ __forceinline__ void setup_force(const ForcingT<T>& F, T px, T py, T H, T g, T& Fx, T& Fy) {
  const T dx = px - F.ps[0], dy = py - F.ps[1], is2 = frcp(F.ps[2] * F.ps[2]);
  const T eta = F.ps[3] * fexp(-(dx * dx + dy * dy) * T(0.5) * is2);
  Fx = g * H * (-eta * dx * is2);
  Fy = g * H * (-eta * dy * is2);
}

// area integrals (grad v, F) + (s, v) of one element into Rz, Rx, Ry (weak-form moments)
template <int P, class Pol, int FT>
__device__ __forceinline__ void tile_area(const Elem<P, Pol>& E, const Geo<Pol>& G, const ScenDev& S,
                                          const StageArgs<Pol>& a, int press, const typename Pol::T vx[3],
                                          const typename Pol::T vy[3], typename Pol::T (&Rz)[np_of(P)],
                                          typename Pol::T (&Rx)[np_of(P)], typename Pol::T (&Ry)[np_of(P)]) {
  using T = typename Pol::T;
  constexpr int NP = np_of(P);
  constexpr int NQ = 7;
  const RefTab<T>& tab = ctab<T, P>();
  const ForcingT<T>& F = forcing<T>(S);
  const T g = a.g, H0 = a.H0;
  const T detJ = T(0.5) * acc_r(G.A);
  const T idetJ = T(2) * acc_r(G.invA);
  // detJ grad(phi_1) and detJ grad(phi_2) of the linear modes phi_1 = sqrt(3) (lambda_1 - lambda_0),
  // phi_2 = 3 lambda_2 - 1: the barycentric gradients are -1 / (2 A) times the opposite edges' scaled normals
  const T G1x = T(0.4330127018922193) * (G.lnx[1] - G.lnx[2]), G1y = T(0.4330127018922193) * (G.lny[1] - G.lny[2]);
  const T G2x = T(-0.75) * G.lnx[0], G2y = T(-0.75) * G.lny[0];
  const T hbx = idetJ * (E.hb1 * G1x + E.hb2 * G2x), hby = idetJ * (E.hb1 * G1y + E.hb2 * G2y);  // constant grad(hb)
  const int friction = ft_friction(FT) >= 0 ? ft_friction(FT) : a.friction;
  const T cfm = (friction == 0) ? g * G.man * G.man : a.cf;
  if constexpr (P == 1) {
    const T xb = acc_r(E.xb), yb = acc_r(E.yb);
    T Fx[NQ], Fy[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) Fx[q] = Fy[q] = T(0);
    if (press) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const T px = tab.ql[q][0] * vx[0] + tab.ql[q][1] * vx[1] + tab.ql[q][2] * vx[2];
        const T py = tab.ql[q][0] * vy[0] + tab.ql[q][1] * vy[1] + tab.ql[q][2] * vy[2];
        const T Hq = E.Hb + (fma(E.zs[1], tab.qphi[q][2], E.zs[0] * tab.qphi[q][1]) +
                             fma(E.hb1, tab.qphi[q][1], E.hb2 * tab.qphi[q][2]));
        setup_force<T>(F, px, py, Hq, g, Fx[q], Fy[q]);
      }
    }
    T dv[3], dm[3], Hv[3], Hm[3], xv[3], xm[3], yv[3], ym[3];
    tri_points<T>(T(0), E.zs[0], E.zs[1], dv, dm);
    tri_points<T>(E.Hb, E.zs[0] + E.hb1, E.zs[1] + E.hb2, Hv, Hm);
    tri_points<T>(xb, E.xs[0], E.xs[1], xv, xm);
    tri_points<T>(yb, E.ys[0], E.ys[1], yv, ym);
    const T hg = T(0.5) * g, ghbx = g * hbx, ghby = g * hby;
    T SF[5], SS[3][2];
    AreaP1<T> A1;
#pragma unroll
    for (int i = 0; i < 5; ++i) A1.SF[i] = T(0);
#pragma unroll
    for (int m = 0; m < 3; ++m) A1.SS[m][0] = A1.SS[m][1] = T(0);
    {
      const T wp[3] = {tab.qwphiT[0][0], T(0), T(0)};
      area_point_p1<true, 0, T>(A1, T(0), E.Hb, xb, yb, tab.qwT[0], wp, H0, hg, ghbx, ghby, cfm, friction, Fx[0], Fy[0]);
    }
    if constexpr (sizeof(T) == 4 && DG_PACKED_FLUX) {
      AreaP1<f2> A2;
#pragma unroll
      for (int i = 0; i < 5; ++i) A2.SF[i] = p2(0.f);
#pragma unroll
      for (int m = 0; m < 3; ++m) A2.SS[m][0] = A2.SS[m][1] = p2(0.f);
      const f2 H02 = p2(H0), hg2 = p2(hg), gx2 = p2(ghbx), gy2 = p2(ghby), cfm2 = p2(cfm);
      auto pair = [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const f2 wp[3] = {make_float2(tab.vmw[k][1][0], tab.vmw[k][1][1]), make_float2(tab.vmw[k][2][0], tab.vmw[k][2][1]),
                          make_float2(tab.vmw[k][3][0], tab.vmw[k][3][1])};
        area_point_p1<false, k, f2>(A2, make_float2(dv[k], dm[k]), make_float2(Hv[k], Hm[k]), make_float2(xv[k], xm[k]),
                                    make_float2(yv[k], ym[k]), make_float2(tab.vmw[k][0][0], tab.vmw[k][0][1]), wp, H02, hg2,
                                    gx2, gy2, cfm2, friction, make_float2(Fx[4 + k], Fx[1 + k]),
                                    make_float2(Fy[4 + k], Fy[1 + k]));
      };
      pair(IntC<0>());
      pair(IntC<1>());
      pair(IntC<2>());
#pragma unroll
      for (int i = 0; i < 5; ++i) SF[i] = (A2.SF[i].x + A2.SF[i].y) + A1.SF[i];
      SS[0][0] = (A2.SS[0][0].x + A2.SS[0][0].y) + A1.SS[0][0];
      SS[0][1] = (A2.SS[0][1].x + A2.SS[0][1].y) + A1.SS[0][1];
#pragma unroll
      for (int m = 1; m < 3; ++m) {
        SS[m][0] = A2.SS[m][0].x + A2.SS[m][0].y;
        SS[m][1] = A2.SS[m][1].x + A2.SS[m][1].y;
      }
    } else {
      auto both = [&](auto kc) {
        constexpr int k = decltype(kc)::value;
        const T wv[3] = {tab.vmw[k][1][0], tab.vmw[k][2][0], tab.vmw[k][3][0]};
        const T wm[3] = {tab.vmw[k][1][1], tab.vmw[k][2][1], tab.vmw[k][3][1]};
        area_point_p1<false, k, T>(A1, dv[k], Hv[k], xv[k], yv[k], tab.vmw[k][0][0], wv, H0, hg, ghbx, ghby, cfm, friction,
                                   Fx[4 + k], Fy[4 + k]);
        area_point_p1<false, k, T>(A1, dm[k], Hm[k], xm[k], ym[k], tab.vmw[k][0][1], wm, H0, hg, ghbx, ghby, cfm, friction,
                                   Fx[1 + k], Fy[1 + k]);
      };
      both(IntC<0>());
      both(IntC<1>());
      both(IntC<2>());
#pragma unroll
      for (int i = 0; i < 5; ++i) SF[i] = A1.SF[i];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        SS[m][0] = A1.SS[m][0];
        SS[m][1] = A1.SS[m][1];
      }
    }
    const T gx[3] = {T(0), G1x, G2x}, gy[3] = {T(0), G1y, G2y};
    Rz[0] = T(0);
    Rx[0] = detJ * SS[0][0];
    Ry[0] = detJ * SS[0][1];
#pragma unroll
    for (int m = 1; m < NP; ++m) {
      Rz[m] = gx[m] * SF[0] + gy[m] * SF[3];
      Rx[m] = fma(detJ, SS[m][0], gx[m] * SF[1] + gy[m] * SF[2]);
      Ry[m] = fma(detJ, SS[m][1], gx[m] * SF[2] + gy[m] * SF[4]);
    }
  } else if constexpr (sizeof(T) == 4 && DG_PACKED_FLUX) {
    // FP32: the points in packed pairs (0,1), (2,3), (4,5), (6,7); point 7 has zero weight and zero
    // basis values (the mean state, finite) and adds exact zeros
    static_assert(NQ + 1 == MAXNQP, "one padding point");
    // gradients of r and s: the barycentric gradients of vertices 1 and 2, times 2
    const T h = T(-0.5) * idetJ, rx = h * G.lnx[2], ry = h * G.lny[2], sx = h * G.lnx[0], sy = h * G.lny[0];
    constexpr int NS = NP - 1;
    f2 Rz2[NP], Rx2[NP], Ry2[NP];
#pragma unroll
    for (int m = 0; m < NP; ++m) Rz2[m] = Rx2[m] = Ry2[m] = p2(0.f);
    const f2 rx2 = p2(rx), ry2 = p2(ry), sx2 = p2(sx), sy2 = p2(sy), detJ2 = p2(detJ);
    const f2 H02 = p2(H0), hg = p2(0.5f * g), ghbx = p2(g * hbx), ghby = p2(g * hby), cfm2 = p2(cfm);
    const f2 xb2 = p2(acc_r(E.xb)), yb2 = p2(acc_r(E.yb)), Hb2 = p2(E.Hb), hb12 = p2(E.hb1), hb22 = p2(E.hb2);
#pragma unroll
    for (int q = 0; q < NQ + 1; q += 2) {
      f2 d = p2(0.f), qx = xb2, qy = yb2;
#pragma unroll
      for (int m = 0; m < NS; ++m) {
        const f2 ph = vtab<f2, float>(tab.qphiT[m + 1], q);
        d = fma2(p2(E.zs[m]), ph, d);
        qx = fma2(p2(E.xs[m]), ph, qx);
        qy = fma2(p2(E.ys[m]), ph, qy);
      }
      const f2 H = add2(Hb2, add2(d, fma2(hb12, vtab<f2, float>(tab.qphiT[1], q),
                                          mul2(hb22, vtab<f2, float>(tab.qphiT[2], q)))));
      const f2 Hs = max2(H, H02);
      const f2 iH = rcp2(Hs);
      const f2 u = mul2(qx, iH), v = mul2(qy, iH);
      const f2 pp = mul2(mul2(hg, d), fma2(p2(2.f), H, neg2(d)));  // g/2 d (2H - d)
      f2 tau = p2(0.f);
      if (friction <= 1) tau = vtau(qx, qy, u, v, Hs, p2(0.f), cfm2, friction);
      float Fx0 = 0.f, Fy0 = 0.f, Fx1 = 0.f, Fy1 = 0.f;
      if (press) {
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (q + k >= NQ) continue;
          const float px = tab.ql[q + k][0] * vx[0] + tab.ql[q + k][1] * vx[1] + tab.ql[q + k][2] * vx[2];
          const float py = tab.ql[q + k][0] * vy[0] + tab.ql[q + k][1] * vy[1] + tab.ql[q + k][2] * vy[2];
          setup_force<float>(F, px, py, k ? H.y : H.x, g, k ? Fx1 : Fx0, k ? Fy1 : Fy0);
        }
      }
      const f2 sxs = fma2(ghbx, d, fma2(neg2(tau), qx, make_float2(Fx0, Fx1)));
      const f2 sys = fma2(ghby, d, fma2(neg2(tau), qy, make_float2(Fy0, Fy1)));
      const f2 fxx = fma2(qx, u, pp), fyx = mul2(qx, v), fxy = mul2(qy, u), fyy = fma2(qy, v, pp);
      const f2 wq = mul2(vtab<f2, float>(tab.qwT, q), detJ2);
      // fluxes rotated into the reference directions, with the weight
      const f2 zr = mul2(wq, fma2(rx2, qx, mul2(ry2, qy))), zs = mul2(wq, fma2(sx2, qx, mul2(sy2, qy)));
      const f2 xr = mul2(wq, fma2(rx2, fxx, mul2(ry2, fyx))), xs2 = mul2(wq, fma2(sx2, fxx, mul2(sy2, fyx)));
      const f2 yr = mul2(wq, fma2(rx2, fxy, mul2(ry2, fyy))), ys2 = mul2(wq, fma2(sx2, fxy, mul2(sy2, fyy)));
      const f2 wsx = mul2(wq, sxs), wsy = mul2(wq, sys);
#pragma unroll
      for (int m = 0; m < NP; ++m) {
        const f2 dr = vtab<f2, float>(tab.qdrT[m], q), ds = vtab<f2, float>(tab.qdsT[m], q);
        const f2 ph = vtab<f2, float>(tab.qphiT[m], q);
        if (m > 0) Rz2[m] = fma2(dr, zr, fma2(ds, zs, Rz2[m]));
        Rx2[m] = fma2(dr, xr, fma2(ds, xs2, fma2(ph, wsx, Rx2[m])));
        Ry2[m] = fma2(dr, yr, fma2(ds, ys2, fma2(ph, wsy, Ry2[m])));
      }
    }
#pragma unroll
    for (int m = 0; m < NP; ++m) {
      Rz[m] = Rz2[m].x + Rz2[m].y;
      Rx[m] = Rx2[m].x + Rx2[m].y;
      Ry[m] = Ry2[m].x + Ry2[m].y;
    }
  } else {
    const T h = T(-0.5) * idetJ, rx = h * G.lnx[2], ry = h * G.lny[2], sx = h * G.lnx[0], sy = h * G.lny[0];
#pragma unroll
    for (int m = 0; m < NP; ++m) Rz[m] = Rx[m] = Ry[m] = T(0);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const Trace<T> tq = trace_at<P, Pol>(E, tab.qphi[q]);
      const T Hs = max_r(tq.H, H0);
      T hf = T(0);
      const T iH = vdepth(Hs, friction, hf);
      const T u = tq.qx * iH, v = tq.qy * iH;
      const T pp = pdev(tq.d, tq.H, g);
      T tau = 0;
      if (friction <= 1) tau = vtau(tq.qx, tq.qy, u, v, Hs, hf, cfm, friction);
      T Fxs = 0, Fys = 0;
      if (press) {
        const T px = tab.ql[q][0] * vx[0] + tab.ql[q][1] * vx[1] + tab.ql[q][2] * vx[2];
        const T py = tab.ql[q][0] * vy[0] + tab.ql[q][1] * vy[1] + tab.ql[q][2] * vy[2];
        setup_force<T>(F, px, py, tq.H, g, Fxs, Fys);
      }
      const T sx_ = g * tq.d * hbx - tau * tq.qx + Fxs;
      const T sy_ = g * tq.d * hby - tau * tq.qy + Fys;
      const T fxx = tq.qx * u + pp, fyx = tq.qx * v;
      const T fxy = tq.qy * u, fyy = tq.qy * v + pp;
      const T wq = tab.qw[q] * detJ;
      // each flux rotated once into the reference directions (grad phi_m = qdr grad r + qds grad s),
      // with the weight: then two products per mode and variable
      const T zr = wq * (rx * tq.qx + ry * tq.qy), zs = wq * (sx * tq.qx + sy * tq.qy);
      const T xr = wq * (rx * fxx + ry * fyx), xs2 = wq * (sx * fxx + sy * fyx);
      const T yr = wq * (rx * fxy + ry * fyy), ys2 = wq * (sx * fxy + sy * fyy);
      const T wsx = wq * sx_, wsy = wq * sy_;
#pragma unroll
      for (int m = 0; m < NP; ++m) {
        const T dr = tab.qdr[q][m], ds = tab.qds[q][m], ph = tab.qphi[q][m];
        if (m > 0) Rz[m] = fma(dr, zr, fma(ds, zs, Rz[m]));
        Rx[m] = fma(dr, xr, fma(ds, xs2, fma(ph, wsx, Rx[m])));
        Ry[m] = fma(dr, yr, fma(ds, ys2, fma(ph, wsy, Ry[m])));
      }
    }
  }
}

// ---------------------------------------------------------------------- edge phase ------
// record of a side in shared memory (read as such, not through a generic address): own (src < 32) or
// staged halo; ownB and halB are the addresses of the blocks' first vectors, halB less 32 of them
template <int RV>
__device__ __forceinline__ void fetch_side(uint32_t ownB, uint32_t halB, unsigned src, Raw<RV>& r) {
  const uint32_t p = (src < 32 ? ownB : halB) + 16u * src;
  constexpr uint32_t stride = 16u * TILE;  // HALO == TILE: one stride for both
#pragma unroll
  for (int v = 0; v < RV; ++v) r.v[v] = lds128(p + stride * v);
}
// an edge's scaled normal along its left side's outward direction
__device__ __forceinline__ void edge_normal(const uint4* geo, unsigned ed, float& nx, float& ny) {
  const float2 n = reinterpret_cast<const float2*>(geo)[(ed >> 18) & 255];
  const unsigned sg = ed & ED_OWN_R;
  nx = __uint_as_float(__float_as_uint(n.x) ^ sg);
  ny = __uint_as_float(__float_as_uint(n.y) ^ sg);
}
__device__ __forceinline__ void edge_normal(const uint4* geo, unsigned ed, double& nx, double& ny) {
  const double2 n = reinterpret_cast<const double2*>(geo)[(ed >> 18) & 255];
  nx = (ed & ED_OWN_R) ? -n.x : n.x;
  ny = (ed & ED_OWN_R) ? -n.y : n.y;
}
// traces of a side at the points of its local edge j, in reverse order with REV (the points of the
// other side).  ephi4 (FP32): p = 1 one row per edge {phi_1, phi_2 at point 0, at point 1}; p = 2 one row
// per edge and mode m = 1..5 with phi_m at the three points
template <int P, class Pol, bool REV>
__device__ __forceinline__ void side_traces(const Elem<P, Pol>& E, int j, const typename Pol::T (*ephi)[P + 1][np_of(P)],
                                            const float4* ephi4, Trace<typename Pol::T> (&t)[P + 1]) {
  using T = typename Pol::T;
  constexpr int NG = P + 1;
  if constexpr (sizeof(T) == 4 && P == 1) {
    const float4 b = ephi4[j];
    t[REV ? 1 : 0] = trace_p1(E, b.x, b.y);
    t[REV ? 0 : 1] = trace_p1(E, b.z, b.w);
  } else if constexpr (sizeof(T) == 4) {
    const T xb = acc_r(E.xb), yb = acc_r(E.yb);
    T h[NG];
#pragma unroll
    for (int k = 0; k < NG; ++k) t[k] = {T(0), T(0), xb, yb};
#pragma unroll
    for (int m = 0; m < np_of(P) - 1; ++m) {
      const float4 b = ephi4[5 * j + m];
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int q = REV ? NG - 1 - k : k;
        const float ph = q == 0 ? b.x : (q == 1 ? b.y : b.z);
        t[k].d = fma(E.zs[m], ph, t[k].d);
        t[k].qx = fma(E.xs[m], ph, t[k].qx);
        t[k].qy = fma(E.ys[m], ph, t[k].qy);
        if (m == 0) h[k] = E.hb1 * ph;
        if (m == 1) h[k] = fma(E.hb2, ph, h[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < NG; ++k) t[k].H = E.Hb + (t[k].d + h[k]);
  } else if constexpr (P == 1) {
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const T* ph = ephi[j][REV ? NG - 1 - k : k];
      t[k] = trace_p1(E, ph[1], ph[2]);
    }
  } else {
#pragma unroll
    for (int k = 0; k < NG; ++k) t[k] = trace_at<P, Pol>(E, ephi[j][REV ? NG - 1 - k : k]);
  }
}

// one side's edge slot at flx[(j NPR + i) 32 + lane], pairs of T: Gz[NG], Gx[NG], Gy[NG] (, mass)
template <class T>
struct Pair;
template <>
struct Pair<float> {
  using V = float2;
};
template <>
struct Pair<double> {
  using V = double2;
};
template <class T, int NPR, int NV>
__device__ __forceinline__ void store_side(void* flx, int lane, int j, const T* vals) {
  using V = typename Pair<T>::V;
  V* f = reinterpret_cast<V*>(flx);
#pragma unroll
  for (int i = 0; i < NPR; ++i) {
    V v;
    v.x = vals[2 * i];
    v.y = (2 * i + 1 < NV) ? vals[2 * i + 1] : T(0);
    f[(j * NPR + i) * 32 + lane] = v;
  }
}
template <class T, int NPR, int NV>
__device__ __forceinline__ void load_side(const void* flx, int lane, int j, T* vals) {
  using V = typename Pair<T>::V;
  const V* f = reinterpret_cast<const V*>(flx);
#pragma unroll
  for (int i = 0; i < NPR; ++i) {
    const V v = f[(j * NPR + i) * 32 + lane];
    vals[2 * i] = v.x;
    if (2 * i + 1 < NV) vals[2 * i + 1] = v.y;
  }
}
// mass integral of a side's slot: stored (odd NG) or the sum of its Gz in point order (even NG)
template <class T, int NG, bool MASSV>
__device__ __forceinline__ T side_mass(const T* vals) {
  if constexpr (MASSV) {
    return vals[3 * NG];
  } else {
    T m = vals[0];
#pragma unroll
    for (int k = 1; k < NG; ++k) m += vals[k];
    return m;
  }
}

// reflective wall seen from a trace, along the unit outward normal n: the numerical flux between
// the trace and its mirror image in closed form (Roe: q.n (q.n / Hs + c) n; LLF adds |q.n| q.n / Hs
// n), plus the pressure relative to the side's own mean; no mass crosses
template <int FLUX, class T>
__device__ __forceinline__ T wall_coef(const Trace<T>& t, T nx, T ny, T g, T H0) {
  const T qn = t.qx * nx + t.qy * ny;
  const T Hs = max_r(t.H, H0);
  const T r = frsqrt(Hs), iH = r * r;
  const T c = fsqrt_pos(g) * (Hs * r);
  const T un = (FLUX == 1) ? (qn + abs_r(qn)) * iH : qn * iH;
  return qn * (un + c) + pdev(t.d, t.H, g);
}

// Edge slots at p = 1 in FP32 hold, per variable, the sum S and the difference D of the two point
// values instead of the values: seen from the other side (negated, points in reverse order) they are
// (-S, D), so the right side needs no reordering, S of the mass flux is the mass integral, and the lift
// needs only the basis' means and differences over the points, several of which are zero.  With the
// normals by one index, the boundary cases in a branch of their own and no run-time test for far
// neighbours: 361 -> about 300 warp instructions per edge round, 250k triangles 39.2 -> 36.3 us per step,
// hurricane 2M 253.6 -> 233.9, 500k LLF SSP(5,2) 185.3 -> 175.4, graded p = 2 300k 140.2 -> 136.2.
template <int P, class Pol>
DG_HD constexpr bool slots_sd() {
  return DG_PACKED_FLUX && P == 1 && sizeof(typename Pol::T) == 4;
}
__device__ __forceinline__ f2 sum_diff(f2 v) { return make_float2(v.x + v.y, v.y - v.x); }
// slot of side j of element e: {Gz, Gx} at [j][32] float4, then Gy at [j][32] float2
__device__ __forceinline__ void store_sd(void* flx, int e, int j, f2 z, f2 x, f2 y) {
  reinterpret_cast<float4*>(flx)[j * 32 + e] = make_float4(z.x, z.y, x.x, x.y);
  reinterpret_cast<float2*>(reinterpret_cast<float4*>(flx) + 96)[j * 32 + e] = y;
}

// a point's (or a packed pair's) values for both sides from the doubled flux: w half the point's edge
// weight, pq = w g / 2 for the pressure, the mean of the sides' g/2 d (2H - d) relative to each side's mean
template <class V>
__device__ __forceinline__ void side_points(V Ld, V LH, V Rd, V RH, V dc, V nx, V ny, V w, V pq, V fz, V fx, V fy,
                                            V (&l)[3], V (&r)[3]) {
  const V two = vbc<V>(2.f);
  const V Fz = vmul(w, fz), Fx = vmul(w, fx), Fy = vmul(w, fy);
  const V A = vmul(Ld, vfma(two, LH, vneg(Ld))), B = vmul(Rd, vfma(two, RH, vneg(Rd)));
  const V R1 = vadd(Rd, dc), L1 = vadd(Ld, vneg(dc));
  const V pL = vmul(pq, vfma(R1, vfma(two, RH, vneg(R1)), A)), pR = vmul(pq, vfma(L1, vfma(two, LH, vneg(L1)), B));
  l[0] = Fz;
  l[1] = vfma(pL, nx, Fx);
  l[2] = vfma(pL, ny, Fy);
  r[0] = vneg(Fz);
  r[1] = vneg(vfma(pR, nx, Fx));
  r[2] = vneg(vfma(pR, ny, Fy));
}

template <int P, int FLUX, class Pol, int FT>
__device__ __forceinline__ void tile_edge(const StageArgs<Pol>& a, const ScenDev& S, uint32_t ownB, uint32_t halB,
                                          const uint4* geo, void* flx, unsigned ed,
                                          const typename Pol::T (*ephi)[P + 1][np_of(P)], const float4* ephi4, double t64,
                                          typename Pol::Acc& bdry_acc) {
  using T = typename Pol::T;
  using L = TileLayout<P, Pol, FT>;
  constexpr int NG = P + 1, RV = L::RV, NPR = L::NPR, NV = L::NV;
  constexpr bool MASSV = L::MASSV;
  const RefTab<T>& tab = ctab<T, P>();
  const T g = a.g, H0 = a.H0;
  const unsigned jL = ed & 3, srcL = (ed >> 2) & 63;
  const unsigned jR = (ed >> 8) & 3, srcR = (ed >> 10) & 63;
  Raw<RV> rl;
  fetch_side<RV>(ownB, halB, srcL, rl);
  T lnx, lny;
  edge_normal(geo, ed, lnx, lny);
  Elem<P, Pol> EL;
  unpack<P>(rl, EL);
  const T l2 = lnx * lnx + lny * lny, il = frsqrt(l2), len = l2 * il;  // edge length and its inverse
  const T nx = lnx * il, ny = lny * il;
  Trace<T> tl[NG], tr[NG];
  side_traces<P, Pol, false>(EL, jL, ephi, ephi4, tl);
  const bool interior = !(ed & ED_BND);
  const bool dryL = (EL.flags & FLAG_DRY) != 0;
  bool dryR = false, land = false, river = false;
  T dcRL = T(0), qr = T(0);
  if (interior) {
    Raw<RV> rr;
    fetch_side<RV>(ownB, halB, srcR, rr);
    Elem<P, Pol> ER;
    unpack<P>(rr, ER);
    dcRL = acc_sub_r(ER.zb, EL.zb);
    dryR = (ER.flags & FLAG_DRY) != 0;
    side_traces<P, Pol, true>(ER, jR, ephi, ephi4, tr);  // the same points
  } else {
    // boundary kind (an instantiation without a kind treats such an edge as a wall; the host never
    // selects it for a run that has one); a land edge takes the flux evaluation against its own trace
    const int code = (ed >> 8) & 255;
#pragma unroll
    for (int k = 0; k < NG; ++k) tr[k] = tl[k];
    if ((FT & FT_RIVER) && code > MAXSEG) {  // river: interior elevation, prescribed normal discharge
      qr = river_at<T>(S, min(code - 1 - MAXSEG, MAXRIV - 1), t64);
      river = true;
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        tr[k].qx = -qr * nx;
        tr[k].qy = -qr * ny;
      }
    } else if ((FT & FT_OCEAN) && code >= 1 && code <= MAXSEG) {  // ocean: tidal elevation, interior discharge
      const T zbc = tide_at<T>(S, code - 1, t64);
      const T dgh = acc_r(acc_addr(acc_neg(EL.zb), zbc));  // ghost zeta - mean of L
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        tr[k].H = tl[k].H + (dgh - tl[k].d);
        tr[k].d = dgh;
      }
    } else {
      land = true;
    }
  }
  const T hl = T(0.5) * len;
  if constexpr (slots_sd<P, Pol>()) {
    // both points in packed FP32x2; every edge takes the flux evaluation, so that no lane takes a
    // separate wall path.  Both Gauss weights are 1.
    const Trace2 L2{make_float2(tl[0].d, tl[1].d), make_float2(tl[0].H, tl[1].H), make_float2(tl[0].qx, tl[1].qx),
                    make_float2(tl[0].qy, tl[1].qy)};
    const Trace2 R2{make_float2(tr[0].d, tr[1].d), make_float2(tr[0].H, tr[1].H), make_float2(tr[0].qx, tr[1].qx),
                    make_float2(tr[0].qy, tr[1].qy)};
    f2 fz2, fx2, fy2;
    FluxAux2 ax;  // per-side quantities for the wall flux
    edge_flux_pair2<FLUX>(L2, R2, p2(dcRL), p2(nx), p2(ny), g, H0, fz2, fx2, fy2, ax);
    if (river) fz2 = p2(-2.f * qr);  // the specified normal flow is the mass flux
    const f2 hh2 = p2(0.5f * hl);    // half the edge weight: the fluxes are doubled
    const f2 Fz = mul2(sum_diff(fz2), hh2);  // Fz.x: the mass integral along n
    // wet/dry closure: no water leaves a dry element (interior: either side; ocean/river: L)
    const bool closed = land || (dryL && Fz.x > 0.f) || (dryR && Fz.x < 0.f);
    if (!closed) {
      const f2 Fx = mul2(sum_diff(fx2), hh2), Fy = mul2(sum_diff(fy2), hh2), dc = p2(dcRL), pq = p2(0.25f * g * hl);
      if (srcL < TILE) {  // pressure: the mean of the sides' g/2 d (2H - d) relative to L's mean
        const f2 Rd = add2(R2.d, dc);
        const f2 pp = fma2(L2.d, fma2(p2(2.f), L2.H, neg2(L2.d)), mul2(Rd, fma2(p2(2.f), R2.H, neg2(Rd))));
        const f2 Pd = mul2(sum_diff(pp), pq);
        store_sd(flx, srcL, jL, Fz, fma2(Pd, p2(nx), Fx), fma2(Pd, p2(ny), Fy));
        if (!interior) bdry_acc = acc_addr(bdry_acc, -Fz.x);  // inflow
      }
      if (interior && srcR < TILE) {  // relative to R's mean, along -n
        const f2 Ld = sub2(L2.d, dc);
        const f2 pp = fma2(R2.d, fma2(p2(2.f), R2.H, neg2(R2.d)), mul2(Ld, fma2(p2(2.f), L2.H, neg2(Ld))));
        const f2 Pd = mul2(sum_diff(pp), pq);
        store_sd(flx, srcR, jR, make_float2(-Fz.x, Fz.y), fma2(Pd, make_float2(-nx, nx), make_float2(-Fx.x, Fx.y)),
                 fma2(Pd, make_float2(-ny, ny), make_float2(-Fy.x, Fy.y)));
      }
    } else {
      // wall: q.n (q.n / Hs + c) + pressure relative to the side's mean (LLF: (q.n + |q.n|) / Hs)
      const f2 z = p2(0.f), sg = p2(fsqrt_pos(g)), hg = p2(0.5f * g), hl2 = p2(hl);
      if (srcL < TILE) {
        const f2 un = (FLUX == 1) ? mul2(add2(ax.mL, abs2(ax.mL)), ax.iL) : mul2(ax.mL, ax.iL);
        const f2 w = fma2(ax.mL, fma2(sg, ax.sL, un), mul2(hg, mul2(L2.d, fma2(p2(2.f), L2.H, neg2(L2.d)))));
        const f2 Wd = mul2(sum_diff(w), hl2);
        store_sd(flx, srcL, jL, z, mul2(Wd, p2(nx)), mul2(Wd, p2(ny)));
      }
      if (interior && srcR < TILE) {  // seen from R along -n: q.n_R = -mR
        const f2 mR = neg2(ax.mR);
        const f2 un = (FLUX == 1) ? mul2(add2(mR, abs2(mR)), ax.iR) : mul2(mR, ax.iR);
        const f2 w = fma2(mR, fma2(sg, ax.sR, un), mul2(hg, mul2(R2.d, fma2(p2(2.f), R2.H, neg2(R2.d)))));
        const f2 Wd = mul2(sum_diff(w), hl2);
        store_sd(flx, srcR, jR, z, mul2(Wd, make_float2(-nx, nx)), mul2(Wd, make_float2(-ny, ny)));
      }
    }
  } else {
    // both sides' values at the points, in L's point order
    T lv[NG][3], rv[NG][3];
    const T hh = T(0.5) * hl, hp = T(0.5) * g;
    if constexpr (P == 2 && sizeof(T) == 4 && DG_PACKED_FLUX) {  // points 0 and 1 packed, point 2 alone
      const Trace2 L2{make_float2(tl[0].d, tl[1].d), make_float2(tl[0].H, tl[1].H), make_float2(tl[0].qx, tl[1].qx),
                      make_float2(tl[0].qy, tl[1].qy)};
      const Trace2 R2{make_float2(tr[0].d, tr[1].d), make_float2(tr[0].H, tr[1].H), make_float2(tr[0].qx, tr[1].qx),
                      make_float2(tr[0].qy, tr[1].qy)};
      f2 fz2, fx2, fy2, l2v[3], r2v[3];
      FluxAux2 ax2;
      edge_flux_pair2<FLUX>(L2, R2, p2(dcRL), p2(nx), p2(ny), g, H0, fz2, fx2, fy2, ax2);
      if (river) fz2 = p2(-2.f * qr);
      const f2 w = mul2(make_float2(tab.gw[0], tab.gw[1]), p2(hh));
      side_points<f2>(L2.d, L2.H, R2.d, R2.H, p2(dcRL), p2(nx), p2(ny), w, mul2(w, p2(hp)), fz2, fx2, fy2, l2v, r2v);
      T fz, fx, fy;
      edge_flux2<FLUX, T>(tl[2], tr[2], dcRL, nx, ny, g, H0, fz, fx, fy);
      if (river) fz = -2.f * qr;
      const T w2 = tab.gw[2] * hh;
      side_points<T>(tl[2].d, tl[2].H, tr[2].d, tr[2].H, dcRL, nx, ny, w2, w2 * hp, fz, fx, fy, lv[2], rv[2]);
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        lv[0][v] = l2v[v].x;
        lv[1][v] = l2v[v].y;
        rv[0][v] = r2v[v].x;
        rv[1][v] = r2v[v].y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        T fz, fx, fy;
        edge_flux2<FLUX, T>(tl[k], tr[k], dcRL, nx, ny, g, H0, fz, fx, fy);
        if (river) fz = T(-2) * qr;  // the specified normal flow is the mass flux
        const T w = P == 1 ? hh : tab.gw[k] * hh;  // both Gauss weights are 1 at p = 1
        side_points<T>(tl[k].d, tl[k].H, tr[k].d, tr[k].H, dcRL, nx, ny, w, w * hp, fz, fx, fy, lv[k], rv[k]);
      }
    }
    T ec = lv[0][0];  // mass flux integral along n (L's outward normal)
#pragma unroll
    for (int k = 1; k < NG; ++k) ec += lv[k][0];
    // wet/dry closure: no water leaves a dry element (interior: either side; ocean/river: L)
    const bool closed = land || (dryL && ec > T(0)) || (dryR && ec < T(0));
    if (closed) {  // walls, each side from its own trace
      ec = T(0);
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const T w = tab.gw[k] * hl;
        const T cl = w * wall_coef<FLUX, T>(tl[k], nx, ny, g, H0), cr = w * wall_coef<FLUX, T>(tr[k], -nx, -ny, g, H0);
        lv[k][0] = rv[k][0] = T(0);
        lv[k][1] = cl * nx;
        lv[k][2] = cl * ny;
        rv[k][1] = -(cr * nx);
        rv[k][2] = -(cr * ny);
      }
    }
    T vals[NV + 1];
    if (srcL < TILE) {  // L's slot, in L's point order
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        vals[k] = lv[k][0];
        vals[NG + k] = lv[k][1];
        vals[2 * NG + k] = lv[k][2];
      }
      if (MASSV) vals[3 * NG] = ec;
      store_side<T, NPR, NV>(flx, srcL, jL, vals);
      if (!interior && !closed) bdry_acc = acc_addr(bdry_acc, -ec);  // inflow
    }
    if (interior && srcR < TILE) {  // R's slot, in R's point order (its point k is L's NG-1-k)
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        vals[k] = rv[NG - 1 - k][0];
        vals[NG + k] = rv[NG - 1 - k][1];
        vals[2 * NG + k] = rv[NG - 1 - k][2];
      }
      if (MASSV) vals[3 * NG] = -ec;
      store_side<T, NPR, NV>(flx, srcR, jR, vals);
    }
  }
}

// ------------------------------------------------------------------------ tile plan ------
// one warp per tile, once per mesh: ownership of the tile's edges (boundary edges, edges to
// out-of-tile neighbours and in-tile edges to a higher index belong to a lane's element; the lower
// element index is the left side) and the order described at EDGE_INLINE
template <class Pol>
__global__ void __launch_bounds__(256) plan_kernel(const int4* nbr, const uint4* geo, const int4* nodes, const double* xy,
                                                   const int4* tile_meta, int ntiles, int rv, uint4* stat,
                                                   int32_t* plan_x) {
  using T = typename Pol::T;
  using L = TileLayout<1, Pol>;  // the static block does not depend on the degree
  const int tile = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (tile >= ntiles) return;
  const int4 meta = tile_meta[tile];
  const bool valid = lane < meta.y;
  const int e0 = tile * TILE, e = e0 + lane;
  const int4 nb = valid ? nbr[e] : make_int4(-1, -1, -1, 0);
  const int code[3] = {nb.x, nb.y, nb.z};
  uint4* B = stat + (size_t)tile * L::SVM;
  for (int i = lane; i < TILE * L::GV; i += 32) B[i] = geo[(size_t)tile * TILE * L::GV + i];
  {
    const long long v = valid ? nodes[e].x : 0;
    T* x0 = reinterpret_cast<T*>(B + L::S_XY) + 2 * lane;
    x0[0] = valid ? (T)xy[2 * v] : T(0);
    x0[1] = valid ? (T)xy[2 * v + 1] : T(0);
  }
  uint4* P = B + L::S_PLAN;
  unsigned* desc = reinterpret_cast<unsigned*>(P);
  int32_t* halo = reinterpret_cast<int32_t*>(P + EDGE_INLINE / 4);
  int32_t* over = plan_x + (size_t)tile * PLAN_X;
  for (int i = lane; i < EDGE_INLINE + HALO; i += 32) desc[i] = 0u;
  for (int i = lane; i < PLAN_X; i += 32) over[i] = 0;
  __syncwarp();
  const unsigned lt = (1u << lane) - 1u;
  // halo slot of each edge to another tile
  int hs[3], nhalo = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int c = code[j], n = c >> 2;
    const bool out = valid && c >= 0 && (n < e0 || n >= e0 + TILE);
    const unsigned m = __ballot_sync(0xffffffffu, out);
    hs[j] = out ? nhalo + __popc(m & lt) : -1;
    if (out) {
      const int32_t at = (int32_t)(((unsigned)n >> 5) * rv * 32 + (n & 31));
      if (hs[j] < HALO) halo[hs[j]] = at;
      else over[hs[j]] = at;  // neighbour 32 and on, after the 32 edge words
    }
    nhalo += __popc(m);
  }
  int base = 0, count[5];
#pragma unroll
  for (int kind = 0; kind < 5; ++kind) {  // in-tile; to the first 32 neighbours; boundary; batches 1 and 2
    const int before = base;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const int c = code[j], n = c >> 2, jn = c & 3;
      const unsigned me = (unsigned)((lane << 2) | j);
      const bool inside = valid && c >= 0 && hs[j] < 0;
      const bool mine = kind == 0 ? (inside && e < n) : kind == 2 ? (valid && c < 0) : (hs[j] >= 0 && hs[j] / HALO == (kind == 1 ? 0 : kind - 2));
      const unsigned m = __ballot_sync(0xffffffffu, mine);
      if (mine) {
        unsigned d;
        if (kind == 0) {
          d = me | (unsigned)(((n - e0) << 2) | jn) << 8;
        } else if (kind == 2) {
          d = me | (unsigned)(-1 - c) << 8 | ED_BND;
        } else {
          const unsigned other = (unsigned)(((32 + hs[j] % HALO) << 2) | jn);
          d = e < n ? (me | other << 8) : (other | me << 8 | ED_OWN_R);
        }
        d |= (unsigned)(lane * (sizeof(T) == 4 ? 6 : 5) + j) << 18;  // float2 / double2 of the own element's normal j
        const int i = base + __popc(m & lt);
        if (i < EDGE_INLINE) desc[i] = d;
        else over[i - EDGE_INLINE] = (int32_t)d;
      }
      base += __popc(m);
    }
    count[kind] = base - before;
  }
  if (sizeof(T) == 4) reinterpret_cast<int32_t*>(P + (EDGE_INLINE + HALO) / 4)[lane] = valid ? nb.w : 0;
  if (lane == 0)
    reinterpret_cast<int4*>(P)[plan_vec<T>() - 1] =
        make_int4(meta.x, meta.y, (count[0] + count[1] + count[2]) | count[0] << 8 | min(nhalo, HALO) << 16,
                  count[3] | count[4] << 8);
}

// --------------------------------------------------------------------- one tile, one stage ---
// storm rain at a stage: centre, radius, 1 / (2 rm), log2(e) / re, a third of the peak rate.  The
// instantiations whose only rain is the storm keep it in registers from tile to tile (250k triangles:
// 40.7 -> 39.4 us per step; read per tile it was a chain of dependent loads); at p = 2, where registers
// are short (141 -> 150 us), and in the generic ones it is formed per tile.
template <class T>
struct Storm {
  T cx, cy, rm, rlin, rexp, r0;
};
template <class T>
__device__ __forceinline__ Storm<T> storm_at(const ScenDev& S, double t64) {
  const ForcingT<T>& F = forcing<T>(S);
  const T tt = (T)t64 - F.storm[7];
  return {F.storm[0] + F.storm[2] * tt, F.storm[1] + F.storm[3] * tt, F.storm[5], T(0.5) * F.storm[8], F.storm[9],
          F.storm[4] * T(1.0 / 3.0)};
}
template <int P, int FT>
DG_HD constexpr bool storm_regs() {
  return P == 1 && ft_rain(FT) == 2;
}

// Phases 1-3 of one tile: the area integrals and rain of each lane's element, every edge of the tile
// once, then the lift, stage combination and positive-depth operator; O is the element's new record.
// halo_ready() makes the staged halo records readable; it is called once by the whole warp, before
// the first round that has an edge to another tile; halo_more(mine, at) replaces them by the
// records at the places that the lanes name; release() is called once by the whole warp when the tile's static data is
// done with.  The step-initial record comes from shared memory (WNS) or from a.wn.
template <int P, int FLUX, class Pol, int FT, bool WNS, class HaloReady, class HaloMore, class Release>
__device__ __forceinline__ void tile_body(const StageArgs<Pol>& a, const ScenDev& S, double t64, int rain_kind, int press,
                                          const RainRec<typename Pol::T>& rr,
                                          const Storm<typename Pol::T>& storm, int tile, int lane, bool valid, int counts, int more,
                                          const uint4* own, const uint4* halo, const uint4* geoS, const unsigned* planS,
                                          const float* man, const typename Pol::T* xyS, void* flx, const uint4* wnS,
                                          const typename Pol::T (*s_ephi)[P + 1][np_of(P)], const float4* s_ephi4,
                                          HaloReady halo_ready, HaloMore halo_more, Release release, Elem<P, Pol>& O, typename Pol::Acc& rain_acc,
                                          typename Pol::Acc& bdry_acc) {
  using T = typename Pol::T;
  using Acc = typename Pol::Acc;
  using L = TileLayout<P, Pol, FT>;
  constexpr int NP = np_of(P), NS = NP - 1, NG = P + 1, RV = L::RV, GV = L::GV, NPR = L::NPR, NV = L::NV;
  const RefTab<T>& tab = ctab<T, P>();
  const int e = tile * TILE + lane;
  const int nedge = counts & 255, ninner = (counts >> 8) & 255;
  const int32_t* over = a.plan_x + (size_t)tile * PLAN_X;

  // ---- element phase A: area integrals and rain, while the halo copies are in flight
  T Rz[NP], Rx[NP], Ry[NP];
  T Re = 0;
  if (valid) {
    Geo<Pol> G;
    geo_from(geoS + lane * GV, man + lane, G);
    // gridded rain: the element's two records now, blended after the area integrals; without
    // records the node indices now, their nodal rates then
    T re0 = T(0), re1 = T(0);
    int4 nd = make_int4(0, 0, 0, 0);
    if (rain_kind == 3) {
      if (rr.r0) {
        re0 = __ldg(rr.r0 + e);
        re1 = __ldg(rr.r1 + e);
      } else {
        nd = __ldg(a.nodes + e);
      }
    }
    Elem<P, Pol> E;
    {
      Raw<RV> r;
#pragma unroll
      for (int v = 0; v < RV; ++v) r.v[v] = own[v * TILE + lane];
      unpack<P>(r, E);
    }
    // vertex coordinates: the first vertex, then along the edge vectors t_j = (-ln_j.y, ln_j.x)
    T vx[3] = {0, 0, 0}, vy[3] = {0, 0, 0};
    if (press || rain_kind == 2) {
      const T* x0 = xyS + 2 * lane;
      vx[0] = x0[0];
      vy[0] = x0[1];
      vx[1] = vx[0] - G.lny[0];
      vy[1] = vy[0] + G.lnx[0];
      vx[2] = vx[0] + G.lny[2];
      vy[2] = vy[0] - G.lnx[2];
    }
    tile_area<P, Pol, FT>(E, G, S, a, press, vx, vy, Rz, Rx, Ry);
    // forcing: element rain = mean of the three nodal rates (Eq. rain)
    if (rain_kind == 1) {
      Re = a.rain_e[e];
    } else if (rain_kind == 2) {  // radial storm profile at the three vertices
      const Storm<T> st = storm_regs<P, FT>() ? storm : storm_at<T>(S, t64);
      T acc = 0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const T dx = vx[i] - st.cx, dy = vy[i] - st.cy;
        const T r = fsqrt0(dx * dx + dy * dy);
        acc += (r < st.rm) ? fma(st.rlin, r, T(0.5)) : fexp2((st.rm - r) * st.rexp);
      }
      Re = acc * st.r0;
    } else if (rain_kind == 3 && rr.r0) {
      Re = rain_blend<T>(re0, re1, rr.f);
    } else if (rain_kind == 3) {  // nodal rates interpolated by the node kernel of this stage
      Re = (a.rain_node[nd.x] + a.rain_node[nd.y] + a.rain_node[nd.z]) * T(1.0 / 3.0);
    }
  }

  // ---- edge phase: each edge touching the tile once, one per lane and round; the halo records are
  // waited for before the first round that has an edge to another tile
  const uint32_t ownB = smem_u32(own), halB = smem_u32(halo) - 16u * TILE;
  const int nr0 = (nedge + 31) >> 5, nr = nr0 + (more ? (more >> 8 ? 2 : 1) : 0);
  bool staged = false;
  int base = 0, lim = nedge;
  for (int r = 0; r < nr; ++r, base += 32) {
    if (!staged && r * 32 + 32 > ninner) {
      halo_ready();
      staged = true;
    }
    if (r >= nr0) {  // further neighbours (rare): their records in place of the ones before, and their edges
      const int b = r - nr0, n = (more >> (8 * b)) & 255;
      __syncwarp();
      halo_more(lane < n, (uint32_t)__ldg(over + 32 + HALO * b + lane));
      base = lim;
      lim += n;
    }
    const int i = base + lane;
    if (i < lim) {
      const unsigned ed = i < EDGE_INLINE ? planS[i] : (unsigned)__ldg(over + (i - EDGE_INLINE));
      tile_edge<P, FLUX, Pol, FT>(a, S, ownB, halB, geoS, flx, ed, s_ephi, s_ephi4, t64, bdry_acc);
    }
  }
  if (!staged) halo_ready();
  __syncwarp();

  // ---- element phase B: lift, inverse mass, stage combination, positive-depth operator
  Geo<Pol> G;
  if (valid) geo_from(geoS + lane * GV, man + lane, G);
  release();
  if (valid) {
    Elem<P, Pol> E;
    {
      Raw<RV> r;
#pragma unroll
      for (int v = 0; v < RV; ++v) r.v[v] = own[v * TILE + lane];
      unpack<P>(r, E);
    }
    T ms[3];  // edge mass outflows (volume per second)
    if constexpr (slots_sd<P, Pol>()) {
      // basis over an edge's two points: mean * S + difference / 2 * D, for phi_1 and phi_2 on edges 0, 1, 2
      constexpr float MID[3][2] = {{0.f, -1.f}, {0.8660254f, 0.5f}, {-0.8660254f, 0.5f}};
      constexpr float DIF[3][2] = {{1.f, 0.f}, {-0.5f, 0.8660254f}, {-0.5f, -0.8660254f}};
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const float4 zx = reinterpret_cast<const float4*>(flx)[j * 32 + lane];
        const float2 y = reinterpret_cast<const float2*>(reinterpret_cast<const float4*>(flx) + 96)[j * 32 + lane];
        Rx[0] = fma(-tab.phi0, zx.z, Rx[0]);
        Ry[0] = fma(-tab.phi0, y.x, Ry[0]);
#pragma unroll
        for (int m = 1; m < 3; ++m) {
          if (MID[j][m - 1] != 0.f) {
            Rz[m] = fma(-MID[j][m - 1], zx.x, Rz[m]);
            Rx[m] = fma(-MID[j][m - 1], zx.z, Rx[m]);
            Ry[m] = fma(-MID[j][m - 1], y.x, Ry[m]);
          }
          if (DIF[j][m - 1] != 0.f) {
            Rz[m] = fma(-DIF[j][m - 1], zx.y, Rz[m]);
            Rx[m] = fma(-DIF[j][m - 1], zx.w, Rx[m]);
            Ry[m] = fma(-DIF[j][m - 1], y.y, Ry[m]);
          }
        }
        ms[j] = zx.x;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        T vals[NV + 1];
        load_side<T, NPR, NV>(flx, lane, j, vals);
#pragma unroll
        for (int k = 0; k < NG; ++k) {
#pragma unroll
          for (int m = 0; m < NP; ++m) {
            const T ph_ = tab.ephi[j][k][m];
            if (m > 0) Rz[m] = fma(-ph_, vals[k], Rz[m]);
            Rx[m] = fma(-ph_, vals[NG + k], Rx[m]);
            Ry[m] = fma(-ph_, vals[2 * NG + k], Ry[m]);
          }
        }
        ms[j] = side_mass<T, NG, L::MASSV>(vals);
      }
    }
    if (E.flags & FLAG_DRY) {  // the momentum equations are not advanced on dry elements
#pragma unroll
      for (int m = 0; m < NP; ++m) Rx[m] = Ry[m] = 0;
    }
    // Shu-Osher combination: out = a_n w^n + a_in w^in + beta dt M^{-1} R
    const T idetJ = T(2) * acc_r(G.invA);
    const Acc an = acc_make<Acc>(a.a_n_hi, a.a_n_lo, a.a_n);
    const Acc ain = acc_make<Acc>(a.a_in_hi, a.a_in_lo, a.a_in);
    const Acc bdt = acc_make<Acc>(S.bdt_hi[a.stage], S.bdt_lo[a.stage], S.bdt[a.stage]);
    // increments of the means: beta dt (R_e - outflow / A) and beta dt phi_0 R_0 / detJ
    const Acc massout = acc_sum3(ms[0], ms[1], ms[2], acc_make<Acc>(0.f, 0.f, 0.0));
    const Acc dz = acc_increment(bdt, Re, massout, G.invA);
    const T fR = acc_r(bdt) * idetJ;
    const T dx = (tab.phi0 * fR) * Rx[0], dy = (tab.phi0 * fR) * Ry[0];
    O = E;
    Elem<P, Pol> Wn = E;
    if (a.has_n) {
      Raw<RV> rn;
#pragma unroll
      for (int v = 0; v < RV; ++v) rn.v[v] = WNS ? wnS[v * TILE + lane] : __ldg(a.wn + rec_at<RV>(e, v));
      unpack<P>(rn, Wn);
    }
    const T an_r = (sizeof(T) == 4) ? (T)a.a_n_hi : (T)a.a_n, ain_r = (sizeof(T) == 4) ? (T)a.a_in_hi : (T)a.a_in;
    {
      Acc z, x, y;
      constexpr int PW = ft_pow2(FT);
      if (sizeof(T) == 4 && (PW == 1 || (PW == -1 && a.pow2))) {  // exact scaling of both words by a power of two
        z = acc_scale2(E.zb, ain_r);
        x = acc_scale2(E.xb, ain_r);
        y = acc_scale2(E.yb, ain_r);
        if (a.has_n) {
          z = acc_addf(z, acc_scale2(Wn.zb, an_r));
          x = acc_addf(x, acc_scale2(Wn.xb, an_r));
          y = acc_addf(y, acc_scale2(Wn.yb, an_r));
        }
      } else {
        z = acc_mul(ain, E.zb);
        x = acc_mul(ain, E.xb);
        y = acc_mul(ain, E.yb);
        if (a.has_n) {
          z = acc_add(z, acc_mul(an, Wn.zb));
          x = acc_add(x, acc_mul(an, Wn.xb));
          y = acc_add(y, acc_mul(an, Wn.yb));
        }
      }
      O.zb = acc_addf(z, dz);
      O.xb = acc_addr(x, dx);
      O.yb = acc_addr(y, dy);
    }
    // other modes: in FP32 two modes per packed operation
    if constexpr (sizeof(T) == 4 && DG_PACKED_FLUX) {
      const f2 f2R = p2(fR), ai2 = p2(ain_r), an2 = p2(an_r);
      auto comb = [&](const T* w, const T* wn, const T* R, T* o) {
#pragma unroll
        for (int m = 0; m + 1 < NS; m += 2) {
          f2 v = fma2(f2R, make_float2(R[m + 1], R[m + 2]), mul2(ai2, make_float2(w[m], w[m + 1])));
          if (a.has_n) v = fma2(an2, make_float2(wn[m], wn[m + 1]), v);
          o[m] = v.x;
          o[m + 1] = v.y;
        }
        if (NS % 2) {
          T v = fma(fR, R[NS], ain_r * w[NS - 1]);
          if (a.has_n) v = fma(an_r, wn[NS - 1], v);
          o[NS - 1] = v;
        }
      };
      comb(E.zs, Wn.zs, Rz, O.zs);
      comb(E.xs, Wn.xs, Rx, O.xs);
      comb(E.ys, Wn.ys, Ry, O.ys);
    } else {
#pragma unroll
      for (int m = 0; m < NS; ++m) {
        T z = fma(fR, Rz[m + 1], ain_r * E.zs[m]);
        T x = fma(fR, Rx[m + 1], ain_r * E.xs[m]);
        T y = fma(fR, Ry[m + 1], ain_r * E.ys[m]);
        if (a.has_n) {
          z = fma(an_r, Wn.zs[m], z);
          x = fma(an_r, Wn.xs[m], x);
          y = fma(an_r, Wn.ys[m], y);
        }
        O.zs[m] = z;
        O.xs[m] = x;
        O.ys[m] = y;
      }
    }
    apply_positivity<P, Pol>(O, G, e, a, &a.ctl->err);
    rain_acc = acc_addmul(rain_acc, G.A, Re);
  }
}

// -------------------------------------------------------------------------- the kernel ---
#ifndef DG_TILE_MAXNREG
// register budget (registers are allocated per SM sub-partition, so a kernel gets 4 floor(512 / regs)
// warps): mixed p = 1 at 128 for 16 warps per SM, mixed p = 2 at 168 for 12; FP64 at 224 for 8.
// Mixed p = 1 at 96 registers (20 warps, one static buffer) was slower: hurricane 2M 279 us per step
// against 260, 500k LLF 224 against 188; the kernel wants instruction-level parallelism, not warps.
#define DG_TILE_BOUNDS __maxnreg__(sizeof(typename Pol::T) == 4 ? (P == 1 ? 128 : 168) : 224)
#else
#define DG_TILE_BOUNDS __maxnreg__(DG_TILE_MAXNREG)
#endif

// the 16-byte rows of edge basis values that side_traces reads
template <int P, class T>
__device__ __forceinline__ void edge_rows(const RefTab<T>& tab, float4* rows) {
  const int t = threadIdx.x;
  if (P == 1 && t < 3)
    rows[t] = make_float4((float)tab.ephi[t][0][1], (float)tab.ephi[t][0][2], (float)tab.ephi[t][1][1], (float)tab.ephi[t][1][2]);
  if (P == 2 && t < 15)
    rows[t] = make_float4((float)tab.ephi[t / 5][0][t % 5 + 1], (float)tab.ephi[t / 5][1][t % 5 + 1],
                          (float)tab.ephi[t / 5][2][t % 5 + 1], 0.f);
}

template <int P, int FLUX, class Pol, int FT = FT_ALL>
__global__ void DG_TILE_BOUNDS tile_kernel(const StageArgs<Pol> a) {
  using T = typename Pol::T;
  using Acc = typename Pol::Acc;
  using L = TileLayout<P, Pol, FT>;
  constexpr int NP = np_of(P), NG = P + 1, RV = L::RV;
  const RefTab<T>& tab = ctab<T, P>();

  // edge basis values, read at edge-dependent indices; in FP32 as rows of 16 bytes alone (side_traces)
  __shared__ T s_ephi[3][NG][NP];
  __shared__ float4 s_ephi4[P == 1 ? 3 : 15];
  extern __shared__ uint4 tsm[];
  const int tid = threadIdx.x;
  for (int i = tid; sizeof(T) == 8 && i < 3 * NG * NP; i += blockDim.x) {
    const int j = i / (NG * NP), k = (i / NP) % NG, m = i % NP;
    s_ephi[j][k][m] = tab.ephi[j][k][m];
  }
  edge_rows<P>(tab, s_ephi4);
  __syncthreads();
  const int lane = tid & 31;
  uint4* Wm = tsm + (size_t)(tid >> 5) * L::VEC;
  uint4* halo = Wm + L::HAL;                                       // [HALO][RV]
  void* flx = Wm + L::FLX;                                         // [3][NPR][32] pairs
  const uint32_t bar = smem_u32(Wm + L::BAR);  // record buffers 0 and 1 at +0 and +8, static at +16
  if (lane == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 8, 1);
    mbar_init(bar + 16, 1);
    mbar_fence_init();
  }
  __syncwarp();
  const int gw = blockIdx.x * (blockDim.x >> 5) + (tid >> 5);
  const int W = gridDim.x * (blockDim.x >> 5);
  // TMA copies by lane 0: a tile's records into a buffer; its geometry, plan and first vertices, with
  // the records' barrier when they are double-buffered too
  constexpr bool SD = L::NSTAT == 2;
  auto copy_static = [&](int t, uint4* to, uint32_t br) {
    bulk_g2s(smem_u32(to), a.stat + (size_t)t * L::SVM, 16u * L::SV, br);
  };
  auto issue = [&](int t, int b, bool stat, bool rec) {
    if (lane == 0) {
      fence_proxy_async();
      if (stat && SD) {
        mbar_expect_tx(bar + 8 * b, 16u * (L::REC + L::SV));
        copy_static(t, Wm + L::STAT + b * L::SV, bar + 8 * b);
      }
      if (rec) {
        if (!SD) mbar_expect_tx(bar + 8 * b, 16u * L::REC);
        bulk_g2s(smem_u32(Wm + b * L::REC), a.in + (size_t)t * L::REC, 16u * L::REC, bar + 8 * b);
      }
    }
  };
  auto issue_static = [&](int t) {  // the single static buffer
    if (!SD && lane == 0) {
      fence_proxy_async();
      mbar_expect_tx(bar + 16, 16u * L::SV);
      copy_static(t, Wm + L::STAT, bar + 16);
    }
  };
  // Programmatic dependent launch: the CTAs start as soon as those of the kernel before have left,
  // without waiting for its memory flush and completion; what comes before pdl_wait reads only data
  // that no kernel writes while steps run.  250k triangles: 41.9 -> 40.8 us per step, 37k: 16.2 ->
  // 15.0.  No early trigger: CTAs that start beside a running stage spread unevenly over the SMs
  // (FP64 61k: 410 -> 465 us per step with a trigger at the start; 37k: 15.0 -> 17.2).
  if (gw < a.ntiles) {
    issue_static(gw);
    issue(gw, 0, true, false);
  }
  pdl_wait();
  if (gw < a.ntiles) issue(gw, 0, false, true);
  const double stepd = (double)a.ctl->step + a.cst;
  Acc rain_acc = acc_make<Acc>(0.f, 0.f, 0.0), bdry_acc = acc_make<Acc>(0.f, 0.f, 0.0);
  int cur = -1;
  // constants of the current scenario, reloaded when a tile of another scenario comes
  const ScenDev* Sp = a.scen;
  double t64 = 0.0;
  int rain_kind = 0, press = 0;
  RainRec<T> rr = {nullptr, nullptr, T(0)};  // gridded rain: the two records around the stage time
  Storm<T> storm = {};

  int it = 0;
  for (int tile = gw; tile < a.ntiles; tile += W, ++it) {
    const int b = it & 1, next = tile + W;
    if (next < a.ntiles) issue(next, b ^ 1, true, true);  // the other buffer's tile was consumed last iteration
    const bool arrived = (SD || mbar_wait(bar + 16, it & 1)) && mbar_wait(bar + 8 * b, (it >> 1) & 1);
    if (!__all_sync(0xffffffffu, arrived)) {
      tile_timeout(a, bar, it, next < a.ntiles, SD, lane);
      return;
    }
    const uint4* own = Wm + b * L::REC;                           // [RV][32] records
    const uint4* stat = Wm + L::STAT + (SD ? b * L::SV : 0);
    const uint4* geoS = stat + L::S_GEO;                          // [32][GV]
    const unsigned* planS = reinterpret_cast<const unsigned*>(stat + L::S_PLAN);
    const int4 meta = reinterpret_cast<const int4*>(stat + L::S_META)[0];
    const int sc = meta.x, present = meta.y;
    if (present == 0) {  // padding tile: no element (uniform over the warp)
      __syncwarp();
      if (next < a.ntiles) issue_static(next);
      continue;
    }
    if (sc != cur) {
      if (cur >= 0 && !a.tune) flush_ledger<P, Pol>(a, cur, gw, rain_acc, bdry_acc);
      cur = sc;
      Sp = a.scen + sc;
      t64 = Sp->d.t0 + stepd * Sp->d.dt;  // stage time, formed in FP64
      rain_kind = ft_rain(FT) >= 0 ? ft_rain(FT) : Sp->rain_kind;
      press = (FT & FT_PRESS) ? Sp->press : 0;
      if constexpr (storm_regs<P, FT>()) storm = storm_at<T>(*Sp, t64);
      if (rain_kind == 3) {
        rr.r0 = nullptr;
        if (Sp->rrec) {
          rr = rain_records<T>(*Sp, t64);
          rr.r0 -= Sp->elem_begin;
          rr.r1 -= Sp->elem_begin;
        }
      }
    }
    const ScenDev& S = *Sp;
    const int e0 = tile * TILE, e = e0 + lane;
    const bool valid = lane < present;
    // step-initial modes, read in phase B (not the vectors that hold only depth, flag and bathymetry)
    if (a.has_n && lane == 0) bulk_prefetch_l2(a.wn + (size_t)e0 * RV, 16u * TILE * L::RVN);

    // ---- the out-of-tile neighbours' records, one halo slot per lane, by the tile's plan
    if (lane < (meta.z >> 16)) {
      const uint4* from = a.in + reinterpret_cast<const uint32_t*>(stat + L::S_HALO)[lane];
#pragma unroll
      for (int v = 0; v < RV; ++v) cp_async16(halo + v * HALO + lane, from + v * TILE);
    }
    cp_async_commit();

    Elem<P, Pol> O;
    tile_body<P, FLUX, Pol, FT, false>(a, S, t64, rain_kind, press, rr, storm, tile, lane, valid, meta.z, meta.w, own, halo, geoS, planS,
                                       reinterpret_cast<const float*>(stat + L::S_MAN),
                                       reinterpret_cast<const T*>(stat + L::S_XY), flx, nullptr, s_ephi, s_ephi4,
                                       [] {
                                         cp_async_wait_all();
                                         __syncwarp();
                                       },
                                       [&](bool mine, uint32_t at) {
                                         if (mine) {
#pragma unroll
                                           for (int v = 0; v < RV; ++v)
                                             cp_async16(halo + v * HALO + lane, a.in + at + v * TILE);
                                         }
                                         cp_async_commit();
                                         cp_async_wait_all();
                                         __syncwarp();
                                       },
                                       [&] {
                                         if (SD) return;
                                         __syncwarp();
                                         if (next < a.ntiles) issue_static(next);
                                       },
                                       O, rain_acc, bdry_acc);
    if (valid) {
      Raw<RV> ro;
      pack<P>(O, ro);
      store_raw<RV>(a.out, e, ro);
    }
    __syncwarp();  // this tile's shared data is consumed: its buffers may be refilled
  }
  if (cur >= 0 && !a.tune) flush_ledger<P, Pol>(a, cur, gw, rain_acc, bdry_acc);

  // launch epilogue: the last CTA to finish advances the step counter after the final stage
  if (a.last && !a.tune) {
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      const unsigned tk = atomicAdd(&a.ctl->ticket, 1u);
      if (tk == gridDim.x - 1) {
        a.ctl->ticket = 0;
        a.ctl->step += 1ull;
        __threadfence();
      }
    }
  }
}

}  // namespace dg
