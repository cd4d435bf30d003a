// step.cu -- the VP-LBM time step for sm_103a.
//
// One time step is two launches that write disjoint nodes:
//   * the special kernel: the SIM points (stress of Sec. 2.3.2 at the
//     sampled fluid node from its pre-collision populations, S_i sigma n_i
//     and its moment, Eq. defFf), the nodes on the lattice edges (side
//     conditions of Sec. 3.1/3.2), and the tiles of the force region around
//     the body (penalized nodes and the MEM link terms of Eq. MMEL /
//     Eq. fluidtorque).  Its SIM and region blocks add their force terms into
//     exact fixed-point sums, which one extra block of the next step's launch
//     records.  For a moving body every block of that launch applies the FP64
//     rigid-body update (Eqs. dep1, theta2) for itself, and the region tiles
//     rasterise the mask of the body's current position (each tile with a
//     one-node halo).
//   * the bulk kernel: every other node -- pull streaming (Eq. eqBd) and the
//     BGK/TRT collision (Eq. TRT) of fluid nodes whose sources all lie inside
//     the lattice; no mask, no side conditions, no forces.  It comes in
//     several launch forms with identical results (bulk32x2_kernel for FP32,
//     bulk_kernel for FP64, bulk16_kernel and bulk16x4_kernel for 16-bit storage).
// Where the body stands still and the compute type is FP32, two time steps can
// be one launch over the same nodes (pair.cuh).
// For the first step after a pre-collision state the special kernel updates
// every tile.
#include "vplbm_internal.cuh"

namespace vplbm {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------
// exact force sums
// ---------------------------------------------------------------------------
template <typename T>
struct FixAcc {
  long long f[3][Fix<T>::kWords];
  __device__ __forceinline__ FixAcc() {
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int k = 0; k < Fix<T>::kWords; ++k) f[q][k] = 0;
  }
  __device__ __forceinline__ void add(int q, T v) {
    long long w[Fix<T>::kWords];
    Fix<T>::split(v, w);
#pragma unroll
    for (int k = 0; k < Fix<T>::kWords; ++k) f[q][k] += w[k];
  }
};

// the sum of a 64-bit integer over the warp, by three 32-bit warp reductions
// of its 24-, 24- and 16-bit pieces (a butterfly takes ten shuffles)
__device__ __forceinline__ long long warp_sum(long long v) {
  const unsigned lo = __reduce_add_sync(kFull, (unsigned)v & 0xffffffu);
  const unsigned mid = __reduce_add_sync(kFull, (unsigned)(v >> 24) & 0xffffffu);
  const int hi = __reduce_add_sync(kFull, (int)(v >> 48));
  return (long long)((unsigned long long)lo + ((unsigned long long)mid << 24) +
                     ((unsigned long long)(long long)hi << 48));
}

// adds the warp's fixed-point words into acc[slot][word] for the three
// quantities starting at slot base (a low word as two: Fix<double>)
template <typename T>
__device__ __forceinline__ void warp_add(const FixAcc<T> &a, unsigned long long *acc, int base) {
  constexpr int W = Fix<T>::kWords;
  long long any = 0;
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int k = 0; k < W; ++k) any |= a.f[q][k];
  if (!__any_sync(kFull, any != 0)) return;
  // a lane per accumulator word: one instruction adds them all (from lane 0, word
  // after word, a 512 x 256 FP32 airfoil took 4.28 us per step, 4.09 so; the FP64
  // disk channel 15.8 and 15.2)
  const int lane = threadIdx.x & 31;
  long long mine = 0;
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int k = 0; k < W; ++k) {
      const long long v = warp_sum(a.f[q][k]);
      if (k == 0) {
        if (lane == kSlotWords * q) mine = v;
      } else {
        if (lane == kSlotWords * q + 1) mine = v >> 26;
        if (lane == kSlotWords * q + 2) mine = v & Fix<double>::kLowMask;
      }
    }
  if (lane < 3 * kSlotWords && mine)
    atomicAdd(acc + kSlotWords * base + lane, (unsigned long long)mine);
}

// The force terms are written with named roundings, so that a state gives the
// same bits in a single step and in either step of a pair, whatever the
// compiler would fuse around them.
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float rrcp(float a) { return __frcp_rn(a); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double rrcp(double a) { return __drcp_rn(a); }

// the nine populations of a node, passed by value
template <typename T>
struct Offsets {
  T h[9];
};

// ---------------------------------------------------------------------------
// SIM (Sec. 2.3.2)
// ---------------------------------------------------------------------------

// The part of the stress beyond -(1/3) I at a fluid node,
// sigma + (1/3) I = -(rho - 1)/3 I - (1 - 1/(2 tau+)) sum c c (f - feq),
// from its pre-collision offsets h, in the compute type (all terms are small).
// The second moment of the equilibrium's offset is (rho - 1)/3 I plus
// rho u u - u_ref u_ref, three products as in collide(), so the sum over the
// populations needs only the offsets' own second moment (about 40 operations
// where summing c c (h_a - heq_a) took 200: FP64's SIM blocks were bound by it).
template <typename T>
struct Stress {
  T xx, xy, yy;
};
template <typename T>
__device__ __forceinline__ Stress<T> stress_of(const Offsets<T> &f, const StepArgs &p) {
  const Lattice &L = p.L;
  const Consts<T> c(p);
  const T(&h)[9] = f.h;
  const T s1 = radd(h[1], h[3]), s2 = radd(h[2], h[4]), s5 = radd(h[5], h[7]), s6 = radd(h[6], h[8]);
  const T d5 = radd(h[5], -h[7]), d6 = radd(h[6], -h[8]), diag = radd(s5, s6);
  const T drho = radd(radd(h[0], radd(s1, s2)), diag);
  const T djx = rfma((T)0.5, lat_bf<T>(L, 0), radd(radd(h[1], -h[3]), radd(d5, -d6)));
  const T djy = rfma((T)0.5, lat_bf<T>(L, 1), radd(radd(h[2], -h[4]), radd(d5, d6)));
  const T inv = rrcp(radd((T)1, drho));
  const T dux = rmul(rfma(drho, -c.urx, djx), inv), duy = rmul(rfma(drho, -c.ury, djy), inv);
  const T ux = radd(c.urx, dux), uy = radd(c.ury, duy);
  const T third = rmul(drho, (T)(1.0 / 3.0));
  const T pxx = radd(radd(radd(s1, diag), -third), -rfma(djx, ux, rmul(c.urx, dux)));
  const T pyy = radd(radd(radd(s2, diag), -third), -rfma(djy, uy, rmul(c.ury, duy)));
  const T pxy = radd(radd(s5, -s6), -rfma(djx, uy, rmul(c.urx, duy)));
  return Stress<T>{rfma(-c.sim_s, pxx, -third), rmul(-c.sim_s, pxy), rfma(-c.sim_s, pyy, -third)};
}

// the pre-collision offsets of node (i, j) of the level that buf holds
template <typename S, bool kGather>
struct FieldNode {
  const S *buf;
  const typename Store<S>::T *prev;
  const Lattice &L;
  __device__ __forceinline__ void operator()(int i, int j,
                                             Offsets<typename Store<S>::T> &f) const {
#pragma unroll
    for (int a = 0; a < 9; ++a) f.h[a] = pre_pop<S, kGather>(buf, prev, L, a, i, j);
  }
};

// mask byte of node (i, j) (inside the lattice) as SIM sees it: chi, or for a
// moving body (a disk; t given) the predicate of Eq. fcar on the current body, since
// the force-region tiles rewrite chi during the step
__device__ __forceinline__ uint8_t solid_at(const StepArgs &p, const NearTest *t, int i, int j) {
  if (t) return disk_contains(*t, i, j) ? kSolid : (uint8_t)0;
  return p.chi[(int64_t)j * p.L.pitch + i];
}

// first fluid node of q_k = (qi, qj) + k c_a, k = 0..3, inside the lattice
// (the four mask bytes are loaded together)
__device__ __forceinline__ bool sim_walk(const StepArgs &p, const NearTest *t, int a, int qi,
                                         int qj, int &oi, int &oj) {
  const Lattice &L = p.L;
  uint8_t m[4];
  bool in[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int ii = qi + k * cx_of(a), jj = qj + k * cy_of(a);
    in[k] = ii >= 0 && ii < L.nx && jj >= 0 && jj < L.ny;
    m[k] = in[k] ? solid_at(p, t, ii, jj) : (uint8_t)kSolid;
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (!in[k]) return false;
    if (!(m[k] & kSolid)) {
      oi = qi + k * cx_of(a);
      oj = qj + k * cy_of(a);
      return true;
    }
  }
  return false;
}

template <typename T>
__device__ __forceinline__ void sim_geom(const SimPoint &sp, T &dx, T &dy, T &nx, T &ny, T &s);
template <>
__device__ __forceinline__ void sim_geom<double>(const SimPoint &sp, double &dx, double &dy,
                                                 double &nx, double &ny, double &s) {
  dx = sp.dx; dy = sp.dy; nx = sp.nx; ny = sp.ny; s = sp.s;
}
template <>
__device__ __forceinline__ void sim_geom<float>(const SimPoint &sp, float &dx, float &dy,
                                                float &nx, float &ny, float &s) {
  dx = sp.f_dx; dy = sp.f_dy; nx = sp.f_nx; ny = sp.f_ny; s = sp.f_s;
}

// The sampled nodes of SIM point sp for the reference point (bxg, byg): the
// nearest node (both nodes when the point lies exactly half-way: the
// coordinates are compared in FP64), each walked along the direction closest
// to the normal to the first fluid node.  Returns their count (1, 2 or 4; 0
// when a walk finds no fluid node), the nodes packed i | j << 16 in the order
// the stress sum takes them.
__device__ __forceinline__ int sim_candidates(const StepArgs &p, const NearTest *t,
                                              const SimPoint &sp, double bxg, double byg,
                                              uint32_t (&cand)[4]) {
  const double x = bxg + sp.dx, y = byg + sp.dy;
  const double rx = floor(x + 0.5), ry = floor(y + 0.5);
  const int ncx = (rx == x + 0.5) ? 2 : 1, ncy = (ry == y + 0.5) ? 2 : 1;
  int n = 0;
  for (int u = 0; u < ncy; ++u)
    for (int v = 0; v < ncx; ++v) {
      int qi, qj;
      if (!sim_walk(p, t, sp.dir, (int)rx - v, (int)ry - u, qi, qj)) return 0;
      cand[n++] = (uint32_t)qi | ((uint32_t)qj << 16);
    }
  return n;
}

// The walks of a fixed body's SIM points, once when the body is placed (the
// mask never changes afterwards): one thread per point.
__global__ void sim_cache_kernel(const StepArgs p) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= p.n_sim) return;
  SimPoint *sp = const_cast<SimPoint *>(p.sim_pts) + q;
  uint32_t cand[4] = {0u, 0u, 0u, 0u};
  const int n = sim_candidates(p, nullptr, *sp, p.body_src->xg, p.body_src->yg, cand);
#pragma unroll
  for (int k = 0; k < 4; ++k) sp->cand[k] = cand[k];
  sp->n_cand = n;
}

// S (sigma + I/3) n and its moment of SIM point sp, from the stress summed over
// its n sampled nodes
template <typename T>
__device__ __forceinline__ FixAcc<T> sim_sum(const SimPoint &sp, const Stress<T> sig, int n) {
  FixAcc<T> r;
  // mean over 1, 2 or 4 candidates: an exact power-of-two scaling
  const T inv = (n == 1) ? (T)1 : ((n == 2) ? (T)0.5 : (T)0.25);
  T dx, dy, nx, ny, sl;
  sim_geom<T>(sp, dx, dy, nx, ny, sl);
  const T sxx = rmul(sig.xx, inv), sxy = rmul(sig.xy, inv), syy = rmul(sig.yy, inv);
  const T tx = rmul(sl, rfma(sxx, nx, rmul(sxy, ny)));
  const T ty = rmul(sl, rfma(sxy, nx, rmul(syy, ny)));
  r.add(0, tx);
  r.add(1, ty);
  r.add(2, rfma(dx, ty, -rmul(dy, tx)));
  return r;
}

// The stress at SIM point sp extrapolated linearly along its sampling direction
// from the sampled node (qi, qj) and the next one (sim_order 1)
template <typename T>
__device__ __forceinline__ Stress<T> extrapolate(const SimPoint &sp, double bxg, double byg, int qi,
                                              int qj, Stress<T> s3, const Stress<T> next) {
  const double x = bxg + sp.dx, y = byg + sp.dy;
  const int c2 = cx_of(sp.dir) * cx_of(sp.dir) + cy_of(sp.dir) * cy_of(sp.dir);
  const T t = (T)(((x - qi) * cx_of(sp.dir) + (y - qj) * cy_of(sp.dir)) / (double)c2);
  s3.xx = rfma(t, radd(next.xx, -s3.xx), s3.xx);
  s3.xy = rfma(t, radd(next.xy, -s3.xy), s3.xy);
  s3.yy = rfma(t, radd(next.yy, -s3.yy), s3.yy);
  return s3;
}

// The force terms of SIM point sp from its n sampled nodes cand; node(i, j, f) gives the pre-collision offsets
// of a node at the step's level.  The -(1/3) S n part sums to a constant of
// the polygon added when the sums are finalized.
template <typename T, typename Node>
__device__ __forceinline__ FixAcc<T> sim_terms(const StepArgs &p, const NearTest *t,
                                               const SimPoint &sp, double bxg, double byg,
                                               const uint32_t (&cand)[4], int n,
                                               const Node &node) {
  T sig[3] = {0, 0, 0};
  for (int k = 0; k < n; ++k) {
    const int qi = (int)(cand[k] & 0xffffu), qj = (int)(cand[k] >> 16);
    Offsets<T> f;
    node(qi, qj, f);
    Stress<T> s3 = stress_of<T>(f, p);
    if (p.sim_order == 1) {
      // first order: extrapolated to the point along the direction from
      // the next node, where that node is fluid and inside the lattice
      const int ni = qi + cx_of(sp.dir), nj = qj + cy_of(sp.dir);
      if (ni >= 0 && ni < p.L.nx && nj >= 0 && nj < p.L.ny && !(solid_at(p, t, ni, nj) & kSolid)) {
        node(ni, nj, f);
        s3 = extrapolate<T>(sp, bxg, byg, qi, qj, s3, stress_of<T>(f, p));
      }
    }
    sig[0] = radd(sig[0], s3.xx);
    sig[1] = radd(sig[1], s3.xy);
    sig[2] = radd(sig[2], s3.yy);
  }
  return n > 0 ? sim_sum<T>(sp, Stress<T>{sig[0], sig[1], sig[2]}, n) : FixAcc<T>();
}

// One SIM integration point: its sampled nodes (walked now, or for a fixed
// body found when it was placed) and its force terms.
template <typename S, bool kGather>
__device__ __noinline__ FixAcc<typename Store<S>::T> sim_point(const StepArgs &p, const S *buf,
                                                               const BodyState &body, int q,
                                                               bool &missing) {
  using T = typename Store<S>::T;
  const SimPoint &sp = p.sim_pts[q];
  uint32_t cand[4] = {sp.cand[0], sp.cand[1], sp.cand[2], sp.cand[3]};
  const double bxg = body.xg, byg = body.yg;
  const NearTest near(body);
  const NearTest *t = p.raster ? &near : nullptr;  // a moving body: its predicate, not chi
  const int n = sp.n_cand >= 0 ? sp.n_cand : sim_candidates(p, t, sp, bxg, byg, cand);
  missing = n <= 0;
  p.sim_nodes[q] = n > 0 ? (int)(cand[0] >> 16) * p.L.nx + (int)(cand[0] & 0xffffu) : -1;
  return sim_terms<T>(p, t, sp, bxg, byg, cand, n,
                      FieldNode<S, kGather>{buf, static_cast<const T *>(p.prev_src), p.L});
}

// ---------------------------------------------------------------------------
// the mask of a moving body, rasterised tile by tile (Eq. fcar)
// ---------------------------------------------------------------------------
// Solid bits of one tile and a one-node halo around it: the predicate of
// Eq. fcar on the body at the step's time level, evaluated by the tile's own
// block, so that no single block re-rasterises the body between steps.
struct TileMask {
  uint8_t s[kTileY + 2][kTileX + 2];
};

// A block of the special kernel takes a tile of kThreads nodes, or with FP64
// storage one of its eight 32-node slices: the FP64 lanes of an SM (two) are what
// its blocks wait for, and one warp per block spreads them over all SMs (the
// disk channel's step, 20 tiles: 32 -> 28 us, and 15 us with one link per lane
// in mem_terms; FP32 tiles in slices of 128 or 64 gain nothing and a moving
// disk's step loses 0.3 and 0.7 us of 10.0).  Nodes are numbered within the tile,
// x fastest.
template <typename S>
constexpr int kSlices = sizeof(S) == 8 ? 8 : 1;
struct Slice {
  int first, count;  // the block's nodes of the tile
};

__device__ __forceinline__ void tile_solid(const StepArgs &p, const BodyState &body, int ti,
                                           int tj, Slice sl, TileMask &tm) {
  const Lattice &L = p.L;
  const NearTest near(body);
  // the slice's rows and columns with their halo (a slice shorter than a row
  // lies within one)
  const int x0 = sl.first % kTileX, y0 = sl.first / kTileX;
  const int w = min(sl.count, kTileX) + 2, h = (sl.count + kTileX - 1) / kTileX + 2;
  for (int q = threadIdx.x; q < w * h; q += blockDim.x) {
    const int hx = x0 + q % w, hy = y0 + q / w;
    int gi = ti * kTileX + hx - 1, gj = tj * kTileY + hy - 1;
    // halo nodes across a periodic side are the nodes there; beyond another
    // side they are never a neighbour (neighbour() gives false)
    if (L.bc[0] == VPLBM_PERIODIC) gi = gi < 0 ? gi + L.nx : (gi >= L.nx ? gi - L.nx : gi);
    if (L.bc[2] == VPLBM_PERIODIC) gj = gj < 0 ? gj + L.ny : (gj >= L.ny ? gj - L.ny : gj);
    const bool in = gi >= 0 && gi < L.nx && gj >= 0 && gj < L.ny;
    tm.s[hy][hx] = (in && disk_contains(near, gi, gj)) ? kSolid : (uint8_t)0;
  }
}

// mask byte (solid bit and interface bit) of the tile node (tx, ty) at (i, j)
__device__ __forceinline__ uint8_t tile_mask_byte(const Lattice &L, const TileMask &tm, int i,
                                                  int j, int tx, int ty) {
  const uint8_t self = tm.s[ty + 1][tx + 1];
  bool iface = false;
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    int ni, nj;
    if (neighbour(L, a, i, j, ni, nj) && tm.s[ty + 1 + cy_of(a)][tx + 1 + cx_of(a)] != self)
      iface = true;
  }
  return (uint8_t)(self | (iface ? kInterface : 0));
}

// ---------------------------------------------------------------------------
// MEM (Sec. 2.3.1)
// ---------------------------------------------------------------------------

// The links of node (i, j) (bit a: the neighbour along a lies in the lattice and
// in the other phase), from chi or from the tile's mask when it rasterises its
// own.  Off the edges the eight bytes are loaded together with the node's own
// populations: the links' latency is then not added to theirs.
__device__ __forceinline__ uint32_t node_links(const StepArgs &p, int i, int j, bool solid,
                                               const TileMask *tm, int tx = 0, int ty = 0) {
  const Lattice &L = p.L;
  const uint8_t self = solid ? kSolid : (uint8_t)0;
  uint32_t links = 0;
  if (i > 0 && i < L.nx - 1 && j > 0 && j < L.ny - 1 && !tm) {
    uint8_t m[9];
#pragma unroll
    for (int a = 1; a < 9; ++a) m[a] = p.chi[(int64_t)(j + cy_of(a)) * L.pitch + i + cx_of(a)];
#pragma unroll
    for (int a = 1; a < 9; ++a) links |= (uint32_t)((m[a] ^ self) & kSolid) << a;
    return links;
  }
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    int ni, nj;
    if (!neighbour(L, a, i, j, ni, nj)) continue;
    const uint8_t m = tm ? tm->s[ty + 1 + cy_of(a)][tx + 1 + cx_of(a)]
                         : p.chi[(int64_t)nj * L.pitch + ni];
    links |= (uint32_t)((m ^ self) & kSolid) << a;
  }
  return links;
}

// The link terms of a warp's interface nodes (Eq. MMEL): for each lattice
// neighbour of the other phase, the fluid end adds (c_a - u_Gamma) f~_a and
// the solid end subtracts its own (c_a - u_Gamma) f~_a, with x_Gamma the link
// midpoint and u_Gamma the rigid velocity there; torques about the reference
// point (Eq. fluidtorque).  f~ = h~ + E is split so that the E parts, which
// cancel in pairs around a fixed body, are rounded exactly.
//
// A warp holds a few interface nodes with a few links each: walking the eight
// directions with most lanes idle was the longest part of a special block
// (2.7 us in FP32, some 400 FP64 operations in FP64).  Every lane takes one link
// of the warp instead: listed in shared memory, or without a list (nullptr)
// found from the lanes' link counts by shuffles, for kernels that run beside
// others which need the L1 that the list would take (the FP16 batch 12.9 us per
// lattice step without lists, 13.5 with them).  Every lane of the warp calls; a
// lane's sums are of the links it took (their order and place do not matter: the
// sums are exact).
template <typename T>
struct LinkList {
  T post[8][32];       // o[1 .. 8] of the lanes with links
  uint16_t link[256];  // lane | direction << 5 | solid << 9
};
template <typename T, bool kList>
__device__ __forceinline__ FixAcc<T> mem_terms(const StepArgs &p, const BodyState &body,
                                               const T (&o)[9], int i, int j, bool solid,
                                               uint32_t links, LinkList<T> *list) {
  FixAcc<T> acc;
  __syncwarp();  // the lanes come from divergent updates; unmerged they would run all this in turn
  if (!__any_sync(kFull, links != 0)) return acc;
  const int lane = threadIdx.x & 31;
  const int n = __popc(links);
  int end = n;  // links of the lanes up to this one
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int v = __shfl_up_sync(kFull, end, d);
    if (lane >= d) end += v;
  }
  const int total = __shfl_sync(kFull, end, 31);
  if constexpr (kList) {
    int at = end - n;
#pragma unroll
    for (int a = 1; a < 9; ++a)
      if (links >> a & 1u) {
        list->post[a - 1][lane] = o[a];
        list->link[at++] = (uint16_t)(lane | a << 5 | (solid ? 1 << 9 : 0));
      }
    __syncwarp();
  }
  const uint32_t mine = links | (solid ? 1u : 0u);  // bit 0: the node's phase
  const Lattice &L = p.L;
  const BodyRef<T> b(body);
#pragma unroll 1
  for (int first = 0; first < total; first += 32) {
    const int t = first + lane;
    int from = 0, a = 1;  // the link's lane and direction
    bool in_solid;
    T post;
    if constexpr (kList) {
      const uint32_t e = t < total ? list->link[t] : 1u << 5;
      from = (int)(e & 31u);
      a = (int)(e >> 5 & 15u);
      in_solid = e >> 9;
      post = list->post[a - 1][from];
    } else {
      // the lane of link t is the first whose end lies beyond t
#pragma unroll
      for (int d = 16; d > 0; d >>= 1)
        if (__shfl_sync(kFull, end, from + d - 1) <= t) from += d;
      from &= 31;
      const uint32_t bits = __shfl_sync(kFull, mine, from);
      const int before = __shfl_sync(kFull, end - n, from);
      uint32_t rest = bits & ~1u;  // its directions from the one taken on
#pragma unroll
      for (int k = 0; k < 7; ++k)
        if (k < t - before) rest &= rest - 1u;
      a = __ffs((int)rest) - 1;
      in_solid = bits & 1u;
      post = __shfl_sync(kFull, o[1], from);
#pragma unroll
      for (int q = 2; q < 9; ++q) {
        const T v = __shfl_sync(kFull, o[q], from);
        if (a == q) post = v;
      }
    }
    const int ni = __shfl_sync(kFull, i, from), nj = __shfl_sync(kFull, j, from);
    if (t >= total) continue;
    const T cx = (T)cx_of(a), cy = (T)cy_of(a);
    const T sg = in_solid ? (T)-1 : (T)1;
    const T rx = radd(radd((T)ni, -b.xg), rmul((T)0.5, cx));
    const T ry = radd(radd((T)nj, -b.yg), rmul((T)0.5, cy));
    const T vx = radd(cx, -rfma(-b.om, ry, b.ux)), vy = radd(cy, -rfma(b.om, rx, b.uy));
    const T ah = rmul(sg, post), aw = rmul(sg, LatC<T>::E(L, a));
    const T lxh = rmul(vx, ah), lyh = rmul(vy, ah), lxw = rmul(vx, aw), lyw = rmul(vy, aw);
    acc.add(0, lxh);
    acc.add(0, lxw);
    acc.add(1, lyh);
    acc.add(1, lyw);
    acc.add(2, rfma(rx, lyh, -rmul(ry, lxh)));
    acc.add(2, rfma(rx, lyw, -rmul(ry, lxw)));
  }
  if constexpr (kList) __syncwarp();
  return acc;
}

// The volume-integral terms of one solid node (Eq. Angotforce, reading R19):
// the penalization force (pen_x, pen_y) on the fluid, reversed, and its moment
// about the reference point.
template <typename T>
__device__ __forceinline__ FixAcc<T> vol_terms(const BodyRef<T> b, int i, int j, T pen_x, T pen_y) {
  FixAcc<T> vol;
  const T fx = -pen_x, fy = -pen_y;
  vol.add(0, fx);
  vol.add(1, fy);
  vol.add(2, rfma(radd((T)i, -b.xg), fy, -rmul(radd((T)j, -b.yg), fx)));
  return vol;
}

// ---------------------------------------------------------------------------
// rigid body and the force sums' bookkeeping
// ---------------------------------------------------------------------------

// A moving body at the step's time level, into b (shared memory), by one warp.
// With the previous step's sums pending (finalize_prev) it is the previous
// level's state updated with them (Eqs. dep1 and theta2, explicit trapezoid in
// time), lanes 0, 1 and 2 taking x, y and the rotation; lanes 0 .. 8 return that
// step's nine totals.  Every block of a launch computes it for itself: the
// earlier scheme, in which the last block of the step (found by a ticket) did
// this for all, added a fence, two rounds to L2 and a half-empty GPU to every
// step's chain.
template <typename T>
__device__ __forceinline__ double moving_body(const StepArgs &p, BodyState &b, bool &ok) {
  constexpr int kBodyWords = (int)(sizeof(BodyState) / sizeof(unsigned long long));
  static_assert(sizeof(BodyState) % sizeof(unsigned long long) == 0 && kBodyWords <= 32,
                "BodyState in 8-byte words, one per lane");
  const int lane = threadIdx.x & 31, k = min(lane, 2);
  const BodyState *from = p.finalize_prev ? p.body_prev : p.body_src;
  // all loads are issued together
  unsigned long long w = 0;
  long long w0 = 0, w1 = 0, w2 = 0;
  if (lane < kBodyWords) w = __ldcg(reinterpret_cast<const unsigned long long *>(from) + lane);
  if (p.finalize_prev && lane < kAccSlots) {
    const unsigned long long *slot = p.acc_prev + kSlotWords * lane;
    w0 = (long long)__ldcg(slot);
    if (Fix<T>::kWords > 1) {
      w1 = (long long)__ldcg(slot + 1);
      w2 = (long long)__ldcg(slot + 2);
    }
  }
  const double inv = __ldg(p.rigid->inv + k), acc = __ldg(p.rigid->acc + k);
  if (lane < kBodyWords) reinterpret_cast<unsigned long long *>(&b)[lane] = w;
  __syncwarp();
  ok = true;
  if (!p.finalize_prev) return 0.0;
  double tot = Fix<T>::value(w0, w1, w2);
  if (lane >= 3 && lane < 6) tot += p.sim_const[lane - 3];
  const double force = __shfl_sync(kFull, tot, b.estimator == VPLBM_SIM ? 3 + k : k);
  const double v0 = k == 0 ? b.ux : k == 1 ? b.uy : b.omega;
  const double x0 = k == 0 ? b.xg : k == 1 ? b.yg : b.theta;
  const double v1 = v0 + fma(force, inv, acc);
  const double x1 = x0 + 0.5 * (v0 + v1);
  // a body that left the lattice or moved a node in one step stays where it was
  // (and one block flags the run as unstable)
  const double r = 0.5 * b.length, far = (double)((k == 0 ? p.L.nx : p.L.ny) - 1);
  const bool fine = k == 2 || (x1 - r >= 0.0 && x1 + r <= far && fabs(x1 - x0) < 1.0);
  ok = __all_sync(kFull, fine);
  __syncwarp();
  if (ok) {
    if (lane == 0) {
      b.ux = v1;
      b.xg = x1;
      b.f_ux = (float)v1;
      b.f_xg = (float)x1;
    } else if (lane == 1) {
      b.uy = v1;
      b.yg = x1;
      b.f_uy = (float)v1;
      b.f_yg = (float)x1;
    } else if (lane == 2) {
      b.omega = v1;
      b.theta = x1;
      b.f_omega = (float)v1;
    }
  }
  __syncwarp();
  return tot;
}

// The bookkeeping of a moving body's step by one warp: with sums pending, the
// body at this level, the history row, running sums and step counter; and the
// force region of this level's body, for the next launch.
template <typename T>
__device__ __forceinline__ void record_moving(const StepArgs &p, BodyState &b,
                                              ForceRegion *region) {
  const int lane = threadIdx.x & 31;
  bool ok;
  const double tot = moving_body<T>(p, b, ok);
  if (lane == 0)
    *region = make_region(p.L, b.xg, b.yg, 0.5 * b.length, p.ntiles_x, p.ntiles_y, kTileX);
  if (!p.finalize_prev) return;
  constexpr int kBodyWords = (int)(sizeof(BodyState) / sizeof(unsigned long long));
  if (lane < kBodyWords)
    reinterpret_cast<unsigned long long *>(p.body_src)[lane] =
        reinterpret_cast<const unsigned long long *>(&b)[lane];
  const bool do_sim = p.prev_sim != 0;
  const long long step = __ldcg(p.dev_step);
  __syncwarp();
  if (lane < kHistCols) {
    // MEM (0-2) and the volume integral (6-8) every step, SIM (3-5) when due
    const bool have = lane < 3 || lane >= 6 || do_sim;
    p.hist[kHistCols * (step % p.hist_len) + lane] =
        have ? tot : __longlong_as_double(0x7ff8000000000000LL);
    if (have && lane < 6) p.sums[lane] += tot;
  } else if (lane == 16) {
    p.counts[0] += 1;
  } else if (lane == 17 && do_sim) {
    p.counts[1] += 1;
  } else if (lane == 18) {
    *p.dev_step = step + 1;
  } else if (lane == 19 && !ok) {
    atomicOr(p.status, kStatusUnstable);
  }
}

// Force bookkeeping of the previous launch (a fixed body): the
// fixed-point sums of its step, or of the two steps of a pair, become the
// steps' history rows and are added to the running sums in step order; the
// step counter advances and the sums are cleared for reuse two launches later.
// Runs in one block beside the next launch's work, or alone at the end of a
// call.  Loads are spread over threads and issued together.
template <typename T>
__device__ void finalize(const StepArgs &p) {
  const int tid = threadIdx.x;
  const int rows = p.prev_rows;
  __shared__ double tot[2][kAccSlots];
  const bool do_sim = p.prev_sim != 0;
  // A warp per row (or one warp for both in turn).  Each row's words and the
  // step counter are loaded together; the code is kept short, since a lone
  // finalizing launch mostly waits for its instructions.
  const int lane = tid & 31;
#pragma unroll 1
  for (int row = tid >> 5; row < rows; row += blockDim.x >> 5) {
    unsigned long long *acc = row ? p.acc2_prev : p.acc_prev;
    long long step = 0;
    double v = 0.0;
    if (lane < kHistCols) {
      const unsigned long long *slot = acc + kSlotWords * lane;
      const long long w0 = (long long)__ldcg(slot);
      const long long w1 = (long long)__ldcg(slot + 1);
      const long long w2 = (long long)__ldcg(slot + 2);
      step = __ldcg(p.dev_step) + row;
      v = Fix<T>::value(w0, w1, w2);
      const bool is_sim = lane >= 3 && lane < 6;
      if (is_sim) v += p.sim_const[lane - 3];
      // MEM (0-2) and the volume integral (6-8) every step, SIM (3-5) when due;
      // not the first of two steps in a ring of one row, which the second's warp
      // writes with no order between them
      if (rows - row <= p.hist_len)
        p.hist[kHistCols * (step % p.hist_len) + lane] =
            !is_sim || do_sim ? v : __longlong_as_double(0x7ff8000000000000LL);
      tot[row][lane] = v;
    }
    __syncwarp();
    if (lane < kAccWords) acc[lane] = 0ull;
  }
  __syncthreads();
  if (tid < 6) {
    if (tid < 3 || do_sim) {
      double v = p.sums[tid] + tot[0][tid];
      if (rows > 1) v += tot[1][tid];
      p.sums[tid] = v;
    }
  } else if (tid == 6 || (tid == 7 && do_sim)) {
    p.counts[tid - 6] += rows;
  } else if (tid == 8) {
    *p.dev_step += rows;  // read above by both rows before the barrier
  }
}

// ---------------------------------------------------------------------------
// node update
// ---------------------------------------------------------------------------

// Coefficients 3 w_a of the odd part of the forcing term, for the axis
// directions (k1 = 3 w_1 = 1/3) and the diagonals (k2 = 3 w_5 = 1/12), in the
// compute type with 2 k1 + 4 k2 = 1 exactly, so that the forcing adds exactly
// its momentum.
template <typename T>
struct OddW;
template <>
struct OddW<double> {
  static constexpr double k1 = 1.0 / 3.0;
  static constexpr double k2 = (1.0 - 2.0 * (1.0 / 3.0)) / 4.0;  // exact: 2 k1 + 4 k2 = 1
};
template <>
struct OddW<float> {
  static constexpr float k1 = 0x1.555556p-2f;  // 1/3 rounded
  static constexpr float k2 = 0x1.555554p-4f;  // (1 - 2 k1) / 4, exactly
};
template <typename T>
__device__ __forceinline__ constexpr T odd_w(int a) {
  return a <= 4 ? OddW<T>::k1 : OddW<T>::k2;
}

// The update is written over a value type V: double for FP64 lattices, and for
// FP32 compute the packed f32x2 instructions of sm_100 and later (one
// instruction for two nodes).  The special kernels update a single node with
// the same packed instructions, the node in both lanes: the compiler fuses
// some packed multiplies with a following add (even when the PTX names a
// rounding mode), so only the same instruction sequence gives a node the same
// bits in every kernel.
struct F2 {
  float2 v;
};
__device__ __forceinline__ unsigned long long f2_bits(F2 a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.v.x), "f"(a.v.y));
  return r;
}
__device__ __forceinline__ F2 bits_f2(unsigned long long r) {
  F2 a;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a.v.x), "=f"(a.v.y) : "l"(r));
  return a;
}
__device__ __forceinline__ F2 vpair(float x, float y) { return F2{make_float2(x, y)}; }
__device__ __forceinline__ F2 vsame(float x) { return F2{make_float2(x, x)}; }
__device__ __forceinline__ F2 vadd(F2 a, F2 b) { return F2{__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ F2 vmul(F2 a, F2 b) { return F2{__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) { return F2{__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ F2 vsub(F2 a, F2 b) {
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
  return bits_f2(r);
}
__device__ __forceinline__ float vlo(F2 a) { return a.v.x; }
__device__ __forceinline__ float vhi(F2 a) { return a.v.y; }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
template <typename V>
struct Val;
template <>
struct Val<F2> {
  using T = float;
  static __device__ __forceinline__ F2 splat(float c) { return vsame(c); }
};
template <>
struct Val<double> {
  using T = double;
  static __device__ __forceinline__ double splat(double c) { return c; }
};
__device__ __forceinline__ bool rho_bad(float r) { return !(r > 0.f) || !isfinite(r); }
__device__ __forceinline__ bool rho_bad(double r) { return !(r > 0.0) || !isfinite(r); }

// 1 / a by Newton's iteration y <- y + y (1 - a y) from the hardware's
// approximation (relative error below 2^-22; the error squares), two FMAs, where
// the correctly rounded division's range checks and fix-ups cost several times
// that.  The result is the correctly rounded one for every float between 2^-20
// and 2^20 (all of them were compared with __frcp_rn); densities are near 1.
__device__ __forceinline__ F2 vrcp(F2 a) {
  float x, y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(a.v.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a.v.y));
  const F2 r = vpair(x, y);
  return vfma(r, vfma(vmul(a, vsame(-1.0f)), r, vsame(1.0f)), r);
}
__device__ __forceinline__ double vrcp(double a) { return near_rcp(a); }

// Sums and differences of the opposite pairs (a, opp(a)), a = 1, 2, 5, 6, and
// the moments of the offsets: drho = rho - 1 and (djx, djy) = j - u_ref.
template <typename V>
struct Moments {
  V s[4], d[4], drho, djx, djy;
  __device__ __forceinline__ explicit Moments(const V (&h)[9]) {
    s[0] = vadd(h[1], h[3]);
    d[0] = vsub(h[1], h[3]);
    s[1] = vadd(h[2], h[4]);
    d[1] = vsub(h[2], h[4]);
    s[2] = vadd(h[5], h[7]);
    d[2] = vsub(h[5], h[7]);
    s[3] = vadd(h[6], h[8]);
    d[3] = vsub(h[6], h[8]);
    drho = vadd(vadd(h[0], vadd(s[0], s[1])), vadd(s[2], s[3]));
    djx = vadd(d[0], vsub(d[2], d[3]));
    djy = vadd(d[1], vadd(d[2], d[3]));
  }
};

// BGK/TRT collision with the forcing term (Eq. TRT), into o.  The equilibrium
// enters through its offset heq = feq(rho, u) - E, written with the small
// quantities drho, du = u - u_ref and dj = rho u - u_ref only.  Its second
// moments are three products,
//   X = rho u_x^2 - u_ref,x^2 = dj_x u_x + u_ref,x du_x, Y alike, and
//   P = rho u_x u_y - u_ref,x u_ref,y = dj_x u_y + u_ref,x du_y,
// from which the even parts follow, heq+ = w [drho - 1.5 (X + Y) + 4.5 X_a]
// with X_1 = X, X_2 = Y, X_5,6 = X + Y +- 2 P; the odd parts are
// heq- = 3 w c.dj.  (FP64 runs at about 1/58 of the FP32 rate on this part and
// FP32 is bound by its FMA pipe in the kernels that fuse two steps, so the
// operation count is what both pay for: 76 operations per node, where the form
// with (c.u)^2 and c.u per direction took 115 and a division.)
//
// The odd rates sm_k1 = 3 w_1 s- and sm_k2 = 3 w_5 s- satisfy
// sm_k1 + 2 sm_k2 = s-/2 exactly (api.cu), so that the odd equilibrium carries
// exactly the node's momentum: rounded independently they would make every
// collision add about 1e-8 of the momentum offset, a bias that compounds step
// after step.  The
// rest population takes what the moving populations' even parts give up,
// o_0 = h_0 - 2 sum (even change of a pair's population): equal to the
// relaxation of h_0 towards heq_0 (plus F_0) in exact arithmetic, and
// conserving mass exactly up to the rounding of that sum.  kForce = false
// drops the forcing term (G = 0: a fluid node without body force), kRef = false
// the terms of u_ref (zero).
//
// kHalves writes a pair as half its sum and half its difference, o_a,b = P +- M,
// and the rest population as what they leave of rho: eight operations fewer than
// adding the changes to h, for FP64 (bound by its operation count) where it rounds
// no worse than the form with (c.u)^2.  That is s- >= 1/2: M then takes
// (1 - s-)/2 <= 1/4 of the difference, an exact coefficient.  Below, the rounding
// of the difference itself enters at half its size and the coefficient is rounded:
// momentum error of a collision at s- = 0.17, in 1e-18: 3.2 with a bias of 1.7 for
// halves, 1.6 for the form with (c.u)^2, 1.5 for changes added to h; at s- = 0.51
// 2.6, 2.9 and 2.0; at s- = 1.5 4.7, 7.7 and 4.4.
template <typename V, bool kForce, bool kRef = true, bool kHalves = false>
__device__ __forceinline__ void collide(const V (&h)[9], const Moments<V> &m, V djx, V djy, V ux,
                                        V uy, V dux, V duy, V gx, V gy,
                                        const Consts<typename Val<V>::T> &c, V (&o)[9]) {
  using T = typename Val<V>::T;
  auto k = [](T v) { return Val<V>::splat(v); };
  const V X = kRef ? vfma(djx, ux, vmul(k(c.urx), dux)) : vmul(djx, ux);
  const V Y = kRef ? vfma(djy, uy, vmul(k(c.ury), duy)) : vmul(djy, uy);
  const V P = kRef ? vfma(djx, uy, vmul(k(c.urx), duy)) : vmul(djx, uy);
  const V t = vadd(X, Y);
  const V axis = vmul(k(c.sp_w1), vfma(k((T)-1.5), t, m.drho));
  const V diag = vmul(k(c.sp_w5), vfma(k((T)3), t, m.drho));
  V even{};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int a = q < 2 ? q + 1 : q + 3, b = opp_of(a);
    // s+ heq+ of the pair and c.dj
    const V ep = q == 0   ? vfma(k(c.sp_45w1), X, axis)
                 : q == 1 ? vfma(k(c.sp_45w1), Y, axis)
                 : q == 2 ? vfma(k(c.sp_9w5), P, diag)
                          : vfma(k(-c.sp_9w5), P, diag);
    const V cdj = q == 0 ? djx : q == 1 ? djy : q == 2 ? vadd(djx, djy) : vsub(djy, djx);
    V dp = vfma(k(kHalves ? (T)0.5 + c.nsp_half : c.nsp_half), m.s[q], ep);
    V dm = vfma(k(kHalves ? (T)0.5 + c.nsm_half : c.nsm_half), m.d[q],
                vmul(k(q < 2 ? c.sm_k1 : c.sm_k2), cdj));
    if (kForce) {
      // F_a = w [3 c.G + 9 (c.u)(c.G) - 3 u.G], even and odd parts
      const V cu = q == 0 ? ux : q == 1 ? uy : q == 2 ? vadd(ux, uy) : vsub(uy, ux);
      const V cg = q == 0 ? gx : q == 1 ? gy : q == 2 ? vadd(gx, gy) : vsub(gy, gx);
      const V ug = vfma(ux, gx, vmul(uy, gy));
      const T w = (T)w_of(a);
      dp = vfma(k(c.a_plus * w * (T)9), vmul(cu, cg), vfma(k(c.a_plus * w * (T)-3), ug, dp));
      dm = vfma(k(c.a_minus), vmul(k(odd_w<T>(a)), cg), dm);
    }
    even = q == 0 ? dp : vadd(even, dp);
    o[a] = vadd(kHalves ? dp : vadd(h[a], dp), dm);
    o[b] = vsub(kHalves ? dp : vadd(h[b], dp), dm);
  }
  o[0] = vfma(k((T)-2), even, kHalves ? m.drho : h[0]);
}

// The update of fluid nodes (no penalization): moments, velocity and the
// collision, from the pre-collision offsets h of a node (FP64), a node pair or
// one node in both lanes (FP32); kForce adds the uniform body force, kRef = false
// leaves out u_ref = 0 (seven operations; FP64 lattices store offsets from rest);
// kHalves: see collide().  Returns rho.
template <typename V, bool kForce, bool kRef = true, bool kHalves = false>
__device__ __forceinline__ V fluid_update(const Lattice &L, const Consts<typename Val<V>::T> &cst,
                                          const V (&h)[9], V (&o)[9]) {
  using T = typename Val<V>::T;
  const Moments<V> m(h);
  const V rho = vadd(Val<V>::splat((T)1), m.drho);
  const V inv = vrcp(rho);
  V djx = m.djx, djy = m.djy, gx{}, gy{};
  if (kForce) {
    gx = Val<V>::splat(lat_bf<T>(L, 0));
    gy = Val<V>::splat(lat_bf<T>(L, 1));
    djx = vfma(Val<V>::splat((T)0.5), gx, djx);
    djy = vfma(Val<V>::splat((T)0.5), gy, djy);
  }
  const V dux = vmul(kRef ? vfma(m.drho, Val<V>::splat(-cst.urx), djx) : djx, inv);
  const V duy = vmul(kRef ? vfma(m.drho, Val<V>::splat(-cst.ury), djy) : djy, inv);
  const V ux = kRef ? vadd(Val<V>::splat(cst.urx), dux) : dux;
  const V uy = kRef ? vadd(Val<V>::splat(cst.ury), duy) : duy;
  collide<V, kForce, kRef, kHalves>(h, m, djx, djy, ux, uy, dux, duy, gx, gy, cst, o);
  return rho;
}

// ---------------------------------------------------------------------------
// 16-bit storage keeps the arithmetic it began with, bit for bit: every stored
// value is rounded to 16 bits, so any change of FP32 rounding flips some of
// them and the run follows another rounding history (instantaneous forces move
// by 1e-3, where the form above moves FP32 lattices by 1e-6).  Per pair
// (a, opp(a))
//   s+ heq+ = s+ w K + 4.5 s+ w X,  X = drho (c.u)^2 + (c.du)(c.u + c.u_ref),
//   K = drho (1 - 1.5 |u|^2) - 1.5 (|u|^2 - |u_ref|^2),
// the odd part is -s- (h- - k (drho c.u + c.du)), and the rest population
// takes the even changes' remainder.
// ---------------------------------------------------------------------------
template <bool kForce>
__device__ __forceinline__ void collide16(const F2 (&h)[9], F2 drho, F2 dux, F2 duy, F2 gx, F2 gy,
                                          const Consts<float> &c, F2 (&o)[9]) {
  using V = F2;
  using T = float;
  const V urx = vsame(c.urx), ury = vsame(c.ury);
  const V ux = vadd(urx, dux), uy = vadd(ury, duy);
  const V uu = vfma(ux, ux, vmul(uy, uy));
  const V dsu = vfma(dux, vadd(ux, urx), vmul(duy, vadd(uy, ury)));
  const V m15 = vsame((T)-1.5);
  const V K = vfma(m15, dsu, vmul(drho, vfma(m15, uu, vsame((T)1))));
  V ug{};
  if (kForce) ug = vfma(ux, gx, vmul(uy, gy));
  const V nsph = vsame((T)-0.5 * c.s_plus), nsm = vsame(-c.s_minus), half = vsame((T)0.5);
  V even = vsame((T)0);
#pragma unroll
  for (int a = 1; a <= 6; ++a) {
    if (a == 3 || a == 4) continue;
    const int b = opp_of(a);
    const T w = (T)w_of(a);
    const V k = vsame(odd_w<T>(a));
    // c.u, c.du for the four directions 1 (1,0), 2 (0,1), 5 (1,1), 6 (-1,1)
    V cu, cdu;
    if (a == 1) {
      cu = ux;
      cdu = dux;
    } else if (a == 2) {
      cu = uy;
      cdu = duy;
    } else if (a == 5) {
      cu = vadd(ux, uy);
      cdu = vadd(dux, duy);
    } else {
      cu = vsub(uy, ux);
      cdu = vsub(duy, dux);
    }
    const V csu = vadd(cu, vsame((T)cx_of(a) * c.urx + (T)cy_of(a) * c.ury));
    const V dc = vmul(drho, cu);
    const V X = vfma(dc, cu, vmul(cdu, csu));
    const V P = vfma(vsame((T)4.5 * c.s_plus * w), X, vmul(vsame(c.s_plus * w), K));
    V dp = vfma(nsph, vadd(h[a], h[b]), P);
    // -s- (h- - heq-), h- = (h_a - h_b) / 2, heq- = k (drho c.u + c.du)
    V dm = vmul(nsm, vsub(vmul(half, vsub(h[a], h[b])), vmul(k, vadd(dc, cdu))));
    if (kForce) {
      V cg;
      if (a == 1)
        cg = gx;
      else if (a == 2)
        cg = gy;
      else if (a == 5)
        cg = vadd(gx, gy);
      else
        cg = vsub(gy, gx);
      dp = vfma(vsame(c.a_plus * w * (T)9), vmul(cu, cg), vfma(vsame(c.a_plus * w * (T)-3), ug, dp));
      dm = vfma(vsame(c.a_minus), vmul(k, cg), dm);
    }
    even = vadd(even, dp);
    o[a] = vadd(vadd(h[a], dp), dm);
    o[b] = vsub(vadd(h[b], dp), dm);
  }
  o[0] = vfma(vsame((T)-2), even, h[0]);
}

// moments of nine offsets in the order of the 16-bit forms
__device__ __forceinline__ void moments16(const F2 (&h)[9], F2 &drho, F2 &djx, F2 &djy) {
  drho = vadd(vadd(vadd(h[0], h[1]), vadd(h[2], h[3])),
              vadd(vadd(vadd(h[4], h[5]), vadd(h[6], h[7])), h[8]));
  djx = vadd(vadd(vsub(h[1], h[3]), vsub(h[5], h[6])), vsub(h[8], h[7]));
  djy = vadd(vadd(vsub(h[2], h[4]), vsub(h[5], h[7])), vsub(h[6], h[8]));
}

template <bool kForce>
__device__ __forceinline__ F2 fluid_update16(const Lattice &L, const Consts<float> &cst,
                                             const F2 (&h)[9], F2 (&o)[9]) {
  F2 drho, djx, djy;
  moments16(h, drho, djx, djy);
  const F2 rho = vadd(vsame(1.0f), drho);
  const F2 inv = vrcp(rho);
  F2 gx{}, gy{};
  if (kForce) {
    gx = vsame(lat_bf<float>(L, 0));
    gy = vsame(lat_bf<float>(L, 1));
    djx = vfma(vsame(0.5f), gx, djx);
    djy = vfma(vsame(0.5f), gy, djy);
  }
  collide16<kForce>(h, drho, vmul(vfma(drho, vsame(-cst.urx), djx), inv),
                    vmul(vfma(drho, vsame(-cst.ury), djy), inv), gx, gy, cst, o);
  return rho;
}

// the fluid update of storage form S
template <typename S, bool kForce, typename V>
__device__ __forceinline__ V update_fluid(const Lattice &L,
                                          const Consts<typename Val<V>::T> &cst,
                                          const V (&h)[9], V (&o)[9]) {
  if constexpr (sizeof(S) == 2)
    return fluid_update16<kForce>(L, cst, h, o);
  else if constexpr (sizeof(S) == 8)
    return cst.urx != 0.0 || cst.ury != 0.0 ? fluid_update<V, kForce>(L, cst, h, o)
           : cst.halves                     ? fluid_update<V, kForce, false, true>(L, cst, h, o)
                                            : fluid_update<V, kForce, false>(L, cst, h, o);
  else
    return fluid_update<V, kForce>(L, cst, h, o);
}

// a single node's value as V (in both lanes) and back
template <typename T>
struct NodeVal;
template <>
struct NodeVal<float> {
  using V = F2;
  static __device__ __forceinline__ float get(F2 v) { return vlo(v); }
};
template <>
struct NodeVal<double> {
  using V = double;
  static __device__ __forceinline__ double get(double v) { return v; }
};

// Moments, penalized velocity and force density of one node (Eqs. updatestep
// .. updatestepm: G = -rho (chi/eta)(u - u_s) in the rearranged form
// -(chi/eta)(j - rho u_s)/(1 + chi dt/(2 eta)), plus the body force), then
// the collision; a fluid node gets the same bits as from the bulk kernels.
// (pen_x, pen_y): the penalization part of G (solid nodes only).  Returns true
// for a non-finite or non-positive density.
template <typename S, bool kForce, typename T>
__device__ __forceinline__ bool update_node(const T (&h)[9], uint8_t mask, int i, int j,
                                            const Lattice &L, const BodyState *body,
                                            const Consts<T> &cst, T (&o)[9], T &pen_x,
                                            T &pen_y) {
  using N = NodeVal<T>;
  using V = typename N::V;
  pen_x = pen_y = (T)0;
  V hv[9], ov[9], rho;
#pragma unroll
  for (int a = 0; a < 9; ++a) hv[a] = Val<V>::splat(h[a]);
  if (!(mask & kSolid)) {
    rho = update_fluid<S, kForce>(L, cst, hv, ov);
  } else {
    const Moments<V> m(hv);
    V drho = m.drho, jx = m.djx, jy = m.djy;
    if constexpr (sizeof(S) == 2) moments16(hv, drho, jx, jy);
    rho = vadd(Val<V>::splat((T)1), drho);
    const T bfx = lat_bf<T>(L, 0), bfy = lat_bf<T>(L, 1);
    const T djx = N::get(vfma(Val<V>::splat((T)0.5), Val<V>::splat(bfx), jx));
    const T djy = N::get(vfma(Val<V>::splat((T)0.5), Val<V>::splat(bfy), jy));
    T usx, usy;
    solid_velocity<T>(*body, i, j, usx, usy);
    const T k = cst.half_pen, r = N::get(rho), dr = N::get(drho);
    const T den = r + k * r;
    // the momentum defect j - rho u_s, from the offsets' first moment
    const T defx = djx - dr * usx + (cst.urx - usx);
    const T defy = djy - dr * usy + (cst.ury - usy);
    // u - u_ref = (j + k rho u_s)/(rho (1 + k)) - u_ref, written as
    // (u_s - u_ref) + (j - rho u_s)/(rho (1 + k)): the large part is exact
    // and the small one keeps its relative precision (k rho u_s alone
    // would carry an FP32 rounding of 1e-3 into the division by k rho);
    // G = -(chi/eta)(j - rho u_s)/(1 + k)
    T ex, ey;
    if constexpr (sizeof(S) == 2) {
      ex = defx / den;
      ey = defy / den;
      const T pen = (T)2 * k;
      pen_x = -pen * defx / ((T)1 + k);
      pen_y = -pen * defy / ((T)1 + k);
    } else {
      const T inv = N::get(vrcp(Val<V>::splat(den)));
      ex = defx * inv;
      ey = defy * inv;
      pen_x = cst.pen * defx;
      pen_y = cst.pen * defy;
    }
    const T dux = (usx - cst.urx) + ex, duy = (usy - cst.ury) + ey;
    const V vx = Val<V>::splat(dux), vy = Val<V>::splat(duy);
    const V gx = Val<V>::splat(bfx + pen_x), gy = Val<V>::splat(bfy + pen_y);
    if constexpr (sizeof(S) == 2) {
      collide16<true>(hv, drho, vx, vy, gx, gy, cst, ov);
    } else {
      // rho u - u_ref with the penalized velocity
      const V ux = Val<V>::splat(usx + ex), uy = Val<V>::splat(usy + ey);
      collide<V, true>(hv, m, vfma(drho, ux, vx), vfma(drho, uy, vy), ux, uy, vx, vy, gx, gy, cst, ov);
    }
  }
#pragma unroll
  for (int a = 0; a < 9; ++a) o[a] = N::get(ov[a]);
  return rho_bad(N::get(rho));
}

// ---------------------------------------------------------------------------
// stochastic rounding of the stored populations (the _SR storage forms)
// ---------------------------------------------------------------------------
// hash of the level being written: the rounding counter, which the special
// kernel advances by one per step
__device__ __forceinline__ uint32_t sr_level(const StepArgs &p, int step = 0) {
  const unsigned long long n = __ldg(p.rng_src) + (unsigned long long)step;
  return pcg_hash((uint32_t)n ^ (uint32_t)(n >> 32));
}

// The random bits of a node pair (the nodes 2q and 2q + 1 of the linear index
// j * pitch + i; a row starts at an even index, the pitch being a multiple of
// 64) for the eighteen values it stores: four hashes, and nine words made of
// distinct exclusive-ors of them, one word per population.  The low half of
// population a's word serves the even node, the high half the odd one (the
// lanes of the conversion).  Distinct subsets of independent uniform words
// are pairwise independent, so any two roundings of the pair are
// uncorrelated.  Every kernel that stores a node draws the same bits.
struct SrBits {
  uint32_t h[4];
  __device__ __forceinline__ SrBits(uint32_t level, uint32_t pair) {
#pragma unroll
    for (int q = 0; q < 4; ++q) h[q] = pcg_hash(level + pair * 4u + (uint32_t)q);
  }
  __device__ __forceinline__ uint32_t word(int a) const {
    switch (a) {
      case 0: return h[0];
      case 1: return h[1];
      case 2: return h[2];
      case 3: return h[3];
      case 4: return h[0] ^ h[1];
      case 5: return h[2] ^ h[3];
      case 6: return h[0] ^ h[2];
      case 7: return h[1] ^ h[3];
      default: return h[0] ^ h[3];
    }
  }
};

// stores population value v of node `node`, rounded to the storage type (to
// nearest, or stochastically with the bits of the node's pair)
template <typename S, bool kSR>
__device__ __forceinline__ void store_pop(S *ptr, typename Store<S>::T v, const SrBits *r, int a,
                                          uint32_t node) {
  if constexpr (sizeof(S) == 2 && kSR) {
    const uint32_t w = r->word(a);
    *reinterpret_cast<unsigned short *>(ptr) =
        (unsigned short)(Stochastic<S>::pair(v, v, (node & 1u) ? w >> 16 : w) & 0xffffu);
  } else {
    Store<S>::st(ptr, v);
  }
}

// pre-collision populations of an edge node, with the side conditions
template <typename S, bool kGather>
__device__ __forceinline__ void edge_pops(const S *src, const typename Store<S>::T *prev,
                                          const Lattice &L, int i, int j,
                                          typename Store<S>::T (&h)[9]) {
#pragma unroll
  for (int a = 0; a < 9; ++a) h[a] = pre_pop<S, kGather>(src, prev, L, a, i, j);
}

// What a node of the force region leaves for its warp's force terms: its
// post-collision values, links and penalization force.
template <typename T>
struct NodeForces {
  T o[9], pen_x = 0, pen_y = 0;
  uint32_t links = 0;
  bool solid = false;
};

// The pre-collision populations of a node of the special kernel (with the side
// conditions where needed).
template <typename S, bool kGather>
__device__ __forceinline__ void special_load(const StepArgs &p, int i, int j,
                                             typename Store<S>::T (&h)[9]) {
  using T = typename Store<S>::T;
  const Lattice &L = p.L;
  const S *__restrict__ src = static_cast<const S *>(p.src);
  if (kGather && i > 0 && i < L.nx - 1 && j > 0 && j < L.ny - 1) {
    const int64_t node = (int64_t)j * L.pitch + i;
#pragma unroll
    for (int a = 0; a < 9; ++a)
      h[a] = Store<S>::ld(src + (int64_t)a * L.plane + node - cy_of(a) * L.pitch - cx_of(a));
  } else {
    edge_pops<S, kGather>(src, static_cast<const T *>(p.prev_src), L, i, j, h);
  }
}

// One node of the special kernel: keep the outlet column, update and store.
template <typename S>
__device__ __forceinline__ bool special_node(const StepArgs &p, const BodyState *body,
                                             const typename Store<S>::T (&h)[9], int i, int j,
                                             bool in_reg, const TileMask *tm, int tx, int ty,
                                             NodeForces<typename Store<S>::T> &nf) {
  using T = typename Store<S>::T;
  const Lattice &L = p.L;
  S *dst = static_cast<S *>(p.dst);
  const int64_t node = (int64_t)j * L.pitch + i;
  if (i == L.nx - 1 && L.bc[1] == VPLBM_OUTLET_CONVECTIVE) {
    // the outlet column's pre-collision values, for the next step
    T *pd = static_cast<T *>(p.prev_dst);
    pd[0 * L.ny + j] = h[3];
    pd[1 * L.ny + j] = h[6];
    pd[2 * L.ny + j] = h[7];
  }
  uint8_t m;
  if (tm) {
    // a moving body's tile: its mask byte from the tile's predicate, kept in
    // chi for the read-backs
    m = tile_mask_byte(L, *tm, i, j, tx, ty);
    p.chi[node] = m;
  } else {
    m = p.chi[node];
  }
  // FP64's long update hides the links' loads; elsewhere only interface nodes
  // look for theirs
  if (in_reg && ((sizeof(S) == 8 && !tm) || (m & kInterface)))
    nf.links = node_links(p, i, j, m & kSolid, tm, tx, ty);
  nf.solid = m & kSolid;
  T(&o)[9] = nf.o;
  const Consts<T> cst(p);
  const bool bad =
      L.has_bf ? update_node<S, true>(h, m, i, j, L, body, cst, o, nf.pen_x, nf.pen_y)
               : update_node<S, false>(h, m, i, j, L, body, cst, o, nf.pen_x, nf.pen_y);
  if (sizeof(S) == 2 && p.sr) {
    const SrBits r(sr_level(p), (uint32_t)node >> 1);
#pragma unroll
    for (int a = 0; a < 9; ++a)
      store_pop<S, true>(dst + (int64_t)a * L.plane + node, o[a], &r, a, (uint32_t)node);
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a)
      store_pop<S, false>(dst + (int64_t)a * L.plane + node, o[a], nullptr, a, (uint32_t)node);
  }
  return bad;
}

// ---------------------------------------------------------------------------
// special kernel: SIM blocks, then blocks of edge nodes, then the
// force-region tiles (or, for the first step, every tile)
// ---------------------------------------------------------------------------
// The special kernels of lattices stepped side by side share the SMs with the
// bulk kernels, whose bytes in flight need the register file: for a fixed
// body with FP32 compute the special kernel is then capped at 64 registers (four
// blocks per SM), at the price of a few spilled values.  A moving body's special
// kernel is on the step's critical path (its force feeds the next step), and so
// is that of a lattice stepped alone: they keep all the registers they want
// (kMinBlocks 1).
template <typename S>
constexpr int kSpecialMinBlocks = sizeof(S) <= 4 ? 4 : 1;

template <typename S, bool kGather, int kMinBlocks, bool kList>
__global__ void __launch_bounds__(kThreads / kSlices<S>, kMinBlocks)
    special_kernel(const StepArgs p) {
  using T = typename Store<S>::T;
  constexpr int kBlock = kThreads / kSlices<S>;
  __shared__ TileMask tmask;
  __shared__ BodyState moving;
  __shared__ LinkList<T> lists[kList ? kBlock / 32 : 1];
  const Lattice &L = p.L;
  const int b = blockIdx.x / kSlices<S>;
  const Slice slice{(int)(blockIdx.x % kSlices<S>) * kBlock, kBlock};
  const int tid = slice.first + threadIdx.x;  // within the tile's nodes
  const ForceRegion reg = *p.reg_src;
  const bool moves = kList && p.raster;  // a moving body (special_t)
  if (p.sr && b == 0 && tid == 0) *p.rng_dst = *p.rng_src + 1ull;  // the next level's counter
  if ((p.finalize_prev || moves) && b == (int)(gridDim.x / kSlices<S>) - 1) {
    // the previous step's force sums, beside this step's work
    if (slice.first != 0) return;
    if (!moves) {
      finalize<T>(p);
    } else if (threadIdx.x < 32) {
      if (threadIdx.x < kAccWords) p.acc_next[threadIdx.x] = 0ull;
      record_moving<T>(p, moving, p.reg_dst);
    }
    return;
  }
  // a moving body's state at this level, by the block's first warp
  bool ok;
  const BodyState *body = moves ? &moving : p.body_src;

  if (b < p.sim_blocks) {
    // ---- SIM points of this level ----
    if (moves) {
      if (threadIdx.x < 32) moving_body<T>(p, moving, ok);
      __syncthreads();
    }
    const int q = b * p.sim_per_block + tid;
    FixAcc<T> acc;
    bool missing = false;
    if (tid < p.sim_per_block && q < p.n_sim)
      acc = sim_point<S, kGather>(p, static_cast<const S *>(p.src), *body, q, missing);
    __syncwarp();
    if (__any_sync(kFull, missing) && (tid & 31) == 0) atomicOr(p.status, kStatusSimMissing);
    warp_add(acc, p.acc, 3);
  } else if (!p.all_tiles && b < p.sim_blocks + p.edge_blocks) {
    // ---- one edge node per thread (nodes of force-region tiles excluded) ----
    const int e = (b - p.sim_blocks) * kThreads + tid;
    bool bad = false;
    if (e < edge_count(L.nx, L.ny)) {
      int i, j;
      edge_node(e, L.nx, L.ny, i, j);
      const int ti = i / kTileX, tj = j / kTileY;
      const bool in_reg = ti >= reg.ti0 && ti <= reg.ti1 && tj >= reg.tj0 && tj <= reg.tj1;
      if (!in_reg) {
        NodeForces<T> unused;
        T h[9];
        special_load<S, kGather>(p, i, j, h);
        bad = special_node<S>(p, p.body_src, h, i, j, false, nullptr, 0, 0, unused);
      }
    }
    if (__any_sync(kFull, bad) && (tid & 31) == 0) atomicOr(p.status, kStatusUnstable);
  } else {
    // ---- a whole tile: every tile (first step) or a force-region tile ----
    int ti, tj;
    const int r = b - p.sim_blocks;
    if (p.all_tiles) {
      ti = r % p.ntiles_x;
      tj = r / p.ntiles_x;
    } else {
      const int k = r - p.edge_blocks;
      if (k >= reg.count) return;  // spare slot (moving bodies)
      const int rw = reg.ti1 - reg.ti0 + 1;
      ti = reg.ti0 + k % rw;
      tj = reg.tj0 + k / rw;
    }
    const bool in_reg = ti >= reg.ti0 && ti <= reg.ti1 && tj >= reg.tj0 && tj <= reg.tj1;
    const int tx = tid % kTileX, ty = tid / kTileX;
    const int i = ti * kTileX + tx, j = tj * kTileY + ty;
    const bool inside = i < L.nx && j < L.ny;
    T h[9];
    if (inside) special_load<S, kGather>(p, i, j, h);
    // a moving body: its state, and the region tiles rasterise its mask at this
    // level, while the populations arrive
    const bool raster = moves && in_reg;  // uniform over the block
    if (raster) {
      if (threadIdx.x < 32) moving_body<T>(p, moving, ok);
      __syncthreads();
      tile_solid(p, moving, ti, tj, slice, tmask);
      __syncthreads();
    }
    bool bad = false;
    NodeForces<T> nf;
    if (inside)
      bad = special_node<S>(p, body, h, i, j, in_reg, raster ? &tmask : nullptr, tx, ty, nf);
    __syncwarp();
    if (__any_sync(kFull, bad) && (tid & 31) == 0) atomicOr(p.status, kStatusUnstable);
    if (!in_reg) return;  // uniform over the block
    LinkList<T> *list = nullptr;
    if constexpr (kList) list = lists + (threadIdx.x >> 5);
    warp_add(mem_terms<T, kList>(p, *body, nf.o, i, j, nf.solid, nf.links, list), p.acc, 0);
    FixAcc<T> vol;
    if (nf.solid) vol = vol_terms<T>(BodyRef<T>(*body), i, j, nf.pen_x, nf.pen_y);
    warp_add(vol, p.acc, 6);
  }
}

// ---------------------------------------------------------------------------
// bulk kernel: every node off the lattice edges and outside the force-region
// tiles -- fluid nodes whose pull sources all lie inside the lattice.
// ---------------------------------------------------------------------------
template <typename S, bool kForce, int kTiles>
__global__ void __launch_bounds__(kThreads * kTiles) bulk_kernel(const StepArgs p) {
  using T = typename Store<S>::T;
  const Lattice &L = p.L;
  const int ti = blockIdx.x;
  const int i = ti * kTileX + threadIdx.x;
  const int j = blockIdx.y * (kTileY * kTiles) + threadIdx.y;  // a block is kTiles tiles high
  const int tj = j / kTileY;
  if (i < 1 || i > L.nx - 2 || j < 1 || j > L.ny - 2) return;  // edge nodes: special kernel
  const S *__restrict__ src = static_cast<const S *>(p.src);
  S *__restrict__ dst = static_cast<S *>(p.dst);
  const int64_t node = (int64_t)j * L.pitch + i;
  // the populations are requested before the force-region bounds are known,
  // so that their latency is not added to that of the bounds
  T h[9];
#pragma unroll
  for (int a = 0; a < 9; ++a)
    h[a] = Store<S>::ld(src + (int64_t)a * L.plane + node - cy_of(a) * L.pitch - cx_of(a));
  {
    const ForceRegion reg = *p.reg_src;
    if (ti >= reg.ti0 && ti <= reg.ti1 && tj >= reg.tj0 && tj <= reg.tj1) return;  // special kernel
  }
  T o[9];
  const T rho = update_fluid<S, kForce>(L, Consts<T>(p), h, o);
#pragma unroll
  for (int a = 0; a < 9; ++a) Store<S>::st(dst + (int64_t)a * L.plane + node, o[a]);
  if (rho_bad(rho)) atomicOr(p.status, kStatusUnstable);
}

// ---------------------------------------------------------------------------
// bulk kernel for FP32 storage: two adjacent nodes per thread, one 64-bit
// load and one 64-bit store per plane, the +-x neighbour from the next lane by
// a shuffle, and the collision of both nodes in packed f32x2 arithmetic (the
// special kernel updates its fluid nodes with the same arithmetic, one node
// in both lanes).  A tile row of 128 nodes is two warps; a block is kTiles
// tiles high.
// ---------------------------------------------------------------------------
template <bool kForce, int kTiles>
__global__ void __launch_bounds__(kThreads / 2 * kTiles) bulk32x2_kernel(const StepArgs p) {
  const Lattice &L = p.L;
  const int ti = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const int i = ti * kTileX + 2 * threadIdx.x;  // the thread's nodes i, i + 1
  const int j = blockIdx.y * (kTileY * kTiles) + threadIdx.y;
  const int tj = j / kTileY;
  // every lane loads from inside its row (clamped), so that the shuffles see
  // all lanes; results of clamped lanes are never stored.  Rows start on
  // 256-byte boundaries (the pitch is a multiple of 64 values).
  const int ic = i < L.pitch - 2 ? i : L.pitch - 2;
  const float *__restrict__ src = static_cast<const float *>(p.src);
  F2 h[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    int r = j - cy_of(a);
    r = r < 0 ? 0 : (r > L.ny - 1 ? L.ny - 1 : r);
    const float *row = src + (int64_t)a * L.plane + (int64_t)r * L.pitch;
    const float2 v = __ldg(reinterpret_cast<const float2 *>(row + ic));
    if (cx_of(a) == 0) {
      h[a] = vpair(v.x, v.y);
    } else if (cx_of(a) > 0) {  // sources i - 1 (the left lane's second value), i
      float left = __shfl_up_sync(0xffffffffu, v.y, 1);
      if (lane == 0) left = ic >= 1 ? __ldg(row + ic - 1) : 0.f;
      h[a] = vpair(left, v.x);
    } else {  // sources i + 1, i + 2 (the right lane's first value)
      float right = __shfl_down_sync(0xffffffffu, v.x, 1);
      if (lane == 31) right = ic + 2 < L.pitch ? __ldg(row + ic + 2) : 0.f;
      h[a] = vpair(v.y, right);
    }
  }
  {
    const ForceRegion reg = *p.reg_src;
    if (ti >= reg.ti0 && ti <= reg.ti1 && tj >= reg.tj0 && tj <= reg.tj1) return;  // special kernel
  }
  if (j < 1 || j > L.ny - 2) return;  // edge rows: special kernel
  const bool ok0 = i >= 1 && i <= L.nx - 2, ok1 = i + 1 <= L.nx - 2;
  if (!ok0 && !ok1) return;
  F2 o[9];
  const F2 rho = update_fluid<float, kForce>(L, Consts<float>(p), h, o);
  float *dst = static_cast<float *>(p.dst) + (int64_t)j * L.pitch + i;
  if (ok0 && ok1) {
#pragma unroll
    for (int a = 0; a < 9; ++a)
      *reinterpret_cast<float2 *>(dst + (int64_t)a * L.plane) = make_float2(vlo(o[a]), vhi(o[a]));
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      if (ok0) dst[(int64_t)a * L.plane] = vlo(o[a]);
      if (ok1) dst[(int64_t)a * L.plane + 1] = vhi(o[a]);
    }
  }
  if ((ok0 && rho_bad(vlo(rho))) || (ok1 && rho_bad(vhi(rho)))) atomicOr(p.status, kStatusUnstable);
}

// ---------------------------------------------------------------------------
// bulk kernel for 16-bit storage: eight nodes per thread.  HBM stays busy
// only with enough bytes in flight per SM, and a thread holds what it loads
// in registers until it is used; with 2-byte values the registers, not the
// threads, cap what is in flight.  So each thread takes the nodes i .. i+7
// (i a multiple of 8) of a tile row, a half-warp per row and one warp per
// 128 x 2 tile: one aligned 128-bit load per plane brings eight values, kept
// packed (four 32-bit words per plane, 36 registers for 8 nodes: 144 bytes
// in flight per thread).  For c_x = +1 (sources i-1 .. i+6) and c_x = -1
// (sources i+1 .. i+8) the value beyond the thread's eight comes from the
// next lane of the half-warp by a shuffle (one extra 2-byte load at the
// row's edge) and a funnel shift realigns the words.  The nodes are collided
// two at a time in packed f32x2 (collide2) and leave in one 128-bit store per
// plane.  96 registers, 20 one-warp blocks per SM: about 90 KB in flight per
// SM.
// ---------------------------------------------------------------------------
template <typename S>
struct Pair16;
template <>
struct Pair16<__half> {
  static __device__ __forceinline__ float lo(uint32_t w) {
    return __half2float(__ushort_as_half((unsigned short)(w & 0xffffu)));
  }
  static __device__ __forceinline__ float hi(uint32_t w) {
    return __half2float(__ushort_as_half((unsigned short)(w >> 16)));
  }
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
};
template <>
struct Pair16<__nv_bfloat16> {
  static __device__ __forceinline__ float lo(uint32_t w) { return __uint_as_float(w << 16); }
  static __device__ __forceinline__ float hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }
  static __device__ __forceinline__ uint32_t pack(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
};

// (lo half of b, hi half of a) -> the pair starting one value later
__device__ __forceinline__ uint32_t shift16(uint32_t a, uint32_t b) {
  return __funnelshift_r(a, b, 16);
}

// the update of the node pair whose pre-collision values are the packed
// words w[a], nodes `node` and `node + 1`; returns the packed post-collision
// words (rounded to nearest, or stochastically with the level's bits) and rho
template <typename S, bool kForce, bool kSR>
__device__ __forceinline__ F2 collide_pair16(const StepArgs &p, const uint32_t (&w)[9],
                                             uint32_t (&out)[9], uint32_t level, uint32_t node) {
  using P = Pair16<S>;
  F2 h[9];
#pragma unroll
  for (int a = 0; a < 9; ++a) h[a] = vpair(P::lo(w[a]), P::hi(w[a]));
  F2 o[9];
  const F2 rho = update_fluid<S, kForce>(p.L, Consts<float>(p), h, o);
  if constexpr (kSR) {
    const SrBits r(level, node >> 1);
#pragma unroll
    for (int a = 0; a < 9; ++a) out[a] = Stochastic<S>::pair(vlo(o[a]), vhi(o[a]), r.word(a));
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) out[a] = P::pack(vlo(o[a]), vhi(o[a]));
  }
  return rho;
}

template <typename S, bool kForce, bool kSR, int kMinBlocks>
__global__ void __launch_bounds__(32, kMinBlocks) bulk16_kernel(const StepArgs p) {
  const int ti = blockIdx.x, tj = blockIdx.y;
  const Lattice &L = p.L;
  const int lane = threadIdx.x & 15;               // lane within the tile row
  const int i = ti * kTileX + 8 * lane;            // the thread's nodes i .. i + 7
  const int j = tj * kTileY + (threadIdx.x >> 4);  // half-warp per tile row
  // every lane loads from inside its row (clamped), so that the shuffles see
  // all lanes; results of clamped lanes are never stored.  Rows and planes
  // start on 16-byte boundaries (the pitch is a multiple of 64 values).
  const int ic = i < L.pitch - 8 ? i : L.pitch - 8;
  const S *__restrict__ src = static_cast<const S *>(p.src);
  uint32_t w[4][9];  // sources of the node pairs (i, i+1) .. (i+6, i+7), packed
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    int r = j - cy_of(a);
    r = r < 0 ? 0 : (r > L.ny - 1 ? L.ny - 1 : r);
    const S *row = src + (int64_t)a * L.plane + (int64_t)r * L.pitch;
    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(row + ic));
    if (cx_of(a) == 0) {
      w[0][a] = v.x;
      w[1][a] = v.y;
      w[2][a] = v.z;
      w[3][a] = v.w;
    } else if (cx_of(a) > 0) {  // sources i-1 (the left lane's last value) .. i+6
      uint32_t left = __shfl_up_sync(0xffffffffu, v.w, 1, 16);
      if (lane == 0)
        left = ic >= 1 ? ((uint32_t)__ldg(reinterpret_cast<const unsigned short *>(row + ic - 1)) << 16)
                       : 0u;
      w[0][a] = shift16(left, v.x);
      w[1][a] = shift16(v.x, v.y);
      w[2][a] = shift16(v.y, v.z);
      w[3][a] = shift16(v.z, v.w);
    } else {  // sources i+1 .. i+8 (the right lane's first value)
      uint32_t right = __shfl_down_sync(0xffffffffu, v.x, 1, 16);
      if (lane == 15)
        right = ic + 8 < L.pitch ? (uint32_t)__ldg(reinterpret_cast<const unsigned short *>(row + ic + 8))
                                 : 0u;
      w[0][a] = shift16(v.x, v.y);
      w[1][a] = shift16(v.y, v.z);
      w[2][a] = shift16(v.z, v.w);
      w[3][a] = shift16(v.w, right);
    }
  }
  {
    const ForceRegion reg = *p.reg_src;
    if (ti >= reg.ti0 && ti <= reg.ti1 && tj >= reg.tj0 && tj <= reg.tj1) return;  // special kernel
  }
  if (j < 1 || j > L.ny - 2) return;  // edge rows: special kernel
  const int n_ok_lo = i >= 1 ? 0 : 1;                    // first node to store
  const int n_ok_hi = L.nx - 2 - i < 7 ? L.nx - 2 - i : 7;  // last node to store
  if (n_ok_hi < n_ok_lo) return;
  uint32_t out[4][9];
  bool bad = false;
  const uint32_t level = kSR ? sr_level(p) : 0u;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const F2 r = collide_pair16<S, kForce, kSR>(p, w[k], out[k], level,
                                           (uint32_t)((int64_t)j * L.pitch + i + 2 * k));
    bad |= (2 * k >= n_ok_lo && 2 * k <= n_ok_hi && rho_bad(vlo(r))) ||
           (2 * k + 1 >= n_ok_lo && 2 * k + 1 <= n_ok_hi && rho_bad(vhi(r)));
  }
  S *dst = static_cast<S *>(p.dst) + (int64_t)j * L.pitch + i;
  if (n_ok_lo == 0 && n_ok_hi == 7) {
#pragma unroll
    for (int a = 0; a < 9; ++a)
      *reinterpret_cast<uint4 *>(dst + (int64_t)a * L.plane) =
          make_uint4(out[0][a], out[1][a], out[2][a], out[3][a]);
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      unsigned short *d = reinterpret_cast<unsigned short *>(dst + (int64_t)a * L.plane);
#pragma unroll
      for (int n = 0; n < 8; ++n)
        if (n >= n_ok_lo && n <= n_ok_hi)
          d[n] = (unsigned short)(n & 1 ? out[n >> 1][a] >> 16 : out[n >> 1][a] & 0xffffu);
    }
  }
  if (bad) atomicOr(p.status, kStatusUnstable);
}

// The same update with four nodes per thread (one 64-bit load per plane, one
// warp per tile row, 80 registers): a variant for the tuner.
template <typename S, bool kForce, bool kSR>
__global__ void __launch_bounds__(32 * kTileY, 12) bulk16x4_kernel(const StepArgs p) {
  const int ti = blockIdx.x, tj = blockIdx.y;
  const Lattice &L = p.L;
  const int lane = threadIdx.x;
  const int i = ti * kTileX + 4 * lane;  // the thread's nodes i .. i + 3
  const int j = tj * kTileY + threadIdx.y;
  // every lane loads from inside its row (clamped), so that the shuffles see
  // all 32 lanes; results of clamped lanes are never stored.  Rows and planes
  // start on 8-byte boundaries (the pitch is a multiple of 64 values).
  const int ic = i < L.pitch - 4 ? i : L.pitch - 4;
  const S *__restrict__ src = static_cast<const S *>(p.src);
  uint32_t wa[9], wb[9];  // sources of nodes (i, i+1) and (i+2, i+3), packed
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    int r = j - cy_of(a);
    r = r < 0 ? 0 : (r > L.ny - 1 ? L.ny - 1 : r);
    const S *row = src + (int64_t)a * L.plane + (int64_t)r * L.pitch;
    const uint2 w = __ldg(reinterpret_cast<const uint2 *>(row + ic));
    if (cx_of(a) == 0) {
      wa[a] = w.x;
      wb[a] = w.y;
    } else if (cx_of(a) > 0) {  // sources i-1 (the left lane's last value) .. i+2
      uint32_t left = __shfl_up_sync(0xffffffffu, w.y, 1);
      if (lane == 0)
        left = ic >= 1 ? ((uint32_t)__ldg(reinterpret_cast<const unsigned short *>(row + ic - 1)) << 16)
                       : 0u;
      wa[a] = shift16(left, w.x);
      wb[a] = shift16(w.x, w.y);
    } else {  // sources i+1 .. i+4 (the right lane's first value)
      uint32_t right = __shfl_down_sync(0xffffffffu, w.x, 1);
      if (lane == 31)
        right = ic + 4 < L.pitch ? (uint32_t)__ldg(reinterpret_cast<const unsigned short *>(row + ic + 4))
                                 : 0u;
      wa[a] = shift16(w.x, w.y);
      wb[a] = shift16(w.y, right);
    }
  }
  {
    const ForceRegion reg = *p.reg_src;
    if (ti >= reg.ti0 && ti <= reg.ti1 && tj >= reg.tj0 && tj <= reg.tj1) return;  // special kernel
  }
  if (j < 1 || j > L.ny - 2) return;  // edge rows: special kernel
  bool ok[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) ok[k] = i + k >= 1 && i + k <= L.nx - 2;
  if (!ok[0] && !ok[1] && !ok[2] && !ok[3]) return;
  S *dst = static_cast<S *>(p.dst) + (int64_t)j * L.pitch + i;
  // the two pairs one after the other, each stored as soon as it is done
  bool bad = false;
  const uint32_t level = kSR ? sr_level(p) : 0u;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    uint32_t o[9];
    const F2 r = collide_pair16<S, kForce, kSR>(p, half ? wb : wa, o, level,
                                           (uint32_t)((int64_t)j * L.pitch + i + 2 * half));
    const bool ok0 = ok[2 * half], ok1 = ok[2 * half + 1];
    S *d2 = dst + 2 * half;
    if (ok0 && ok1) {
#pragma unroll
      for (int a = 0; a < 9; ++a) *reinterpret_cast<uint32_t *>(d2 + (int64_t)a * L.plane) = o[a];
    } else {
#pragma unroll
      for (int a = 0; a < 9; ++a) {
        unsigned short *d = reinterpret_cast<unsigned short *>(d2 + (int64_t)a * L.plane);
        if (ok0) d[0] = (unsigned short)(o[a] & 0xffffu);
        if (ok1) d[1] = (unsigned short)(o[a] >> 16);
      }
    }
    bad |= (ok0 && rho_bad(vlo(r))) || (ok1 && rho_bad(vhi(r)));
  }
  if (bad) atomicOr(p.status, kStatusUnstable);
}

#include "pair.cuh"

template <typename S, bool kGather>
cudaError_t special_t(const StepArgs &a, cudaStream_t s) {
  const int tiles = a.all_tiles ? a.ntiles_x * a.ntiles_y : a.edge_blocks + a.region_slots;
  const int blocks = (a.sim_blocks + tiles + (a.finalize_prev || a.raster ? 1 : 0)) * kSlices<S>;
  constexpr int kBlock = kThreads / kSlices<S>;
  if (a.raster || sizeof(S) == 8)
    special_kernel<S, kGather, 1, true><<<blocks, kBlock, 0, s>>>(a);
  else if (a.uncapped)
    special_kernel<S, kGather, 1, false><<<blocks, kBlock, 0, s>>>(a);
  else
    special_kernel<S, kGather, kSpecialMinBlocks<S>, false><<<blocks, kBlock, 0, s>>>(a);
  return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(64) finalize_kernel(const StepArgs p) {
  __shared__ BodyState moving;
  if (!p.raster) {
    finalize<T>(p);
    return;
  }
  // a moving body: into the state and region that the next launch starts from;
  // all its sums are cleared, so that it starts at any of them
  if (threadIdx.x >= 32) return;
  record_moving<T>(p, moving, const_cast<ForceRegion *>(p.reg_src));
  if (threadIdx.x < kAccWords) {
    p.acc_prev[threadIdx.x] = 0ull;
    p.acc[threadIdx.x] = 0ull;
    p.acc_next[threadIdx.x] = 0ull;
  }
}

// chi of a moving body on the force-region tiles, tile by tile as the special
// kernel rasterises it
__global__ void __launch_bounds__(kThreads) mask_kernel(const StepArgs p) {
  __shared__ TileMask tm;
  const ForceRegion reg = *p.reg_src;
  const int k = blockIdx.x;
  if (k >= reg.count) return;
  const int rw = reg.ti1 - reg.ti0 + 1;
  const int ti = reg.ti0 + k % rw, tj = reg.tj0 + k / rw;
  tile_solid(p, *p.body_src, ti, tj, Slice{0, kThreads}, tm);
  __syncthreads();
  const int tx = threadIdx.x % kTileX, ty = threadIdx.x / kTileX;
  const int i = ti * kTileX + tx, j = tj * kTileY + ty;
  if (i < p.L.nx && j < p.L.ny)
    p.chi[(int64_t)j * p.L.pitch + i] = tile_mask_byte(p.L, tm, i, j, tx, ty);
}

template <typename S, bool kForce, bool kSR>
cudaError_t bulk16_v(int variant, const StepArgs &a, cudaStream_t s) {
  static_assert(kTileX == 8 * 16 && kTileY == 2, "bulk16_kernel maps a tile onto one warp");
  const dim3 grid(a.ntiles_x, a.ntiles_y);
  switch (variant) {
    case 0: bulk16_kernel<S, kForce, kSR, 20><<<grid, dim3(32), 0, s>>>(a); break;  // 8 nodes, 96 regs
    case 1: bulk16_kernel<S, kForce, kSR, 16><<<grid, dim3(32), 0, s>>>(a); break;  // 8 nodes, 126 regs
    case 2: bulk16x4_kernel<S, kForce, kSR><<<grid, dim3(32, kTileY), 0, s>>>(a); break;  // 4 nodes
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <typename S, bool kForce>
cudaError_t bulk_v(int variant, const StepArgs &a, cudaStream_t s) {
  if constexpr (sizeof(S) == 2) {
    return a.sr ? bulk16_v<S, kForce, true>(variant, a, s) : bulk16_v<S, kForce, false>(variant, a, s);
  } else if constexpr (sizeof(S) == 4) {
    const int k = variant == 0 ? 1 : (variant == 1 ? 2 : 4);  // tiles per block
    if (variant < 0 || variant > 2) return cudaErrorInvalidValue;
    const dim3 grid(a.ntiles_x, (a.ntiles_y + k - 1) / k), block(kTileX / 2, kTileY * k);
    if (k == 1) bulk32x2_kernel<kForce, 1><<<grid, block, 0, s>>>(a);
    else if (k == 2) bulk32x2_kernel<kForce, 2><<<grid, block, 0, s>>>(a);
    else bulk32x2_kernel<kForce, 4><<<grid, block, 0, s>>>(a);
  } else {
    const int k = variant == 0 ? 1 : (variant == 1 ? 2 : 4);  // tiles per block
    if (variant < 0 || variant > 2) return cudaErrorInvalidValue;
    const dim3 grid(a.ntiles_x, (a.ntiles_y + k - 1) / k), block(kTileX, kTileY * k);
    if (k == 1) bulk_kernel<S, kForce, 1><<<grid, block, 0, s>>>(a);
    else if (k == 2) bulk_kernel<S, kForce, 2><<<grid, block, 0, s>>>(a);
    else bulk_kernel<S, kForce, 4><<<grid, block, 0, s>>>(a);
  }
  return cudaGetLastError();
}

template <typename S>
cudaError_t bulk_t(int variant, const StepArgs &a, cudaStream_t s) {
  return a.L.has_bf ? bulk_v<S, true>(variant, a, s) : bulk_v<S, false>(variant, a, s);
}

}  // namespace

cudaError_t launch_special(int dtype, bool gather, const StepArgs &a, cudaStream_t s) {
  switch (dtype) {
    case VPLBM_F64: return gather ? special_t<double, true>(a, s) : special_t<double, false>(a, s);
    case VPLBM_F32: return gather ? special_t<float, true>(a, s) : special_t<float, false>(a, s);
    case VPLBM_F16_OFS: return gather ? special_t<__half, true>(a, s) : special_t<__half, false>(a, s);
    case VPLBM_BF16_OFS:
      return gather ? special_t<__nv_bfloat16, true>(a, s) : special_t<__nv_bfloat16, false>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_pair(int dtype, const StepArgs &a, cudaStream_t s) {
  switch (dtype) {
    case VPLBM_F32: return pair_t<float>(a, s);
    case VPLBM_F16_OFS: return pair_t<__half>(a, s);
    case VPLBM_BF16_OFS: return pair_t<__nv_bfloat16>(a, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_finalize(int dtype, const StepArgs &a, cudaStream_t s) {
  if (dtype == VPLBM_F64)
    finalize_kernel<double><<<1, 64, 0, s>>>(a);
  else
    finalize_kernel<float><<<1, 64, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_mask(const StepArgs &a, cudaStream_t s) {
  mask_kernel<<<a.region_slots, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_sim_cache(const StepArgs &a, cudaStream_t s) {
  if (a.n_sim <= 0) return cudaSuccess;
  sim_cache_kernel<<<(a.n_sim + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_bulk(int dtype, int variant, const StepArgs &a, cudaStream_t s) {
  switch (dtype) {
    case VPLBM_F64: return bulk_t<double>(variant, a, s);
    case VPLBM_F32: return bulk_t<float>(variant, a, s);
    case VPLBM_F16_OFS: return bulk_t<__half>(variant, a, s);
    case VPLBM_BF16_OFS: return bulk_t<__nv_bfloat16>(variant, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace vplbm
