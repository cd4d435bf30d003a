// pair.cuh -- two time steps in one pass over the populations (FP32 compute:
// FP32 and 16-bit storage; a fixed body or none).  Included by step.cu, whose
// node update, MEM and SIM terms it uses.
//
// A step reads and writes every population once, 72 bytes per node in FP32,
// and the single-step kernels run at the copy rate of HBM: only fewer passes
// make the step faster.  Two steps per pass halve the traffic at the price of
// recomputing the first step on a one-node rim of every tile.  One launch
// holds, on disjoint nodes,
//   * the special blocks, first in the grid: the SIM points of both levels,
//     the frame of the two outermost rows and columns, and the box around the
//     body; one more block finalizes the previous launch's force sums;
//   * the bulk blocks: all other nodes, whose two steps are plain fluid
//     updates.
// Every value between the two steps is rounded to the storage type as a store
// and a load would, so a pair gives the bits of two single steps.

// ---------------------------------------------------------------------------
// pair bulk kernel.  A warp takes a strip of 64 nodes, two per lane, and
// marches up pair_rows rows: the first step of row q, then the second step of
// row q - 1, whose sources are the first step's rows q - 2 .. q.  A population
// is needed one row later (c_y = 0), two rows later (c_y = 1) or at once
// (c_y = -1), so nine node pairs per lane hold everything between the steps:
// no barriers and no exchange through shared memory.  The +-x sources come
// from the neighbouring lanes by shuffles; the outermost lanes are the rim in
// x (30 of 32 lanes store).
//
// In FP32 the kernel is bound by HBM, which wants many bytes in flight: each
// lane copies its own cells two rows ahead into a ring in shared memory
// (cp.async), so that what is in flight holds no registers.  In 16-bit storage
// it is bound by the FMA pipe (62 % busy) and one row prefetched in registers is
// enough.  Measured, us per step and lattice, five 2048 x 1024 lattices in FP32:
// 22.9 in single steps (0.97 of the copy rate), 14.0 with the next row held in
// registers, 13.15 with a ring of three rows and 13.8 with one of four (shared
// memory taken from L1), 13.06 with four blocks per SM (96 registers, which five
// need, spill in the special blocks: 13.15), 12.8 with the warps numbered over the
// whole grid (kPairWarps); 11.3 is the traffic of a pair at the copy rate.
// ---------------------------------------------------------------------------
template <typename S>
struct Cell;  // a lane's two nodes of one plane in storage form
template <>
struct Cell<float> {
  using Raw = uint2;
  static __device__ __forceinline__ F2 pair(Raw v) {
    return vpair(__uint_as_float(v.x), __uint_as_float(v.y));
  }
  // the pair one node to the left (its first node from the left lane), ...
  static __device__ __forceinline__ F2 from_left(Raw v) {
    return vpair(__uint_as_float(__shfl_up_sync(kFull, v.y, 1)), __uint_as_float(v.x));
  }
  // ... and one to the right
  static __device__ __forceinline__ F2 from_right(Raw v) {
    return vpair(__uint_as_float(v.y), __uint_as_float(__shfl_down_sync(kFull, v.x, 1)));
  }
  static __device__ __forceinline__ Raw pack(F2 v) {
    return make_uint2(__float_as_uint(vlo(v)), __float_as_uint(vhi(v)));
  }
};
template <typename S>
struct Cell16 {
  using Raw = uint32_t;
  using P = Pair16<S>;
  static __device__ __forceinline__ F2 pair(Raw v) { return vpair(P::lo(v), P::hi(v)); }
  static __device__ __forceinline__ F2 from_left(Raw v) {
    return pair(shift16(__shfl_up_sync(kFull, v, 1), v));
  }
  static __device__ __forceinline__ F2 from_right(Raw v) {
    return pair(shift16(v, __shfl_down_sync(kFull, v, 1)));
  }
  static __device__ __forceinline__ Raw pack(F2 v) { return P::pack(vlo(v), vhi(v)); }
};
template <>
struct Cell<__half> : Cell16<__half> {};
template <>
struct Cell<__nv_bfloat16> : Cell16<__nv_bfloat16> {};

// pre-collision values of the lane's nodes from the cells of the nine source
// planes (rows already chosen)
template <typename S>
__device__ __forceinline__ void cell_pull(const typename Cell<S>::Raw (&v)[9], F2 (&h)[9]) {
#pragma unroll
  for (int a = 0; a < 9; ++a)
    h[a] = cx_of(a) == 0  ? Cell<S>::pair(v[a])
           : cx_of(a) > 0 ? Cell<S>::from_left(v[a])
                          : Cell<S>::from_right(v[a]);
}

// A density is good (finite and positive) when its bits less one, unsigned, are
// below this: the kernel keeps the largest value seen and looks at it once.
constexpr uint32_t kRhoBits = 0x7f7fffffu;

// the fluid update of the lane's nodes: post-collision values in storage form;
// node0: linear index of the first node (the stochastic bits' key); watch: bits
// of the nodes whose density is looked at
template <typename S, bool kForce, bool kSR>
__device__ __forceinline__ void cell_update(const StepArgs &p, const Consts<float> &cst,
                                            const F2 (&h)[9], typename Cell<S>::Raw (&o)[9],
                                            uint32_t level, uint32_t node0, uint32_t watch,
                                            uint32_t &worst) {
  F2 q[9];
  const F2 rho = update_fluid<S, kForce>(p.L, cst, h, q);
  if (watch & 1u) worst = max(worst, __float_as_uint(vlo(rho)) - 1u);
  if (watch & 2u) worst = max(worst, __float_as_uint(vhi(rho)) - 1u);
  if constexpr (kSR) {
    const SrBits r(level, node0 >> 1);
#pragma unroll
    for (int a = 0; a < 9; ++a) o[a] = Stochastic<S>::pair(vlo(q[a]), vhi(q[a]), r.word(a));
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) o[a] = Cell<S>::pack(q[a]);
  }
}

// Warps per block, numbered over the whole grid (strips of a run of rows, then of
// the next): with a block's four strips side by side the last block of a run held
// up to three idle warps (1024 x 512, 17 strips: 5.8 us per step, 4.9 without;
// 3614 x 1946, 61 strips: 45.5 and 44.9; 8192 x 4096, 137 strips: 204.2 and 202.3).
constexpr int kPairWarps = 4;
constexpr int kPairStore = 60;   // nodes a warp stores per row
constexpr int kPairStages = 3;   // rows of the ring
constexpr int kPairAhead = kPairStages - 1;
constexpr int kPairMinBlocks = 4;
// 16-bit rows are small enough to be prefetched in registers, one row ahead
template <typename S>
constexpr bool kRing = sizeof(S) == 4;

// (the memory clobber keeps the ring's reads and later copies into the same stage
// in program order)
template <typename Raw>
__device__ __forceinline__ void copy_async(Raw *smem, const void *global) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem)),
               "l"(global), "n"(sizeof(Raw))
               : "memory");
}

template <typename S, bool kForce, bool kSR>
__device__ __forceinline__ void pair_bulk(
    const StepArgs &p, int strip, int run,
    typename Cell<S>::Raw (*ring)[9][32 * kPairWarps]) {
  using Raw = typename Cell<S>::Raw;
  const Lattice &L = p.L;
  const int lane = threadIdx.x & 31;
  const int i = 2 + strip * kPairStore + 2 * (lane - 1);  // the lane's nodes i, i + 1
  const int r0 = 2 + run * p.pair_rows;
  if (r0 >= L.ny - 2) return;  // the warp lies beyond the last run of rows
  const int r1 = min(r0 + p.pair_rows, L.ny - 2);
  // the nodes that the lane stores (bits), outside / inside the rows of the
  // box (its columns start and end on pairs)
  uint32_t own = i <= L.nx - 3 ? (i + 1 <= L.nx - 3 ? 3u : 1u) : 0u;
  if (lane == 0 || lane == 31) own = 0;
  const bool in_box = i >= p.box[0] && i <= p.box[1];
  if (r0 >= p.box[2] && r1 - 1 <= p.box[3] && __all_sync(kFull, in_box || !own)) return;
  // lanes beyond the row load inside it.  Addresses are a base per plane, the
  // same for the whole grid, and one 32-bit byte offset per lane and row (a
  // plane holds fewer than 2^30 nodes: api.cu, pair_plan).
  const uint32_t row_bytes = (uint32_t)L.pitch * (uint32_t)sizeof(S);
  const char *const src0 = static_cast<const char *>(p.src);
  char *const dst0 = static_cast<char *>(p.dst);
  const int64_t plane = L.plane * (int64_t)sizeof(S);
  const uint32_t col_in = (uint32_t)(min(i, L.pitch - 2) * (int)sizeof(S));
  const Consts<float> cst(p);
  const uint32_t level1 = kSR ? sr_level(p, 0) : 0u, level2 = kSR ? sr_level(p, 1) : 0u;
  uint32_t worst = 0;
  Raw e[9] = {}, late[3] = {};  // e: sources of the second step; late: c_y = 1, one row old
  auto cell_of = [&](int a, int q) {  // the cell of plane a that row q pulls from
    return reinterpret_cast<const Raw *>(src0 + (a * plane - cy_of(a) * (int64_t)row_bytes) +
                                         ((uint32_t)q * row_bytes + col_in));
  };
  auto fetch = [&](int q) {  // row q into the ring
    if (q <= r1) {
#pragma unroll
      for (int a = 0; a < 9; ++a)
        copy_async(&ring[(uint32_t)q % kPairStages][a][threadIdx.x], cell_of(a, q));
    }
    asm volatile("cp.async.commit_group;");
  };
  Raw next[9];
  if constexpr (kRing<S>) {
#pragma unroll
    for (int k = 0; k < kPairAhead; ++k) fetch(r0 - 1 + k);
  } else {
#pragma unroll
    for (int a = 0; a < 9; ++a) next[a] = __ldg(cell_of(a, r0 - 1));
  }
#pragma unroll 1
  for (int q = r0 - 1; q <= r1; ++q) {
    F2 h[9];
    if constexpr (kRing<S>) {
      fetch(q + kPairAhead);
      asm volatile("cp.async.wait_group %0;" ::"n"(kPairAhead) : "memory");
      Raw v[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) v[a] = ring[(uint32_t)q % kPairStages][a][threadIdx.x];
      cell_pull<S>(v, h);
    } else {
      cell_pull<S>(next, h);
      if (q < r1) {
#pragma unroll
        for (int a = 0; a < 9; ++a) next[a] = __ldg(cell_of(a, q + 1));
      }
    }
    Raw o[9];
    const uint32_t first = (uint32_t)q * (uint32_t)L.pitch + (uint32_t)i;
    const uint32_t st1 = q < r0 || q >= r1 || (in_box && q >= p.box[2] && q <= p.box[3]) ? 0u : own;
    cell_update<S, kForce, kSR>(p, cst, h, o, level1, first, st1, worst);
    // populations that move down are needed in this row's place at once
    e[4] = o[4];
    e[7] = o[7];
    e[8] = o[8];
    if (q > r0) {
      Raw o2[9];
      cell_pull<S>(e, h);
      const uint32_t st = in_box && q - 1 >= p.box[2] && q - 1 <= p.box[3] ? 0u : own;
      cell_update<S, kForce, kSR>(p, cst, h, o2, level2, first - (uint32_t)L.pitch, st, worst);
      const uint32_t off = (uint32_t)(q - 1) * row_bytes + (uint32_t)i * (uint32_t)sizeof(S);
      if (st == 3u) {
#pragma unroll
        for (int a = 0; a < 9; ++a) *reinterpret_cast<Raw *>(dst0 + a * plane + off) = o2[a];
      } else if (st) {  // the first node alone
#pragma unroll
        for (int a = 0; a < 9; ++a)
          *reinterpret_cast<S *>(dst0 + a * plane + off) = *reinterpret_cast<const S *>(&o2[a]);
      }
    }
    e[0] = o[0];
    e[1] = o[1];
    e[3] = o[3];
    e[2] = late[0];
    e[5] = late[1];
    e[6] = late[2];
    late[0] = o[2];
    late[1] = o[5];
    late[2] = o[6];
  }
  if (worst >= kRhoBits) atomicOr(p.status, kStatusUnstable);
}

// ---------------------------------------------------------------------------
// special blocks.  A block takes a tile of 128 nodes, one per thread: the first
// step on all of them into shared memory, the second on the tile without its
// one-node rim.  Box tiles are 16 x 8 (penalization and the MEM and
// volume-integral terms of both levels), frame tiles 32 x 4 along the rows and
// 4 x 32 along the columns (side conditions; fluid only: the box keeps clear of
// the frame).  SIM of the first level reads the stored field as single steps
// do; SIM of the second level recomputes the nine populations that stream into
// a sampled node, one lane each, three points per warp.  These blocks are
// latency-bound and few, and share the SMs with the bulk blocks: the update is
// in the code once, in a loop over the two steps (or over a point's sampled
// nodes), so that they stay in the instruction cache.
// ---------------------------------------------------------------------------
constexpr int kPairThreads = 32 * kPairWarps;
constexpr int kBoxW = 16, kBoxH = 8;      // box tile with its rim
constexpr int kFrameL = 32, kFrameD = 4;  // frame tile with its rim: length, depth
constexpr int kSimGroups = 3;             // SIM points per warp, second level
static_assert(kBoxW * kBoxH == kPairThreads && kFrameL * kFrameD == kPairThreads, "one node per thread");

// the nine populations of a node after the first step, in storage precision,
// as the second step reads them back
template <typename S, bool kSR>
__device__ __forceinline__ void stored_pops(float (&o)[9], uint32_t level, uint32_t node) {
  if constexpr (sizeof(S) == 2) {
    const SrBits r(level, node >> 1);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      S t;
      store_pop<S, kSR>(&t, o[a], &r, a, node);
      if constexpr (std::is_same<S, __half>::value)
        o[a] = __half2float(t);
      else
        o[a] = __bfloat162float(t);
    }
  }
}

// the first step's tile in shared memory, read by unwrapped node coordinates
struct TileSrc {
  const float (*post)[kPairThreads];
  int i0, j0, log_w;
  __device__ __forceinline__ float operator()(int a, int i, int j) const {
    return post[a][((j - j0) << log_w) + (i - i0)];
  }
};

struct PairGrid {
  int sim1, sim2, frame_x, frame_y, box_x, box_y, special;
};
__host__ __device__ inline PairGrid pair_grid(const StepArgs &p) {
  PairGrid g{};
  if (p.sim_blocks) {
    g.sim1 = (p.n_sim + kPairThreads - 1) / kPairThreads;
    g.sim2 = (p.n_sim + kPairWarps * kSimGroups - 1) / (kPairWarps * kSimGroups);
  }
  const int len = kFrameL - 2;
  g.frame_x = (p.L.nx + len - 1) / len;      // tiles of each pair of rows
  g.frame_y = (p.L.ny - 4 + len - 1) / len;  // tiles of each pair of columns
  if (p.box[1] >= p.box[0]) {
    g.box_x = (p.box[1] - p.box[0] + kBoxW - 2) / (kBoxW - 2);
    g.box_y = (p.box[3] - p.box[2] + kBoxH - 2) / (kBoxH - 2);
  }
  g.special = g.sim2 + g.box_x * g.box_y + 2 * g.frame_x + 2 * g.frame_y + g.sim1 +
              (p.finalize_prev ? 1 : 0);
  return g;
}

template <typename S, bool kForce, bool kSR>
__device__ __forceinline__ void pair_special(const StepArgs &p, const PairGrid &g, int b,
                                             float (*post)[kPairThreads],
                                             float (*old)[kPairThreads], LinkList<float> *list) {
  const Lattice &L = p.L;
  const int tid = threadIdx.x, lane = tid & 31;
  const BodyState *body = p.body_src;
  const S *__restrict__ src = static_cast<const S *>(p.src);
  const float *prev = static_cast<const float *>(p.prev_src);
  const Consts<float> cst(p);
  // ---- what the thread's node is ----
  const bool sim2 = b < g.sim2;
  const bool frame = !sim2 && b >= g.sim2 + g.box_x * g.box_y;
  if (b >= g.special - (p.finalize_prev ? 1 : 0)) {
    finalize<float>(p);
    return;
  }
  if (b >= g.sim2 + g.box_x * g.box_y + 2 * g.frame_x + 2 * g.frame_y) {
    // SIM of the first level
    const int q = (b - (g.special - (p.finalize_prev ? 1 : 0) - g.sim1)) * kPairThreads + tid;
    FixAcc<float> acc;
    bool missing = false;
    if (q < p.n_sim) acc = sim_point<S, true>(p, src, *body, q, missing);
    if (__any_sync(kFull, missing) && lane == 0) atomicOr(p.status, kStatusSimMissing);
    warp_add(acc, p.acc, 3);
    return;
  }
  int i = 0, j = 0, log_w = 0, i0 = 0, j0 = 0, iters = 2;
  bool active = false, own = false;  // updated in the first step; in the second
  const SimPoint *sp = nullptr;
  const int dir = lane % 9, group = lane / 9;  // SIM of the second level: source node and point
  if (sim2) {
    const int q = (b * kPairWarps + (tid >> 5)) * kSimGroups + group;
    if (lane < 9 * kSimGroups && q < p.n_sim) sp = p.sim_pts + q;
    iters = __reduce_max_sync(kFull, sp ? sp->n_cand * (1 + p.sim_order) : 0);
  } else if (frame) {
    b -= g.sim2 + g.box_x * g.box_y;
    const int len = kFrameL - 2;
    const bool along_x = b < 2 * g.frame_x;
    int last;  // last node along the tile's length
    if (along_x) {
      const bool top = b >= g.frame_x;
      i0 = (top ? b - g.frame_x : b) * len - 1;
      j0 = (top ? L.ny - 2 : 0) - 1;
      log_w = 5;
      last = L.nx - 1;
    } else {
      b -= 2 * g.frame_x;
      const bool right = b >= g.frame_y;
      i0 = (right ? L.nx - 2 : 0) - 1;
      j0 = 2 + (right ? b - g.frame_y : b) * len - 1;
      log_w = 2;
      last = L.ny - 3;
    }
    const int ex = tid & ((1 << log_w) - 1), ey = tid >> log_w;
    i = i0 + ex;
    j = j0 + ey;
    own = along_x ? (ex >= 1 && ex < kFrameL - 1 && i <= last && ey >= 1 && ey < kFrameD - 1)
                  : (ey >= 1 && ey < kFrameL - 1 && j <= last && ex >= 1 && ex < kFrameD - 1);
    // rim nodes beyond a periodic side are the nodes there; beyond another
    // side, and past the last node's rim, there are none
    active = (along_x ? i <= last + 1 : j <= last + 1) &&
             (L.bc[0] == VPLBM_PERIODIC || (i >= 0 && i < L.nx)) &&
             (L.bc[2] == VPLBM_PERIODIC || (j >= 0 && j < L.ny));
  } else {
    b -= g.sim2;
    const int ex = tid & (kBoxW - 1), ey = tid / kBoxW;
    i = p.box[0] + (b % g.box_x) * (kBoxW - 2) + ex - 1;
    j = p.box[2] + (b / g.box_x) * (kBoxH - 2) + ey - 1;
    active = i <= p.box[1] + 1 && j <= p.box[3] + 1;
    own = ex >= 1 && ex < kBoxW - 1 && ey >= 1 && ey < kBoxH - 1 && i <= p.box[1] && j <= p.box[3];
  }
  Stress<float> sig{0.f, 0.f, 0.f}, near{0.f, 0.f, 0.f};
  bool bad = false;
  uint8_t m = 0;
  uint32_t links = 0;
  if (!sim2 && !frame && active) {
    m = p.chi[(int64_t)j * L.pitch + i];
    links = node_links(p, i, j, m & kSolid, nullptr);
  }
#pragma unroll 1
  for (int it = 0; it < iters; ++it) {
    const bool second = !sim2 && it == 1;  // the second step of a tile
    int k = 0, qi = 0, qj = 0;
    bool next_node = false;  // SIM of first order: the node behind the sampled one
    if (sim2) {
      k = p.sim_order ? it >> 1 : it;
      next_node = p.sim_order && (it & 1);
      active = sp && k < sp->n_cand;
      if (active) {
        const uint32_t c = sp->cand[k];
        qi = (int)(c & 0xffffu);
        qj = (int)(c >> 16);
        if (next_node) {
          qi += cx_of(sp->dir);
          qj += cy_of(sp->dir);
        }
        i = qi - cx_of(dir);
        j = qj - cy_of(dir);
      }
    }
    float h[9], o[9], px, py;
    const int gi = frame ? wrap(i, L.nx) : i, gj = frame ? wrap(j, L.ny) : j;
    const int64_t node = (int64_t)gj * L.pitch + gi;
    // ---- pre-collision populations ----
    if (second) {
      if (own) {
        const int row = frame ? 1 << log_w : kBoxW;
        if (gi > 0 && gi < L.nx - 1 && gj > 0 && gj < L.ny - 1) {
#pragma unroll
          for (int a = 0; a < 9; ++a) h[a] = post[a][tid - cy_of(a) * row - cx_of(a)];
        } else {
          const TileSrc tile{post, i0, j0, log_w};
          const bool at_out = i == L.nx - 1;
          const bool outlet = at_out && L.bc[1] == VPLBM_OUTLET_CONVECTIVE;
          const bool free_out = at_out && L.bc[1] == VPLBM_OUTLET_FREE;
#pragma unroll
          for (int a = 0; a < 9; ++a) {
            const float f =
                gather_from<float>(tile, L, a, cx_of(a) < 0 && (outlet || free_out) ? i - 1 : i, j);
            // the convective condition of gather(), on the level before
            h[a] = cx_of(a) < 0 && outlet
                       ? (old[outlet_slot(a)][tid] + L.uc_f * f) / (1.0f + L.uc_f)
                       : f;
          }
          if (outlet) {
            float *pd = static_cast<float *>(p.prev_dst);
            pd[0 * L.ny + j] = h[3];
            pd[1 * L.ny + j] = h[6];
            pd[2 * L.ny + j] = h[7];
          }
        }
      }
    } else if (active) {
      if (gi > 0 && gi < L.nx - 1 && gj > 0 && gj < L.ny - 1) {
#pragma unroll
        for (int a = 0; a < 9; ++a)
          h[a] = Store<S>::ld(src + (int64_t)a * L.plane + node - cy_of(a) * L.pitch - cx_of(a));
      } else {
#pragma unroll
        for (int a = 0; a < 9; ++a) h[a] = gather(src, prev, L, a, gi, gj);
        old[0][tid] = h[3];
        old[1][tid] = h[6];
        old[2][tid] = h[7];
      }
    }
    // ---- the update ----
    const bool update = second ? own : active;
    if (update) {
      if (sim2) m = p.chi[node];
      bad |= update_node<S, kForce>(h, m, gi, gj, L, body, cst, o, px, py) && own;
    }
    __syncwarp();  // fluid and solid lanes meet again
    const uint32_t level = kSR ? sr_level(p, second ? 1 : 0) : 0u;
    if (sim2) {
      // the populations streaming into (qi, qj), exchanged within the group
      if (active) stored_pops<S, kSR>(o, level, (uint32_t)node);
      float v = o[0];
#pragma unroll
      for (int a = 1; a < 9; ++a)
        if (dir == a) v = o[a];
      Offsets<float> f;
#pragma unroll
      for (int a = 0; a < 9; ++a) f.h[a] = __shfl_sync(kFull, v, group * 9 + a);
      if (active) {
        const Stress<float> s3 = stress_of<float>(f, p);
        if (next_node) {
          if (!(p.chi[(int64_t)qj * L.pitch + qi] & kSolid))
            near = extrapolate<float>(*sp, body->xg, body->yg, qi - cx_of(sp->dir),
                                      qj - cy_of(sp->dir), near, s3);
        } else {
          near = s3;
        }
        if (next_node || !p.sim_order) {
          sig.xx = radd(sig.xx, near.xx);
          sig.xy = radd(sig.xy, near.xy);
          sig.yy = radd(sig.yy, near.yy);
        }
      }
      continue;
    }
    if (!frame) {
      // from the values before rounding
      unsigned long long *sums = second ? p.acc2 : p.acc;
      warp_add(mem_terms<float, true>(p, *body, o, i, j, m & kSolid, own ? links : 0u, list), sums, 0);
      FixAcc<float> vol;
      if (own && (m & kSolid)) vol = vol_terms<float>(BodyRef<float>(*body), i, j, px, py);
      warp_add(vol, sums, 6);
    }
    if (!second) {
      if (active) {
        stored_pops<S, kSR>(o, level, (uint32_t)node);
#pragma unroll
        for (int a = 0; a < 9; ++a) post[a][tid] = o[a];
      }
      __syncthreads();
    } else if (own) {
      S *dst = static_cast<S *>(p.dst);
      const SrBits r(level, (uint32_t)node >> 1);
#pragma unroll
      for (int a = 0; a < 9; ++a)
        store_pop<S, kSR>(dst + (int64_t)a * L.plane + node, o[a], &r, a, (uint32_t)node);
    }
  }
  if (sim2) {
    FixAcc<float> acc;
    if (sp && dir == 0 && sp->n_cand > 0) acc = sim_sum<float>(*sp, sig, sp->n_cand);
    warp_add(acc, p.acc2, 3);
    return;
  }
  if (__any_sync(kFull, bad) && lane == 0) atomicOr(p.status, kStatusUnstable);
}

template <typename S, bool kForce, bool kSR>
__global__ void __launch_bounds__(kPairThreads, kPairMinBlocks) pair_kernel(const StepArgs p) {
  using Raw = typename Cell<S>::Raw;
  constexpr size_t kPopBytes = 12 * kPairThreads * sizeof(float);
  constexpr size_t kTileBytes = kPopBytes + kPairWarps * sizeof(LinkList<float>);
  constexpr size_t kRingBytes = kRing<S> ? sizeof(Raw[kPairStages][9][kPairThreads]) : 0;
  __shared__ __align__(16) unsigned char smem[kRingBytes > kTileBytes ? kRingBytes : kTileBytes];
  const PairGrid g = pair_grid(p);
  const int b = blockIdx.x;
  if (kSR && b == 0 && threadIdx.x == 0) *p.rng_dst = *p.rng_src + 2ull;  // the next launch's counter
  if (b < g.special) {
    float(*post)[kPairThreads] = reinterpret_cast<float(*)[kPairThreads]>(smem);
    LinkList<float> *lists = reinterpret_cast<LinkList<float> *>(smem + kPopBytes);
    pair_special<S, kForce, kSR>(p, g, b, post, post + 9, lists + (threadIdx.x >> 5));
    return;
  }
  const int warp = (b - g.special) * kPairWarps + (int)(threadIdx.x >> 5);
  pair_bulk<S, kForce, kSR>(p, warp % p.pair_strips, warp / p.pair_strips,
                            reinterpret_cast<Raw(*)[9][kPairThreads]>(smem));
}

template <typename S, bool kForce>
cudaError_t pair_f(StepArgs a, cudaStream_t s) {
  a.pair_strips = (a.L.nx - 4 + kPairStore - 1) / kPairStore;
  const int warps = a.pair_strips * ((a.L.ny - 4 + a.pair_rows - 1) / a.pair_rows);
  const int blocks = pair_grid(a).special + (warps + kPairWarps - 1) / kPairWarps;
  if constexpr (sizeof(S) == 2) {
    if (a.sr) {
      pair_kernel<S, kForce, true><<<blocks, kPairThreads, 0, s>>>(a);
      return cudaGetLastError();
    }
  }
  pair_kernel<S, kForce, false><<<blocks, kPairThreads, 0, s>>>(a);
  return cudaGetLastError();
}

template <typename S>
cudaError_t pair_t(const StepArgs &a, cudaStream_t s) {
  return a.L.has_bf ? pair_f<S, true>(a, s) : pair_f<S, false>(a, s);
}
