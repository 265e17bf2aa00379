// Special nodes of a 2D level update: the outer nodes a level rebuilds from
// its parent (eqs. spaceInt, rescff) and the TN nodes it takes from its child
// (eqs. filterFneq, rescfc), rebuilt, collided and stored here in one go, in
// blocks of the level update's own launch.
//
// In the AA pattern a node's update reads and writes only the node's own
// cells, so these nodes need no order against the rest of their level: a
// coarse step of a 2D run is a chain of one capture and the level updates,
// without a rebuild before every update, a restriction beside it, and the
// stream forks that ran them side by side.  A small run is bound by the
// latency of that chain (a kernel of a few blocks costs about two
// microseconds whatever it does), a large one saves the pass of the rebuilt
// populations through memory.
// A run with few special nodes (E.wide: a chain of small launches) spreads a
// node over lanes -- four for an outer node, one per tap of its stencil,
// sixteen for a TN node, one per child under the filter -- that exchange sums
// by shuffles, so that no lane walks dependent loads; with many (a large
// batch) a lane takes a whole node, which issues a fourth of the
// instructions.  The sums are formed in the same order either way.
// Per coarse step, against a rebuild before every update and a restriction
// on a second stream: 128 x 64 run with a refined slab 19.7 -> 12.4 us (22.6
// with one lane per node), 592^2 binary16 run of three levels 59.2 -> 43.6;
// 33 runs of 512^2 + 513^2 327 -> 332 us in binary32, 207 -> 202 in binary16
// (one lane per node; 357 and 219 with several).
#pragma once

template <class L>
struct NoEdge {};
template <class L>
using EdgeArg = std::conditional_t<L::D == 2, Edge2d, NoEdge<L>>;

template <class L>
__device__ __forceinline__ int edge_slices(const NoEdge<L>&) { return 0; }
__device__ __forceinline__ int edge_slices(const Edge2d& E) { return E.nz; }

// Nodes the special blocks of the launch take.
template <class L>
__device__ __forceinline__ bool edge_node(const LevelView&, const NoEdge<L>&, int, int) {
  return false;
}
__device__ __forceinline__ bool edge_node(const LevelView& v, const Edge2d& E, int x, int y) {
  if (E.nb && ((!v.per[0] && (x == 0 || x == v.n[0] - 1)) ||
               (!v.per[1] && (y == 0 || y == v.n[1] - 1))))
    return true;
  return E.nt && x >= v.tn_lo[0] && x <= v.tn_hi[0] && y >= v.tn_lo[1] && y <= v.tn_hi[1];
}

// Sums over the lanes of a group, the same bits in every lane.
__device__ __forceinline__ float lanes_sum4(unsigned mask, float a) {
  a = __fadd_rn(a, __shfl_xor_sync(mask, a, 1));
  return __fadd_rn(a, __shfl_xor_sync(mask, a, 2));
}

// Outer node k of run `run` before its collision: position and populations.
template <int LANES>
__device__ __forceinline__ void edge_rebuild(const LevelView& v, const RefF& R, const Edge2d& E,
                                             int run, int k, int sub, unsigned mask, int& x, int& y,
                                             float (&g)[D2Q9::Q]) {
  using L = D2Q9;
  // (components picked without indexing the parameters: an indexed parameter
  // is copied to local memory by every thread of the launch)
  auto pick = [](const auto& q, int ax) { return ax == 0 ? q[0] : q[1]; };
  int f = 0;
  while (f + 1 < E.nf && k >= E.b_start[f + 1]) ++f;
  const int a = E.b_axis[f], b = 1 - a;
  const int xb = E.b_lo[f] + (k - E.b_start[f]);  // along the face
  const int xa = E.b_side[f] ? pick(v.n, a) - 1 : 0;
  x = a == 0 ? xa : xb;
  y = a == 0 ? xb : xa;
  // eq. spaceInt: taps at parent positions (xb >> 1) - 1 + tap; an even node
  // takes its co-located parent node (tap 1) alone
  const float* h = E.hist + run * E.run_stride + E.r_start[f];
  float m[3], f1[L::Q];
  auto weight = [&](int tap) {
    return (xb & 1) ? ((tap == 0 || tap == 3) ? -1.0f / 16.0f : 9.0f / 16.0f)
                    : (tap == 1 ? 1.0f : 0.0f);
  };
  auto place = [&](int tap) {
    const int p = (xb >> 1) - 1 + tap;
    // (ring entries start one parent cell before the box)
    return pick(E.p_boxed, b) ? p + 1 : wrapi(p, pick(E.p_n, b));
  };
  auto fill = [&](auto val) {
#pragma unroll
    for (int j = 0; j < 3; ++j) m[j] = val(j);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) f1[i] = val(4 + i);
  };
  if constexpr (LANES == 4) {
    const float w = weight(sub);
    const float* hp = h + place(sub);
    fill([&](int j) {
      return lanes_sum4(mask, w != 0.0f ? __fmul_rn(w, hp[j * E.K]) : 0.0f);
    });
  } else {
    const int p0 = place(0), p1 = place(1), p2 = place(2), p3 = place(3);
    if (xb & 1)
      fill([&](int j) {
        const float* hj = h + j * E.K;
        return __fadd_rn(__fadd_rn(__fmul_rn(-1.0f / 16.0f, hj[p0]), __fmul_rn(9.0f / 16.0f, hj[p1])),
                         __fadd_rn(__fmul_rn(9.0f / 16.0f, hj[p2]), __fmul_rn(-1.0f / 16.0f, hj[p3])));
      });
    else
      fill([&](int j) { return h[j * E.K + p1]; });
  }
  equilibrium_emit<L>(m[0], m[1], m[2], 0.0f, R, [&](auto I, float g0) {
    constexpr int i = decltype(I)::value;
    g[i] = fmaf(E.resc, f1[i], g0);
  });
}

// TN node k of run `run` before its collision.
template <int LANES, class S>
__device__ __forceinline__ void edge_restrict(const LevelView& v, const RefF& R, const Edge2d& E,
                                              int run, int k, int sub, unsigned mask, int& x,
                                              int& y, float (&g)[D2Q9::Q]) {
  using L = D2Q9;
  auto pick = [](const auto& q, int ax) { return ax == 0 ? q[0] : q[1]; };
  int f = 0;
  while (f + 1 < E.tf && k >= E.t_start[f + 1]) ++f;
  const int a = E.t_axis[f], b = 1 - a;
  const int ra = E.t_ra[f], rb = E.t_lo[f] + (k - E.t_start[f]);
  const LevelView& c = E.child;
  const S* fc = run_cptr<S>(c, run);
  float f1[L::Q], m[3] = {0.0f, 0.0f, 0.0f};
  // child (da, db) off the co-located one: its weighted f^(1) into fw
  auto child = [&](int da, int db, float (&fw)[L::Q]) {
    int ca = 2 * ra + da, cb = 2 * rb + db;
    if (pick(c.per, a)) ca = wrapi(ca, pick(c.n, a));
    if (pick(c.per, b)) cb = wrapi(cb, pick(c.n, b));
    float gc[L::Q], drho, dux, duy, duz;
    load_pre<L, S>(fc, c.plane, node_addr<L>(c, a == 0 ? ca : cb, a == 0 ? cb : ca, 0), E.cpar,
                   c.es, gc);
    split_neq<L>(gc, R, drho, dux, duy, duz, fw);
    const float w = (da == 0 ? 0.5f : 0.25f) * (db == 0 ? 0.5f : 0.25f);  // (exact)
#pragma unroll
    for (int i = 0; i < L::Q; ++i) fw[i] = __fmul_rn(w, fw[i]);
    if (da == 0 && db == 0) {
      m[0] = drho;
      m[1] = dux;
      m[2] = duy;
    }
  };
  // three rows along the face's tangent; each adds its children in the order
  // (0, -1) + (+1), then the rows are added the same way
  if constexpr (LANES == 16) {  // lane 4 row + normal offset, both 0 .. 2
    const int da = (sub & 3) - 1, db = (sub >> 2) - 1;
    if (da < 2 && db < 2)
      child(da, db, f1);
    else
#pragma unroll
      for (int i = 0; i < L::Q; ++i) f1[i] = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) m[i] = __shfl_sync(mask, m[i], 5, 16);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
      f1[i] = lanes_sum4(mask, f1[i]);
      f1[i] = __fadd_rn(f1[i], __shfl_xor_sync(mask, f1[i], 4));
      f1[i] = __fadd_rn(f1[i], __shfl_xor_sync(mask, f1[i], 8));
    }
  } else {
    float r1[L::Q], t[L::Q];
#pragma unroll 1
    for (int db = -1; db <= 1; ++db) {
      child(-1, db, r1);
      child(0, db, t);
#pragma unroll
      for (int i = 0; i < L::Q; ++i) r1[i] = __fadd_rn(r1[i], t[i]);
      child(1, db, t);
#pragma unroll
      for (int i = 0; i < L::Q; ++i) {
        r1[i] = __fadd_rn(r1[i], t[i]);
        f1[i] = db == -1 ? r1[i] : __fadd_rn(f1[i], r1[i]);
      }
    }
  }
  equilibrium_emit<L>(m[0], m[1], m[2], 0.0f, R, [&](auto I, float g0) {
    constexpr int i = decltype(I)::value;
    g[i] = fmaf(E.t_resc, f1[i], g0);
  });
  auto pc = [&](int ax, int r) {  // parent coordinate
    if (pick(E.t_boxed, ax)) {
      r += pick(E.t_org, ax);
      if (pick(v.per, ax)) r = wrapi(r, pick(v.n, ax));
    }
    return r;
  };
  x = pc(0, a == 0 ? ra : rb);
  y = pc(1, a == 0 ? rb : ra);
}

template <bool WIDE, class S, int COLL, int PAR, bool MOV>
__device__ __forceinline__ void edge_update(const LevelView& v, float omega, const RefF& R,
                                            const Edge2d& E) {
  using L = D2Q9;
  constexpr int BL = WIDE ? 4 : 1, TL = WIDE ? 16 : 1;  // lanes per outer and TN node
  // (32 bits: the host keeps the lanes of all special nodes below 2^31)
  unsigned t = ((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                   (blockDim.x * blockDim.y) + threadIdx.y * blockDim.x + threadIdx.x;
  const int lane = (int)(t & 31);  // (blocks hold whole warps)
  // outer nodes of every run first, padded to whole warps
  const unsigned bl = ((unsigned)E.nb * v.batch * BL + 31) & ~31u;
  int x, y, lanes, sub;
  float g[L::Q];
  unsigned run;
  if (t < bl) {
    const unsigned item = t / BL;
    run = item / max(E.nb, 1);
    if (run >= (unsigned)v.batch) return;  // whole groups leave
    lanes = BL;
    sub = lane & (BL - 1);
    edge_rebuild<BL>(v, R, E, (int)run, (int)(item - run * E.nb), sub, 0xfu << (lane & 28), x, y,
                     g);
  } else {
    t -= bl;
    const unsigned item = t / TL;
    run = item / max(E.nt, 1);
    if (run >= (unsigned)v.batch || E.nt == 0) return;
    lanes = TL;
    sub = lane & (TL - 1);
    edge_restrict<TL, S>(v, R, E, (int)run, (int)(item - run * E.nt), sub, 0xffffu << (lane & 16),
                         x, y, g);
  }
  S* fp = run_ptr<S>(v, (int)run);
  const NodeAddr ad = node_addr<L>(v, x, y, 0);
  collide_emit<L, COLL, MOV>(g, omega, R, [&](auto I, float val) {
    constexpr int i = decltype(I)::value;
    if ((i & (lanes - 1)) != sub) return;  // the lanes share the stores
    if constexpr (PAR == 0)
      Store<S>::st(fp + (long long)opp<L>(i) * v.plane + v.es * ad.at(0, 0, 0), val);
    else
      Store<S>::st(
          fp + (long long)i * v.plane + v.es * ad.at(L::c(i, 0), L::c(i, 1), L::c(i, 2)), val);
  });
}

// The special blocks' part of an update kernel; true in those blocks.
template <class L, class S, int COLL, int PAR, bool MOV>
__device__ __forceinline__ bool edge_block(const LevelView& v, float omega, const RefF& R,
                                           const EdgeArg<L>& E) {
  if constexpr (L::D == 2) {
    if ((int)blockIdx.z < E.nz) {
      if (E.wide)
        edge_update<true, S, COLL, PAR, MOV>(v, omega, R, E);
      else
        edge_update<false, S, COLL, PAR, MOV>(v, omega, R, E);
      return true;
    }
  }
  return false;
}
