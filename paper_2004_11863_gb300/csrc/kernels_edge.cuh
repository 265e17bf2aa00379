// Special nodes of a 2D level update: the outer nodes a level rebuilds from
// its parent (eqs. spaceInt, rescff) and the TN nodes it takes from its child
// (eqs. filterFneq, rescfc), rebuilt, collided and stored here in one go.
//
// In the AA pattern a node's update reads and writes only the node's own
// cells, so these nodes need no order against the rest of their level: a
// coarse step of a 2D run is a chain of one capture and the level updates,
// without a rebuild before every update and a restriction beside it.
//
// Few of them (edges_few) go into leading blocks of the update's own launch: a
// small run is bound by the latency of its chain of launches (a kernel of a
// few blocks costs about two microseconds whatever it does).  A node is then
// spread over lanes -- four for an outer node, one per tap of its stencil,
// sixteen for a TN node, one per child under the filter -- that exchange sums
// by shuffles, so that no lane walks dependent loads.  Many of them (a large
// batch) go into a launch of their own beside the update's, one lane a node,
// which issues a fourth of the instructions: compiled into the update that
// path sets its registers (binary32 update 40 and 160 to 208 bytes of spills,
// now 39 to 40 and none; 33 runs of 512^2 + 513^2 354 -> 333 us a step, 1024 of
// 128 x 64 with a refined slab 924 -> 855).  The sums are formed in the same
// order either way.
// Per coarse step, against a rebuild before every update and a restriction
// on a second stream: the 128 x 64 run 20.4 -> 11.3 us, 592^2 binary16 run of
// three levels 68 -> 43, 33 runs of 512^2 + 513^2 362 -> 333 in binary32,
// 247 -> 203 in binary16.
// The line between the two (lanes of the fine and of the coarse level's
// launch; us a step within the update, beside it with one lane a node, beside
// it with several): 512^2 + 513^2, 1 run (8 k, 16 k) 18.6, 20.9, 17.9; 4 runs
// (33 k, 65 k) 40.9, 40.2, 42.0; 8 runs (66 k, 131 k) 84.1, 82.1, 85.2; 12 runs
// (98 k, 197 k) 130.8, 127.2, 132.2; 128 x 64, 8 runs (8 k, 16 k) 14.9, 20.7,
// 17.1; 64 runs (66 k, 131 k) 40.2, 41.6, 42.1.
//
// Levels with sensors, whose velocity pass needs the special nodes' velocity
// before the update, take a launch of their own for any number, which writes
// it (512^2 + 513^2, sensors on level 0: 38 -> 28 us a step against a rebuild
// into the planes before it and a second one in the update).
#pragma once

// What an update kernel is told of them: nothing (3D, and 2D levels without
// any), the nodes it leaves alone (EdgeCount), or those its own leading blocks
// take (Edge2d).
template <class L>
struct NoEdge {};

template <class E>
__device__ __forceinline__ int edge_slices(const E&) { return 0; }
__device__ __forceinline__ int edge_slices(const Edge2d& E) { return E.nz; }

// Nodes that other threads take.
template <class L>
__device__ __forceinline__ bool edge_node(const LevelView&, const NoEdge<L>&, int, int) {
  return false;
}
__device__ __forceinline__ bool edge_node(const LevelView& v, const EdgeCount& E, int x, int y) {
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

// Special node t (lanes included) of runs run0 .. run0 + runs - 1, parity par;
// du: its velocity deviation goes there too, when given.
template <bool WIDE, class S, int COLL, bool MOV>
__device__ __forceinline__ void edge_update(const LevelView& v, float omega, const RefF& R,
                                            const Edge2d& E, int par, float* du, unsigned t,
                                            int run0, int runs) {
  using L = D2Q9;
  constexpr int BL = WIDE ? 4 : 1, TL = WIDE ? 16 : 1;  // lanes per outer and TN node
  const int lane = (int)(t & 31);  // (t of a warp's first lane is a multiple of 32)
  // outer nodes of every run first, padded to whole warps
  const unsigned bl = ((unsigned)E.nb * runs * BL + 31) & ~31u;
  int x, y, lanes, sub;
  float g[L::Q];
  unsigned run;
  if (t < bl) {
    const unsigned item = t / BL;
    run = item / max(E.nb, 1);
    if (run >= (unsigned)runs) return;  // whole groups leave
    const int k = (int)(item - run * E.nb);
    run += run0;
    lanes = BL;
    sub = lane & (BL - 1);
    edge_rebuild<BL>(v, R, E, (int)run, k, sub, 0xfu << (lane & 28), x, y, g);
  } else {
    t -= bl;
    const unsigned item = t / TL;
    run = item / max(E.nt, 1);
    if (run >= (unsigned)runs || E.nt == 0) return;
    const int k = (int)(item - run * E.nt);
    run += run0;
    lanes = TL;
    sub = lane & (TL - 1);
    edge_restrict<TL, S>(v, R, E, (int)run, k, sub, 0xffffu << (lane & 16), x, y, g);
  }
  S* fp = run_ptr<S>(v, (int)run);
  const NodeAddr ad = node_addr<L>(v, x, y, 0);
  if (du != nullptr && sub == 0) {
    float drho, u[3];
    deviations<L>(g, R, drho, u[0], u[1], u[2]);
    float* d = du + (long long)run * L::D * v.plane + ad.at(0, 0, 0);
    d[0] = u[0];
    d[v.plane] = u[1];
  }
  collide_emit<L, COLL, MOV>(g, omega, R, [&](auto I, float val) {
    constexpr int i = decltype(I)::value;
    if ((i & (lanes - 1)) != sub) return;  // the lanes share the stores
    if (par == 0)
      Store<S>::st(fp + (long long)opp<L>(i) * v.plane + v.es * ad.at(0, 0, 0), val);
    else
      Store<S>::st(
          fp + (long long)i * v.plane + v.es * ad.at(L::c(i, 0), L::c(i, 1), L::c(i, 2)), val);
  });
}

// The special blocks' part of an update kernel; true in those blocks.
template <class L, class S, int COLL, int PAR, bool MOV, class E>
__device__ __forceinline__ bool edge_block(const LevelView&, float, const RefF&, const E&) {
  return false;
}
template <class L, class S, int COLL, int PAR, bool MOV>
__device__ __forceinline__ bool edge_block(const LevelView& v, float omega, const RefF& R,
                                           const Edge2d& E) {
  if ((int)blockIdx.z >= E.nz) return false;
  // (blocks hold whole warps)
  const unsigned t = ((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                         (blockDim.x * blockDim.y) + threadIdx.y * blockDim.x + threadIdx.x;
  edge_update<true, S, COLL, MOV>(v, omega, R, E, PAR, nullptr, t, 0, v.batch);
  return true;
}

// The special nodes of a level update in a launch of their own, run by run.
template <bool WIDE, class S, int COLL, bool MOV>
__global__ void __launch_bounds__(64)
    k_edges(LevelView v, float omega, RefF R, const __grid_constant__ Edge2d E, int par,
            float* du) {
  edge_update<WIDE, S, COLL, MOV>(v, omega, R, E, par, du,
                                  blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y, 1);
}
