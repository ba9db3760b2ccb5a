// Q-split kernels: the step as two kernels whose parallel index is (r-node,
// Q-node) instead of the fused kernel's r-node alone.
//
//   collide_kernel  pull, collide and write of all populations, from complete
//                   moment planes of the state (Sec. VI-C update)
//   moments_kernel  pull-read of all populations -> moment planes (Sec. VI-A,
//                   VI-B; Theta of Sec. III)
//
// A warp takes 32 consecutive r-nodes and one Q-node at a time; the warps of a
// block share the r-nodes and divide the Q-nodes. The collision of a Q-node
// needs no other Q-node's populations, so its warps never wait for each other
// after the block has formed U; the moments sum over the Q-nodes in a fixed
// order (each warp its own Q-nodes in order, then the warps in order), which
// does not depend on where a node lies in a grid, a tile or a slab.
//
// Against the fused kernel the populations are read twice, but a grid of a few
// thousand nodes spreads over the whole GPU (64 x 64 nodes are 16 tiles of the
// fused kernel, and 4096 warps of work per 32 Q-nodes here), there is no chain
// over the Q-nodes with two barriers each, and no arrival sums on the ring of a
// tile. FP64 takes these kernels at every size: they need half of the fused
// kernel's FP64 operations, which bound it (2 lanes per clock and SM).
//
// Operation count in FP64: the shift difference of a pulled population is the
// same for the members of a Q-displacement group and constant per Q-node, so the
// moments add its sum once, after the sum of the stored values that it nearly
// cancels (in any precision: it is also the most exact order), and the FP64
// collision adds (1 - 2 beta) times it to the group's equilibrium term instead of
// shifting every population, and takes delta psi from the moment planes. The FP32
// collision shifts and sums the populations themselves: its mass would otherwise
// drift by the rounding of the summed shifts, 1e-8 of the polymer's per step. FP16
// storage works in stored units (the deviation times a power of two)
// throughout, so no population is scaled or unscaled.
//
// Bound by: FP64, the FP64 pipe (82% busy in the collision); FP32 and FP16 storage,
// the latency of a launch and of one round of loads on small grids, and on large ones
// the loads in flight: a warp loads the next Q-node's populations into each register
// as soon as the present one has used it. Measured on GB300, us per step, before
// (fused, or two passes with one thread per node) and now: FP64, 52 Q-nodes, 64 x 64
// nodes 1085 and 109; FP64, 32 Q-nodes, 512 x 512 4739 and 3071; FP32, 32 Q-nodes,
// 64 x 64 61.8 and 12.1; 72 x 72 78 and 15.2; 128 x 128 64 and 35; 1000 x 750 1433 and
// 1426 (4.85 GB read and written and 2.43 GB read again: 5.1 TB/s); FP16 storage, the
// same grid, 1283 and 1193.
#include <algorithm>
#include <type_traits>

#include "tfkt_fused.cuh"

namespace tfkt {
namespace {

constexpr int QN = 32;       // r-nodes of a group (one warp wide)
constexpr int CW = 8;        // warps of a collide block

__host__ __device__ constexpr int opposite(int i) {
  for (int j = 0; j < 25; ++j) {
    const V4 c = c25(i), d = c25(j);
    if (d.rx == -c.rx && d.ry == -c.ry && d.qx == -c.qx && d.qy == -c.qy) return j;
  }
  return -1;
}
// Slot of a Q-displacement group that moves in Q in the per-Q-node tables.
__host__ __device__ constexpr int qslot(int g) { return g < 4 ? g : g - 1; }

// The node of a lane: row-major index k over the grid. A lane past the last node
// repeats it: it reads the same values and stores the same results.
struct Node {
  int x, y;
};
__device__ __forceinline__ Node lane_node(int nx, int ny) {
  const uint32_t total = (uint32_t)nx * (uint32_t)ny;
  uint32_t k = (blockIdx.x * blockDim.z + threadIdx.z) * QN + threadIdx.x;
  Node n;
  if (k >= total) k = total - 1;
  n.y = (int)(k / (uint32_t)nx);
  n.x = (int)(k - (uint32_t)n.y * (uint32_t)nx);
  return n;
}

// Byte offsets of the nine pull sources of a node within a plane of elements of
// `es` bytes, the size of a stored population. 32 bits are enough: two buffers of at
// least 34 planes fit the GPU's memory, so such a plane is below 2^32 bytes.
struct Offs {
  uint32_t o[9];
};
__device__ __forceinline__ Offs pull_offsets(const Node& nd, int nx, int ny, uint32_t pitch,
                                             uint32_t es) {
  const uint32_t x = nd.x * es, xm = (nd.x == 0 ? nx - 1 : nd.x - 1) * es;
  const uint32_t xp = (nd.x == nx - 1 ? 0 : nd.x + 1) * es;
  pitch *= es;
  const uint32_t y = nd.y * pitch, ym = (nd.y == 0 ? ny - 1 : nd.y - 1) * pitch;
  const uint32_t yp = (nd.y == ny - 1 ? 0 : nd.y + 1) * pitch;
  Offs f;
  f.o[0] = ym + xm; f.o[1] = ym + x; f.o[2] = ym + xp;
  f.o[3] = y + xm;  f.o[4] = y + x;  f.o[5] = y + xp;
  f.o[6] = yp + xm; f.o[7] = yp + x; f.o[8] = yp + xp;
  return f;
}
// The planes of a buffer, addressed by plane index and byte offset. The size of a
// plane of stored populations is 32 bits too: an address is a 32 x 32 + 64 bit
// multiply-add and a 64-bit add (with 64-bit element arithmetic the address
// computations were three quarters of the instructions). The FP32 planes beside FP16
// populations may be larger and are addressed in 64 bits.
template <typename T>
struct Planes {
  char* p;
  uint64_t bytes;   // of a plane
  __device__ __forceinline__ Planes(const void* base, size_t plane)
      : p((char*)base), bytes(plane * sizeof(T)) {}
  // element at byte offset o of plane k; o counts in elements of type E
  template <typename E = T>
  __device__ __forceinline__ T& at(uint32_t k, uint32_t o) const {
    static_assert(sizeof(T) >= sizeof(E), "");
    if constexpr (sizeof(T) == sizeof(E))
      return *reinterpret_cast<T*>((p + o) + (uint64_t)k * (uint32_t)bytes);
    else
      return *reinterpret_cast<T*>((p + (uint64_t)o * (sizeof(T) / sizeof(E))) + k * bytes);
  }
};
// The same value in every lane, told to the compiler as warp-uniform, so that what
// depends on it (plane addresses, branches) stays in uniform registers.
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// The 25 pulled populations of Q-node q, in their stored form. A group whose
// source leaves the Q-disk (src < 0) takes the node's own opposite velocities.
template <typename S>
__device__ __forceinline__ void pull25(S (&h)[25], const Planes<S>& src, const int (&srow)[8], int q,
                                       const Offs& off) {
  const uint32_t own = 9 + 25 * q;
  static_for<0, 5>([&](auto I) {
    constexpr int i = I;
    constexpr V4 c = c25(i);
    h[i] = src.at(own + i, off.o[shift_index(-c.rx, -c.ry)]);
  });
  static_for<0, 9>([&](auto GI) {
    constexpr int g = GI;
    if constexpr (g != 4) {
      const int e = srow[qslot(g)];
      if (e >= 0) {
        static_for<5, 20>([&](auto I) {
          constexpr int i = I;
          constexpr V4 c = c25(i);
          if constexpr (qgroup(c) == g) h[i] = src.at(e + i, off.o[shift_index(-c.rx, -c.ry)]);
        });
      } else {
        static_for<5, 20>([&](auto I) {
          constexpr int i = I;
          if constexpr (qgroup(c25(i)) == g) h[i] = src.at(own + opposite(i), off.o[4]);
        });
      }
    }
  });
}

// One pulled population, its group's bounce as a select: for loads that follow the
// use of a register one by one.
template <int I, typename S>
__device__ __forceinline__ S pull1(const Planes<S>& src, const int (&srow)[8], int q, const Offs& off) {
  constexpr V4 c = c25(I);
  const uint32_t own = 9 + 25 * q;
  if constexpr (qgroup(c) == 4) {
    return src.at(own + I, off.o[shift_index(-c.rx, -c.ry)]);
  } else {
    const int e = srow[qslot(qgroup(c))];
    return src.at(e >= 0 ? e + I : own + opposite(I), e >= 0 ? off.o[shift_index(-c.rx, -c.ry)] : off.o[4]);
  }
}

// A Q-node's table entry, read by every lane of the warp (one address: a broadcast).
template <typename real>
__device__ __forceinline__ void load_src(int (&s)[8], const QRow<real>* r) {
  const int4 a = reinterpret_cast<const int4*>(r->src)[0], b = reinterpret_cast<const int4*>(r->src)[1];
  s[0] = uniform(a.x); s[1] = uniform(a.y); s[2] = uniform(a.z); s[3] = uniform(a.w);
  s[4] = uniform(b.x); s[5] = uniform(b.y); s[6] = uniform(b.z); s[7] = uniform(b.w);
}

// Adds the Q-node's shift differences to its pulled populations (in stored units).
template <typename real>
__device__ __forceinline__ void add_shifts(real (&h)[25], const QRow<real>* row) {
  real d[8];
  load_vec<8>(d, row->bd);
  static_for<5, 20>([&](auto I) {
    constexpr int i = I;
    h[i] += d[qslot(qgroup(c25(i)))];
  });
}

// The four velocities (+-1, +-1) of a component pair.
template <int CA, int CB>
struct Pair {
  static constexpr int a = CA, b = CB;
  static constexpr int pp = pair_vel(CA, CB, 1, 1), pm = pair_vel(CA, CB, 1, -1);
  static constexpr int mp = pair_vel(CA, CB, -1, 1), mm = pair_vel(CA, CB, -1, -1);
};

// The six component pairs: (rx,ry) (rx,qx) (rx,qy) (ry,qx) (ry,qy) (qx,qy).
template <int PR>
using PairOf = Pair<(PR < 3 ? 0 : (PR < 5 ? 1 : 2)), (PR == 0 ? 1 : (PR == 1 || PR == 3 ? 2 : 3))>;

// ------------------------------------------------------------------ moments
// Whether the shift differences are folded into the moments and the equilibria (see
// above) or added to every pulled population.
template <typename real>
constexpr bool FOLD = std::is_same<real, double>::value;

template <typename real, typename S, int MAXW>
__global__ void __launch_bounds__(QN * MAXW, sizeof(real) == 8 ? 1 : 32 / MAXW) moments_kernel(KernelArgs<real> a) {
  const int lane = threadIdx.x, w = uniform(threadIdx.y), W = blockDim.y;
  const int nq = a.nq;
  const size_t P = a.plane;
  const Node nd = lane_node(a.nx, a.ny);
  const Offs off = pull_offsets(nd, a.nx, a.ny, (uint32_t)a.pitch, sizeof(S));
  const uint32_t n = off.o[4];   // the node itself
  const Planes<S> src(a.src, P);
  const Planes<real> M(a.M, P);
  let_successor_start();
  int srow[8];
  if (w < nq) load_src(srow, a.tab.row + w);
  wait_for_predecessor();
  // this warp's sums over its Q-nodes: delta rho, J_x, J_y, Theta
  real sum[6] = {0, 0, 0, 0, 0, 0};
  int q = w;
#pragma unroll 1
  for (; q < nq; q += W) {
    const QRow<real>* row = a.tab.row + q;
    if (q != w) load_src(srow, row);
    S hr[25];
    pull25(hr, src, srow, q, off);
    real h[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) h[i] = from_store<real>(hr[i]);
    real dpsi = h[0], rx = 0, ry = 0;
    {
      using K = Pair<0, 1>;
      const real d1 = h[K::pp] - h[K::mm], d2 = h[K::pm] - h[K::mp];
      dpsi += (h[K::pp] + h[K::mm]) + (h[K::pm] + h[K::mp]);
      rx = d1 + d2;
      ry = d1 - d2;
    }
    static_for<2, 2>([&](auto C) {   // (rx, qx), (rx, qy)
      using K = Pair<0, decltype(C)::value>;
      const real p = h[K::pp] + h[K::pm], m = h[K::mp] + h[K::mm];
      dpsi += p + m;
      rx += p - m;
    });
    static_for<2, 2>([&](auto C) {   // (ry, qx), (ry, qy)
      using K = Pair<1, decltype(C)::value>;
      const real p = h[K::pp] + h[K::pm], m = h[K::mp] + h[K::mm];
      dpsi += p + m;
      ry += p - m;
    });
    {
      using K = Pair<2, 3>;
      dpsi += (h[K::pp] + h[K::mm]) + (h[K::pm] + h[K::mp]);
    }
    dpsi += row->dpsi;   // last: it nearly cancels the sum of the stored values
    if constexpr (!std::is_same<S, real>::value) {   // stored units -> deviations
      dpsi *= a.pinv;
      rx *= a.pinv;
      ry *= a.pinv;
    }
    M.template at<S>(q, n) = dpsi;
    sum[0] += dpsi;
    sum[1] += rx;
    sum[2] += ry;
    sum[3] += dpsi * row->tq[0];
    sum[4] += dpsi * row->tq[1];
    sum[5] += dpsi * row->tq[2];
  }
  if (q == nq) {   // the solvent follows the last Q-node in the warps' order
    const Planes<SolventT<S>> ssrc(solvent_planes<S>(a.src, P, nq), P);
    real ds = 0, jx = 0, jy = 0;
    static_for<0, 9>([&](auto I) {
      constexpr int i = I;
      const real v = from_store<real>(ssrc.template at<S>(i, off.o[shift_index(-c9x(i), -c9y(i))]));
      ds += v;
      acc<c9x(i)>(jx, v);
      acc<c9y(i)>(jy, v);
    });
    sum[0] += ds;
    sum[1] += jx;
    sum[2] += jy;
  }
  __shared__ real part[6][MAXW][QN];   // a group of 32 nodes has W rows, at z W
  const int g0 = threadIdx.z * W;
#pragma unroll
  for (int j = 0; j < 6; ++j) part[j][g0 + w][lane] = sum[j];
  __syncthreads();
  for (int j = w; j < 6; j += W) {
    real s = part[j][g0][lane];
    for (int v = 1; v < W; ++v) s += part[j][g0 + v][lane];
    M.template at<S>(nq + j, n) = j < 3 ? s : a.hl2h * s;
  }
}

// ------------------------------------------------------------------ collide
// UPASS: U is read from its planes, which a velocity pass has written.
template <typename real, typename S, bool STRESS, bool UPASS = false>
__global__ void __launch_bounds__(QN * CW, 2) collide_kernel(KernelArgs<real> a) {
  __shared__ real su_[CW][2][5][QN];   // one part per group of 32 nodes
  auto& su = su_[threadIdx.z];
  const int lane = threadIdx.x, w = uniform(threadIdx.y), W = blockDim.y;
  const int nq = a.nq;
  const size_t P = a.plane;
  const Node nd = lane_node(a.nx, a.ny);
  const Offs off = pull_offsets(nd, a.nx, a.ny, (uint32_t)a.pitch, sizeof(S));
  const uint32_t n = off.o[4];   // the node itself
  const Planes<real> M(a.M, P);
  const Planes<S> src(a.src, P), dst(a.dst, P);

  // the first Q-node's loads, in flight while the block forms U
  const int q0 = blockIdx.y * W + w, dq = gridDim.y * W;
  S hr[25];
  real mn[4], dpsi = 0;
  int srow[8];
  auto load_moments = [&](int q) {
    mn[0] = M.template at<S>(q, off.o[5]);
    mn[1] = M.template at<S>(q, off.o[3]);
    mn[2] = M.template at<S>(q, off.o[7]);
    mn[3] = M.template at<S>(q, off.o[1]);
    if constexpr (FOLD<real> && !STRESS) dpsi = M.template at<S>(q, n);
  };
  let_successor_start();
  if (q0 < nq) load_src(srow, a.tab.row + q0);
  wait_for_predecessor();
  if (q0 < nq) {
    pull25(hr, src, srow, q0, off);
    load_moments(q0);
  }

  // U of the block's nodes and of their four neighbours
  for (int k = w; k < 5; k += W) {
    const int x = k == 1 ? (nd.x == a.nx - 1 ? 0 : nd.x + 1) : (k == 2 ? (nd.x == 0 ? a.nx - 1 : nd.x - 1) : nd.x);
    const int y = k == 3 ? (nd.y == a.ny - 1 ? 0 : nd.y + 1) : (k == 4 ? (nd.y == 0 ? a.ny - 1 : nd.y - 1) : nd.y);
    real ux, uy;
    if constexpr (UPASS) {
      const size_t m = (size_t)y * a.pitch + x;
      ux = a.U[m];
      uy = a.U[P + m];
    } else {
      velocity_at(a, a.M, x, y, ux, uy);
    }
    su[0][k][lane] = ux;
    su[1][k][lane] = uy;
  }
  __syncthreads();
  const real Ux = su[0][0][lane], Uy = su[1][0][lane];
  const real G00 = real(0.5) * (su[0][1][lane] - su[0][2][lane]);   // d_x U_x
  const real G01 = real(0.5) * (su[1][1][lane] - su[1][2][lane]);   // d_x U_y
  const real G10 = real(0.5) * (su[0][3][lane] - su[0][4][lane]);   // d_y U_x
  const real G11 = real(0.5) * (su[1][3][lane] - su[1][4][lane]);   // d_y U_y

  // weights of the momenta: 3 x the mixed equilibrium's momentum (1 - r) f* + r f^eq
  // times 2 beta w (w = 1/36) is wa J(g) + wb J_eq
  const real tw = a.tb * real(1.0 / 36.0), tw3 = real(3) * tw;
  real wa, wb;
  if constexpr (STRESS) {   // both targets carry the equilibrium momenta
    wa = 0;
    wb = tw3 * a.pscale;
  } else {
    wa = tw3 * a.omr * a.c2 * a.inv_c2p1;
    wb = tw3 * (a.omr * a.inv_c2p1 + a.r) * a.pscale;
  }

  int q = q0;
#pragma unroll 1
  for (; q < nq; q += dq) {
    const QRow<real>* row = a.tab.row + q;
    real h[25];
#pragma unroll
    for (int i = 0; i < 25; ++i) h[i] = from_store<real>(hr[i]);
    constexpr bool FOLDED = FOLD<real> && !STRESS;
    real bd[8] = {};
    if constexpr (FOLDED) load_vec<8>(bd, row->bd);
    else add_shifts(h, row);
    const bool more = q + dq < nq;
    if (more) load_src(srow, row + dq);
    // Moments of g in stored units. FOLDED: the momenta, and psi from the moment planes.
    // Otherwise delta psi is the sum of the shifted populations themselves, so that the
    // collision conserves mass exactly as it is stored (the rounded shifts cancel between
    // Q-nodes; the rounded sums in the moment planes do not), and for STRESS the second
    // moments from the same terms.
    real ps = h[0], jg[4] = {0, 0, 0, 0}, t[4] = {0, 0, 0, 0}, t2[6];
    if constexpr (FOLDED) {
      jg[2] = row->dq[0];
      jg[3] = row->dq[1];
    }
    static_for<0, 6>([&](auto PR) {
      using K = PairOf<decltype(PR)::value>;
      if constexpr (!STRESS) {
        const real d1 = h[K::pp] - h[K::mm], d2 = h[K::pm] - h[K::mp];
        jg[K::a] += d1 + d2;
        jg[K::b] += d1 - d2;
      }
      if constexpr (!FOLDED) {
        const real s1 = h[K::pp] + h[K::mm], s2 = h[K::pm] + h[K::mp];
        ps += s1 + s2;
        if constexpr (STRESS) {
          t[K::a] += s1 + s2;
          t[K::b] += s1 + s2;
          t2[PR] = s1 - s2;
        }
      }
    });
    real wd = 0;   // 2 beta w delta psi, in stored units
    if constexpr (FOLDED) {
      wd = tw * a.pscale * dpsi;
    } else {
      dpsi = ps * a.pinv;
      wd = tw * ps;
    }
    const real psi = row->psi0 + dpsi;
    const real qg = row->hq[0] * (mn[0] - mn[1]) + row->hq[1] * (mn[2] - mn[3]);   // Q . grad psi
    const real Qx = row->q[0], Qy = row->q[1];
    const real jrex = psi * Ux + row->cf[0] * qg;
    const real jrey = psi * Uy + row->cf[1] * qg;
    const real jqex = psi * (Qx * G00 + Qy * G10 - row->kf[0]);
    const real jqey = psi * (Qx * G01 + Qy * G11 - row->kf[1]);
    real m[4] = {wb * jrex, wb * jrey, wb * jqex, wb * jqey};
    const uint32_t own = 9 + 25 * q;
    auto put = [&](auto I, real v) {
      dst.at(own + decltype(I)::value, n) = to_store<S>(v);
      if (more) hr[decltype(I)::value] = pull1<decltype(I)::value>(src, srow, q + dq, off);
    };
    if (more) load_moments(q + dq);
    if constexpr (!STRESS) {
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] += wa * jg[k];
      put(std::integral_constant<int, 0>(), a.om2b * h[0] + real(12) * wd);   // w0 / w = 12
      static_for<0, 6>([&](auto PR) {
        using K = PairOf<decltype(PR)::value>;
        auto one = [&](auto I, real e) { put(I, a.om2b * h[decltype(I)::value] + e); };
        using pp = std::integral_constant<int, K::pp>;
        using pm = std::integral_constant<int, K::pm>;
        using mp = std::integral_constant<int, K::mp>;
        using mm = std::integral_constant<int, K::mm>;
        const real ma = m[K::a], mb = m[K::b];
        if constexpr (FOLDED) {
          // the constant term of a Q-displacement group: 2 beta w dpsi + (1 - 2 beta) shift
          auto base = [&](auto I) {
            constexpr int g = qgroup(c25(decltype(I)::value));
            if constexpr (g == 4) return wd;
            else return wd + bd[qslot(g)];
          };
          one(pp(), base(pp()) + (ma + mb));
          one(pm(), base(pm()) + (ma - mb));
          one(mp(), base(mp()) - (ma - mb));
          one(mm(), base(mm()) - (ma + mb));
        } else {
          // the r-momentum first: the Q-momentum, of the drift at rest, is the larger one
          one(pp(), wd + ma + mb);
          one(pm(), wd + ma - mb);
          one(mp(), wd - ma + mb);
          one(mm(), wd - ma - mb);
        }
      });
    } else {
      // the second-order Hermite terms of f**: per axis sk, per pair sp, and s0
      const real kf = tw * a.omr * a.c2 * a.inv_c2p1;
      const real eq = ps * real(1.0 / 3.0);
      real sk[4], tr = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const real dk = t[k] - eq;
        tr += dk;
        sk[k] = real(4.5) * kf * dk;
      }
      const real s0 = real(-1.5) * kf * tr;
      put(std::integral_constant<int, 0>(), a.om2b * h[0] + real(12) * (wd + s0));
      static_for<0, 6>([&](auto PR) {
        using K = PairOf<decltype(PR)::value>;
        const real sp = real(9) * kf * t2[PR], e = wd + (sk[K::a] + sk[K::b] + s0);
        put(std::integral_constant<int, K::pp>(), a.om2b * h[K::pp] + (e + sp + m[K::a] + m[K::b]));
        put(std::integral_constant<int, K::mm>(), a.om2b * h[K::mm] + (e + sp - m[K::a] - m[K::b]));
        put(std::integral_constant<int, K::pm>(), a.om2b * h[K::pm] + (e - sp + m[K::a] - m[K::b]));
        put(std::integral_constant<int, K::mp>(), a.om2b * h[K::mp] + (e - sp - m[K::a] + m[K::b]));
      });
    }
  }

  // ---- the solvent follows the last Q-node in the warps' order
  if (q != nq) return;
  const real rho = a.rho0 + M.template at<S>(nq + M_DRHO, n);
  const real force = rho * a.tab.arow[nd.y];
  using SS = SolventT<S>;
  const Planes<SS> ssrc(solvent_planes<S>(a.src, P, nq), P), sdst(solvent_planes<S>(a.dst, P, nq), P);
  real hs[9], drs = 0;
  static_for<0, 9>([&](auto I) {
    constexpr int i = I;
    hs[i] = from_store<real>(ssrc.template at<S>(i, off.o[shift_index(-c9x(i), -c9y(i))]));
    drs += hs[i];
  });
  const real rs = real(1) + drs;
  if constexpr (STRESS) {
    // P(f) - rho_S c_s^2 I = [2 tau2 (P(g) - P_eq) + tau2 (F U + U F)] / (2 tau2 + 1) + rho_S U U
    const real cs2 = real(1) / real(3);
    real pxx = 0, pxy = 0, pyy = 0;
    static_for<0, 9>([&](auto I) {
      constexpr int i = I;
      acc<c9x(i) * c9x(i)>(pxx, hs[i]);
      acc<c9x(i) * c9y(i)>(pxy, hs[i]);
      acc<c9y(i) * c9y(i)>(pyy, hs[i]);
    });
    const real dxx = pxx - drs * cs2 - rs * Ux * Ux, dxy = pxy - rs * Ux * Uy;
    const real dyy = pyy - drs * cs2 - rs * Uy * Uy;
    const real fxx = (a.c2 * dxx + a.tau2 * real(2) * force * Ux) * a.inv_c2p1 + rs * Ux * Ux;
    const real fxy = (a.c2 * dxy + a.tau2 * force * Uy) * a.inv_c2p1 + rs * Ux * Uy;
    const real fyy = a.c2 * dyy * a.inv_c2p1 + rs * Uy * Uy;
    const real usq = Ux * Ux + Uy * Uy;
    static_for<0, 9>([&](auto I) {
      constexpr int i = I;
      constexpr real cx = real(c9x(i)), cy = real(c9y(i));
      const real cu = cx * Ux + cy * Uy;
      const real pneq = fxx * (cx * cx - cs2) + real(2) * fxy * cx * cy + fyy * (cy * cy - cs2);
      const real fss_dev = real(w9(i)) * (drs + real(3) * rs * cu + real(4.5) * pneq);
      const real feq_dev = real(w9(i)) * (drs + rs * (real(3) * cu + real(4.5) * cu * cu - real(1.5) * usq));
      const real srcterm = real(w9(i)) * (real(3) * (cx - Ux) + real(9) * cu * cx) * force;
      const real hp = a.om2b * hs[i] + a.tb * (a.omr * fss_dev + a.r * feq_dev) + a.omb * srcterm;
      sdst.template at<S>(i, n) = to_store<SS>(hp);
    });
  } else {
    real jsx = 0, jsy = 0;
    static_for<0, 9>([&](auto I) {
      constexpr int i = I;
      acc<c9x(i)>(jsx, hs[i]);
      acc<c9y(i)>(jsy, hs[i]);
    });
    const real jfx = (a.c2 * jsx + rs * Ux + a.tau2 * force) * a.inv_c2p1;
    const real jfy = (a.c2 * jsy + rs * Uy) * a.inv_c2p1;
    const real usx = jfx / rs, usy = jfy / rs;
    const real vx = a.omr * usx + a.r * Ux, vy = a.omr * usy + a.r * Uy;
    const real sq = a.omr * (usx * usx + usy * usy) + a.r * (Ux * Ux + Uy * Uy);
    static_for<0, 9>([&](auto I) {
      constexpr int i = I;
      real cus = 0, cu = 0, cv = 0;
      acc<c9x(i)>(cus, usx); acc<c9y(i)>(cus, usy);
      acc<c9x(i)>(cu, Ux);   acc<c9y(i)>(cu, Uy);
      acc<c9x(i)>(cv, vx);   acc<c9y(i)>(cv, vy);
      // Guo source (3 (c - U) + 9 (c . U) c) . (force, 0)
      real gx = -real(3) * Ux;
      acc<c9x(i)>(gx, real(3) + real(9) * cu);
      const real feq_dev = real(w9(i)) * (drs + rs * (real(3) * cv +
                                                      real(4.5) * (a.omr * cus * cus + a.r * cu * cu) -
                                                      real(1.5) * sq));
      const real hp = a.om2b * hs[i] + a.tb * feq_dev + a.omb * real(w9(i)) * gx * force;
      sdst.template at<S>(i, n) = to_store<SS>(hp);
    });
  }
}

// Blocks of g groups of 32 nodes that cover the grid.
inline uint32_t node_blocks(const int nx, const int ny, int g) {
  return (uint32_t)(((size_t)nx * ny + (size_t)QN * g - 1) / ((size_t)QN * g));
}

}  // namespace

// Host-side per-Q-node table of the Q-split kernels.
template <typename real>
std::vector<QRow<real>> build_rows(const Lattice& L, const HostTables& t) {
  std::vector<QRow<real>> rows(L.nq);
  const double s = polymer_scale(L), b = 1.0 / (2.0 * L.tau1 + 1.0);
  const double hl2h = 0.5 * L.H * L.ell * L.ell;
  for (int q = 0; q < L.nq; ++q) {
    QRow<real>& r = rows[q];
    double dpsi = 0, dqx = 0, dqy = 0;
    for (int i = 0; i < 25; ++i) {
      const V4 c = c25(i);
      const double d = t.delta[(size_t)q * 25 + i];
      dpsi += d;
      dqx += c.qx * d;
      dqy += c.qy * d;
      if (qgroup(c) == 4) continue;
      // the first plane of the source Q-node, or ~(first plane of q) where the pull bounces
      const int e = t.pull[(size_t)q * 25 + i];
      r.src[qslot(qgroup(c))] = e >= 0 ? e - i : ~(9 + 25 * q);
      const bool folded = FOLD<real> && L.qe_model == TFKT_QE_MOMENTUM;
      r.bd[qslot(qgroup(c))] = (real)(s * d * (folded ? 1.0 - 2.0 * b : 1.0));
    }
    r.dpsi = (real)(s * dpsi);
    r.dq[0] = (real)(s * dqx);
    r.dq[1] = (real)(s * dqy);
    r.psi0 = (real)t.psi0[q];
    r.q[0] = (real)t.qx[q];
    r.q[1] = (real)t.qy[q];
    r.hq[0] = (real)(0.5 * t.qx[q]);
    r.hq[1] = (real)(0.5 * t.qy[q]);
    r.kf[0] = (real)(L.kappa * t.fx[q]);
    r.kf[1] = (real)(L.kappa * t.fy[q]);
    r.cf[0] = (real)(L.tau_m * hl2h * t.fx[q]);
    r.cf[1] = (real)(L.tau_m * hl2h * t.fy[q]);
    r.tq[0] = (real)(t.fx[q] * t.qx[q]);
    r.tq[1] = (real)(t.fx[q] * t.qy[q]);
    r.tq[2] = (real)(t.fy[q] * t.qy[q]);
    r.pad = 0;
  }
  return rows;
}

// `n` tasks over at most `most` warps in as few rounds as possible, the warps
// equally loaded.
static int even_warps(int n, int most) {
  const int rounds = (n + most - 1) / most;
  return (n + rounds - 1) / rounds;
}
// From here on a grid fills the GPU several times over with blocks of four groups of
// nodes, whose warps read longer runs of a plane.
constexpr size_t MANY_GROUPS = 8 * 2 * 152;

// Warps that share a node's moment sums. Up to one block of 32 nodes per SM the
// sums are a chain of loads and every warp shortens it (64 x 64 nodes, 32 Q-nodes,
// FP32, us per step: 16.8 with 8 warps, 14.0 with 16, 12.8 with 32); with more
// blocks the smaller ones spread better (128 x 128: 33.8, 36.4, 40.5), and a large
// grid wants few (the kernel alone, us: 333 x 777 nodes with 9 Q-nodes 79 with 8, 66
// with 2; 999 x 1411 with 12 404 and 341; 512 x 512 in FP64 with 32 751, and 727 with 4)
// unless a node has many Q-nodes (512 x 512 with 156 720 with 8, 797 with 2). The number
// sets the order of the sums, so it depends on the whole run, not on a slab of it.
int moment_warps(const Lattice& L) {
  const size_t ny = L.ny_global > 0 ? L.ny_global : L.ny;
  const size_t groups = (L.nx * ny + QN - 1) / QN;
  const bool fp64 = L.precision == TFKT_FP64;
  const int most = groups <= 152 ? (fp64 ? 16 : 32)
                 : groups <= 2 * 152 ? 16
                 : groups < MANY_GROUPS || L.nq >= 64 ? 8 : (fp64 ? 4 : 2);
  return even_warps(L.nq + 1, most);
}

// A collision forms U at a node and its four neighbours for every group of Q-nodes. In FP64
// that is a fifth of the operations of a run with one Q-node, the pipe's that bounds it, and
// from a grid that fills the GPU on a pass that forms each U once pays for its launch: us per
// step, 1024 x 1024 nodes, one Q-node 1194 without and 971 with it (stress model 1425 and
// 1192), 256 x 256 (below the line) 90. The whole run decides, so that a
// slab does as it does.
bool velocity_pass(const Lattice& L) {
  const size_t ny = L.ny_global > 0 ? L.ny_global : L.ny;
  return L.precision == TFKT_FP64 && L.nq < 4 && (L.nx * ny + QN - 1) / QN >= MANY_GROUPS;
}

template <typename real, typename S>
cudaError_t launch_moments(const KernelArgs<real>& a, cudaStream_t s, bool dependent) {
  auto go = [&](auto MW) {
    constexpr int mw = decltype(MW)::value;
    const int w = a.mom_warps, g = mw / w;
    return launch(moments_kernel<real, S, mw>, node_blocks(a.nx, a.ny, g), dim3(QN, w, g), 0, s, dependent,
                  a);
  };
  if (a.mom_warps <= 8) return go(std::integral_constant<int, 8>());
  if constexpr (sizeof(real) == 4)
    if (a.mom_warps > 16) return go(std::integral_constant<int, 32>());
  return go(std::integral_constant<int, 16>());
}

// How the collision's Q-nodes are divided: over the warps of a block (the fewer, the
// longer the runs of a plane that a block reads) and, where a grid does not fill the
// GPU, over `split` blocks. A block's time is its prologue (about 1.5 Q-nodes' worth)
// and its Q-nodes per warp; the number of waves follows from the two blocks that are
// resident on an SM. `shared`: the launch runs beside others that fill the GPU. The
// choice does not change any result. us per step in FP32: 64 x 64 nodes with 32 Q-nodes
// 19.1 with one block, 14.0 with 2, 13.2 with 3, 13.4 with 4; 128 x 128: 40.2, 36.4, 34.6,
// 36.1. The kernel alone on large grids, 8 and 2 warps: 333 x 777 nodes with 9 Q-nodes 147
// and 114, 1000 x 750 with 32 978 and 939; FP64, 512 x 512, 2385 and with 4 warps 2350.
template <typename real, typename S>
cudaError_t launch_step(const KernelArgs<real>& a, cudaStream_t s, bool dependent, bool shared) {
  const int tasks = a.nq + 1;   // the Q-nodes and the solvent
  const bool many = shared || node_blocks(a.nx, a.ny, 1) >= MANY_GROUPS;
  const int w = even_warps(tasks, !many ? CW : (sizeof(real) == 8 ? 4 : 2)), g = CW / w;
  const uint32_t nb = node_blocks(a.nx, a.ny, g);
  const size_t slots = 2 * 152;
  int split = 1;
  double best = 1e300;
  for (int k = 1; k <= 8 && (k - 1) * w < tasks && !many; ++k) {
    const double waves = (double)((nb * (size_t)k + slots - 1) / slots);
    const double cost = waves * (1.5 + std::max(1.0, (double)tasks / (k * w)));
    if (cost < best) {
      best = cost;
      split = k;
    }
  }
  const dim3 grid(nb, split), block(QN, w, g);
  if constexpr (sizeof(real) == 8)
    if (a.u_pass) {
      const cudaError_t e = launch_velocity<real>(a, s);
      if (e != cudaSuccess) return e;
      if (a.qe == TFKT_QE_STRESS)
        return launch(collide_kernel<real, S, true, true>, grid, block, 0, s, dependent, a);
      return launch(collide_kernel<real, S, false, true>, grid, block, 0, s, dependent, a);
    }
  if (a.qe == TFKT_QE_STRESS)
    return launch(collide_kernel<real, S, true>, grid, block, 0, s, dependent, a);
  return launch(collide_kernel<real, S, false>, grid, block, 0, s, dependent, a);
}

#define TFKT_INSTANTIATE_SPLIT(real, S)                                                   \
  template cudaError_t launch_moments<real, S>(const KernelArgs<real>&, cudaStream_t, bool);  \
  template cudaError_t launch_step<real, S>(const KernelArgs<real>&, cudaStream_t, bool, bool);
TFKT_INSTANTIATE_SPLIT(double, double)
TFKT_INSTANTIATE_SPLIT(float, float)
TFKT_INSTANTIATE_SPLIT(float, __half)
template std::vector<QRow<double>> build_rows<double>(const Lattice&, const HostTables&);
template std::vector<QRow<float>> build_rows<float>(const Lattice&, const HostTables&);

}  // namespace tfkt
