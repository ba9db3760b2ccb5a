// Device kernels of the two-fluid kinetic step (arXiv 2201.10132, Sec. VI-VII).
//
// Storage: structure-of-arrays planes of ny rows x pitch elements, x fastest.
// Population planes 0..8 hold the solvent (D2Q9), plane 9 + 25 q + i the
// polymer velocity i at Q-node q (D4Q25). A buffer holds post-collision g'
// values that have not been streamed yet, stored as deviations from rest:
// g' - w_i (solvent, rho_0 = 1) and g' - w_i psi0(q) (polymer). The pull at
// node r reads g'_i(r - c_r, q - Qdot_i), or g'_{-i}(r, q) when q - Qdot_i
// leaves the Q-disk (bounce-back), and adds the shift difference delta(q, i).
//
// Moment planes M: delta psi(q) (q < nq), then delta rho (total), J_x, J_y
// (total momentum of g), and delta Theta_xx, xy, yy = (H ell^2 / 2) sum_q
// delta psi phi_q Q Q, all of the pulled (pre-collision) state.
#include <type_traits>

#include "tfkt_internal.cuh"

namespace tfkt {

namespace {

// The nine pull offsets of node (x, y): source displaced by (sx, sy).
struct Offsets {
  size_t o[9];
};

__device__ __forceinline__ Offsets node_offsets(int x, int y, int nx, int ny, size_t pitch) {
  const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  const size_t rm = (size_t)ym * pitch, r0 = (size_t)y * pitch, rp = (size_t)yp * pitch;
  Offsets f;
  f.o[0] = rm + xm; f.o[1] = rm + x; f.o[2] = rm + xp;
  f.o[3] = r0 + xm; f.o[4] = r0 + x; f.o[5] = r0 + xp;
  f.o[6] = rp + xm; f.o[7] = rp + x; f.o[8] = rp + xp;
  return f;
}

// ------------------------------------------------------------------ init
// g = f^eq of the initial fields (Sec. VI-D): rho_S = 1, psi = psi0(q),
// U = base flow + perturbation, J^r_eq = psi U, J^Q_eq = psi (Q . grad U -
// kappa Q) (grad_r psi = 0). Each value is written to the slot that the
// first pull reads for it, so the first step starts from exactly this state.
// For the same reason the pulled populations of a node are its own stored
// values: the kernel also writes the state's moment planes M, rebuilding each
// value from its stored form, so the moments need no second pass over the
// populations. Contexts whose steps sum the moments in another order (the Q-split
// kernels) leave the sums out and run the moments pass.
template <typename real, typename S, bool MOMENTS>
__global__ void __launch_bounds__(256) init_kernel(KernelArgs<real> a) {
  using SS = SolventT<S>;
  SS* __restrict__ sdst = solvent_planes<S>(a.dst, a.plane, a.nq);
  S* __restrict__ dst = (S*)a.dst;
  const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  const int nx = a.nx, ny = a.ny;
  auto U0 = [&](int xx, int yy, real& ux, real& uy) {
    const size_t k = (size_t)yy * nx + xx;
    ux = a.tab.urow[yy] + (a.perturb ? real(a.perturb[k]) : real(0));
    uy = a.perturb ? real(a.perturb[(size_t)nx * ny + k]) : real(0);
  };
  const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  real ux, uy, uxa, uya, uxb, uyb;
  U0(x, y, ux, uy);
  U0(xp, y, uxa, uya);
  U0(xm, y, uxb, uyb);
  const real G00 = real(0.5) * (uxa - uxb), G01 = real(0.5) * (uya - uyb);
  U0(x, yp, uxa, uya);
  U0(x, ym, uxb, uyb);
  const real G10 = real(0.5) * (uxa - uxb), G11 = real(0.5) * (uya - uyb);
  const Offsets off = node_offsets(x, y, nx, ny, a.pitch);
  const size_t P = a.plane;
  const real usq = ux * ux + uy * uy;
  real drho = 0, jx = 0, jy = 0;
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const real cu = real(c9x(i)) * ux + real(c9y(i)) * uy;
    const real h = real(w9(i)) * (real(3) * cu + real(4.5) * cu * cu - real(1.5) * usq);
    const SS st = to_store<SS>(h);
    sdst[(size_t)i * P + off.o[shift_index(-c9x(i), -c9y(i))]] = st;
    if (MOMENTS) {
      const real v = from_store<real>(st);
      drho += v;
      jx += real(c9x(i)) * v;
      jy += real(c9y(i)) * v;
    }
  }
  real txx = 0, txy = 0, tyy = 0;
  for (int q = 0; q < a.nq; ++q) {
    const real Qx = a.tab.qx[q], Qy = a.tab.qy[q], psi = a.tab.psi0[q];
    const real Fx = a.tab.fx[q], Fy = a.tab.fy[q];
    const real jrx = psi * ux, jry = psi * uy;
    const real jqx = psi * (Qx * G00 + Qy * G10 - a.kappa * Fx);
    const real jqy = psi * (Qx * G01 + Qy * G11 - a.kappa * Fy);
    real dpsi = 0, rx = 0, ry = 0;
#pragma unroll
    for (int i = 0; i < 25; ++i) {
      const V4 c = c25(i);
      const real h = real(w25(i)) * real(3) *
                     (jrx * real(c.rx) + jry * real(c.ry) + jqx * real(c.qx) + jqy * real(c.qy));
      const int e = a.tab.pull[q * 25 + i];
      const size_t o = e >= 0 ? off.o[shift_index(-c.rx, -c.ry)] : off.o[4];
      const int p = e >= 0 ? e : ~e;
      const S st = to_store<S>((h - a.tab.delta[q * 25 + i]) * a.pscale);
      dst[(size_t)p * P + o] = st;
      if (MOMENTS) {
        const real v = from_store<real>(st) * a.pinv + a.tab.delta[q * 25 + i];
        dpsi += v;
        rx += real(c.rx) * v;
        ry += real(c.ry) * v;
      }
    }
    if (!MOMENTS) continue;
    a.M[(size_t)q * P + off.o[4]] = dpsi;
    drho += dpsi;
    jx += rx;
    jy += ry;
    txx += dpsi * Fx * Qx;
    txy += dpsi * Fx * Qy;
    tyy += dpsi * Fy * Qy;
  }
  if (!MOMENTS) return;
  const size_t n = off.o[4];
  const int nq = a.nq;
  a.M[(size_t)(nq + M_DRHO) * P + n] = drho;
  a.M[(size_t)(nq + M_JX) * P + n] = jx;
  a.M[(size_t)(nq + M_JY) * P + n] = jy;
  a.M[(size_t)(nq + M_THXX) * P + n] = a.hl2h * txx;
  a.M[(size_t)(nq + M_THXY) * P + n] = a.hl2h * txy;
  a.M[(size_t)(nq + M_THYY) * P + n] = a.hl2h * tyy;
}

// ------------------------------------------------------------- observers
template <typename real>
__global__ void __launch_bounds__(256) velocity_kernel(KernelArgs<real> a) {
  const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  real ux, uy, rho;
  mixture_velocity(a, x, y, ux, uy, rho);
  const size_t n = (size_t)y * a.pitch + x;
  a.U[n] = ux;
  a.U[a.plane + n] = uy;
}

// Per-node observables (Sec. VII): rho_S, psi_tot, U, C, Theta, Q_rms, vorticity, the
// ones in `mask`, in FP64 from sums over the Q-nodes: the second moments behind C_xy and
// Theta_xy cancel between Q-nodes of opposite sign, which FP32 sums would resolve only
// to ~1e-7 of the diagonal ones. FP64 arithmetic, 2 lanes per clock and SM, would bound
// the kernel of FP32 contexts: rho_s, U and C of 1024 x 1024 nodes with 32 Q-nodes took
// 767 us (the velocity pass included). There the sums of psi, psi Q Q run over the stored
// deviations in three floats each, which keep what every product and sum rounds away
// (two-sum: Knuth; cascaded: Ogita, Rump and Oishi 2005), and meet the sums of psi0 in
// FP64 at the end: 247 us; with 9 Q-nodes 284 and 159. Two floats per sum (161 and
// 75 us) leave 2^-48 of a sum, more than FP64 sums do; three leave less (2^-70), so the
// result is rounded three times where an FP64 sum is at every Q-node. Theta (the spring
// force is no short binary fraction) and nodes with non-finite or overflowing values are
// summed in FP64. What bounds it: the FP32 issue rate, about 80 instructions per Q-node,
// and about 40 FP64 operations per node after the sums.
constexpr uint32_t FIELDS_PSUM = (1u << TFKT_F_RHO_S) | (1u << TFKT_F_PSI_TOT) | (1u << TFKT_F_CXX) |
                                 (1u << TFKT_F_CXY) | (1u << TFKT_F_CYY) | (1u << TFKT_F_QRMS);
constexpr uint32_t FIELDS_CONF = (1u << TFKT_F_CXX) | (1u << TFKT_F_CXY) | (1u << TFKT_F_CYY) |
                                 (1u << TFKT_F_QRMS);
constexpr uint32_t FIELDS_STRESS = (1u << TFKT_F_THXX) | (1u << TFKT_F_THXY) | (1u << TFKT_F_THYY);

// From this many Q-nodes on: with one the three floats' set-up and end cost more than they save
// (C of 1024 x 1024 nodes, us: 206 with them, 170 in FP64; with 4 138 and 166).
constexpr int EXACT_SUMS_NQ = 4;

// A sum kept in three floats.
struct ExactSum {
  float hi = 0, lo = 0, rest = 0;
  // a += x; returns what the addition rounds away (exact)
  static __device__ __forceinline__ float two_sum(float& a, float x) {
    const float s = __fadd_rn(a, x), b = __fsub_rn(s, a);
    const float r = __fadd_rn(__fsub_rn(a, __fsub_rn(s, b)), __fsub_rn(x, b));
    a = s;
    return r;
  }
  __device__ __forceinline__ void add(float x) {
    rest = __fadd_rn(rest, two_sum(lo, two_sum(hi, x)));
  }
  __device__ __forceinline__ void add(float m, float w) {   // m w: a product and its rounding error
    const float x = __fmul_rn(m, w);
    add(x);
    rest = __fadd_rn(rest, two_sum(lo, __fmaf_rn(m, w, -x)));
  }
  __device__ __forceinline__ double value() const { return (double)hi + ((double)lo + (double)rest); }
};

// Staged once per block: the weights Q Q (xx, xy, yy) of the Q-nodes, exact in FP32
// (quarters of small integers), behind the sums of psi0 with the weights 1, Q Q.
struct FieldRow {
  float w[3];
};
constexpr size_t FIELD_HEAD = 4 * sizeof(double);

__device__ __forceinline__ void stage_field_rows(const KernelArgs<float>& a, double* s0, FieldRow* row) {
  for (int q = threadIdx.y * TX + threadIdx.x; q < a.nq; q += TX * TY) {
    const float Qx = a.tab.qx[q], Qy = a.tab.qy[q];
    row[q] = {{Qx * Qx, Qx * Qy, Qy * Qy}};
  }
  static_assert(TX == 32 && TY >= 4, "one warp per sum of psi0");
  const int j = threadIdx.y;
  if (j >= 4) return;
  double s = 0;
  for (int q = threadIdx.x; q < a.nq; q += 32) {
    const float Qx = a.tab.qx[q], Qy = a.tab.qy[q];
    s += double(a.tab.psi0[q]) * double(j == 0 ? 1.0f : j == 1 ? Qx * Qx : j == 2 ? Qx * Qy : Qy * Qy);
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  if (threadIdx.x == 0) s0[j] = s;
}

// s: sum of delta psi, then of delta psi Q Q (xx, xy, yy) where asked.
template <bool CONF>
__device__ __forceinline__ void exact_sums(const KernelArgs<float>& a, const FieldRow* row, size_t n,
                                           ExactSum (&s)[4]) {
  const size_t P = a.plane;
  const float* mp = a.M + n;
  // the planes four at a time, so that several loads are in flight
  for (int q0 = 0; q0 < a.nq; q0 += 4) {
    float m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = mp[(size_t)(q0 + k < a.nq ? q0 + k : q0) * P];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (q0 + k >= a.nq) break;
      s[0].add(m[k]);
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (CONF) s[1 + j].add(m[k], row[q0 + k].w[j]);
    }
  }
}

template <typename real>
__device__ __forceinline__ void fp64_sums(const KernelArgs<real>& a, size_t n, bool conf, bool stress,
                                       double (&s)[7]) {
  for (int j = 0; j < 7; ++j) s[j] = 0;
  for (int q = 0; q < a.nq; ++q) {
    const double p = double(a.tab.psi0[q]) + double(a.M[(size_t)q * a.plane + n]);
    const double Qx = a.tab.qx[q], Qy = a.tab.qy[q];
    s[0] += p;
    if (conf) {
      s[1] += p * Qx * Qx;
      s[2] += p * Qx * Qy;
      s[3] += p * Qy * Qy;
    }
    if (stress) {
      const double Fx = a.tab.fx[q], Fy = a.tab.fy[q];
      s[4] += p * Fx * Qx;
      s[5] += p * Fx * Qy;
      s[6] += p * Fy * Qy;
    }
  }
}

template <typename real>
__global__ void __launch_bounds__(256) fields_kernel(KernelArgs<real> a, uint32_t mask,
                                                     double* out) {
  extern __shared__ __align__(16) unsigned char field_smem[];
  const bool sums = mask & (FIELDS_PSUM | FIELDS_STRESS);
  const bool conf = mask & FIELDS_CONF, stress = mask & FIELDS_STRESS;
  const int nq = a.nq;
  const bool exact = sums && !stress && nq >= EXACT_SUMS_NQ;
  double* s0 = reinterpret_cast<double*>(field_smem);
  FieldRow* row = reinterpret_cast<FieldRow*>(field_smem + FIELD_HEAD);
  if constexpr (std::is_same<real, float>::value)
    if (exact) {
      stage_field_rows(a, s0, row);
      __syncthreads();
    }
  const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  const size_t P = a.plane, n = (size_t)y * a.pitch + x;
  const size_t N = (size_t)a.nx * a.ny, k = (size_t)y * a.nx + x;
  double f[TFKT_NFIELDS];
  f[TFKT_F_UX] = a.U[n];
  f[TFKT_F_UY] = a.U[P + n];
  const real drho = a.M[(size_t)(nq + M_DRHO) * P + n];
  const int xm = x == 0 ? a.nx - 1 : x - 1, xp = x == a.nx - 1 ? 0 : x + 1;
  const int ym = y == 0 ? a.ny - 1 : y - 1, yp = y == a.ny - 1 ? 0 : y + 1;
  const bool vort = mask & (1u << TFKT_F_VORT);
  double s[7] = {};
  bool done = !sums;
  if constexpr (std::is_same<real, float>::value)
    if (exact) {
      ExactSum es[4];
      if (conf) exact_sums<true>(a, row, n, es);
      else exact_sums<false>(a, row, n, es);
      done = true;   // unless a sum left the range of FP32 or met a non-finite value
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        s[j] = s0[j] + es[j].value();
        done = done && isfinite(es[j].hi);
      }
    }
  if (!done) fp64_sums(a, n, conf, stress, s);
  const double pt = s[0], l2 = a.l2, hh = 0.5 * double(a.H) * l2;
  f[TFKT_F_RHO_S] = double(a.rho0) + double(drho) - pt;
  f[TFKT_F_PSI_TOT] = pt;
  if (conf) {
    const double cxx = pt != 0 ? l2 * s[1] / pt : 0, cxy = pt != 0 ? l2 * s[2] / pt : 0,
                 cyy = pt != 0 ? l2 * s[3] / pt : 0;
    f[TFKT_F_CXX] = cxx;
    f[TFKT_F_CXY] = cxy;
    f[TFKT_F_CYY] = cyy;
    if (mask & (1u << TFKT_F_QRMS)) f[TFKT_F_QRMS] = sqrt(cxx + cyy);
  }
  f[TFKT_F_THXX] = hh * s[4];
  f[TFKT_F_THXY] = hh * s[5];
  f[TFKT_F_THYY] = hh * s[6];
  if (vort) {
    const double duy_dx = 0.5 * (double(a.U[P + (size_t)y * a.pitch + xp]) -
                                 double(a.U[P + (size_t)y * a.pitch + xm]));
    const double dux_dy =
        0.5 * (double(a.U[(size_t)yp * a.pitch + x]) - double(a.U[(size_t)ym * a.pitch + x]));
    f[TFKT_F_VORT] = duy_dx - dux_dy;
  }
  int slot = 0;
#pragma unroll
  for (int j = 0; j < TFKT_NFIELDS; ++j)
    if (mask & (1u << j)) out[(size_t)(slot++) * N + k] = f[j];
}

template <typename real>
__global__ void __launch_bounds__(256) psi_kernel(KernelArgs<real> a, double* out) {
  const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  const size_t n = (size_t)y * a.pitch + x, k = (size_t)y * a.nx + x;
  for (int q = 0; q < a.nq; ++q)
    out[k * a.nq + q] = double(a.tab.psi0[q]) + double(a.M[(size_t)q * a.plane + n]);
}

// Stored populations with the storage shift added back, as doubles.
template <typename real, typename S>
__global__ void __launch_bounds__(256) populations_kernel(KernelArgs<real> a, double* out) {
  const S* src = (const S*)a.src;
  const SolventT<S>* ssrc = solvent_planes<S>(a.src, a.plane, a.nq);
  const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
  if (x >= a.nx || y >= a.ny) return;
  const size_t n = (size_t)y * a.pitch + x, k = (size_t)y * a.nx + x,
               N = (size_t)a.nx * a.ny;
  for (int i = 0; i < 9; ++i)
    out[(size_t)i * N + k] = w9(i) + from_store<double>(ssrc[(size_t)i * a.plane + n]);
  for (int q = 0; q < a.nq; ++q)
    for (int i = 0; i < 25; ++i) {
      const int p = 9 + 25 * q + i;
      out[(size_t)p * N + k] = w25(i) * double(a.tab.psi0[q]) +
                               from_store<double>(src[(size_t)p * a.plane + n]) * double(a.pinv);
    }
}

// Global diagnostics: per-block FP64 partial sums over a fixed node
// partition (grid-stride, fixed order), then one block sums the partials in
// block order: the result does not depend on scheduling.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) v += __shfl_down_sync(0xffffffffu, v, s);
  return v;
}

// Maximum of non-negative values (|u|^2, Q_rms) that keeps a NaN once it has
// met one (fmax would drop it), so that a non-finite node shows in the maximum
// diagnostics too. For IEEE values with the sign bit clear the order of the
// bit patterns read as unsigned integers is the numeric order, and every NaN
// (of either sign) lies above +inf: one integer maximum.
__device__ __forceinline__ float nan_max(float m, float v) {
  return __uint_as_float(max(__float_as_uint(m), __float_as_uint(v)));
}
__device__ __forceinline__ double nan_max(double m, double v) {
  return __longlong_as_double((long long)max((unsigned long long)__double_as_longlong(m),
                                             (unsigned long long)__double_as_longlong(v)));
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) v = nan_max(v, __shfl_down_sync(0xffffffffu, v, s));
  return v;
}
// Diagnostics reduced by maximum rather than by sum.
__host__ __device__ constexpr bool diag_is_max(int j) {
  return j == TFKT_D_U2_MAX || j == TFKT_D_QRMS_MAX;
}

// Block partials of the global diagnostics (Sec. VII follows the enstrophy
// and Q_rms): sums, and the maxima of |u|^2 (a Mach-number guard, since the
// lattice scheme holds only for |u| well below c_s) and of Q_rms. A block takes whole rows, a thread every DIAG_THREADS-th
// node of a row. Per node only what the sums need is formed, in the context's
// precision and as deviations from the rest state (sum_q delta psi, and
// sum_q delta psi Q^2 for Q_rms); the rest-state constants are added once.
// Values are summed in that precision along a row segment of one thread and
// in FP64 across segments, blocks and the final reduction: FP64 arithmetic,
// slow on this GPU, stays out of the per-node work of FP32 contexts, while
// FP64 contexts keep FP64 throughout.
// |Q|^2 of every Q-node is staged in shared memory; a node's moment planes
// are loaded eight at a time so that several loads are in flight per thread
// (the sums still run in Q-node order).
template <typename real>
__global__ void __launch_bounds__(DIAG_THREADS) diag_partial_kernel(KernelArgs<real> a,
                                                                    double* partials) {
  extern __shared__ unsigned char diag_smem[];
  real* q2 = reinterpret_cast<real*>(diag_smem);
  const int nq = a.nq;
  const size_t P = a.plane;
  for (int q = threadIdx.x; q < nq; q += DIAG_THREADS) {
    const real Qx = a.tab.qx[q], Qy = a.tab.qy[q];
    q2[q] = Qx * Qx + Qy * Qy;
  }
  __syncthreads();
  real s0 = 0;   // sum_q psi0(q) |Q|^2 of the rest state
  for (int q = 0; q < nq; ++q) s0 += a.tab.psi0[q] * q2[q];
  double acc[TFKT_NDIAG] = {};
  for (int y = blockIdx.x; y < a.ny; y += gridDim.x) {
    const int ym = y == 0 ? a.ny - 1 : y - 1, yp = y == a.ny - 1 ? 0 : y + 1;
    real r[TFKT_NDIAG] = {};
    for (int x = threadIdx.x; x < a.nx; x += DIAG_THREADS) {
      const size_t n = (size_t)y * a.pitch + x;
      real dpt = 0, sq = 0;
      const real* mp = a.M + n;
      int q = 0;
      for (; q + 8 <= nq; q += 8) {
        real m[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) m[k] = mp[(size_t)(q + k) * P];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          dpt += m[k];
          sq += m[k] * q2[q + k];
        }
      }
      for (; q < nq; ++q) {
        const real m = mp[(size_t)q * P];
        dpt += m;
        sq += m * q2[q];
      }
      const real drho = a.M[(size_t)(nq + M_DRHO) * P + n];
      const real pt = a.psi_tot0 + dpt, rho = a.rho0 + drho;
      const real ux = a.U[n], uy = a.U[P + n];
      const int xm = x == 0 ? a.nx - 1 : x - 1, xp = x == a.nx - 1 ? 0 : x + 1;
      const real w = real(0.5) * (a.U[P + (size_t)y * a.pitch + xp] - a.U[P + (size_t)y * a.pitch + xm]) -
                     real(0.5) * (a.U[(size_t)yp * a.pitch + x] - a.U[(size_t)ym * a.pitch + x]);
      r[TFKT_D_MASS_S] += drho - dpt;   // rho_s minus its rest value rho0 - psi_tot0
      r[TFKT_D_MASS_P] += dpt;          // psi_tot minus psi_tot0
      r[TFKT_D_PX] += rho * ux;
      r[TFKT_D_PY] += rho * uy;
      r[TFKT_D_KE] += real(0.5) * rho * (ux * ux + uy * uy);
      r[TFKT_D_ENSTROPHY] += real(0.5) * w * w;
      const real qrms = pt != real(0) ? sqrt(a.l2 * (s0 + sq) / pt) : real(0);
      r[TFKT_D_QRMS_MEAN] += qrms;
      r[TFKT_D_EY2] += uy * uy;
      r[TFKT_D_U2_MAX] = nan_max(r[TFKT_D_U2_MAX], ux * ux + uy * uy);
      r[TFKT_D_QRMS_MAX] = nan_max(r[TFKT_D_QRMS_MAX], qrms);
    }
#pragma unroll
    for (int j = 0; j < TFKT_NDIAG; ++j)
      acc[j] = diag_is_max(j) ? nan_max(acc[j], double(r[j])) : acc[j] + double(r[j]);
  }
  __shared__ double red[DIAG_THREADS / 32][TFKT_NDIAG];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < TFKT_NDIAG; ++j) {
    const double v = diag_is_max(j) ? warp_max(acc[j]) : warp_sum(acc[j]);
    if (lane == 0) red[warp][j] = v;
  }
  __syncthreads();
  if (threadIdx.x < TFKT_NDIAG) {
    const int j = threadIdx.x;
    double s = 0;
    for (int w = 0; w < DIAG_THREADS / 32; ++w)
      s = diag_is_max(j) ? nan_max(s, red[w][j]) : s + red[w][j];
    partials[(size_t)blockIdx.x * TFKT_NDIAG + j] = s;
  }
}

// base_s, base_p: the masses of the rest state, N (rho0 - psi_tot0) and N psi_tot0.
// One warp per diagnostic: lanes stride over the block partials, then a fixed
// shuffle tree (the order does not depend on scheduling).
__global__ void diag_final_kernel(const double* partials, int nblocks, double inv_n, double base_s,
                                  double base_p, double* out) {
  const int j = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (j >= TFKT_NDIAG) return;
  const bool mx = diag_is_max(j);
  double s = 0;
  for (int b = lane; b < nblocks; b += 32) {
    const double v = partials[(size_t)b * TFKT_NDIAG + j];
    s = mx ? nan_max(s, v) : s + v;
  }
  s = mx ? warp_max(s) : warp_sum(s);
  if (lane == 0) {
    if (j == TFKT_D_MASS_S) s += base_s;
    if (j == TFKT_D_MASS_P) s += base_p;
    if (j == TFKT_D_QRMS_MEAN) s *= inv_n;
    if (j == TFKT_D_U2_MAX) s = sqrt(s);   // reported as max |u|
    out[j] = s;
  }
}

inline dim3 node_grid(int nx, int ny) { return dim3((nx + TX - 1) / TX, (ny + TY - 1) / TY); }

}  // namespace

template <typename real, typename S>
cudaError_t launch_init(const KernelArgs<real>& a, bool moments, cudaStream_t s) {
  const dim3 grid = node_grid(a.nx, a.ny), block(TX, TY);
  if (moments) init_kernel<real, S, true><<<grid, block, 0, s>>>(a);
  else init_kernel<real, S, false><<<grid, block, 0, s>>>(a);
  return cudaGetLastError();
}
template <typename real>
cudaError_t launch_velocity(const KernelArgs<real>& a, cudaStream_t s) {
  velocity_kernel<real><<<node_grid(a.nx, a.ny), dim3(TX, TY), 0, s>>>(a);
  return cudaGetLastError();
}
template <typename real>
cudaError_t launch_fields(const KernelArgs<real>& a, uint32_t mask, double* out, cudaStream_t s) {
  const size_t smem = sizeof(real) == 4 ? FIELD_HEAD + (size_t)a.nq * sizeof(FieldRow) : 0;
  cudaError_t e = allow_dynamic_smem(fields_kernel<real>, smem);
  if (e != cudaSuccess) return e;
  fields_kernel<real><<<node_grid(a.nx, a.ny), dim3(TX, TY), smem, s>>>(a, mask, out);
  return cudaGetLastError();
}
template <typename real>
cudaError_t launch_psi(const KernelArgs<real>& a, double* out, cudaStream_t s) {
  psi_kernel<real><<<node_grid(a.nx, a.ny), dim3(TX, TY), 0, s>>>(a, out);
  return cudaGetLastError();
}
template <typename real, typename S>
cudaError_t launch_populations(const KernelArgs<real>& a, double* out, cudaStream_t s) {
  populations_kernel<real, S><<<node_grid(a.nx, a.ny), dim3(TX, TY), 0, s>>>(a, out);
  return cudaGetLastError();
}
template <typename real>
cudaError_t launch_diag(const KernelArgs<real>& a, double* partials, int nblocks, double* out,
                        cudaStream_t s) {
  diag_partial_kernel<real><<<nblocks, DIAG_THREADS, (size_t)a.nq * sizeof(real), s>>>(a, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const double N = (double)a.nx * a.ny;
  diag_final_kernel<<<1, 32 * TFKT_NDIAG, 0, s>>>(partials, nblocks, 1.0 / N,
                                     N * ((double)a.rho0 - (double)a.psi_tot0), N * (double)a.psi_tot0,
                                     out);
  return cudaGetLastError();
}

#define TFKT_INSTANTIATE_POP(real, S)                                                          \
  template cudaError_t launch_init<real, S>(const KernelArgs<real>&, bool, cudaStream_t);     \
  template cudaError_t launch_populations<real, S>(const KernelArgs<real>&, double*,          \
                                                   cudaStream_t);
#define TFKT_INSTANTIATE(real)                                                                 \
  template cudaError_t launch_velocity<real>(const KernelArgs<real>&, cudaStream_t);          \
  template cudaError_t launch_fields<real>(const KernelArgs<real>&, uint32_t, double*,        \
                                           cudaStream_t);                                     \
  template cudaError_t launch_psi<real>(const KernelArgs<real>&, double*, cudaStream_t);      \
  template cudaError_t launch_diag<real>(const KernelArgs<real>&, double*, int, double*,      \
                                         cudaStream_t);
TFKT_INSTANTIATE(float)
TFKT_INSTANTIATE(double)
TFKT_INSTANTIATE_POP(double, double)
TFKT_INSTANTIATE_POP(float, float)
TFKT_INSTANTIATE_POP(float, __half)

}  // namespace tfkt
