// Explicit right-hand side of one RK3 sub-step (Sec. 2.2, delta form):
//   r_i = dt [ -gamma_k N_i(u) - zeta_k N_prev_i - alpha_k G_i p + (alpha_k / Re) L u_i + alpha_k f_i ]
// N is the divergence-form convection of Eq. (NSmomentum) with 2nd-order central differences on
// the staggered grid: fluxes at faces / edges from arithmetic averages in x and z and
// distance-weighted linear interpolation in y.  L is the viscous operator (uniform second
// differences in x and z, the three-point non-uniform formula in y).  G is the pressure gradient.
//
// RhsFxK: the FP64 form, in 64-bit fixed point.  The mixed form (FP32): RhsTiledK where nx is a
// multiple of 32, else RhsK, one thread per (i, j) of one z-plane, j = 0..ny (row ny only writes the v
// wall row).  T is the arithmetic type, TR the storage type of r and N.
#include "ns_internal.cuh"

namespace {

struct RhsArgs {
  const double* __restrict__ u;
  const double* __restrict__ v;
  const double* __restrict__ w;
  const double* __restrict__ p;
  void* ru;
  void* rv;
  void* rw;
  void* nu;
  void* nv;
  void* nw;
  const double* __restrict__ gc;
  const double* __restrict__ rt;  // per-j assembly coefficients of this sub-step (RT_* rows)
  const float* __restrict__ rtf;  // the same rows in float (read by the FP32 form)
  // inflow / outflow in x (bl = 1): boundary planes, index k * rows + j
  int bl;
  const double* __restrict__ u_out;
  const double* __restrict__ v_in;
  const double* __restrict__ v_out;
  const double* __restrict__ w_in;
  const double* __restrict__ w_out;
  int nx, ny, nz;
  double idx, idz, idx2, idz2;
  double dt, gam, zet, alp, inv_re, fx;
  double cprev;     // zeta_k / gamma_(k-1): weight of the stored (pre-multiplied) N of sub-step k-1
  const StepK* sk;  // dt-dependent constants of this sub-step (device; read by the Dyn variants)
  StepK kc;         // the same values as kernel arguments (read by the fixed-dt variants)
};

}  // namespace

namespace {

// The right-hand side at (i, j, k): u, w of cell row j (j < ny) and v of face row j (zero on the walls);
// stored if `store`
template <typename T, typename TR>
__device__ __forceinline__ void rhs_cell(const RhsArgs& a, int i, int j, int k, T dt, bool store) {
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const int ip = (i + 1 == nx) ? 0 : i + 1;
  const int im = (i == 0) ? nx - 1 : i - 1;
  const int kp = (k + 1 == nz) ? 0 : k + 1;
  const int km = (k == 0) ? nz - 1 : k - 1;
  const int ny1 = ny + 1;
  const int G = ny + 1;  // stride of the coefficient arrays

  // x-neighbours: periodic wrap, or (bl) the outflow plane / linear ghosts of the boundary faces
  const bool bl = a.bl != 0;
  const int ipx = bl ? i + 1 : ip, imx = bl ? i - 1 : im;
  auto U = [&](int ii, int jj, int kk) -> T {
    if (ii == nx) return from_double<T>(__ldg(a.u_out + (long)kk * ny + jj));
    if (ii < 0) return (T)0;
    return from_double<T>(__ldg(a.u + ((long)kk * ny + jj) * nx + ii));
  };
  auto V = [&](int ii, int jj, int kk) -> T {
    if (ii == nx) return from_double<T>(2.0 * __ldg(a.v_out + (long)kk * ny1 + jj) - __ldg(a.v + ((long)kk * ny1 + jj) * nx + nx - 1));
    if (ii < 0) return from_double<T>(2.0 * __ldg(a.v_in + (long)kk * ny1 + jj) - __ldg(a.v + ((long)kk * ny1 + jj) * nx));
    return from_double<T>(__ldg(a.v + ((long)kk * ny1 + jj) * nx + ii));
  };
  auto W = [&](int ii, int jj, int kk) -> T {
    if (ii == nx) return from_double<T>(2.0 * __ldg(a.w_out + (long)kk * ny + jj) - __ldg(a.w + ((long)kk * ny + jj) * nx + nx - 1));
    if (ii < 0) return from_double<T>(2.0 * __ldg(a.w_in + (long)kk * ny + jj) - __ldg(a.w + ((long)kk * ny + jj) * nx));
    return from_double<T>(__ldg(a.w + ((long)kk * ny + jj) * nx + ii));
  };
  auto Pp = [&](int ii, int jj, int kk) -> T {
    if (ii < 0 || ii == nx) return (T)0;
    return from_double<T>(__ldg(a.p + ((long)kk * ny + jj) * nx + ii));
  };
  auto C = [&](int f, int jj) -> T { return from_double<T>(__ldg(a.gc + f * G + jj)); };

  const T idx = (T)a.idx, idz = (T)a.idz, idx2 = (T)a.idx2, idz2 = (T)a.idz2;
  const T alp = (T)a.alp;
  const T avis = (T)(a.alp * a.inv_re);
  // N is stored pre-multiplied by cn = -dt gamma_k, as in the tiled form; the stored N of the
  // previous sub-step enters with zeta_k / gamma_(k-1)
  const T cn = -dt * (T)a.gam, cpn = (T)a.cprev;
  const T half = (T)0.5, quarter = (T)0.25, two = (T)2;

  TR* ru = (TR*)a.ru;
  TR* rv = (TR*)a.rv;
  TR* rw = (TR*)a.rw;
  TR* nu = (TR*)a.nu;
  TR* nv = (TR*)a.nv;
  TR* nw = (TR*)a.nw;

  if (j < ny) {
    const long cc = ((long)k * ny + j) * nx + i;
    const T idy = C(GC_IDY, j);
    // ---------------- u at (xf_i, yc_j, zc_k)
    {
      const T u0 = U(i, j, k), uxp = U(ipx, j, k), uxm = U(imx, j, k);
      const T uzp = U(i, j, kp), uzm = U(i, j, km);
      const T uyp = (j + 1 < ny) ? U(i, j + 1, k) : (T)0;
      const T uym = (j > 0) ? U(i, j - 1, k) : (T)0;
      const T sr = u0 + uxp, sl = uxm + u0;
      const T nux = (sr * sr - sl * sl) * (quarter * idx);
      T ft = 0, fb = 0;
      if (j + 1 < ny) {
        const T ut = C(GC_WLO, j + 1) * u0 + C(GC_WHI, j + 1) * uyp;
        ft = ut * (V(imx, j + 1, k) + V(i, j + 1, k));
      }
      if (j > 0) {
        const T ub = C(GC_WLO, j) * uym + C(GC_WHI, j) * u0;
        fb = ub * (V(imx, j, k) + V(i, j, k));
      }
      const T nuy = (ft - fb) * (half * idy);
      const T nuz = ((u0 + uzp) * (W(imx, j, kp) + W(i, j, kp)) - (uzm + u0) * (W(imx, j, k) + W(i, j, k))) *
                    (quarter * idz);
      const T n = nux + nuy + nuz;
      const T ac = C(GC_AC, j), cy = C(GC_CC, j);
      const T lap = (uxp - two * u0 + uxm) * idx2 + (uzp - two * u0 + uzm) * idz2 + ac * uym -
                    (ac + cy) * u0 + cy * uyp;
      const T gp = (Pp(i, j, k) - Pp(imx, j, k)) * idx;
      const T nt = cn * n;
      T r = dt * (-alp * gp + avis * lap + (T)(a.alp * a.fx)) + nt;
      if (a.zet != 0.0) r += cpn * (T)nu[cc];
      const bool fixed = bl && i == 0;  // inflow face
      if (store) {
        ru[cc] = fixed ? (TR)0 : (TR)r;
        nu[cc] = fixed ? (TR)0 : (TR)nt;
      }
    }
    // ---------------- w at (xc_i, yc_j, zf_k)
    {
      const T w0 = W(i, j, k), wxp = W(ipx, j, k), wxm = W(imx, j, k);
      const T wzp = W(i, j, kp), wzm = W(i, j, km);
      const T wyp = (j + 1 < ny) ? W(i, j + 1, k) : (T)0;
      const T wym = (j > 0) ? W(i, j - 1, k) : (T)0;
      const T fr = (U(ipx, j, km) + U(ipx, j, k)) * (w0 + wxp);
      const T fl = (U(i, j, km) + U(i, j, k)) * (wxm + w0);
      const T nwx = (fr - fl) * (quarter * idx);
      T gt = 0, gb = 0;
      if (j + 1 < ny) gt = (V(i, j + 1, km) + V(i, j + 1, k)) * (C(GC_WLO, j + 1) * w0 + C(GC_WHI, j + 1) * wyp);
      if (j > 0) gb = (V(i, j, km) + V(i, j, k)) * (C(GC_WLO, j) * wym + C(GC_WHI, j) * w0);
      const T nwy = (gt - gb) * (half * idy);
      const T cf = w0 + wzp, cb = wzm + w0;
      const T nwz = (cf * cf - cb * cb) * (quarter * idz);
      const T n = nwx + nwy + nwz;
      const T ac = C(GC_AC, j), cy = C(GC_CC, j);
      const T lap = (wxp - two * w0 + wxm) * idx2 + (wzp - two * w0 + wzm) * idz2 + ac * wym -
                    (ac + cy) * w0 + cy * wyp;
      const T gp = (Pp(i, j, k) - Pp(i, j, km)) * idz;
      const T nt = cn * n;
      T r = dt * (-alp * gp + avis * lap) + nt;
      if (a.zet != 0.0) r += cpn * (T)nw[cc];
      if (store) {
        rw[cc] = (TR)r;
        nw[cc] = (TR)nt;
      }
    }
  }
  // ---------------- v at (xc_i, yf_j, zc_k)
  {
    const long cf = ((long)k * ny1 + j) * nx + i;
    if (j == 0 || j == ny) {
      if (store) rv[cf] = nv[cf] = (TR)0;
      return;
    }
    const T v0 = V(i, j, k), vxp = V(ipx, j, k), vxm = V(imx, j, k);
    const T vzp = V(i, j, kp), vzm = V(i, j, km);
    const T vyp = V(i, j + 1, k), vym = V(i, j - 1, k);
    const T wl = C(GC_WLO, j), wh = C(GC_WHI, j);
    const T fr = (wl * U(ipx, j - 1, k) + wh * U(ipx, j, k)) * (v0 + vxp);
    const T fl = (wl * U(i, j - 1, k) + wh * U(i, j, k)) * (vxm + v0);
    const T nvx = (fr - fl) * (half * idx);
    const T ct = v0 + vyp, cb = vym + v0;
    const T ihc = C(GC_IHC, j);
    const T nvy = (ct * ct - cb * cb) * (quarter * ihc);
    const T gf = (v0 + vzp) * (wl * W(i, j - 1, kp) + wh * W(i, j, kp));
    const T gb = (vzm + v0) * (wl * W(i, j - 1, k) + wh * W(i, j, k));
    const T nvz = (gf - gb) * (half * idz);
    const T n = nvx + nvy + nvz;
    const T af = C(GC_AF, j), cyf = C(GC_CF, j);
    const T lap = (vxp - two * v0 + vxm) * idx2 + (vzp - two * v0 + vzm) * idz2 + af * vym -
                  (af + cyf) * v0 + cyf * vyp;
    const T gp = (Pp(i, j, k) - Pp(i, j - 1, k)) * ihc;
    const T nt = cn * n;
    T r = dt * (-alp * gp + avis * lap) + nt;
    if (a.zet != 0.0) r += cpn * (T)nv[cf];
    if (store) {
      rv[cf] = (TR)r;
      nv[cf] = (TR)nt;
    }
  }
}

// One thread per (i, j): the FP32 form on grids the tile does not fit.  Dyn: the sub-step constants
// are read from device memory (a step graph that outlives changes of dt); otherwise from the kernel
// arguments, where they cost no registers.
template <typename T, typename TR, bool Dyn>
struct RhsK {
  struct Args {
    RhsArgs a;
  };
  static constexpr int kThreads = 128;
  static constexpr int kMinBlocks = 7;
  static Args make(RhsArgs a) { return Args{a}; }
  static __device__ __forceinline__ void run(const Args& a_, const dim3 bid_, const dim3) {
    const RhsArgs& a = a_.a;
    const long q = (long)bid_.x * blockDim.x + threadIdx.x;
    if (q >= (long)a.nx * (a.ny + 1)) return;
    const int j = (int)(q / a.nx);
    rhs_cell<T, TR>(a, (int)(q - (long)j * a.nx), j, bid_.y, (T)(Dyn ? a.sk->dt : a.kc.dt), true);
  }
};

// ---------------------------------------------------------------------------------------------
// Tiled form of the same right-hand side in FP32 (mixed form).  A block of TX x TZ threads owns a TX (x) by TZ (z)
// column of cells and marches along y over [jb, je).  Four rolling planes of u, v, w, p (with a
// one-cell halo in x and z, periodic wrap) sit in shared memory.  Every product the
// divergence-form convection needs is computed once per tile and then differenced:
//   centre squares  Q1 = (u_i + u_{i+1})^2, Q2 = (v_j + v_{j+1})^2, Q3 = (w_k + w_{k+1})^2
//   edge fluxes     Fuv = u(yf_j) (v_{i-1} + v_i)       at (xf_i, yf_j)
//                   Fuw = (u_{k-1} + u_k)(w_{i-1} + w_i) at (xf_i, zf_k)
//                   Fvw = (v_{k-1} + v_k) w(yf_j)       at (yf_j, zf_k)
// (factors 1/2, 1/4 of the averages are folded into the difference weights).  y-face fluxes of
// face j+1 become those of face j in the next step; Q2 of centre j is kept in a register.
// ---------------------------------------------------------------------------------------------
constexpr int RT_X = 32;
constexpr int RT_Z = 8;
constexpr int RT_PX = RT_X + 2;   // plane pitch (x halo on both sides)
constexpr int RT_PZ = RT_Z + 2;
constexpr int RT_PLANE = RT_PX * RT_PZ;
constexpr int RT_NPL = 4;         // rolling planes per field

struct RhsTile {
  using T = float;
  T pl[4][RT_NPL][RT_PLANE];                 // u, v, w, p planes (j mod 4), index (kk+1)*RT_PX + (ii+1)
  T fuv[2][RT_Z][RT_X + 1];                  // Fuv on y-face (parity), x = i0 .. i0+TX
  T fvw[2][RT_Z + 1][RT_X];                  // Fvw on y-face (parity), z = k0 .. k0+TZ
  T q1[RT_Z][RT_X + 1];                      // x = i0-1 .. i0+TX-1
  T q3[RT_Z + 1][RT_X];                      // z = k0-1 .. k0+TZ-1
  T fuw[RT_Z + 1][RT_X + 1];                 // x = i0 .. i0+TX, z = k0 .. k0+TZ
  T rt[RT_NPL][RT_COUNT];                    // per-row assembly coefficients of row j (j mod 4)
  T wf[RT_NPL];                              // RHO = WHI / WLO of face j (j mod 4), zero at the walls
};

// 8-byte global -> shared copy that completes asynchronously (cp.async, waited for by
// cp.async.wait_all); with valid false nothing is read and the 8 bytes are zero-filled
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, bool valid) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(valid ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all8() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// State values enter by the hardware conversion (one instruction on the FP64 pipe, which the FP32
// RHS leaves idle) instead of the integer-pipe d2f_rn (about a dozen instructions on this issue-bound
// kernel).
template <bool Dyn>
struct RhsTiledK {
  using T = float;
  struct Args {
    RhsArgs a;
    int jchunk;
  };
  static constexpr int kThreads = RT_X * RT_Z;
  // 6 blocks of up to 40 registers (the kernel waits on memory and shared memory, so occupancy pays
  // more than registers: 0.314 ms at 6 blocks against 0.338 at 5, 0.352 at 4 and 0.434 at 3), or 4
  // of up to 64 when the sub-step constants come from device memory (fewer spill)
  static constexpr int kMinBlocks = Dyn ? 4 : 6;
  static Args make(RhsArgs a, int jchunk) { return Args{a, jchunk}; }
  static __device__ __forceinline__ void run(const Args& a_, const dim3 bid_, const dim3 gdim_) {
    const RhsArgs& a = a_.a;
    const int i0 = bid_.x * RT_X, k0 = bid_.y * RT_Z;
    const int jb = bid_.z * a_.jchunk;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  RhsTile& S = *reinterpret_cast<RhsTile*>(smem_raw);
  const int nx = a.nx, ny = a.ny, nz = a.nz, ny1 = ny + 1, G = ny + 1;
  const int tx = threadIdx.x, tz = threadIdx.y, tid = tz * RT_X + tx;
  const int je = min(jb + a_.jchunk, ny);
  const int jlast = (je == ny) ? ny : je - 1;  // v rows: the last chunk also writes face ny

  auto P = [&](int f, int j, int kk, int ii) -> T& { return S.pl[f][j & 3][(kk + 1) * RT_PX + ii + 1]; };

  // Plane loads.  Each thread owns up to two positions of the (RT_PZ x RT_PX) halo plane and
  // loads all four fields there, so the index arithmetic (wrap, offsets) is done once per thread
  // and only j changes between planes.  u, w, p share the offset of a centre; v has its own.
  // Positions on the x boundary of an inflow / outflow domain take the boundary planes instead.
  constexpr int kPos = (RT_PLANE + RT_X * RT_Z - 1) / (RT_X * RT_Z);
  long oc[kPos], ov[kPos];
  int pos[kPos];  // plane index e, -1 if unused, or -(e + 2) for an x-boundary halo position
#pragma unroll
  for (int r = 0; r < kPos; ++r) {
    const int e = tid + r * RT_X * RT_Z;
    pos[r] = -1;
    oc[r] = 0;
    ov[r] = 0;
    if (e < RT_PLANE) {
      const int kk = e / RT_PX - 1, ii = e % RT_PX - 1;
      int gi = i0 + ii, gk = k0 + kk;
      gk = gk < 0 ? gk + nz : (gk >= nz ? gk - nz : gk);
      if (a.bl && (gi < 0 || gi >= nx)) {
        pos[r] = -(e + 2);
        oc[r] = gk;
      } else {
        gi = gi < 0 ? gi + nx : (gi >= nx ? gi - nx : gi);
        pos[r] = e;
        oc[r] = (long)gk * ny * nx + gi;
        ov[r] = (long)gk * ny1 * nx + gi;
      }
    }
  }
  auto load_plane = [&](int j) {
    const bool jc = j >= 0 && j < ny, jv = j >= 0 && j <= ny;
    const long jo = (long)j * nx;
#pragma unroll
    for (int r = 0; r < kPos; ++r) {
      if (pos[r] >= 0) {
        const int e = pos[r];
        const long o = oc[r] + jo, q = ov[r] + jo;
        T vu = (T)0, vv = (T)0, vw = (T)0, vp = (T)0;
        if (jc) {
          vu = __double2float_rn(__ldg(a.u + o));
          vw = __double2float_rn(__ldg(a.w + o));
          vp = __double2float_rn(__ldg(a.p + o));
        }
        if (jv) vv = __double2float_rn(__ldg(a.v + q));
        S.pl[0][j & 3][e] = vu;
        S.pl[1][j & 3][e] = vv;
        S.pl[2][j & 3][e] = vw;
        S.pl[3][j & 3][e] = vp;
      } else if (pos[r] < -1) {
        // x-boundary halo: outflow plane of u, linear ghosts of v and w, nothing for p
        const int e = -pos[r] - 2;
        const int gk = (int)oc[r];
        const bool out = i0 + e % RT_PX - 1 >= nx;
        T vu = (T)0, vv = (T)0, vw = (T)0;
        if (out && jc) vu = from_double<T>(__ldg(a.u_out + (long)gk * ny + j));
        if (jv) {
          const double b = __ldg((out ? a.v_out : a.v_in) + (long)gk * ny1 + j);
          vv = from_double<T>(2.0 * b - __ldg(a.v + ((long)gk * ny1 + j) * nx + (out ? nx - 1 : 0)));
        }
        if (jc) {
          const double b = __ldg((out ? a.w_out : a.w_in) + (long)gk * ny + j);
          vw = from_double<T>(2.0 * b - __ldg(a.w + ((long)gk * ny + j) * nx + (out ? nx - 1 : 0)));
        }
        S.pl[0][j & 3][e] = vu;
        S.pl[1][j & 3][e] = vv;
        S.pl[2][j & 3][e] = vw;
        S.pl[3][j & 3][e] = (T)0;
      }
    }
  };
  // Each product loop gives every thread the item q = tid first (every loop has at least 256
  // items); that item's tile offsets are worked out once, before the march in y, and only the few
  // items q >= 256 take the general index arithmetic: the FP32 RHS is issue-bound.
  const int hk = tid / (RT_X + 1), hi = tid % (RT_X + 1);   // items of the (RT_X + 1)-wide loops
  const int gk = tid / RT_X, gi = tid % RT_X;               // items of the RT_X-wide loops
  const int eA = (hk + 1) * RT_PX + hi + 1, fA = hk * (RT_X + 1) + hi;
  const int eB = (gk + 1) * RT_PX + gi + 1, fB = gk * RT_X + gi;
  auto PL = [&](int f, int j) -> T* { return S.pl[f][j & 3]; };
  // y-face fluxes on face jf, zero on the walls, each divided by the interpolation weight WLO_jf
  // (which the difference weights carry): Fuv = (u_{j-1} + RHO u_j)(v_{i-1} + v_i) and
  // Fvw = (v_{k-1} + v_k)(w_{j-1} + RHO w_j), one FMA, one add and one product each
  // Every product loop has NT <= n < 2 NT items: thread tid takes item tid, and the n - NT items past
  // NT go to the threads from `off` on: Fuv and Q1's extra items to warp 0, Fvw and Q3's to warp 1
  // and Fuw's to warps 2 and 3, so that the four SM sub-partitions (warp w issues on sub-partition w
  // mod 4) share them (0.242 -> 0.237 ms).
  constexpr int NT = RT_X * RT_Z;
  auto second = [&](int n, int off) {
    const int x = tid - off;
    return (x >= 0 && x < n - NT) ? NT + x : -1;
  };
  auto face_fluxes = [&](int jf) {
    const bool inner = jf >= 1 && jf <= ny - 1;
    const T rho = S.wf[jf & 3];
    auto fuv_at = [&](int q) {
      const int kk = q / (RT_X + 1), ii = q % (RT_X + 1);
      T f = 0;
      if (inner)
        f = (P(0, jf - 1, kk, ii) + rho * P(0, jf, kk, ii)) * (P(1, jf, kk, ii - 1) + P(1, jf, kk, ii));
      S.fuv[jf & 1][kk][ii] = f;
    };
    auto fvw_at = [&](int q) {
      const int kk = q / RT_X, ii = q % RT_X;
      T f = 0;
      if (inner)
        f = (P(1, jf, kk - 1, ii) + P(1, jf, kk, ii)) * (P(2, jf - 1, kk, ii) + rho * P(2, jf, kk, ii));
      S.fvw[jf & 1][kk][ii] = f;
    };
    const T* u0 = PL(0, jf - 1);
    const T* u1 = PL(0, jf);
    const T* v1 = PL(1, jf);
    const T* w0 = PL(2, jf - 1);
    const T* w1 = PL(2, jf);
    (&S.fuv[jf & 1][0][0])[fA] = inner ? (u0[eA] + rho * u1[eA]) * (v1[eA - 1] + v1[eA]) : (T)0;
    (&S.fvw[jf & 1][0][0])[fB] = inner ? (v1[eB - RT_PX] + v1[eB]) * (w0[eB] + rho * w1[eB]) : (T)0;
    if (const int q = second(RT_Z * (RT_X + 1), 0); q >= 0) fuv_at(q);
    if (const int q = second((RT_Z + 1) * RT_X, 32); q >= 0) fvw_at(q);
  };
  // centre-plane products of plane j (Q1, Q3, Fuw)
  auto centre_products = [&](int j) {
    auto q1_at = [&](int q) {
      const int kk = q / (RT_X + 1), ii = q % (RT_X + 1) - 1;
      const T s = P(0, j, kk, ii) + P(0, j, kk, ii + 1);
      S.q1[kk][ii + 1] = s * s;
    };
    auto q3_at = [&](int q) {
      const int kk = q / RT_X - 1, ii = q % RT_X;
      const T s = P(2, j, kk, ii) + P(2, j, kk + 1, ii);
      S.q3[kk + 1][ii] = s * s;
    };
    auto fuw_at = [&](int q) {
      const int kk = q / (RT_X + 1), ii = q % (RT_X + 1);
      S.fuw[kk][ii] = (P(0, j, kk - 1, ii) + P(0, j, kk, ii)) * (P(2, j, kk, ii - 1) + P(2, j, kk, ii));
    };
    const T* u = PL(0, j);
    const T* w = PL(2, j);
    const T s1 = u[eA - 1] + u[eA];  // Q1 item: x = i0 - 1 + hi, z row hk
    (&S.q1[0][0])[fA] = s1 * s1;
    const T s3 = w[eB - RT_PX] + w[eB];  // Q3 item: z = k0 - 1 + gk
    (&S.q3[0][0])[fB] = s3 * s3;
    (&S.fuw[0][0])[fA] = (u[eA - RT_PX] + u[eA]) * (w[eA - 1] + w[eA]);
    if (const int q = second(RT_Z * (RT_X + 1), 0); q >= 0) q1_at(q);
    if (const int q = second((RT_Z + 1) * RT_X, 32); q >= 0) q3_at(q);
    if (const int q = second((RT_Z + 1) * (RT_X + 1), 64); q >= 0) fuw_at(q);
  };

  // r = cn N + cp N_prev + cgx (p_i - p_{i-1}) + cx (f_{i+1} + f_{i-1}) + cz (f_{k+1} + f_{k-1})
  //     + cA f_{j-1} + cC f_{j+1} + cD f (+ cb for u), with every constant pre-multiplied by dt;
  // cn N is formed directly (the difference weights carry cn) and stored as the next N_prev
  auto K = [&](int q) -> T {
    const StepK& sk = Dyn ? *a.sk : a.kc;
    return sk.kf[q];
  };
  const T qidx = K(RK_QIDX), qidz = K(RK_QIDZ);
  const T cp = K(RK_CP), cgx = K(RK_CGX), cgz = K(RK_CGZ), cx = K(RK_CX), cz = K(RK_CZ);
  const T cb = K(RK_CB);
  const bool use_prev = a.zet != 0.0;
  auto R = [&](int f, int jj) -> T {
    return __ldg(a.rtf + f * G + jj);
  };
  T* ru = (T*)a.ru;
  T* rv = (T*)a.rv;
  T* rw = (T*)a.rw;
  T* nu = (T*)a.nu;
  T* nv = (T*)a.nv;
  T* nw = (T*)a.nw;
  const int i = i0 + tx, k = k0 + tz;

  // The per-row coefficients every thread of the block reads (R, and the face weights of the
  // y fluxes) are fetched by a few threads into a small ring in shared memory, one step ahead of
  // their use, instead of by every thread through the read-only path.
  auto fetch_face = [&](int jf) { S.wf[jf & 3] = (jf >= 1 && jf <= ny - 1) ? R(RT_RHO, jf) : (T)0; };
  // prologue: planes jb-1, jb; fluxes of face jb; Q2 of centre jb-1
  load_plane(jb - 1);
  load_plane(jb);
  if (tid == 0) fetch_face(jb);
  __syncthreads();
  face_fluxes(jb);
  T q2prev = 0;
  {
    const T s = P(1, jb - 1, tz, tx) + P(1, jb, tz, tx);
    q2prev = (jb >= 1) ? s * s : (T)0;
  }
  for (int j = jb; j <= jlast; ++j) {
    if (tid < RT_COUNT) S.rt[j & 3][tid] = R(tid, j);
    else if (tid == RT_COUNT) fetch_face(j + 1);
    load_plane(j + 1);
    __syncthreads();
    face_fluxes(j + 1);
    centre_products(j);
    __syncthreads();
    // The three components are assembled in one straight-line block (v also on the wall faces
    // and u, w also on the face row j = ny, where the planes read are zero and the results are
    // not stored), so that the compiler can interleave their three chains.
    const bool vrow = j > 0 && j < ny;  // interior v face
    const bool crow = j < ny;           // a row of cells
    const long cf = ((long)k * ny1 + j) * nx + i;
    const long cc = ((long)k * ny + (crow ? j : 0)) * nx + i;
    const T* rt = S.rt[j & 3];
    // ---------------- v at face j
    const T sv = P(1, j, tz, tx) + P(1, j + 1, tz, tx);
    const T q2 = sv * sv;  // Q2 of centre j (zero planes beyond the top)
    const T nvv = (S.fuv[j & 1][tz][tx + 1] - S.fuv[j & 1][tz][tx]) * rt[RT_HXW] + (q2 - q2prev) * rt[RT_QIHC] +
                  (S.fvw[j & 1][tz + 1][tx] - S.fvw[j & 1][tz][tx]) * rt[RT_HZW];
    q2prev = q2;
    const T v0 = P(1, j, tz, tx);
    T rv_ = nvv + rt[RT_CGY] * (P(3, j, tz, tx) - P(3, j - 1, tz, tx));
    rv_ += cx * (P(1, j, tz, tx + 1) + P(1, j, tz, tx - 1));
    rv_ += cz * (P(1, j, tz + 1, tx) + P(1, j, tz - 1, tx));
    // one FMA per term on r (a sum of the three products first would add an instruction)
    rv_ += rt[RT_AF] * P(1, j - 1, tz, tx);
    rv_ += rt[RT_CF] * P(1, j + 1, tz, tx);
    rv_ += rt[RT_DF] * v0;
    // ---------------- u at (xf_i, yc_j, zc_k)
    const T hym = rt[RT_HYM], hyp = rt[RT_HYP];
    const T cA = rt[RT_AC], cC = rt[RT_CC], cD = rt[RT_DC];
    const T u0 = P(0, j, tz, tx);
    const T nuu = (S.q1[tz][tx + 1] - S.q1[tz][tx]) * qidx +
                  S.fuv[(j + 1) & 1][tz][tx] * hyp + S.fuv[j & 1][tz][tx] * hym +
                  (S.fuw[tz + 1][tx] - S.fuw[tz][tx]) * qidz;
    T ru_ = nuu + cb + cgx * (P(3, j, tz, tx) - P(3, j, tz, tx - 1));
    ru_ += cx * (P(0, j, tz, tx + 1) + P(0, j, tz, tx - 1));
    ru_ += cz * (P(0, j, tz + 1, tx) + P(0, j, tz - 1, tx));
    ru_ += cA * P(0, j - 1, tz, tx);
    ru_ += cC * P(0, j + 1, tz, tx);
    ru_ += cD * u0;
    // ---------------- w at (xc_i, yc_j, zf_k)
    const T w0 = P(2, j, tz, tx);
    const T nww = (S.fuw[tz][tx + 1] - S.fuw[tz][tx]) * qidx +
                  S.fvw[(j + 1) & 1][tz][tx] * hyp + S.fvw[j & 1][tz][tx] * hym +
                  (S.q3[tz + 1][tx] - S.q3[tz][tx]) * qidz;
    T rw_ = nww + cgz * (P(3, j, tz, tx) - P(3, j, tz - 1, tx));
    rw_ += cx * (P(2, j, tz, tx + 1) + P(2, j, tz, tx - 1));
    rw_ += cz * (P(2, j, tz + 1, tx) + P(2, j, tz - 1, tx));
    rw_ += cA * P(2, j - 1, tz, tx);
    rw_ += cC * P(2, j + 1, tz, tx);
    rw_ += cD * w0;
    if (use_prev) {
      if (vrow) rv_ += cp * (T)nv[cf];
      if (crow) {
        ru_ += cp * (T)nu[cc];
        rw_ += cp * (T)nw[cc];
      }
    }
    rv[cf] = vrow ? rv_ : 0;
    nv[cf] = vrow ? nvv : 0;
    if (crow) {
      const bool fixed = a.bl && i == 0;  // inflow face of u
      ru[cc] = fixed ? 0 : ru_;
      nu[cc] = fixed ? 0 : nuu;
      rw[cc] = rw_;
      nw[cc] = nww;
    }
  }

  }
};

// ---------------------------------------------------------------------------------------------
// The FP64 right-hand side in 64-bit fixed point (fx64.cuh).
//
// In FP64 arithmetic the tile was bound by the FP64 pipe: 64.8 instructions a cell of 16 cycles a
// warp, 1.547 ms on 256 x 192 x 256 cells with the pipe 88 % busy.  Here the products and the viscous
// sums run on the integer pipes; the FP64 pipe keeps 13 instructions a cell (pressure gradient, the
// stored N, closing the sum): 0.676 ms, 1257 instructions a warp of cells (with the coefficients), 2.44 a
// cycle; the ALU pipe is 62 % busy, and warps wait at the two barriers of a row, for fixed latencies and for
// the math pipes, in that order.  Tile and block from timings: 32 x 16 cells, two a thread, two blocks an SM
// 0.705; 32 x 16, one a thread (56 registers, 200 bytes spilled) 0.849; 32 x 12 0.773; this one, 27
// warps an SM, 0.677; with the viscous sum converted by the FP64 pipe (18 instructions) 0.704.  r is 3
// to 10 times nearer to the exact sums than FP64 arithmetic was (against extended precision).
//
// A block marches a 32 x 8 (x, z) column along y.  The planes of u, v, w around the row stand in
// shared memory as integers, each plane of each field scaled by its own largest magnitude in the
// tile and cut (towards zero) to 60 bits below it; p stands there in FP64.  Sums whose terms have different scales are sums of products
// with coefficients into which the scales are folded (fx_wcoef).  One warp of the nine does nothing
// else: it forms the coefficients of row j + 1, a term per lane and the scale of each sum from the
// bounds of its terms, while the others work on row j.
//
// A row next to a plane of u, v or w that holds an infinity, a NaN or values near the ends of the
// binary64 range is formed in FP64 arithmetic (rhs_cell), and so is a cell that is quiet beside a larger
// value of its tile: one that, with its neighbours in x and z, keeps fewer than 53 bits of u, v or w
// (FXR_NEAR; of the largest of the tile's three planes, whose scales the sums share).  So the values a sum
// is made of are held as FP64 holds them, against the largest near the cell, and its error is a few
// 2^-60 of the largest terms that the tile's values allow.  The five values rarely are so small together,
// and a call costs a row about 8 us: with the cell and its upper neighbours alone the benchmark's fields took
// 664 us at first, but the flat plate of 384 x 96 x 128 went from 341 to 430 in 80 steps, as values in the first
// tile fall off from the inflow; with all four neighbours 676 (677 without the test) and 338 to 373.  Every
// term of every sum held to 2^-44 of its bound took 720, to 2^-48 1250.
// ---------------------------------------------------------------------------------------------
constexpr int FXR_X = 32, FXR_Z = 8;
constexpr int FXR_PX = FXR_X + 2, FXR_PZ = FXR_Z + 2, FXR_PLANE = FXR_PX * FXR_PZ;
constexpr int FXR_WARPS = FXR_Z;  // worker warps, a z row each; one more forms coefficients
constexpr int FXR_THREADS = 32 * (FXR_WARPS + 1);
constexpr int FXR_NEAR = 20;  // 2^20 in the high word: 53 bits

struct RhsFxTile {
  // u, v, w planes (ring of 5: three in use, one being converted, one arriving as FP64), p planes
  // (ring of 3), index (kk + 1) * FXR_PX + ii + 1
  fx_t pl[3][5][FXR_PLANE];
  double pp[3][FXR_PLANE];
  fx_t fuv[2][FXR_Z][FXR_X + 1];   // the products of RhsTile that neighbours share
  fx_t fvw[2][FXR_Z + 1][FXR_X];
  fx_t fuw[FXR_Z + 1][FXR_X + 1];
  // by row parity: [3][4] terms of n (v, u, w), [3][8] terms of the viscous sums (5 used)
  FxCoef cn[2][12], cr[2][24];
  FxCoef cf[2][4];                 // face parity: weights of u_{j-1}, u_j, w_{j-1}, w_j
  fx_t cb[2];                      // body force, at the scale of u's viscous sum
  double cgy[2];                   // pressure weight of v (zero on the wall)
  int en[2][4];                    // scales of n
  int er[2][4];                    // scales of the viscous sums
  int bad[2];                      // the row takes FP64 arithmetic
  int4 least[2];                   // least high words of u, v, w near a cell (row parity)
  unsigned mag[4][4];              // largest high words of the planes (j mod 4) of u, v, w
};

// The cells of a warp in FP64 arithmetic.  Whole warps make this call, and `store` says which lanes keep the
// result: calls by some lanes of a warp beside others in the fixed-point branch are left out of the kernel.
__device__ __noinline__ void rhs_cells_fp64(const RhsArgs& a, int i, int j, int k, bool store) {
  rhs_cell<double, double>(a, min(i, a.nx - 1), j, k, a.sk->dt, store);
}

struct RhsFxK {
  struct Args {
    RhsArgs a;
    int jchunk;
  };
  static constexpr int kThreads = FXR_THREADS;
  static constexpr int kMinBlocks = 3;  // shared memory holds three; 72 registers

  // exponent of a plane (bit 62 of its integers); zero planes take the lowest
  static __device__ __forceinline__ int plane_e(unsigned m) { return (m == 0 ? 128 : (int)(m >> 20)) + 2; }
  static __device__ __forceinline__ bool plane_ok(unsigned m) { return m == 0 || fx_exponent_ok((int)(m >> 20)); }

  // ---- the coefficient warp ------------------------------------------------------------------
  // One lane's term of a sum: the coefficient mult * p[J * stride] and the scale of its values,
  // max(plane a, plane b) + max(plane c, plane d) + add, where a plane is field | (J offset + 1) << 2
  // and code 15 stands for 0.
  struct Term {
    const double* p;
    int stride;
    double mult;
    int a, b, c, d, add;
  };
  static __device__ __forceinline__ void coef_warp(const RhsArgs& a, RhsFxTile& S, int jb, int je) {
    const int lane = threadIdx.x & 31, G = a.ny + 1, ny = a.ny;
    const double* kd = a.sk->kd;
    enum { U = 0, V = 1, W = 2, LO = 0, AT = 4, UP = 8, ZERO = 15 };
    Term tn, tr;
    auto none = [&](Term& t) {
      t.p = kd;
      t.stride = 0;
      t.mult = 0.0;
      t.a = t.b = U | AT;
      t.c = t.d = ZERO;
      t.add = 0;
    };
    none(tn);
    none(tr);
    {  // n: lanes 4 g + q
      const int g = lane >> 2, q = lane & 3;
      auto flux = [&](Term& t, int f, int at) {  // flux of f v on the face `at` rows above J
        t.a = f | (at ? AT : LO);
        t.b = f | (at ? UP : AT);
        t.c = t.d = V | (at ? UP : AT);
        t.add = -1022;
      };
      auto prod = [&](Term& t, int f, int h) {  // product of plane values of f and h
        t.a = t.b = f | AT;
        t.c = t.d = h | AT;
        t.add = -1021;
      };
      if (g == 0) {
        tn.mult = 1.0;
        if (q == 0) tn.p = kd + RK_HIDX, flux(tn, U, 0);
        if (q == 3) tn.p = kd + RK_HIDZ, flux(tn, W, 0);
        if (q == 1 || q == 2) {  // squares of v at centres J and J - 1
          tn.p = a.rt + RT_QIHC * G;
          tn.stride = 1;
          tn.mult = q == 1 ? 1.0 : -1.0;
          tn.a = tn.c = V | (q == 1 ? AT : LO);
          tn.b = tn.d = V | (q == 1 ? UP : AT);
          tn.add = -1021;
        }
      } else if (g < 3) {
        const int f = g == 1 ? U : W;
        tn.mult = 1.0;
        if (q == 0) tn.p = kd + RK_QIDX, prod(tn, U, f);
        if (q == 3) tn.p = kd + RK_QIDZ, prod(tn, f, W);
        if (q == 1 || q == 2) {  // y fluxes on faces J + 1 and J
          tn.p = a.gc + GC_IDY * G;
          tn.stride = 1;
          tn.mult = (q == 1 ? 0.5 : -0.5) * kd[RK_CN];
          flux(tn, f, q == 1);
        }
      }
    }
    const int gr = lane >> 3, qr = lane & 7;
    if (gr < 3 && qr < 6) {  // viscous sums: lanes 8 g + q: x, z, centre, below, above; u: body force
      const int f = gr == 0 ? V : gr == 1 ? U : W;
      tr.a = tr.b = f | AT;
      tr.mult = 1.0;
      if (qr == 0) tr.p = kd + RK_CX;
      if (qr == 1) tr.p = kd + RK_CZ;
      if (qr >= 2 && qr < 5) {
        const int row = gr == 0 ? (qr == 2 ? RT_DF : qr == 3 ? RT_AF : RT_CF) : (qr == 2 ? RT_DC : qr == 3 ? RT_AC : RT_CC);
        tr.p = a.rt + row * G;
        tr.stride = 1;
        if (qr == 3) tr.a = tr.b = f | LO;
        if (qr == 4) tr.a = tr.b = f | UP;
      }
      if (qr == 5) {
        tr.mult = gr == 1 ? 1.0 : 0.0;
        tr.p = kd + RK_CB;
        tr.a = tr.b = ZERO;
        tr.add = 1023;
      }
    }
    // the scale of a term's values; FX_NONE where they are zero (a factor's planes are)
    auto scale = [&](const Term& t, int J) {
      auto pe = [&](int x, int y) {
        if (x == ZERO) return 0;
        const unsigned m = max(S.mag[(J - 1 + (x >> 2)) & 3][x & 3], S.mag[(J - 1 + (y >> 2)) & 3][y & 3]);
        return m == 0 ? FX_NONE : plane_e(m);
      };
      const int f = pe(t.a, t.b), h = pe(t.c, t.d);
      return f == FX_NONE || h == FX_NONE ? FX_NONE : f + h + t.add;
    };
    auto row = [&](int J) {  // planes J - 1 .. J + 1 are known
      const int par = J & 1;
      const bool wall = J == 0;  // v stays 0 there
      double cn = tn.mult * __ldg(tn.p + (long)J * tn.stride), cr = tr.mult * __ldg(tr.p + (long)J * tr.stride);
      if (wall && lane < 4) cn = 0.0;
      if (wall && gr == 0) cr = 0.0;
      const int etn = scale(tn, J), etr = scale(tr, J);
      const int een = etn == FX_NONE ? FX_NONE : fx_wexp(cn, etn), eer = etr == FX_NONE ? FX_NONE : fx_wexp(cr, etr);
      int mn = een, mr = eer;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        if (o < 4) mn = max(mn, __shfl_xor_sync(NS_FULL_MASK, mn, o));
        mr = max(mr, __shfl_xor_sync(NS_FULL_MASK, mr, o));
      }
      unsigned pn = fx_wpart(cn, een, mn), pr = fx_wpart(cr, eer, mr);
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        if (o < 4) pn += __shfl_xor_sync(NS_FULL_MASK, pn, o);
        pr += __shfl_xor_sync(NS_FULL_MASK, pr, o);
      }
      const int en = fx_wscale(mn, pn), er = fx_wscale(mr, pr);
      bool ok = en >= 128 && en <= 1920 && er >= 128 && er <= 1920;
      if (lane < 9) ok = ok && plane_ok(S.mag[(J - 1 + lane / 3) & 3][lane % 3]);
      if (lane < 12) {
        S.cn[par][lane] = een == FX_NONE ? FxCoef{0, 0} : fx_wcoef(cn, etn, en);
        if ((lane & 3) == 0) S.en[par][lane >> 2] = en;
      }
      if (gr < 3) {
        if (qr < 5) S.cr[par][lane] = eer == FX_NONE ? FxCoef{0, 0} : fx_wcoef(cr, etr, er);
        if (qr == 0) S.er[par][gr] = er;
        if (lane == 13) S.cb[par] = eer == FX_NONE ? 0 : fx_from(cr, er);
      }
      if (lane < 3) {
        const unsigned lo = S.mag[(J - 1) & 3][lane], at = S.mag[J & 3][lane], up = S.mag[(J + 1) & 3][lane];
        const unsigned m = max(at, max(lo, up));
        const int s = FXR_NEAR + plane_e(m) - plane_e(wall && lane == V ? up : at);
        (&S.least[par].x)[lane] = m == 0 ? 0 : s > 30 ? 0x7fffffff : 1 << s;
      }
      const bool good = __all_sync(NS_FULL_MASK, ok);
      if (lane == 0) {
        S.bad[par] = !good;
        S.cgy[par] = wall ? 0.0 : __ldg(a.rt + RT_CGY * G + J);
      }
    };
    auto face = [&](int jf) {  // weights of the interpolation to face jf, brought to the larger scale
      if (lane < 4) {
        const int f = lane < 2 ? U : W;
        FxCoef w{0, 0};  // no flux through the walls
        if (jf >= 1 && jf <= ny - 1) {
          const int e0 = plane_e(S.mag[(jf - 1) & 3][f]), e1 = plane_e(S.mag[jf & 3][f]);
          w = fx_limbs(fx_from(__ldg(a.gc + ((lane & 1) ? GC_WHI : GC_WLO) * G + jf), 1023 + max(e0, e1) - ((lane & 1) ? e1 : e0)));
        }
        S.cf[jf & 1][lane] = w;
      }
    };
    __syncthreads();
    for (int j = jb - 1; j <= jb + 1; ++j) __syncthreads();
    face(jb);
    face(jb + 1);
    row(jb);
    __syncthreads();
    for (int j = jb; j < je; ++j) {
      __syncthreads();
      if (lane < 4) S.mag[(j + 3) & 3][lane] = 0;  // plane j - 1 is done with
      __syncthreads();
      if (j + 1 < je) {
        face(j + 2);
        row(j + 1);
      }
    }
  }

  static __device__ __forceinline__ void run(const Args& a_, const dim3 bid_, const dim3) {
    const RhsArgs& a = a_.a;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    RhsFxTile& S = *reinterpret_cast<RhsFxTile*>(smem_raw);
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int tid = threadIdx.x, lane = tid & 31, wz = tid >> 5;
    const int i0 = bid_.x * FXR_X, k0 = bid_.y * FXR_Z;
    const int jb = bid_.z * a_.jchunk, je = min(jb + a_.jchunk, ny);
    if (wz == FXR_WARPS) {
      if (lane < 16) S.mag[lane >> 2][lane & 3] = 0;
      coef_warp(a, S, jb, je);
      return;
    }
    const int i = i0 + lane, k = k0 + wz;
    const bool active = i < nx && k < nz;  // the last tiles may reach past the grid

    // Plane positions of this thread: row wz of the 10, and a second: rows 8, 9 (warps 0, 1) or the
    // halo columns (warps 2, 3).  gi = -2: nothing there.
    int gk[2], gi[2], pos[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      int row = wz + FXR_Z * r, ii = lane;
      bool any = true;
      if (r == 1 && wz >= 2) {
        any = wz < 4 && lane < FXR_PZ;
        row = any ? lane : 0;
        ii = wz == 2 ? -1 : FXR_X;
      }
      const int kk = k0 + row - 1;
      gk[r] = kk < 0 ? kk + nz : kk >= nz ? kk - nz : kk;
      any = any && kk <= nz && i0 + ii <= nx;  // up to the wrapped neighbour
      gi[r] = any ? i0 + ii : -2;
      pos[r] = row * FXR_PX + ii + 1;
      if (!a.bl) gi[r] = gi[r] == -1 ? nx - 1 : gi[r] == nx ? 0 : gi[r];
    }
    // Plane j of p starts on its way into slot sp
    auto fetch_p = [&](int j, int sp) {
      const bool jc = j >= 0 && j < ny;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (r == 1 && gi[r] == -2) continue;
        const bool in = jc && gi[r] >= 0 && gi[r] < nx;
        cp_async8(S.pp[sp] + pos[r], a.p + (in ? (long)(gk[r] * ny + j) * nx + gi[r] : 0), in);
      }
    };
    // Plane j of u, v, w starts on its way into slot sl
    auto fetch = [&](int j, int sl) {
      const bool jc = j >= 0 && j < ny, jv = j >= 0 && j <= ny;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (r == 1 && gi[r] == -2) continue;
        double* d[3] = {(double*)S.pl[0][sl] + pos[r], (double*)S.pl[1][sl] + pos[r], (double*)S.pl[2][sl] + pos[r]};
        if (gi[r] >= 0 && gi[r] < nx) {
          const long oc = (long)(gk[r] * ny + j) * nx + gi[r];
          cp_async8(d[0], a.u + (jc ? oc : 0), jc);
          cp_async8(d[1], a.v + (jv ? oc + (long)gk[r] * nx : 0), jv);
          cp_async8(d[2], a.w + (jc ? oc : 0), jc);
        } else {
          // nothing, or an x-boundary halo: outflow plane of u, linear ghosts of v and w
          const bool out = gi[r] == nx;
          const int ib = out ? nx - 1 : 0;
          double vu = 0.0, vv = 0.0, vw = 0.0;
          if (jc && gi[r] != -2) {
            const long q = (long)gk[r] * ny + j;
            if (out) vu = __ldg(a.u_out + q);
            vw = 2.0 * __ldg((out ? a.w_out : a.w_in) + q) - __ldg(a.w + q * nx + ib);
          }
          if (jv && gi[r] != -2) {
            const long q = (long)gk[r] * (ny + 1) + j;
            vv = 2.0 * __ldg((out ? a.v_out : a.v_in) + q) - __ldg(a.v + q * nx + ib);
          }
          *d[0] = vu;
          *d[1] = vv;
          *d[2] = vw;
        }
      }
    };
    double pv[2][3];  // this thread's values of the plane that has arrived
    auto gather = [&](int j, int sl) {  // ... join the maxima of plane j
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        unsigned m = 0;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          pv[r][f] = r == 0 || gi[r] != -2 ? ((const double*)S.pl[f][sl])[pos[r]] : 0.0;
          m = max(m, fx_mag(pv[r][f]));
        }
        m = __reduce_max_sync(NS_FULL_MASK, m);
        if (lane == 0) atomicMax(&S.mag[j & 3][f], m);
      }
    };
    auto convert = [&](int j, int sl) {
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const int s = plane_e(S.mag[j & 3][f]);
#pragma unroll
        for (int r = 0; r < 2; ++r)
          if (r == 0 || gi[r] != -2) S.pl[f][sl][pos[r]] = fx_cut(pv[r][f], s);
      }
    };
    // plane element (z row kk, column ii) of this thread's warp: kk relative to its first cell
    const int e0 = (wz + 1) * FXR_PX + lane + 1;

    // y-face fluxes of face jf, its planes jf - 1 and jf in slots sa and sb
    auto face_fluxes = [&](int jf, int sa, int sb) {
      const fx_t *u0 = S.pl[0][sa], *u1 = S.pl[0][sb], *v1 = S.pl[1][sb];
      const fx_t *w0 = S.pl[2][sa], *w1 = S.pl[2][sb];
      const FxCoef cu0 = S.cf[jf & 1][0], cu1 = S.cf[jf & 1][1], cw0 = S.cf[jf & 1][2], cw1 = S.cf[jf & 1][3];
      auto uv = [&](int z, int x) {  // tile row z, column x
        const int e = (z + 1) * FXR_PX + x + 1;
        S.fuv[jf & 1][z][x] = fx_mulhi(fx_interpolate(u0[e], u1[e], cu0, cu1), v1[e - 1] + v1[e]);
      };
      auto vw = [&](int z, int x) {
        const int e = (z + 1) * FXR_PX + x + 1;
        S.fvw[jf & 1][z][x] = fx_mulhi(fx_interpolate(w0[e], w1[e], cw0, cw1), v1[e - FXR_PX] + v1[e]);
      };
      uv(wz, lane);
      vw(wz, lane);
      if (wz == FXR_WARPS - 4) vw(FXR_Z, lane);  // the extra row and column (warps 0 to 3 convert the halo)
      if (wz == FXR_WARPS - 3 && lane < FXR_Z) uv(lane, FXR_X);
    };
    // Fuw of the plane in slot sl
    auto centre_products = [&](int sl) {
      const fx_t *u = S.pl[0][sl], *w = S.pl[2][sl];
      auto uw = [&](int z, int x) {
        const int e = (z + 1) * FXR_PX + x + 1;
        S.fuw[z][x] = fx_mulhi(u[e - FXR_PX] + u[e], w[e - 1] + w[e]);
      };
      uw(wz, lane);
      if (wz == FXR_WARPS - 2) uw(FXR_Z, lane);
      if (wz == FXR_WARPS - 1 && lane <= FXR_Z) uw(lane, FXR_X);
    };
    // (v_j + v_{j+1})^2 of the centre j, at the larger of the planes' scales
    auto square_v = [&](int j, int sa, int sb) {
      const int ea = plane_e(S.mag[j & 3][1]), eb = plane_e(S.mag[(j + 1) & 3][1]), em = max(ea, eb);
      const int da = min(em - ea, 63), db = min(em - eb, 63);
      return fx_sqrhi((S.pl[1][sa][e0] >> da) + (S.pl[1][sb][e0] >> db));
    };

    // ---- prologue: planes jb - 1 .. jb + 1, then (coefficients) the fluxes of face jb.  Slots of planes
    // j - 1, j, j + 1, j + 2, j + 3 and of p's planes j - 1, j:
    int sm = 0, s0 = 1, s1 = 2, s2 = 3, s3 = 4, pm = 0, pc = 1, pn = 2;
    __syncthreads();
    for (int j = jb - 1; j <= jb + 1; ++j) {
      const int q = j - jb + 1;
      fetch(j, q);
      if (q < 2) fetch_p(j, q);
      cp_async_wait_all8();
      gather(j, q);
      __syncthreads();
      convert(j, q);
    }
    if (jb + 1 < je) fetch(jb + 2, s2);
    __syncthreads();
    face_fluxes(jb, sm, s0);
    fx_t q2prev = jb >= 1 ? square_v(jb - 1, sm, s0) : 0;

    const bool use_prev = a.zet != 0.0;
    const double* kd = a.sk->kd;
    const double cp = kd[RK_CP], cgx = kd[RK_CGX], cgz = kd[RK_CGZ];
    double* __restrict__ ru = (double*)a.ru;
    double* __restrict__ rv = (double*)a.rv;
    double* __restrict__ rw = (double*)a.rw;
    double* nu = (double*)a.nu;
    double* nv = (double*)a.nv;
    double* nw = (double*)a.nw;
    for (int j = jb; j < je; ++j) {
      const bool next = j + 1 < je;  // another row follows
      cp_async_wait_all8();
      if (next) gather(j + 2, s2);
      __syncthreads();
      const long cc = ((long)k * ny + j) * nx + i, cf = cc + (long)k * nx;
      if (next) {
        convert(j + 2, s2);
        if (j + 2 < je) fetch(j + 3, s3);
        fetch_p(j + 1, pn);
      }
      double prev[3] = {};  // the stored N of the last sub-step (v, u, w)
      if (use_prev && active) {
        prev[0] = nv[cf];
        prev[1] = nu[cc];
        prev[2] = nw[cc];
      }
      face_fluxes(j + 1, s0, s1);
      centre_products(s0);
      const fx_t q2 = square_v(j, s0, s1);
      __syncthreads();
      const int par = j & 1, f0 = j & 1, f1 = f0 ^ 1;
      bool fp64 = S.bad[par] != 0;  // this cell takes FP64 arithmetic
      if (!fp64) {
        const FxCoef* cn = S.cn[par];
        const FxCoef* cr = S.cr[par];
        // The viscous sum of field f; o: the plane's values at the cell, the z neighbours below and
        // above, the x neighbours before and after
        auto viscous = [&](FxAcc& s, int f, const FxCoef* c, fx_t* o) {
          const fx_t* p = S.pl[f][s0] + e0;
          o[0] = p[0];
          o[1] = p[-FXR_PX];
          o[2] = p[FXR_PX];
          o[3] = p[-1];
          o[4] = p[1];
          fx_wmac(s, o[3] + o[4], c[0]);
          fx_wmac(s, o[1] + o[2], c[1]);
          fx_wmac(s, o[0], c[2]);
          fx_wfold(s);
          fx_wmac(s, S.pl[f][sm][e0], c[3]);
          fx_wmac(s, S.pl[f][s1][e0], c[4]);
        };
        const double* pj = S.pp[pc] + e0;
        const double p0 = pj[0];
        fx_t o[5];
        // the bits of the cell and its neighbours in x and z (as in `viscous`)
        auto bits = [](const fx_t* o) {
          int b = 0;
#pragma unroll
          for (int q = 0; q < 5; ++q) b |= fx_hi(o[q]) ^ (fx_hi(o[q]) >> 31);
          return b;
        };
        int3 size;
        double nd[3], rd[3];  // stored together at the end: the FP64 sums finish meanwhile
        // ---------------- v at face j
        {
          FxAcc n = fx_wacc(0), s = fx_wacc(0);
          fx_wmac(n, S.fuv[f0][wz][lane + 1] - S.fuv[f0][wz][lane], cn[0]);
          fx_wmac(n, S.fvw[f0][wz + 1][lane] - S.fvw[f0][wz][lane], cn[3]);
          fx_wmac(n, q2, cn[1]);
          fx_wmac(n, q2prev, cn[2]);
          viscous(s, 1, cr, o);
          size.y = bits(o);
          if (j == 0) {  // v is zero on the wall: the plane above decides
            const fx_t* p = S.pl[1][s1] + e0;
            const fx_t up[5] = {p[0], p[-FXR_PX], p[FXR_PX], p[-1], p[1]};
            size.y = bits(up);
          }
          nd[0] = fx_to(fx_wsum(n), S.en[par][0]);
          const double dp = p0 - S.pp[pm][e0];
          rd[0] = (fx_to(fx_wsum(s), S.er[par][0]) + fma(S.cgy[par], dp, fma(cp, prev[0], nd[0])));
        }
        // ---------------- u at (xf_i, yc_j, zc_k)
        {
          FxAcc n = fx_wacc(0), s = fx_wacc(S.cb[par]);
          fx_wmac(n, S.fuw[wz + 1][lane] - S.fuw[wz][lane], cn[7]);
          fx_wmac(n, S.fuv[f1][wz][lane], cn[5]);
          fx_wmac(n, S.fuv[f0][wz][lane], cn[6]);
          viscous(s, 0, cr + 8, o);
          size.x = bits(o);
          fx_wmac(n, fx_sqrhi(o[0] + o[4]) - fx_sqrhi(o[3] + o[0]), cn[4]);
          nd[1] = fx_to(fx_wsum(n), S.en[par][1]);
          rd[1] = (fx_to(fx_wsum(s), S.er[par][1]) + fma(cgx, p0 - pj[-1], fma(cp, prev[1], nd[1])));
        }
        // ---------------- w at (xc_i, yc_j, zf_k)
        {
          FxAcc n = fx_wacc(0), s = fx_wacc(0);
          fx_wmac(n, S.fuw[wz][lane + 1] - S.fuw[wz][lane], cn[8]);
          fx_wmac(n, S.fvw[f1][wz][lane], cn[9]);
          fx_wmac(n, S.fvw[f0][wz][lane], cn[10]);
          viscous(s, 2, cr + 16, o);
          size.z = bits(o);
          fx_wmac(n, fx_sqrhi(o[0] + o[2]) - fx_sqrhi(o[1] + o[0]), cn[11]);
          nd[2] = fx_to(fx_wsum(n), S.en[par][2]);
          rd[2] = (fx_to(fx_wsum(s), S.er[par][2]) + fma(cgz, p0 - pj[-FXR_PX], fma(cp, prev[2], nd[2])));
        }
        const int4 least = S.least[par];
        fp64 = size.x < least.x || size.y < least.y || size.z < least.z;
        if (active && !fp64) {
          const bool wall = j == 0, fixed = a.bl && i == 0;  // the wall row of v, the inflow face of u
          nv[cf] = nd[0];
          rv[cf] = wall ? 0.0 : rd[0];
          nu[cc] = fixed ? 0.0 : nd[1];
          ru[cc] = fixed ? 0.0 : rd[1];
          nw[cc] = nd[2];
          rw[cc] = rd[2];
        }
      }
      const bool store64 = active && fp64;
      if (__any_sync(NS_FULL_MASK, store64)) rhs_cells_fp64(a, i, j, k, store64);
      q2prev = q2;
      {  // the rings move on by one plane
        const int t = sm;
        sm = s0;
        s0 = s1;
        s1 = s2;
        s2 = s3;
        s3 = t;
        pm = pc;
        pc = pn;
        pn = 3 - pm - pc;
      }
    }
    if (je == ny) {  // the top wall row of v
      const long cf = ((long)k * (ny + 1) + ny) * nx + i;
      if (active) nv[cf] = rv[cf] = 0.0;
    }
  }
};

}  // namespace

template <typename K>
cudaError_t rhs_attributes(int* bps, size_t smem) {
  const cudaError_t e = set_smem_limit<K>((int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, single_kernel<K>, K::kThreads, smem);
}

cudaError_t rhs_set_attributes(int* bps) {
  cudaError_t e;
  if ((e = rhs_attributes<RhsFxK>(bps + 0, sizeof(RhsFxTile))) != cudaSuccess ||
      (e = rhs_attributes<RhsTiledK<false>>(bps + 1, sizeof(RhsTile))) != cudaSuccess)
    return e;
  return rhs_attributes<RhsTiledK<true>>(bps + 2, sizeof(RhsTile));
}

cudaError_t launch_rhs(ns_ctx* c, int k) {
  LaunchSink s{c, nullptr};
  return stage_rhs(s, k);
}

// Rows of y a block marches: chunks (each re-derives one face and two or three planes) so that the
// blocks fill whole waves of the resident capacity, minimising waves * (rows per chunk + prologue).
// Small grids come down to a row or two a block: the march is one serial chain, and 64 x 64 x 32 cells
// in chunks of six rows filled 44 of 152 SMs.  least: the fewest rows of a chunk (batched instances fill
// the GPU together and keep longer ones).  (Chunks of equal rows in one single wave, some spanning
// two tiles, were slower: neighbouring tiles then march at different y.)
int rhs_chunk(const ns_ctx* c, int tiles, int bps, double prologue, int least) {
  const int ny = c->cfg.ny, resident = c->num_sms * std::max(bps, 1);
  int best_nch = 1;
  double best = 1e300;
  for (int nch = 1; nch <= ny && (nch == 1 || (ny + nch - 1) / nch >= least); ++nch) {
    const int jc = (ny + nch - 1) / nch;
    const long nb = (long)tiles * ((ny + jc - 1) / jc);
    const long waves = (nb + resident - 1) / resident;
    const double cost = (double)waves * (jc + prologue);
    if (cost < best - 1e-9) {
      best = cost;
      best_nch = nch;
    }
  }
  return (ny + best_nch - 1) / best_nch;
}

template <bool Dyn>
cudaError_t emit_tiled(LaunchSink& s, const RhsArgs& a) {
  using K = RhsTiledK<Dyn>;
  const int jchunk = rhs_chunk(s.c, (a.nx / RT_X) * (a.nz / RT_Z), s.c->rhs_bps[Dyn ? 2 : 1], 2.0, s.plan ? 6 : 1);
  return emit<K>(s, K::make(a, jchunk), dim3(a.nx / RT_X, a.nz / RT_Z, (a.ny + jchunk - 1) / jchunk), dim3(RT_X, RT_Z),
                 sizeof(RhsTile));
}

cudaError_t stage_rhs(LaunchSink& s, int k) {
  ns_ctx* c = s.c;
  RhsArgs a;
  a.u = c->f.u;
  a.v = c->f.v;
  a.w = c->f.w;
  a.p = c->f.p;
  a.ru = c->ru;
  a.rv = c->rv;
  a.rw = c->rw;
  a.nu = c->nu;
  a.nv = c->nv;
  a.nw = c->nw;
  a.gc = c->gc;
  a.nx = c->cfg.nx;
  a.ny = c->cfg.ny;
  a.nz = c->cfg.nz;
  a.idx = 1.0 / c->dx;
  a.idz = 1.0 / c->dz;
  a.idx2 = a.idx * a.idx;
  a.idz2 = a.idz * a.idz;
  a.dt = c->cfg.dt;
  a.gam = NS_GAMMA[k];
  a.zet = NS_ZETA[k];
  a.cprev = k > 0 ? NS_ZETA[k] / NS_GAMMA[k - 1] : 0.0;
  a.alp = NS_ALPHA[k];
  a.inv_re = c->cfg.re > 0 ? 1.0 / c->cfg.re : 0.0;
  a.fx = c->cfg.fx;
  a.rt = c->rtab[k];
  a.rtf = c->rtabf[k];
  a.bl = c->bl;
  a.u_out = c->f.u_out;
  a.v_in = c->f.v_in;
  a.v_out = c->f.v_out;
  a.w_in = c->f.w_in;
  a.w_out = c->f.w_out;
  a.sk = c->stepk + k;
  a.kc = c->stepk_h[k];
  if (c->cfg.precision != NS_MIXED) {
    const int tx = (a.nx + FXR_X - 1) / FXR_X, tz = (a.nz + FXR_Z - 1) / FXR_Z;
    const int jchunk = rhs_chunk(c, tx * tz, c->rhs_bps[0], 4.0, s.plan ? 6 : 1);
    return emit<RhsFxK>(s, RhsFxK::Args{a, jchunk}, dim3(tx, tz, (a.ny + jchunk - 1) / jchunk), dim3(FXR_THREADS),
                        sizeof(RhsFxTile));
  }
  if (a.nx % RT_X == 0) return c->dyn_consts ? emit_tiled<true>(s, a) : emit_tiled<false>(s, a);
  const long plane = (long)a.nx * (a.ny + 1);
  dim3 grid((unsigned)((plane + 127) / 128), (unsigned)a.nz);
  return c->dyn_consts ? emit<RhsK<float, float, true>>(s, RhsK<float, float, true>::make(a), grid, 128, 0)
                       : emit<RhsK<float, float, false>>(s, RhsK<float, float, false>::make(a), grid, 128, 0);
}
