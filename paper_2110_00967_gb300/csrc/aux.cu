// aux.cu -- mask rasterisation (Eq. fcar), interface flags, initial state and
// the conversions between the stored offsets and FP64 fields.
#include <cmath>

#include "vplbm_internal.cuh"

namespace vplbm {

namespace {

constexpr int kAuxThreads = 256;

inline int blocks_for(int64_t n) { return (int)((n + kAuxThreads - 1) / kAuxThreads); }

// chi on the box [i0, i1] x [j0, j1] (Eq. fcar: 1 inside or on the body)
__global__ void raster_kernel(Lattice L, const BodyState *body, uint8_t *chi, int i0, int j0,
                              int w, int h) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= w * h) return;
  const int i = i0 + k % w, j = j0 + k / w;
  const BodyState b = *body;
  chi[(int64_t)j * L.pitch + i] = body_contains(b, i, j) ? kSolid : 0;
}

// interface bit: some lattice neighbour (inside the lattice) has the other phase
__global__ void interface_kernel(Lattice L, uint8_t *chi, int i0, int j0, int w, int h) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= w * h) return;
  const int i = i0 + k % w, j = j0 + k / w;
  const uint8_t self = chi[(int64_t)j * L.pitch + i] & kSolid;
  bool iface = false;
#pragma unroll
  for (int a = 1; a < 9; ++a) {
    int ni, nj;
    if (neighbour(L, a, i, j, ni, nj) && ((chi[(int64_t)nj * L.pitch + ni] & kSolid) != self))
      iface = true;
  }
  chi[(int64_t)j * L.pitch + i] = (uint8_t)(self | (iface ? kInterface : 0));
}

// f = feq(1, u0) with u0 = u_in on fluid nodes and the rigid velocity on
// solid nodes; stored as offsets f - E
template <typename S>
__global__ void init_kernel(Lattice L, const BodyState *body, const uint8_t *chi, S *buf,
                            double u0x, double u0y) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= (int64_t)L.nx * L.ny) return;
  const int i = (int)(k % L.nx), j = (int)(k / L.nx);
  const int64_t node = (int64_t)j * L.pitch + i;
  double ux = u0x, uy = u0y;
  if (chi[node] & kSolid) {
    const BodyState b = *body;
    ux = b.ux - b.omega * ((double)j - b.yg);
    uy = b.uy + b.omega * ((double)i - b.xg);
  }
  // feq(1, u0) - E = w (Q(u0) - Q(u_ref)) with Q(u) = 3 c.u + 4.5 (c.u)^2 - 1.5 |u|^2,
  // written with du = u0 - u_ref
  const double dux = ux - L.ur[0], duy = uy - L.ur[1];
  const double dsu = dux * (ux + L.ur[0]) + duy * (uy + L.ur[1]);
#pragma unroll
  for (int a = 0; a < 9; ++a) {
    const double cdu = cx_of(a) * dux + cy_of(a) * duy;
    const double csu = cx_of(a) * (ux + L.ur[0]) + cy_of(a) * (uy + L.ur[1]);
    const double h = w_of(a) * (3.0 * cdu + 4.5 * cdu * csu - 1.5 * dsu);
    buf[(int64_t)a * L.plane + node] = Store<S>::from_double(h);
  }
}

// Read-back kernels cover the rows j0 .. j0 + rows - 1 and write them
// compactly, [rows][nx] per output plane, so that the host read-backs can
// stage a few rows at a time.

// planes a0 .. a0 + na - 1 of the pre-collision populations f = h + E
template <typename S, bool kGather>
__global__ void get_f_kernel(Lattice L, const S *buf, const typename Store<S>::T *prev,
                             double *out, int a0, int na, int j0, int rows) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = (int64_t)L.nx * rows;
  if (k >= n) return;
  const int i = (int)(k % L.nx), j = j0 + (int)(k / L.nx);
#pragma unroll
  for (int a = 0; a < 9; ++a)
    if (a >= a0 && a < a0 + na)
      out[(a - a0) * n + k] = (double)pre_pop<S, kGather>(buf, prev, L, a, i, j) + L.E[a];
}

// Moments of FP32 offsets, exactly: each offset as a 64-bit integer multiple of
// 2^-60 (FP32 values above 2^-37 in magnitude exactly, smaller ones cut off
// below 1e-18), summed as integers with the reference state's part.  rho and j
// are scaled by 2^60, which their quotient does not see.
constexpr int kFixBits = 60;
__device__ __forceinline__ long long fixed60(float h) {
  const uint32_t bits = __float_as_uint(h);
  const int e = (int)(bits >> 23 & 0xffu);
  const unsigned long long m = (unsigned long long)((bits & 0x7fffffu) | 0x800000u) << 35;
  const long long v = (long long)(m >> min(max(125 - e, 0), 63));  // |h| < 1/2: e <= 125
  return (int)bits < 0 ? -v : v;
}

// The double nearest v (a tie away from zero), by integer operations: the
// conversion instruction shares the FP64 lanes.
__device__ __forceinline__ double to_double(long long v) {
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  if (u == 0) return 0.0;
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << lz;                          // leading bit 63
  const unsigned long long r = (m >> 11) + (m >> 10 & 1ull);     // 53 bits, rounded
  // the leading bit of r adds one to the exponent
  return __longlong_as_double((long long)((((unsigned long long)(1085 - lz) << 52) + r) |
                                          ((unsigned long long)v & 0x8000000000000000ull)));
}

// Macroscopic fields of Eqs. updatestep and updatestepm, FP64.  (ox, oy): the
// part of j that the offsets leave out, u_ref plus half the body force, for FP32
// offsets in units of 2^-60.  GB300's two FP64 lanes per SM bound this kernel
// (about 140 FP64 operations per node for nine conversions, the moments and two
// divisions: 246 us for 2048 x 1024, where its traffic takes 19 us); FP32 offsets
// are therefore summed as integers, which rounds less, and a node is left with
// five FP64 operations.  fixed: (ox, oy) fit beside the offsets' sums (six of
// them, below 2.4 in magnitude, in 64 bits of unit 2^-60).
template <typename S, bool kGather>
__global__ void __launch_bounds__(kAuxThreads)
    get_fields_kernel(Lattice L, const S *buf, const typename Store<S>::T *prev,
                      const uint8_t *chi, const BodyState *body, double half_pen, double *rho_o,
                      double *ux_o, double *uy_o, int j0, int rows, long long ox, long long oy,
                      bool fixed) {
  using T = typename Store<S>::T;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= L.nx) return;
  for (int r = blockIdx.y * blockDim.y + threadIdx.y; r < rows; r += gridDim.y * blockDim.y) {
    const int j = j0 + r;
    const int64_t node = (int64_t)j * L.pitch + i, k = (int64_t)r * L.nx + i;
    T h[9];
    if (kGather && i > 0 && i < L.nx - 1 && j > 0 && j < L.ny - 1) {
#pragma unroll
      for (int a = 0; a < 9; ++a)
        h[a] = pop_at(buf, L, a, i - cx_of(a), j - cy_of(a));
    } else {
#pragma unroll
      for (int a = 0; a < 9; ++a) h[a] = pre_pop<S, kGather>(buf, prev, L, a, i, j);
    }
    const uint8_t m = chi[node];
    double rho, jx, jy;  // FP32 offsets: scaled by 2^60
    bool exact = false, near_one;  // near_one: rho between 2^-10 and 2^10
    if constexpr (sizeof(T) == 4) {
      float big = 0.f;
#pragma unroll
      for (int a = 0; a < 9; ++a) big = fmaxf(big, fabsf(h[a]));
      long long v[9];
#pragma unroll
      for (int a = 0; a < 9; ++a) v[a] = fixed60(h[a]);
      const long long s = v[0] + v[1] + v[2] + v[3] + v[4] + v[5] + v[6] + v[7] + v[8] + (1ll << kFixBits);
      // (NaN offsets fail the sum's comparison: fmaxf drops them)
      exact = fixed && big < 0.4f && s > (1ll << (kFixBits - 10)) && h[0] + h[1] + h[2] + h[3] + h[4] + h[5] + h[6] + h[7] + h[8] < 4.f;
      if (exact) {
        rho = to_double(s);
        jx = to_double(v[1] - v[3] + v[5] - v[6] + v[8] - v[7] + ox);
        jy = to_double(v[2] - v[4] + v[5] - v[7] + v[6] - v[8] + oy);
      }
    }
    if (!exact) {
      rho = 1.0 + ((((double)h[0] + (double)h[1]) + ((double)h[2] + (double)h[3])) +
                   (((double)h[4] + (double)h[5]) + ((double)h[6] + (double)h[7])) + (double)h[8]);
      jx = ((double)h[1] - (double)h[3]) + ((double)h[5] - (double)h[6]) + ((double)h[8] - (double)h[7]);
      jy = ((double)h[2] - (double)h[4]) + ((double)h[5] - (double)h[7]) + ((double)h[6] - (double)h[8]);
      jx += L.ur[0] + 0.5 * L.bf[0];
      jy += L.ur[1] + 0.5 * L.bf[1];
    }
    near_one = exact || (uint32_t)(__double2hiint(rho) - (1013 << 20)) < (uint32_t)(20 << 20);
    if (m & kSolid) {
      const BodyState b = *body;
      const double usx = b.ux - b.omega * ((double)j - b.yg);
      const double usy = b.uy + b.omega * ((double)i - b.xg);
      ux_o[k] = (jx + half_pen * rho * usx) / (rho + half_pen * rho);
      uy_o[k] = (jy + half_pen * rho * usy) / (rho + half_pen * rho);
    } else if (near_one) {
      const double inv = near_rcp(rho);
      ux_o[k] = jx * inv;
      uy_o[k] = jy * inv;
    } else {
      ux_o[k] = jx / rho;
      uy_o[k] = jy / rho;
    }
    // 2^-60 rho: the exponent alone (rho is normal)
    rho_o[k] = exact ? __hiloint2double(__double2hiint(rho) - (kFixBits << 20), __double2loint(rho))
                     : rho;
  }
}

template <typename S>
__global__ void set_state_kernel(Lattice L, const double *f, S *buf) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = (int64_t)L.nx * L.ny;
  if (k >= n) return;
  const int i = (int)(k % L.nx), j = (int)(k / L.nx);
  const int64_t node = (int64_t)j * L.pitch + i;
#pragma unroll
  for (int a = 0; a < 9; ++a)
    buf[(int64_t)a * L.plane + node] = Store<S>::from_double(f[a * n + k] - L.E[a]);
}

// outlet column (a = 3, 6, 7 at i = nx - 1) of a pre-collision FP64 field,
// kept as offsets in the compute type
template <typename T>
__global__ void set_prev_kernel(Lattice L, const double *f, T *prev) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= L.ny) return;
  const int64_t n = (int64_t)L.nx * L.ny;
  const int64_t k = (int64_t)j * L.nx + (L.nx - 1);
  prev[0 * L.ny + j] = (T)(f[3 * n + k] - L.E[3]);
  prev[1 * L.ny + j] = (T)(f[6 * n + k] - L.E[6]);
  prev[2 * L.ny + j] = (T)(f[7 * n + k] - L.E[7]);
}

__global__ void get_mask_kernel(Lattice L, const uint8_t *chi, uint8_t *out, int j0, int rows) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= (int64_t)L.nx * rows) return;
  const int i = (int)(k % L.nx), j = j0 + (int)(k / L.nx);
  out[k] = chi[(int64_t)j * L.pitch + i] & kSolid;
}

template <typename S>
cudaError_t get_f_t(bool gather, const Lattice &L, const void *buf, const void *prev_v,
                    double *out, int a0, int na, int j0, int rows, cudaStream_t s) {
  using T = typename Store<S>::T;
  const T *prev = static_cast<const T *>(prev_v);
  const int g = blocks_for((int64_t)L.nx * rows);
  if (gather)
    get_f_kernel<S, true><<<g, kAuxThreads, 0, s>>>(L, (const S *)buf, prev, out, a0, na, j0, rows);
  else
    get_f_kernel<S, false><<<g, kAuxThreads, 0, s>>>(L, (const S *)buf, prev, out, a0, na, j0, rows);
  return cudaGetLastError();
}

template <typename S>
cudaError_t get_fields_t(bool gather, const Lattice &L, const void *buf, const void *prev_v,
                         const uint8_t *chi, const BodyState *body, double half_pen, double *rho,
                         double *ux, double *uy, int j0, int rows, cudaStream_t s) {
  using T = typename Store<S>::T;
  const T *prev = static_cast<const T *>(prev_v);
  // 256 nodes of a row per block, or as many whole rows of a narrow lattice (one
  // row each left most threads idle: 3 x 100000 in FP64 296 us, 17 x 40000 in FP32 134)
  const int w = L.nx < kAuxThreads ? L.nx : kAuxThreads;
  const dim3 b(w, kAuxThreads / w);
  const int high = (rows + (int)b.y - 1) / (int)b.y;
  const dim3 g((L.nx + w - 1) / w, high < 65535 ? high : 65535);
  const double unit = (double)(1ll << kFixBits);
  const double mx = L.ur[0] + 0.5 * L.bf[0], my = L.ur[1] + 0.5 * L.bf[1];
  const bool fixed = fabs(mx) < 4.0 && fabs(my) < 4.0;  // a body force may be larger
  const long long ox = fixed ? llrint(mx * unit) : 0, oy = fixed ? llrint(my * unit) : 0;
  if (gather)
    get_fields_kernel<S, true><<<g, b, 0, s>>>(L, (const S *)buf, prev, chi, body,
                                                         half_pen, rho, ux, uy, j0, rows, ox, oy, fixed);
  else
    get_fields_kernel<S, false><<<g, b, 0, s>>>(L, (const S *)buf, prev, chi, body,
                                                          half_pen, rho, ux, uy, j0, rows, ox, oy, fixed);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_raster(const Lattice &L, const BodyState *body, uint8_t *chi, int i0, int j0,
                          int i1, int j1, cudaStream_t s) {
  const int w = i1 - i0 + 1, h = j1 - j0 + 1;
  if (w <= 0 || h <= 0) return cudaSuccess;
  raster_kernel<<<blocks_for((int64_t)w * h), kAuxThreads, 0, s>>>(L, body, chi, i0, j0, w, h);
  return cudaGetLastError();
}

cudaError_t launch_interface(const Lattice &L, uint8_t *chi, int i0, int j0, int i1, int j1,
                             cudaStream_t s) {
  const int w = i1 - i0 + 1, h = j1 - j0 + 1;
  if (w <= 0 || h <= 0) return cudaSuccess;
  interface_kernel<<<blocks_for((int64_t)w * h), kAuxThreads, 0, s>>>(L, chi, i0, j0, w, h);
  return cudaGetLastError();
}

cudaError_t launch_init(int dtype, const Lattice &L, const BodyState *body, const uint8_t *chi,
                        void *buf, double u0x, double u0y, cudaStream_t s) {
  const int g = blocks_for((int64_t)L.nx * L.ny);
  switch (dtype) {
    case VPLBM_F64: init_kernel<double><<<g, kAuxThreads, 0, s>>>(L, body, chi, (double *)buf, u0x, u0y); break;
    case VPLBM_F32: init_kernel<float><<<g, kAuxThreads, 0, s>>>(L, body, chi, (float *)buf, u0x, u0y); break;
    case VPLBM_F16_OFS: init_kernel<__half><<<g, kAuxThreads, 0, s>>>(L, body, chi, (__half *)buf, u0x, u0y); break;
    case VPLBM_BF16_OFS:
      init_kernel<__nv_bfloat16><<<g, kAuxThreads, 0, s>>>(L, body, chi, (__nv_bfloat16 *)buf, u0x, u0y);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_get_f(int dtype, bool gather, const Lattice &L, const void *buf,
                         const void *prev, double *out, int a0, int na, int j0, int rows,
                         cudaStream_t s) {
  if (rows <= 0 || na <= 0) return cudaSuccess;
  switch (dtype) {
    case VPLBM_F64: return get_f_t<double>(gather, L, buf, prev, out, a0, na, j0, rows, s);
    case VPLBM_F32: return get_f_t<float>(gather, L, buf, prev, out, a0, na, j0, rows, s);
    case VPLBM_F16_OFS: return get_f_t<__half>(gather, L, buf, prev, out, a0, na, j0, rows, s);
    case VPLBM_BF16_OFS: return get_f_t<__nv_bfloat16>(gather, L, buf, prev, out, a0, na, j0, rows, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_get_fields(int dtype, bool gather, const Lattice &L, const void *buf,
                              const void *prev, const uint8_t *chi, const BodyState *body,
                              double half_pen, double *rho, double *ux, double *uy, int j0,
                              int rows, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  switch (dtype) {
    case VPLBM_F64:
      return get_fields_t<double>(gather, L, buf, prev, chi, body, half_pen, rho, ux, uy, j0, rows, s);
    case VPLBM_F32:
      return get_fields_t<float>(gather, L, buf, prev, chi, body, half_pen, rho, ux, uy, j0, rows, s);
    case VPLBM_F16_OFS:
      return get_fields_t<__half>(gather, L, buf, prev, chi, body, half_pen, rho, ux, uy, j0, rows, s);
    case VPLBM_BF16_OFS:
      return get_fields_t<__nv_bfloat16>(gather, L, buf, prev, chi, body, half_pen, rho, ux, uy, j0,
                                         rows, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_set_state(int dtype, const Lattice &L, const double *f, void *buf,
                             cudaStream_t s) {
  const int g = blocks_for((int64_t)L.nx * L.ny);
  switch (dtype) {
    case VPLBM_F64: set_state_kernel<double><<<g, kAuxThreads, 0, s>>>(L, f, (double *)buf); break;
    case VPLBM_F32: set_state_kernel<float><<<g, kAuxThreads, 0, s>>>(L, f, (float *)buf); break;
    case VPLBM_F16_OFS: set_state_kernel<__half><<<g, kAuxThreads, 0, s>>>(L, f, (__half *)buf); break;
    case VPLBM_BF16_OFS:
      set_state_kernel<__nv_bfloat16><<<g, kAuxThreads, 0, s>>>(L, f, (__nv_bfloat16 *)buf);
      break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_set_prev(int dtype, const Lattice &L, const double *f, void *prev,
                            cudaStream_t s) {
  if (dtype == VPLBM_F64)
    set_prev_kernel<double><<<blocks_for(L.ny), kAuxThreads, 0, s>>>(L, f, (double *)prev);
  else
    set_prev_kernel<float><<<blocks_for(L.ny), kAuxThreads, 0, s>>>(L, f, (float *)prev);
  return cudaGetLastError();
}

cudaError_t launch_get_mask(const Lattice &L, const uint8_t *chi, uint8_t *out, int j0, int rows,
                            cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  get_mask_kernel<<<blocks_for((int64_t)L.nx * rows), kAuxThreads, 0, s>>>(L, chi, out, j0, rows);
  return cudaGetLastError();
}

}  // namespace vplbm
