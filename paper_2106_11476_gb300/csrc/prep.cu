// One-time coefficient preparation on the device (Sec. 3.2, 3.3): FP64 for
// everything but the relaxation pair a, b, which is float (relax_ab32).
//
// From the raw per-cell medium (c, rho, beta) and relaxation parameters
// (kappa1, kappa2, d^nu, alpha^nu for nabla_1 and nabla_2) it writes the maps
// the step kernels stream:
//   K = rho c^2, rho, chi (nonlinear factor of Eq. general6),
//   1/kappa1, 1/kappa2,
//   interior a, b (Eqs. relaxation_a, relaxation_b) of every cell, and
//   per-axis a, b inside the boundary strips, where d and alpha follow the
//   two-stage C-PML ramps of Table 1:  X = (X_target - X_0) g + X_0 with
//   g = (x/L)^npow (nu = 1, d), x/L (nu = 1, alpha) and
//   (1 - cos(pi x / L_T)) / 2 over the transition layer (nu >= 2).  In
//   reading C alpha^{nu=1} is blended by that cosine into the C-PML profile
//   d_target (1 - x/L).
// The profile of a face is evaluated at its exact staggered coordinate; the
// relaxation parameters of a face are those of its lower-index cell.
#include "fw2_prep.cuh"
#include <algorithm>
#include <type_traits>

#include "maps.cuh"

namespace fw2 {

namespace {

// tissue index of input cell t (index form)
__device__ __forceinline__ int tissue_at(const PrepParams &Q, long long t) {
  return Q.tissue_wide ? (int)static_cast<const unsigned short *>(Q.tissue_in)[t]
                       : (int)static_cast<const unsigned char *>(Q.tissue_in)[t];
}
// raw parameter of cell t (dense inputs) or of its tissue (index form)
__device__ __forceinline__ long long src_of(const PrepParams &Q, long long t) {
  return Q.tissue_in ? (long long)tissue_at(Q, t) : t;
}
__device__ __forceinline__ long long n_src(const PrepParams &Q) {
  return Q.tissue_in ? (long long)Q.n_tissue : (long long)Q.nx * Q.ny * Q.nz;
}

__device__ __forceinline__ void store(float *p, long long i, double v) { p[i] = (float)v; }
__device__ __forceinline__ void store(__nv_bfloat16 *p, long long i, double v) {
  p[i] = __float2bfloat16_rn((float)v);
}
// FP16 maps: the value times the map's inverse scale (a power of two, exact),
// rounded to float then to half
__device__ __forceinline__ void store(__half *p, long long i, double v, double inv) {
  p[i] = __float2half_rn((float)(v * inv));
}
__device__ __forceinline__ void store(float *p, long long i, double v, double) { store(p, i, v); }
__device__ __forceinline__ void store(__nv_bfloat16 *p, long long i, double v, double) { store(p, i, v); }

// Where the map kernels put a value: stored (scaled for FP16), or, in the
// scan pass of the FP16 maps, folded into this thread's largest magnitude of
// the map; flush() combines the threads' maxima (warp reduction, one atomic
// per warp and map).
template <typename MT, bool SCAN>
struct MapSink {
  const PrepParams &Q;
  float mx[SCAN ? kMapScales : 1];
  __device__ __forceinline__ explicit MapSink(const PrepParams &q) : Q(q) {
    if (SCAN)
      for (int m = 0; m < kMapScales; ++m) mx[m] = 0.f;
  }
  __device__ __forceinline__ void put(int id, void *p, long long i, double v) {
    if constexpr (SCAN) mx[id] = fmaxf(mx[id], (float)fabs(v));
    else store(static_cast<MT *>(p), i, v, Q.inv_scale[id]);
  }
  // decay factor b with 1 - b given: float maps keep b, bf16 and FP16 maps
  // 1 - b (FP16 times the map's inverse scale)
  __device__ __forceinline__ void put_b2(int id, void *p, long long i, float b, float omb) {
    if constexpr (SCAN) {
      mx[id] = fmaxf(mx[id], fabsf(omb));
    } else if constexpr (std::is_same<MT, float>::value) {
      static_cast<float *>(p)[i] = b;
    } else if constexpr (std::is_same<MT, __nv_bfloat16>::value) {
      static_cast<__nv_bfloat16 *>(p)[i] = __float2bfloat16_rn(omb);
    } else {
      static_cast<__half *>(p)[i] = __float2half_rn((float)((double)omb * Q.inv_scale[id]));
    }
  }
  __device__ __forceinline__ void flush() {
    if constexpr (SCAN) {
      const unsigned lane = threadIdx.x & 31;
      for (int m = 0; m < kMapScales; ++m) {
        const unsigned v = __reduce_max_sync(0xffffffffu, __float_as_uint(mx[m]));
        if (lane == 0 && v) atomicMax(Q.f16_max + m, v);
      }
    }
  }
};

// Relaxation coefficients of Eqs. (relaxation_a), (relaxation_b) (Sec. 3.2)
// in float arithmetic, for the cell maps, the C-PML strips and the tissue
// tables alike (GB300's FP64 rate would make the build an order of magnitude
// slower):
//   b = exp(-(d/kappa + alpha) dt),  a = d (b - 1) / (kappa (d + kappa alpha)).
// em = expm1(-(d/kappa + alpha) dt) keeps b - 1 accurate when b is near 1;
// b = 1 + em, 1 - b = -em (what bf16 and FP16 maps store), and
// a = (d/kappa) em / (d + kappa alpha).  A few float ulps from the FP64
// values, far inside the parity bound.  One function everywhere keeps the
// index form bitwise equal to the gathered dense maps, and a strip cell at
// depth 0 (a subdomain's cut side) equal to the interior cell it continues.
__device__ __forceinline__ void relax_ab32(float d, float alpha, float kappa, float ik, float dt, float &a,
                                           float &b, float &omb) {
  const float dk = d * ik;
  const float em = expm1f(-(dk + alpha) * dt);
  b = 1.f + em;
  omb = -em;
  const float den = d + kappa * alpha;
  a = (d == 0.f || den == 0.f) ? 0.f : dk * em / den;
}

// depth (cells, 0..L) into the boundary region of coordinate x on an axis of
// n cells whose outer L cells on each side form the region
__device__ __forceinline__ double depth_of(double x, int n, int L) {
  if (L <= 0) return 0.0;
  const double lo = L - 0.5, hi = n - L - 0.5;
  double d = 0.0;
  if (x < lo) d = lo - x;
  else if (x > hi) d = x - hi;
  return d < (double)L ? d : (double)L;
}

// Profile factors of one depth (Table 1): they depend on the depth alone, so
// they are evaluated once per strip coordinate (profile_kernel, 10 us) and not
// in every cell: the strips were bound by the FP64 cosine and power of each
// cell, 55 ms of three strips at 512^3 (N = 3, bf16) against 10 ms now, 0.93
// against 0.18 ms at 4096^2.
struct Profile {
  double depth;  // cells into the boundary region, 0: interior value
  double gT;     // cosine blend of the transition layer
  double spow;   // (depth / L)^npow
};

__device__ __forceinline__ Profile profile_at(const PrepParams &Q, double depth) {
  Profile f{depth, 1.0, 0.0};
  const int LT = Q.LT, L = Q.LT + Q.LB;
  if (LT > 0 && depth < LT) f.gT = 0.5 * (1.0 - cos(M_PI * depth / LT));
  f.spow = pow(depth / L, Q.npow);
  return f;
}

// C-PML / transition value of parameter X0 at a profile's depth (Table 1).
// nu is 0-based here (nu = 0 is the paper's nu = 1); is_d selects d or alpha.
__device__ __forceinline__ double ramp(const PrepParams &Q, double X0, const Profile &f, int nu, bool is_d) {
  if (f.depth <= 0.0) return X0;
  const int L = Q.LT + Q.LB;
  if (nu == 0 && !is_d && (Q.reading == 2 || Q.reading == 3)) {
    // reading C: the tissue's alpha is blended (cosine over the transition
    // layer) into the C-PML profile d_target (1 - x/L), linear to 0 at the
    // outer edge
    const double a_cfs = Q.d_target * (1.0 - f.depth / L);
    return (1.0 - f.gT) * X0 + f.gT * a_cfs;
  }
  if (nu == 0) {
    if (is_d) return (Q.d_target - X0) * f.spow + X0;
    return (0.0 - X0) * (f.depth / L) + X0;
  }
  if (Q.reading == 3) return X0;  // no transition layer: nu >= 2 kept (unstable, Sec. 3.3)
  return (0.0 - X0) * f.gT + X0;
}

// Profiles of axis q's strip: entry 2 sc of Q.profile[q] for the face, 2 sc +
// 1 for the centre of strip coordinate sc.
__global__ void profile_kernel(const PrepParams Q) {
  const int L = Q.LT + Q.LB, q = blockIdx.y;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 4 * L) return;
  const int ext = q == 0 ? Q.nx : q == 1 ? Q.ny : Q.nz;
  const int sc = t >> 1;
  const int cell = sc < L ? sc : ext - 2 * L + sc;
  const double x = Q.goff[q] + cell + ((t & 1) ? 0.0 : 0.5);
  static_cast<Profile *>(Q.profile)[(long long)q * 4 * L + t] = profile_at(Q, depth_of(x, Q.gext[q], L));
}

template <typename MT, bool SCAN>
__global__ void cell_maps_kernel(const PrepParams Q) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  MapSink<MT, SCAN> out(Q);
  // every thread runs the same number of iterations: the scan pass's warp
  // reduction at the end needs the whole warp
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long t0 = blockIdx.x * (long long)blockDim.x; t0 < n; t0 += stride) {
    const long long t = t0 + threadIdx.x;
    if (t >= n) continue;
    const int i = (int)(t % Q.nx);
    const long long r = t / Q.nx;
    const int j = (int)(r % Q.ny);
    const int k = (int)(r / Q.ny);
    const long long o = (long long)k * Q.plane + (long long)j * Q.pitch + i;
    const double c = Q.c[t], rho = Q.rho[t];
    const double K = rho * c * c;
    out.put(kMsK, Q.K, o, K);
    out.put(kMsRho, Q.rho_o, o, rho);
    if (Q.nl_mode != 0) {
      const double beta = Q.beta[t];
      const double chi = Q.nl_mode != 2 ? (1.0 - 2.0 * beta) / K : -2.0 * beta / K;  // 1, 3: Eq. general6
      out.put(kMsChi, Q.chi, o, chi);
    }
    // the rounded float reciprocal equals the FP64 quotient rounded to float
    // (53 bits are more than 2 x 24 + 2), without two FP64 divisions per cell
    const float k1 = Q.N ? Q.k1[t] : 1.f, k2 = Q.N ? Q.k2[t] : 1.f;
    const float ik1 = __frcp_rn(k1), ik2 = __frcp_rn(k2);
    out.put(kMsIk1, Q.ik1, o, ik1);
    out.put(kMsIk2, Q.ik2, o, ik2);
    const float dt = (float)Q.dt;
    for (int nu = 0; nu < Q.N; ++nu) {
      float a, b, omb;
      relax_ab32(Q.d1[nu * n + t], Q.al1[nu * n + t], k1, ik1, dt, a, b, omb);
      out.put(kMsA1 + nu, Q.a1, nu * Q.npts_alloc + o, a);
      out.put_b2(kMsB1 + nu, Q.b1, nu * Q.npts_alloc + o, b, omb);
      relax_ab32(Q.d2[nu * n + t], Q.al2[nu * n + t], k2, ik2, dt, a, b, omb);
      out.put(kMsA2 + nu, Q.a2, nu * Q.npts_alloc + o, a);
      out.put_b2(kMsB2 + nu, Q.b2, nu * Q.npts_alloc + o, b, omb);
    }
  }
  out.flush();
}

// Tissue-index form: per-tissue coefficient table ([field][tab_stride],
// field order of maps.cuh) with the same arithmetic as the per-cell maps, and
// the index copied into the pitched cell layout.
__global__ void table_kernel(const PrepParams Q) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= Q.n_tissue) return;
  float *T = Q.table_out;
  const int S = Q.tab_stride;  // field stride of this table
  const double c = Q.c[t], rho = Q.rho[t];
  const double K = rho * c * c;
  T[kTabK * S + t] = (float)K;
  T[kTabRho * S + t] = (float)rho;
  if (Q.nl_mode != 0) {
    const double beta = Q.beta[t];
    T[kTabChi * S + t] = (float)(Q.nl_mode != 2 ? (1.0 - 2.0 * beta) / K : -2.0 * beta / K);
  }
  const double k1 = Q.N ? (double)Q.k1[t] : 1.0, k2 = Q.N ? (double)Q.k2[t] : 1.0;
  T[kTabIk1 * S + t] = (float)(1.0 / k1);
  T[kTabIk2 * S + t] = (float)(1.0 / k2);
  const float dt = (float)Q.dt;
  for (int nu = 0; nu < Q.N; ++nu) {
    float a, b, omb;
    relax_ab32(Q.d1[nu * Q.n_tissue + t], Q.al1[nu * Q.n_tissue + t], (float)k1, (float)(1.0 / k1), dt, a, b, omb);
    T[(kTabRelax + nu) * S + t] = a;
    T[(kTabRelax + kTabSlots + nu) * S + t] = b;
    relax_ab32(Q.d2[nu * Q.n_tissue + t], Q.al2[nu * Q.n_tissue + t], (float)k2, (float)(1.0 / k2), dt, a, b, omb);
    T[(kTabRelax + 2 * kTabSlots + nu) * S + t] = a;
    T[(kTabRelax + 3 * kTabSlots + nu) * S + t] = b;
  }
}

__global__ void index_copy_kernel(const PrepParams Q) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % Q.nx);
    const long long r = t / Q.nx;
    const int j = (int)(r % Q.ny);
    const int k = (int)(r / Q.ny);
    const long long o = (long long)k * Q.plane + (long long)j * Q.pitch + i;
    if (Q.tissue_wide) static_cast<unsigned short *>(Q.tissue_out)[o] = (unsigned short)tissue_at(Q, t);
    else static_cast<unsigned char *>(Q.tissue_out)[o] = (unsigned char)tissue_at(Q, t);
  }
}

// One thread per (strip coordinate, other two coordinates) of axis `axis`.
template <typename MT, bool SCAN>
__global__ void strip_maps_kernel(const PrepParams Q, int axis) {
  const int L = Q.LT + Q.LB;
  const int ext[3] = {Q.nx, Q.ny, Q.nz};
  // strip extents: the axis has 2L entries, the others their full extent
  int se[3] = {Q.nx, Q.ny, Q.nz};
  se[axis] = 2 * L;
  const long long total = (long long)se[0] * se[1] * se[2];
  const long long pitch_out = axis == 0 ? 2 * L : Q.pitch;
  MapSink<MT, SCAN> sink(Q);
  // the same number of iterations in every thread (see cell_maps_kernel)
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long t0 = blockIdx.x * (long long)blockDim.x; t0 < total; t0 += stride) {
    const long long t = t0 + threadIdx.x;
    if (t >= total) continue;
    int s[3];
    s[0] = (int)(t % se[0]);
    const long long r = t / se[0];
    s[1] = (int)(r % se[1]);
    s[2] = (int)(r / se[1]);
    int cell[3] = {s[0], s[1], s[2]};
    const int sc = s[axis];
    cell[axis] = sc < L ? sc : ext[axis] - 2 * L + sc;
    const long long src = cell[0] + (long long)Q.nx * (cell[1] + (long long)Q.ny * cell[2]);
    // output index in the strip layout
    long long out;
    if (axis == 0) out = ((long long)s[2] * Q.ny + s[1]) * pitch_out + s[0];
    else if (axis == 1) out = ((long long)s[2] * (2 * L) + s[1]) * pitch_out + s[0];
    else out = ((long long)s[2] * Q.ny + s[1]) * pitch_out + s[0];
    const Profile *prof = static_cast<const Profile *>(Q.profile) + ((long long)axis * 2 * L + sc) * 2;
    const Profile fface = prof[0], fcent = prof[1];
    const long long ri = src_of(Q, src), nr = n_src(Q);
    const float k1 = Q.k1[ri], k2 = Q.k2[ri];
    const float ik1 = __frcp_rn(k1), ik2 = __frcp_rn(k2), dt = (float)Q.dt;  // as cell_maps_kernel
    // the ramped parameters (FP64) through the float coefficients of the cells
    for (int nu = 0; nu < Q.N; ++nu) {
      float a, b, omb;
      const double d1 = ramp(Q, Q.d1[nu * nr + ri], fface, nu, true);
      const double al1 = ramp(Q, Q.al1[nu * nr + ri], fface, nu, false);
      relax_ab32((float)d1, (float)al1, k1, ik1, dt, a, b, omb);
      sink.put(kMsA1 + nu, Q.sa1[axis], nu * Q.strip_nu[axis] + out, a);
      sink.put_b2(kMsB1 + nu, Q.sb1[axis], nu * Q.strip_nu[axis] + out, b, omb);
      const double d2 = ramp(Q, Q.d2[nu * nr + ri], fcent, nu, true);
      const double al2 = ramp(Q, Q.al2[nu * nr + ri], fcent, nu, false);
      relax_ab32((float)d2, (float)al2, k2, ik2, dt, a, b, omb);
      sink.put(kMsA2 + nu, Q.sa2[axis], nu * Q.strip_nu[axis] + out, a);
      sink.put_b2(kMsB2 + nu, Q.sb2[axis], nu * Q.strip_nu[axis] + out, b, omb);
    }
  }
  sink.flush();
}

// Medium scan: count of invalid cells, largest c, and largest c /
// sqrt(kappa1 kappa2) in FP64.  Two passes, both bound by reading the medium:
// the first checks every cell and finds the largest quotient in float, the
// second evaluates in FP64 only the cells whose float quotient is within its
// rounding of that (a cell whose float product leaves float's range always
// is).  Each block reduces before its atomics: two FP64 atomics of every
// thread on one address took 1.6 to 1.7 ms from 2 M cells up, where the two
// passes take 0.04 ms (2 M cells) to 0.26 ms (4096^2).
constexpr float kScanMargin = 1e-5f;  // far above the float quotient's error (about 4 ulp)

struct ScanCell {
  float c, k1, k2;
  bool ok;
};
__device__ __forceinline__ ScanCell scan_cell(const PrepParams &Q, long long t) {
  ScanCell s{0.f, 1.f, 1.f, false};
  if (Q.tissue_in && tissue_at(Q, t) >= Q.n_tissue) return s;
  const long long r = src_of(Q, t);
  s.c = Q.c[r];
  const float rho = Q.rho[r];
  if (Q.N) {
    s.k1 = Q.k1[r];
    s.k2 = Q.k2[r];
  }
  s.ok = isfinite(s.c) && s.c > 0.f && isfinite(rho) && rho > 0.f && isfinite(s.k1) && s.k1 > 0.f &&
         isfinite(s.k2) && s.k2 > 0.f && (Q.nl_mode == 0 || isfinite(Q.beta[r]));
  return s;
}
// float quotient, or -1 where the product or the quotient leaves the normal range
__device__ __forceinline__ float scan_quot(const ScanCell &s) {
  const float kk = s.k1 * s.k2;
  if (!(kk > 1e-30f && kk < 1e30f)) return -1.f;
  const float e = s.c * rsqrtf(kk);
  return (e > 1e-30f && e < 1e30f) ? e : -1.f;
}

__global__ void __launch_bounds__(256) medium_scan_kernel(const PrepParams Q, ScanOut *out) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  float m_e = 0.f, m_c = 0.f;
  int nbad = 0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const ScanCell s = scan_cell(Q, t);
    if (!s.ok) {
      ++nbad;
      continue;
    }
    m_e = fmaxf(m_e, scan_quot(s));
    m_c = fmaxf(m_c, s.c);
  }
  // non-negative floats order like their bits
  const unsigned we = __reduce_max_sync(0xffffffffu, __float_as_uint(m_e));
  const unsigned wc = __reduce_max_sync(0xffffffffu, __float_as_uint(m_c));
  const unsigned wb = __reduce_add_sync(0xffffffffu, (unsigned)nbad);
  __shared__ unsigned red[3][8];
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = we;
    red[1][threadIdx.x >> 5] = wc;
    red[2][threadIdx.x >> 5] = wb;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned e = 0, c = 0, b = 0;
    for (int w = 0; w < 8; ++w) {
      e = max(e, red[0][w]);
      c = max(c, red[1][w]);
      b += red[2][w];
    }
    if (e) atomicMax(&out->quot_bits, e);
    if (c) atomicMax(&out->c_bits, c);
    if (b) atomicAdd(&out->bad, b);
  }
}

__global__ void __launch_bounds__(256) medium_speed_kernel(const PrepParams Q, ScanOut *out) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  const float cut = __uint_as_float(out->quot_bits) * (1.f - kScanMargin);
  double m = 0.0;
  ScanCell last{0.f, 0.f, 0.f, false};  // a uniform medium is one value, not one per cell
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const ScanCell s = scan_cell(Q, t);
    if (!s.ok) continue;
    const float e = scan_quot(s);
    if ((e >= 0.f && e < cut) || (s.c == last.c && s.k1 == last.k1 && s.k2 == last.k2)) continue;
    last = s;
    const double ce = (double)s.c / sqrt((double)s.k1 * (double)s.k2);
    m = ce > m ? ce : m;
  }
  unsigned long long bits = (unsigned long long)__double_as_longlong(m);
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, bits, o);
    bits = x > bits ? x : bits;
  }
  __shared__ unsigned long long red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = bits;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) bits = red[w] > bits ? red[w] : bits;
    // a homogeneous medium has candidates in every block: only a larger value
    // goes to the atomic (the plain read may be old, which costs an atomic)
    if (bits > *reinterpret_cast<volatile unsigned long long *>(&out->speed_bits)) atomicMax(&out->speed_bits, bits);
  }
}

int grid_for(long long n) {
  long long b = (n + 255) / 256;
  if (b > 152 * 32) b = 152 * 32;
  if (b < 1) b = 1;
  return (int)b;
}

}  // namespace

cudaError_t launch_medium_scan(const PrepParams &Q, ScanOut *out, cudaStream_t s) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  // eight blocks per SM: enough loads in flight for the copy bandwidth, few atomics
  const int grid = (int)std::min<long long>((n + 255) / 256, 152 * 8);
  medium_scan_kernel<<<grid, 256, 0, s>>>(Q, out);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  medium_speed_kernel<<<grid, 256, 0, s>>>(Q, out);
  return cudaGetLastError();
}

size_t profile_bytes(const PrepParams &Q) { return sizeof(Profile) * 3 * 4 * (size_t)(Q.LT + Q.LB); }

cudaError_t launch_profiles(const PrepParams &Q, cudaStream_t s) {
  const int L = Q.LT + Q.LB;
  profile_kernel<<<dim3((4 * L + 127) / 128, Q.nd), 128, 0, s>>>(Q);
  return cudaGetLastError();
}

namespace {
template <typename MT, bool SCAN>
cudaError_t launch_strips(const PrepParams &Q, cudaStream_t s) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  const int L = Q.LT + Q.LB;
  if (L > 0 && Q.N > 0) {
    for (int axis = 0; axis < Q.nd; ++axis) {
      long long total = 2LL * L * n / (axis == 0 ? Q.nx : axis == 1 ? Q.ny : Q.nz);
      strip_maps_kernel<MT, SCAN><<<grid_for(total), 256, 0, s>>>(Q, axis);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
  }
  return cudaSuccess;
}
}  // namespace

cudaError_t launch_prep(const PrepParams &Q, int map_kind, cudaStream_t s) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  if (map_kind == 2 || map_kind == 3) {
    table_kernel<<<(Q.n_tissue + 255) / 256, 256, 0, s>>>(Q);
    index_copy_kernel<<<grid_for(n), 256, 0, s>>>(Q);
  } else if (map_kind == 1) {
    cell_maps_kernel<__nv_bfloat16, false><<<grid_for(n), 256, 0, s>>>(Q);
  } else if (map_kind == 4) {
    cell_maps_kernel<__half, false><<<grid_for(n), 256, 0, s>>>(Q);
  } else {
    cell_maps_kernel<float, false><<<grid_for(n), 256, 0, s>>>(Q);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (map_kind == 1) return launch_strips<__nv_bfloat16, false>(Q, s);
  if (map_kind == 4) return launch_strips<__half, false>(Q, s);
  return launch_strips<float, false>(Q, s);
}

cudaError_t launch_prep_scan(const PrepParams &Q, cudaStream_t s) {
  const long long n = (long long)Q.nx * Q.ny * Q.nz;
  cell_maps_kernel<__half, true><<<grid_for(n), 256, 0, s>>>(Q);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_strips<__half, true>(Q, s);
}

}  // namespace fw2
