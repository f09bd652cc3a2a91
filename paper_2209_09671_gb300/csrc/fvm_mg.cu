// Geometric multigrid for the density-weighted pressure operator
//   (L x)_c = sum_faces beta_f (x_c - x_nb) / h_d^2
// and the deterministic reductions the solver and the step use.
//   k_gs                red-black Gauss-Seidel sweep of one colour (i+j+k mod 2)
//   k_residual_restrict residual on the fine level, mean over the children
//   k_prolong           piecewise-constant prolongation, added to the fine level
//   k_gs_prolong        the first sweep after the correction with the prolongation folded in
//   k_gs_zero, k_gs_addp the first sweep from x = 0 and the last one adding x to p (mixed form)
//   k_beta_coarsen      coarse face beta = mean of the fine faces it covers
//   k_coarse_cg         conjugate gradients on a coarsest level too large for the tail
//                       of fvm_tail.cu, one CTA
//   k_residual_norm2    ||b - L x||^2 partial sums
//   k_residual64        mixed form: r = b - L p in double, stored as float
//   k_residual_update   r -= L e in float pairs after p += e (large grids)
//   k_gs_pair           a sweep of each colour in one pass (float, large grids)
//   k_restrict_pairs    float residual and restriction, two cells per load
// The paper names no linear solver; this is the reading used throughout the
// library: V(pre, post) cycles, red first before and black first after the
// coarse correction so that the cycle is a symmetric operator.
#include "fvm_device.cuh"

namespace fvm {

// three float weights passed by value to a kernel
struct W3 {
  float w[3];
};

static inline unsigned grid1d(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// block sum, result broadcast to every thread
__device__ double block_sum_all(double v, double* sh) {
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum_d(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    int nw = (blockDim.x + 31) >> 5;
    double t = (lane < nw) ? sh[lane] : 0.0;
    t = warp_sum_d(t);
    if (lane == 0) sh[32] = t;
  }
  __syncthreads();
  return sh[32];
}

// ---------------------------------------------------------------------------
// One FP64 operation an element (the sum of squares took three, both forms and a
// selection) and eight loads in flight.  256^3 double: 74 -> 43 us.
template <typename T>
__global__ void k_sum_field(const T* a, long long n, int squares,
                            double* partial) {
  dependency_wait();
  __shared__ double sh[33];
  double acc = 0.0;
  const long long st = (long long)gridDim.x * blockDim.x;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += 8 * st) {
    T v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = c + q * st < n ? a[c + q * st] : T(0);
    if (squares) {
#pragma unroll
      for (int q = 0; q < 8; ++q) acc = fma((double)v[q], (double)v[q], acc);
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) acc += (double)v[q];
    }
  }
  double s = block_sum_all(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void k_sum_partials(const double* partial, int nparts,
                               double* out, const int* gate) {
  dependency_wait();
  if (gate && !*gate) return;
  __shared__ double sh[33];
  double acc = 0.0;
  for (int q = threadIdx.x; q < nparts; q += blockDim.x) acc += partial[q];
  double s = block_sum_all(acc, sh);
  if (threadIdx.x == 0) *out = s;
}

void launch_sum_partials(const double* partial, int nparts, double* out, cudaStream_t s,
                         const int* gate) {
  overlap_launch(k_sum_partials, 1, 1024, 0, s, partial, nparts, out, gate);
}

template <typename T>
void launch_sum_field(const T* a, long long n, bool squares, double* partial, double* out,
                      cudaStream_t s) {
  overlap_launch(k_sum_field<T>, kRedBlocks, 256, 0, s, a, n, squares ? 1 : 0, partial);
  launch_sum_partials(partial, kRedBlocks, out, s);
}

// a -= sum / n, with the mean formed once per block while the thread's loads
// are in flight.  256^3: 83 -> 43 us (before: a block for every 256 elements,
// each with its own division and barrier).
__global__ void __launch_bounds__(256) k_sub_mean(double* a, long long n, const double* sum) {
  dependency_wait();
  __shared__ double mean;
  const long long c0 = blockIdx.x * (8LL * 256) + threadIdx.x;
  double v[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = c0 + q * 256 < n ? a[c0 + q * 256] : 0.0;
  if (threadIdx.x == 0) mean = (*sum) / (double)n;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q)
    if (c0 + q * 256 < n) a[c0 + q * 256] = v[q] - mean;
}

void launch_sub_mean(double* a, long long n, const double* sum, cudaStream_t s) {
  overlap_launch(k_sub_mean, grid1d(n, 8 * 256), 256, 0, s, a, n, sum);
}

template <typename T>
__global__ void k_zero(T* a, long long n) {
  dependency_wait();
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c < n) a[c] = T(0);
}

template <typename T>
void launch_zero(T* a, long long n, cudaStream_t s) {
  overlap_launch(k_zero<T>, grid1d(n, 256), 256, 0, s, a, n);
}

// ---------------------------------------------------------------------------
// operator pieces on a level
template <typename T>
struct OpNb {
  int lo[3], hi[3];
  T blo[3], bhi[3];
};

template <typename T>
__device__ __forceinline__ void neighbours(const MGLevel<T>& L, int i, int j, int k, int c,
                                           OpNb<T>& nb) {
  const Geo& g = L.geo;
  const int idx[3] = {i, j, k};
  const int st[3] = {1, g.n[0], g.n[0] * g.n[1]};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int n = g.n[d];
    const int lo = idx[d] == 0 ? c + (n - 1) * st[d] : c - st[d];
    const int hi = idx[d] == n - 1 ? c - (n - 1) * st[d] : c + st[d];
    nb.lo[d] = lo;
    nb.hi[d] = hi;
    nb.blo[d] = L.beta[d][c];
    nb.bhi[d] = (g.bc[d] == WALL && idx[d] == n - 1) ? T(0) : L.beta[d][hi];
  }
}

template <typename T, typename X>
__device__ __forceinline__ X apply_L_at(const MGLevel<T>& L, const X* x, int c,
                                        const OpNb<T>& nb) {
  const Geo& g = L.geo;
  X xc = x[c];
  X out = X(0);
  if (L.wu != T(0)) {
    // one weight for every axis: 13 operations instead of 15
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (g.n[d] == 1) continue;
      out += (X)nb.blo[d] * (xc - x[nb.lo[d]]);
      out += (X)nb.bhi[d] * (xc - x[nb.hi[d]]);
    }
    return out * (X)L.wu;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (g.n[d] == 1) continue;
    out += ((X)nb.blo[d] * (xc - x[nb.lo[d]]) + (X)nb.bhi[d] * (xc - x[nb.hi[d]])) * (X)L.w[d];
  }
  return out;
}

__device__ __forceinline__ void decode_lv(const Geo& g, long long c, int& i, int& j, int& k) {
  const int cc = (int)c;
  const int q = cc / g.n[0];
  i = cc - q * g.n[0];
  k = q / g.n[1];
  j = q - k * g.n[1];
}

// ---------------------------------------------------------------------------
// Gauss-Seidel value of one cell from its right-hand side, the face betas
// and the neighbour values on the low and high side of each axis (axes of
// one cell carry no coupling).  wu: the common weight of the axes (0: w per
// axis).  inv: the cell's reciprocal diagonal, null to form and divide by the
// diagonal.  A double update is bound by the FP64 pipe (2 lanes a clock per
// SM): 8 operations with both, about 27 with neither; a colour sweep of
// 128^3 cells took 50 us before, and the array costs 8 bytes per cell.  In
// float the sweeps are bound by memory, so they divide.
template <typename T>
__device__ __forceinline__ T gs_formula(const Geo& g, const T* w, T wu, T b, const T* blo,
                                        const T* bhi, const T* xlo, const T* xhi,
                                        const T* inv = nullptr) {
  T num, den = T(0);
  if (wu != T(0)) {
    T sum = T(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (g.n[d] == 1) continue;
      sum += blo[d] * xlo[d];
      sum += bhi[d] * xhi[d];
    }
    num = b + sum * wu;
  } else {
    num = b;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (g.n[d] == 1) continue;
      num += (blo[d] * xlo[d] + bhi[d] * xhi[d]) * w[d];
    }
  }
  if (inv) return num * *inv;
  if (wu != T(0)) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (g.n[d] == 1) continue;
      den += blo[d] + bhi[d];
    }
    den *= wu;
  } else {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (g.n[d] == 1) continue;
      den += (blo[d] + bhi[d]) * w[d];
    }
  }
  return num / den;
}

template <typename T>
__device__ __forceinline__ T gs_value(const MGLevel<T>& L, int c, const OpNb<T>& nb, const T* xlo,
                                      const T* xhi) {
  return gs_formula(L.geo, L.w, L.wu, L.b[c], nb.blo, nb.bhi, xlo, xhi,
                    L.inv ? L.inv + c : nullptr);
}

template <typename T>
__global__ void k_inv_diag(MGLevel<T> L) {
  dependency_wait();
  const Geo& g = L.geo;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (i >= g.n[0] || j >= g.n[1] || k >= g.n[2]) return;
  const int c = (k * g.n[1] + j) * g.n[0] + i;
  OpNb<T> nb;
  neighbours(L, i, j, k, c, nb);
  T den = T(0);
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (g.n[d] > 1) den += (nb.blo[d] + nb.bhi[d]) * L.w[d];
  L.inv[c] = T(1) / den;
}

template <typename T>
void launch_inv_diag(const MGLevel<T>& L, cudaStream_t s) {
  const dim3 bs(32, 4, 2);
  const dim3 gs((L.geo.n[0] + 31) / 32, (L.geo.n[1] + 3) / 4, (L.geo.n[2] + 1) / 2);
  overlap_launch(k_inv_diag<T>, gs, bs, 0, s, L);
}

// Gauss-Seidel update of one cell (its colour's neighbours are fixed), which
// are read from x
template <typename T>
__device__ __forceinline__ void gs_point(const MGLevel<T>& L, int i, int j, int k, const T* x) {
  const Geo& g = L.geo;
  const int c = (k * g.n[1] + j) * g.n[0] + i;
  OpNb<T> nb;
  neighbours(L, i, j, k, c, nb);
  T xlo[3], xhi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    xlo[d] = x[nb.lo[d]];
    xhi[d] = x[nb.hi[d]];
  }
  L.x[c] = gs_value(L, c, nb, xlo, xhi);
}

// gate (optional): the sweep does nothing once *gate >= gate_min (the FP64
// solve graph skips the first sweep of every cycle after the first, which
// would repeat the previous cycle's last sweep)
template <typename T>
__global__ void k_gs(MGLevel<T> L, int colour, const int* gate, int gate_min,
                     const T* xin) {
  dependency_wait();
  if (gate && *gate >= gate_min) return;
  const Geo& g = L.geo;
  const int i2 = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (j >= g.n[1] || k >= g.n[2]) return;
  const int i = 2 * i2 + ((colour + j + k) & 1);
  if (xin) {
    // the other colour's first-sweep values move to x: on an axis with walls and
    // an odd number of cells the wrapped neighbour of a wall cell (times beta = 0)
    // has the cell's own colour, so the next sweep reads them there
    const int io = i ^ 1, row = (k * g.n[1] + j) * g.n[0];
    if (io < g.n[0]) L.x[row + io] = xin[row + io];
  }
  if (i >= g.n[0]) return;
  gs_point(L, i, j, k, xin ? xin : L.x);
}

template <typename T>
void launch_gs(const MGLevel<T>& L, int colour, cudaStream_t s, const int* gate, int gate_min,
               const T* xin) {
  const int hx = (L.geo.n[0] + 1) / 2;
  dim3 bs(32, 4, 2);
  dim3 gs((hx + 31) / 32, (L.geo.n[1] + 3) / 4, (L.geo.n[2] + 1) / 2);
  overlap_launch(k_gs<T>, gs, bs, 0, s, L, colour, gate, gate_min, xin);
}

// coarse b = mean over children of (b - L x) on the fine level; coarse x = 0.
// half: the fine level's last sweep was of colour 1, so the residuals of
// those cells are 0 up to the rounding of that sweep; only the children of
// colour 0 are formed (half the FP64 operations: 90 -> 43 us for 128^3 double).
// Not in float: there that rounding is what keeps the restricted residual's
// sum 0, and without it a density ratio of 7900 between the phases slows the
// convergence (1.5e-9 -> 3.1e-8 after five refinements at 256^3).
template <typename T>
__device__ __forceinline__ void restrict_point(const MGLevel<T>& F, const MGLevel<T>& C, int I,
                                               int J, int K, bool half) {
  const long long cc = lin(C.geo, I, J, K);
  T acc = T(0);
  for (int dz = 0; dz < F.f[2]; ++dz)
    for (int dy = 0; dy < F.f[1]; ++dy) {
      const int j = J * F.f[1] + dy, k = K * F.f[2] + dz;
      for (int dx = 0; dx < F.f[0]; ++dx) {
        const int i = I * F.f[0] + dx;
        if (half && ((i + j + k) & 1)) continue;
        const int c = (k * F.geo.n[1] + j) * F.geo.n[0] + i;
        OpNb<T> nb;
        neighbours(F, i, j, k, c, nb);
        acc += F.b[c] - apply_L_at<T, T>(F, F.x, c, nb);
      }
    }
  const int n = F.f[0] * F.f[1] * F.f[2];   // 1, 2, 4 or 8 children
  C.b[cc] = acc * (n == 8 ? T(0.125) : (n == 4 ? T(0.25) : (n == 2 ? T(0.5) : T(1))));
  C.x[cc] = T(0);
}

// one thread per coarse cell on a 3D grid (no index division per thread)
template <typename T>
__global__ void k_residual_restrict(MGLevel<T> F, MGLevel<T> C, int sweep, int half) {
  dependency_wait();
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y * blockDim.y + threadIdx.y;
  const int K = blockIdx.z * blockDim.z + threadIdx.z;
  if (I >= C.geo.n[0] || J >= C.geo.n[1] || K >= C.geo.n[2]) return;
  restrict_point(F, C, I, J, K, half != 0);
  if (sweep && ((I + J + K) & 1) == 0) {
    // the coarse level's first sweep (colour 0 from x = 0) needs only the
    // cell's own right-hand side: taken here, with k_gs's arithmetic
    const int cc = (int)lin(C.geo, I, J, K);
    OpNb<T> nb;
    neighbours(C, I, J, K, cc, nb);
    const T z[3] = {T(0), T(0), T(0)};
    C.x[cc] = gs_value(C, cc, nb, z, z);
  }
}

// The same, float, of a level with one weight that is coarsened by two along each
// axis: the thread's 2 x 2 x 2 cells are four pairs of neighbours in x, so that
// all but twelve of its 44 loads bring two values (the general form takes about
// 76 of one value each).  128 x 128 x 64 to half: 12.7 -> 9.0 us; at 256^3, where the
// 20 bytes a cell come from HBM, 87 us in both forms.  The operations and their
// order are the same.
__global__ void k_restrict_pairs(MGLevel<float> F, MGLevel<float> C, int sweep) {
  dependency_wait();
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int J = blockIdx.y * blockDim.y + threadIdx.y;
  const int K = blockIdx.z * blockDim.z + threadIdx.z;
  if (I >= C.geo.n[0] || J >= C.geo.n[1] || K >= C.geo.n[2]) return;
  const Geo& g = F.geo;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxy = nx * ny;
  const int i = 2 * I, j = 2 * J, k = 2 * K, c = (k * ny + j) * nx + i;
  // from the first cell of the pair, row or plane to the neighbours on both sides
  const bool ex = i + 2 == nx, ey = j + 2 == ny, ez = k + 2 == nz;
  const int xm = i == 0 ? nx - 1 : -1, xp = ex ? 2 - nx : 2;
  const int ym = j == 0 ? (ny - 1) * nx : -nx, yp = ey ? (2 - ny) * nx : 2 * nx;
  const int zm = k == 0 ? (nz - 1) * nxy : -nxy, zp = ez ? (2 - nz) * nxy : 2 * nxy;
  const bool wx = ex && g.bc[0] == WALL, wy = ey && g.bc[1] == WALL, wz = ez && g.bc[2] == WALL;
  const auto two = [](const float* a, int o) { return *reinterpret_cast<const float2*>(a + o); };
  float2 x[4][4], bz[3][2];      // planes k - 1 .. k + 2, rows j - 1 .. j + 2; low z-faces
#pragma unroll
  for (int dy = 0; dy < 2; ++dy) {
    x[0][dy + 1] = two(F.x, c + zm + dy * nx);
    x[3][dy + 1] = two(F.x, c + zp + dy * nx);
    bz[2][dy] = two(F.beta[2], c + zp + dy * nx);
    if (wz) bz[2][dy] = make_float2(0.f, 0.f);
  }
#pragma unroll
  for (int dz = 0; dz < 2; ++dz) {
    x[dz + 1][0] = two(F.x, c + dz * nxy + ym);
    x[dz + 1][3] = two(F.x, c + dz * nxy + yp);
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      x[dz + 1][dy + 1] = two(F.x, c + dz * nxy + dy * nx);
      bz[dz][dy] = two(F.beta[2], c + dz * nxy + dy * nx);
    }
  }
  float acc = 0.f;
#pragma unroll
  for (int dz = 0; dz < 2; ++dz) {
    const int cz = c + dz * nxy;
    float2 by[3] = {two(F.beta[1], cz), two(F.beta[1], cz + nx), two(F.beta[1], cz + yp)};
    if (wy) by[2] = make_float2(0.f, 0.f);
#pragma unroll
    for (int dy = 0; dy < 2; ++dy) {
      const int o = cz + dy * nx;
      const float2 b = two(F.b, o), bx = two(F.beta[0], o), v = x[dz + 1][dy + 1];
      const float bxh = wx ? 0.f : F.beta[0][o + xp];
      const float vl = F.x[o + xm], vh = F.x[o + xp];
      float out = 0.f;
      out += bx.x * (v.x - vl);
      out += bx.y * (v.x - v.y);
      out += by[dy].x * (v.x - x[dz + 1][dy].x);
      out += by[dy + 1].x * (v.x - x[dz + 1][dy + 2].x);
      out += bz[dz][dy].x * (v.x - x[dz][dy + 1].x);
      out += bz[dz + 1][dy].x * (v.x - x[dz + 2][dy + 1].x);
      acc += b.x - out * F.wu;
      out = 0.f;
      out += bx.y * (v.y - v.x);
      out += bxh * (v.y - vh);
      out += by[dy].y * (v.y - x[dz + 1][dy].y);
      out += by[dy + 1].y * (v.y - x[dz + 1][dy + 2].y);
      out += bz[dz][dy].y * (v.y - x[dz][dy + 1].y);
      out += bz[dz + 1][dy].y * (v.y - x[dz + 2][dy + 1].y);
      acc += b.y - out * F.wu;
    }
  }
  const int cc = (K * C.geo.n[1] + J) * C.geo.n[0] + I;
  C.b[cc] = acc * 0.125f;
  float first = 0.f;
  if (sweep && ((I + J + K) & 1) == 0) {
    OpNb<float> nb;
    neighbours(C, I, J, K, cc, nb);
    const float z[3] = {0.f, 0.f, 0.f};
    first = gs_formula(C.geo, C.w, C.wu, acc * 0.125f, nb.blo, nb.bhi, z, z);
  }
  C.x[cc] = first;
}

inline bool restrict_as_pairs(const MGLevel<float>& F, const MGLevel<float>& C, int sweep, dim3 gs,
                              dim3 bs, cudaStream_t s) {
  if (F.f[0] != 2 || F.f[1] != 2 || F.f[2] != 2 || F.wu == 0.f) return false;
  overlap_launch(k_restrict_pairs, gs, bs, 0, s, F, C, sweep);
  return true;
}
inline bool restrict_as_pairs(const MGLevel<double>&, const MGLevel<double>&, int, dim3, dim3,
                              cudaStream_t) {
  return false;
}

// sweep: also take the coarse level's first Gauss-Seidel sweep from x = 0
template <typename T>
void launch_residual_restrict(const MGLevel<T>& F, const MGLevel<T>& C, cudaStream_t s, bool sweep,
                              bool half) {
  const dim3 bs(32, 4, 2);
  const dim3 gs((C.geo.n[0] + 31) / 32, (C.geo.n[1] + 3) / 4, (C.geo.n[2] + 1) / 2);
  if (restrict_as_pairs(F, C, sweep ? 1 : 0, gs, bs, s)) return;
  overlap_launch(k_residual_restrict<T>, gs, bs, 0, s, F, C, sweep ? 1 : 0, half ? 1 : 0);
}

// the coarsening factor of an axis is 1 or 2
__device__ __forceinline__ int coarse_index(int i, int f) { return f == 2 ? (i >> 1) : i; }

template <typename T>
__device__ __forceinline__ void prolong_point(const MGLevel<T>& F, const MGLevel<T>& C, int i,
                                              int j, int k) {
  const long long c = lin(F.geo, i, j, k);
  const long long p = lin(C.geo, coarse_index(i, F.f[0]), coarse_index(j, F.f[1]),
                          coarse_index(k, F.f[2]));
  F.x[c] = F.x[c] + C.x[p];
}

// one thread per fine cell on a 3D grid (no index division per thread)
template <typename T>
__global__ void k_prolong(MGLevel<T> F, MGLevel<T> C) {
  dependency_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (i >= F.geo.n[0] || j >= F.geo.n[1] || k >= F.geo.n[2]) return;
  prolong_point(F, C, i, j, k);
}

template <typename T>
void launch_prolong(const MGLevel<T>& F, const MGLevel<T>& C, cudaStream_t s) {
  const dim3 bs(32, 4, 2);
  const dim3 gs((F.geo.n[0] + 31) / 32, (F.geo.n[1] + 3) / 4, (F.geo.n[2] + 1) / 2);
  overlap_launch(k_prolong<T>, gs, bs, 0, s, F, C);
}

// The first colour sweep after the coarse correction with the
// piecewise-constant prolongation folded in.  A sweep of one colour reads
// only the other colour, so it takes those cells' values plus the coarse
// correction of their parent cells on the fly; the other colour's stored
// values are then overwritten by the next sweep without being read.  The
// pair of sweeps therefore leaves x as k_prolong followed by two k_gs
// launches would, bit for bit, without the prolongation's pass over x.
template <typename T>
__global__ void k_gs_prolong(MGLevel<T> F, MGLevel<T> C, int colour) {
  dependency_wait();
  const Geo& g = F.geo;
  const int i2 = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (j >= g.n[1] || k >= g.n[2]) return;
  const int i = 2 * i2 + ((colour + j + k) & 1);
  if (i >= g.n[0]) return;
  const int c = (k * g.n[1] + j) * g.n[0] + i;
  OpNb<T> nb;
  neighbours(F, i, j, k, c, nb);
  const int idx[3] = {i, j, k};
  T xlo[3], xhi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int n = g.n[d];
    int lo[3] = {i, j, k}, hi[3] = {i, j, k};
    lo[d] = idx[d] == 0 ? n - 1 : idx[d] - 1;
    hi[d] = idx[d] == n - 1 ? 0 : idx[d] + 1;
    const long long pl = lin(C.geo, coarse_index(lo[0], F.f[0]), coarse_index(lo[1], F.f[1]),
                             coarse_index(lo[2], F.f[2]));
    const long long ph = lin(C.geo, coarse_index(hi[0], F.f[0]), coarse_index(hi[1], F.f[1]),
                             coarse_index(hi[2], F.f[2]));
    xlo[d] = F.x[nb.lo[d]] + C.x[pl];
    xhi[d] = F.x[nb.hi[d]] + C.x[ph];
  }
  F.x[c] = gs_value(F, c, nb, xlo, xhi);
}

// The first sweep of a solve that starts from x = 0 (the mixed form's inner
// correction): the other colour's values are 0, so the swept cells take
// gs_formula with zero neighbours and the cells of the other colour are set
// to 0 by the same thread (the pair 2 i2, 2 i2 + 1 of its row), which
// replaces zeroing x in a pass of its own.
template <typename T>
__global__ void k_gs_zero(MGLevel<T> L, int colour) {
  dependency_wait();
  const Geo& g = L.geo;
  const int i2 = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (j >= g.n[1] || k >= g.n[2]) return;
  const int i = 2 * i2 + ((colour + j + k) & 1), io = i ^ 1;
  const int row = (k * g.n[1] + j) * g.n[0];
  if (io < g.n[0]) L.x[row + io] = T(0);
  if (i >= g.n[0]) return;
  OpNb<T> nb;
  neighbours(L, i, j, k, row + i, nb);
  const T z[3] = {T(0), T(0), T(0)};
  L.x[row + i] = gs_value(L, row + i, nb, z, z);
}

// The last sweep of the mixed form's inner correction with p += e folded in:
// the thread adds the new value of its cell and the final value of the other
// colour's cell beside it (not written in this sweep) to the double p.  The
// correction e itself is stored only when the residual is updated with it
// (k_residual_update); the next refinement starts it from 0.
__global__ void k_gs_addp(MGLevel<float> L, int colour, double* p, int store) {
  dependency_wait();
  const Geo& g = L.geo;
  const int i2 = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z * blockDim.z + threadIdx.z;
  if (j >= g.n[1] || k >= g.n[2]) return;
  const int i = 2 * i2 + ((colour + j + k) & 1), io = i ^ 1;
  const int row = (k * g.n[1] + j) * g.n[0];
  if (io < g.n[0]) p[row + io] = p[row + io] + (double)L.x[row + io];
  if (i >= g.n[0]) return;
  OpNb<float> nb;
  neighbours(L, i, j, k, row + i, nb);
  float xlo[3], xhi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    xlo[d] = L.x[nb.lo[d]];
    xhi[d] = L.x[nb.hi[d]];
  }
  const float e = gs_value(L, row + i, nb, xlo, xhi);
  if (store) L.x[row + i] = e;
  p[row + i] = p[row + i] + (double)e;
}

// ---------------------------------------------------------------------------
// Two sweeps in one pass, float: colour a = `first` from x, then colour b from
// the new values, both colours stored to x2.  A colour sweep reads every line of
// x, b and the three betas and writes x: 24 bytes a cell.  A pair in one pass moves
// 24 bytes and a halo, about 33, instead of 48.
//
// A thread owns two neighbouring cells of a row (one of each colour) and walks
// planes upward: the a-cell of plane k from old values, then the b-cell of plane
// k - 1 from new ones.  Values along z stay in registers, those along x come from
// the neighbouring lanes, those along y from global memory (old values) or shared
// memory (new ones).  The outermost lanes, rows and planes of a CTA compute
// a-cells only, for the b-cells beside them: x2 is another array because other
// CTAs still read the old values there.  Every value is that of gs_formula on the
// same operands as in the sweeps one by one, so the results are theirs bit for bit.
//
// A plane's loads are issued a plane ahead into registers and kPairAhead planes
// ahead into L2; what is left is bound by instructions (about 150 per plane and
// warp).  Rings of planes in shared memory filled by 8-byte asynchronous copies
// (bound by L1) or by a bulk copy per row (about 12 cycles each) took half as long
// again.  256^3: a pair 140 us as two sweeps, 101 here (123 with the prolongation, 191
// with p += e); 512 x 512 x 256: 515 and 430.  Below kPairCells, where most of a level stays in L2 and the planes in a
// row count, the sweeps one by one are as fast or faster: melt pool step at
// 256 x 256 x 128 29.3 ms both ways, 192^3 29.2 both, 160^3 18.5 against 18.8 with
// pairs, 128^3 9.6 against 10.3; above, 224 x 224 x 192 36.0 against 35.1, 256^3 46.7
// against 45.5, 512 x 512 x 256 220.6 against 206.7.
constexpr long long kPairCells = 1 << 23;
constexpr int kPairRows = 14;      // rows of a CTA, two of them halo
constexpr int kPairCTAs = 2;       // CTAs per SM
constexpr int kPairAhead = 3;

struct PairTiles {
  int px, py, kz;                  // cell pairs, rows and planes of a CTA
};

template <int S>
__device__ __forceinline__ float pick(float2 v) {
  return S ? v.y : v.x;
}

// gs_formula for one weight on three coupled axes
__device__ __forceinline__ float pair_formula(float wu, float b, const float* lo, const float* hi,
                                              const float* xlo, const float* xhi) {
  float sum = 0.f, den = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    sum += lo[d] * xlo[d];
    sum += hi[d] * xhi[d];
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) den += lo[d] + hi[d];
  den *= wu;
  return (b + sum * wu) / den;
}

__device__ __forceinline__ void prefetch_l2(const float* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// a barrier that the rows reach from different copies of the loop
__device__ __forceinline__ void pair_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// what a plane's step reads, fetched one step ahead
struct PairLoad {
  float2 xn, b, bx, yl, yh, zh;  // (xn, zh: of the plane above)
  float ylo, yhi;                // the a-cell's neighbours in the rows beside
  float cn, clo, chi;            // the coarse corrections of xn, ylo and yhi, added when
                                 // they are used
};

// what a thread carries from plane to plane
struct PairWalk {
  float2 xp, xc, zl;             // old values of planes k - 1 and k; betas below plane k
  float a1, a2;                  // the a-cells of planes k - 1 and k - 2
  float pb, plo[3], phi[3];      // right-hand side and betas of plane k - 1's b-cell
};

// One thread's planes.  Neighbours wrap on walls as on periodic axes: the beta of
// a wall's face is stored as 0 (on the low side of the first cells, where the last
// cells find it by wrapping), and the values it multiplies are finite.
template <bool PROLONG, bool ADDP>
struct PairStep {
  const MGLevel<float>& L;
  const float* xc;               // the coarse correction
  double* p;
  float (*sh)[kPairRows][32];
  int lane, r, cx;               // cx: the pair's parent in a coarse plane
  int dlo, dhi, clo, chi;        // to the rows beside, to their parents
  bool keep;

  __device__ __forceinline__ float2 old(int o, int co) const {
    float2 v = *reinterpret_cast<const float2*>(L.x + o);
    if (PROLONG) {
      const float q = xc[co + cx];
      v.x = v.x + q;
      v.y = v.y + q;
    }
    return v;
  }

  // the loads of a plane at offset o below one at on (parents at co, cn), whose
  // a-cell is component s
  __device__ __forceinline__ PairLoad load(int o, int on, int co, int cn, int s) const {
    PairLoad f;
    f.xn = *reinterpret_cast<const float2*>(L.x + on);
    f.b = *reinterpret_cast<const float2*>(L.b + o);
    f.bx = *reinterpret_cast<const float2*>(L.beta[0] + o);
    f.yl = *reinterpret_cast<const float2*>(L.beta[1] + o);
    f.yh = *reinterpret_cast<const float2*>(L.beta[1] + o + dhi);
    f.zh = *reinterpret_cast<const float2*>(L.beta[2] + on);
    f.ylo = L.x[o + dlo + s];
    f.yhi = L.x[o + dhi + s];
    if (PROLONG) {
      f.cn = xc[cn + cx];
      f.clo = xc[co + clo + cx];
      f.chi = xc[co + chi + cx];
    }
    return f;
  }

  __device__ __forceinline__ void prefetch(int o) const {
    prefetch_l2(L.x + o);
    prefetch_l2(L.b + o);
    prefetch_l2(L.beta[0] + o);
    prefetch_l2(L.beta[1] + o);
    prefetch_l2(L.beta[2] + o);
  }

  // plane k, whose a-cell is component S of the pair; store: plane k - 1, at offset
  // op, is complete
  template <int S>
  __device__ __forceinline__ void run(PairWalk& w, PairLoad f, bool store, int op) const {
    if (PROLONG) {
      f.xn = make_float2(f.xn.x + f.cn, f.xn.y + f.cn);
      f.ylo = f.ylo + f.clo;
      f.yhi = f.yhi + f.chi;
    }
    const float bxr = __shfl_down_sync(0xffffffffu, f.bx.x, 1);
    // the cells beside the a-cell: one is the pair's, one the next lane's
    const float side = S ? __shfl_down_sync(0xffffffffu, w.xc.x, 1)
                         : __shfl_up_sync(0xffffffffu, w.xc.y, 1);
    const float as = S ? __shfl_down_sync(0xffffffffu, w.a1, 1)
                       : __shfl_up_sync(0xffffffffu, w.a1, 1);
    float a;
    {
      const float lo[3] = {pick<S>(f.bx), pick<S>(f.yl), pick<S>(w.zl)};
      const float hi[3] = {S ? bxr : f.bx.y, pick<S>(f.yh), pick<S>(f.zh)};
      const float vlo[3] = {S ? w.xc.x : side, f.ylo, pick<S>(w.xp)};
      const float vhi[3] = {S ? side : w.xc.y, f.yhi, pick<S>(f.xn)};
      a = pair_formula(L.wu, pick<S>(f.b), lo, hi, vlo, vhi);
    }
    sh[S][r][lane] = a;
    // the b-cell of plane k - 1: component S as well; the rows beside it hold that
    // plane's a-cells in component S too
    if (store) {
      const float vlo[3] = {S ? w.a1 : as, sh[S][r - 1][lane], w.a2};
      const float vhi[3] = {S ? as : w.a1, sh[S][r + 1][lane], a};
      const float v = pair_formula(L.wu, w.pb, w.plo, w.phi, vlo, vhi);
      const float2 e = S ? make_float2(w.a1, v) : make_float2(v, w.a1);
      if (!ADDP || keep) *reinterpret_cast<float2*>(L.x2 + op) = e;
      if (ADDP) {
        p[op] = p[op] + (double)e.x;
        p[op + 1] = p[op + 1] + (double)e.y;
      }
    }
    w.pb = pick<1 - S>(f.b);
    w.plo[0] = pick<1 - S>(f.bx);
    w.phi[0] = S ? f.bx.y : bxr;
    w.plo[1] = pick<1 - S>(f.yl);
    w.phi[1] = pick<1 - S>(f.yh);
    w.plo[2] = pick<1 - S>(w.zl);
    w.phi[2] = pick<1 - S>(f.zh);
    w.a2 = w.a1;
    w.a1 = a;
    w.xp = w.xc;
    w.xc = f.xn;
    w.zl = f.zh;
  }

  // planes k0 - 1 .. k1 (plane k1 for its a-cells only) from the a-cell S of plane
  // k0 - 1 on, two at a time so that what was fetched stays where it is
  template <int S>
  __device__ __forceinline__ void march(int k0, int k1, int col, int nz, int nxy, int cnxy,
                                        bool out) const {
    const int n = nz * nxy;
    const auto up = [&](int o) { return plane_above(o, nxy, n); };
    const auto parent = [&](int k) {
      return PROLONG ? coarse_index(k < 0 ? k + nz : (k >= nz ? k - nz : k), L.f[2]) * cnxy : 0;
    };
    int om = (k0 - 2 < 0 ? k0 - 2 + nz : k0 - 2) * nxy + col;
    const int o = up(om);
    int on = up(o), ahead = on;          // planes k + 1 and k + kPairAhead
    for (int q = 1; q < kPairAhead; ++q) ahead = up(ahead);
    PairWalk w = {};
    w.xp = old(om, parent(k0 - 2));
    w.xc = old(o, parent(k0 - 1));
    w.zl = *reinterpret_cast<const float2*>(L.beta[2] + o);
    PairLoad f = load(o, on, parent(k0 - 1), parent(k0), S), h = f;
    int op = (k0 - 2) * nxy + col;       // plane k - 1
    for (int k = k0 - 1;; k += 2) {
      if (k + kPairAhead <= k1) prefetch(ahead);
      if (k < k1) h = load(on, up(on), parent(k + 1), parent(k + 2), 1 - S);
      run<S>(w, f, out && k > k0, op);
      pair_barrier();
      if (k >= k1) break;
      on = up(on);
      ahead = up(ahead);
      op += nxy;
      if (k + 1 + kPairAhead <= k1) prefetch(ahead);
      if (k + 1 < k1) f = load(on, up(on), parent(k + 2), parent(k + 3), S);
      run<1 - S>(w, h, out && k + 1 > k0, op);
      pair_barrier();
      if (k + 1 >= k1) break;
      on = up(on);
      ahead = up(ahead);
      op += nxy;
    }
  }
};

template <bool PROLONG, bool ADDP>
__global__ void __launch_bounds__(32 * kPairRows, kPairCTAs)
    k_gs_pair(MGLevel<float> L, MGLevel<float> C, int first, double* p, int keep, PairTiles t) {
  dependency_wait();
  __shared__ float sh[2][kPairRows][32];   // the a-cells of planes k and k - 1, by component
  const Geo& g = L.geo;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxy = nx * ny, hx = nx >> 1;
  const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
  // this thread's pair and row, wrapped; lanes past the halo repeat its last one,
  // rows past it only keep the barriers
  int i2 = blockIdx.x * t.px - 1 + min(lane, t.px + 1);
  int j = blockIdx.y * t.py - 1 + r;
  const bool out = lane >= 1 && lane <= t.px && i2 < hx && r >= 1 && r <= t.py && j < ny;
  i2 = i2 < 0 ? hx - 1 : (i2 >= hx ? 0 : i2);
  const int par = j + first;
  j = j < 0 ? ny - 1 : (j >= ny ? 0 : j);
  const int jlo = j == 0 ? ny - 1 : j - 1, jhi = j == ny - 1 ? 0 : j + 1;
  const int col = j * nx + 2 * i2;
  const int cnx = C.geo.n[0], cnxy = cnx * C.geo.n[1];
  const int cj = coarse_index(j, L.f[1]);
  const PairStep<PROLONG, ADDP> st = {
      L, C.x, p, sh, lane, r, i2 + cj * cnx, (jlo - j) * nx, (jhi - j) * nx,
      (coarse_index(jlo, L.f[1]) - cj) * cnx, (coarse_index(jhi, L.f[1]) - cj) * cnx, keep != 0};
  const int k0 = blockIdx.z * t.kz, k1 = min(k0 + t.kz, nz);
  if (r > t.py + 1) {
    for (int k = k0 - 1; k <= k1; ++k) pair_barrier();
  } else if ((par + k0 - 1) & 1) {
    st.template march<1>(k0, k1, col, nz, nxy, cnxy, out);
  } else {
    st.template march<0>(k0, k1, col, nz, nxy, cnxy, out);
  }
}

bool pairs_fit(const Geo& g, int fx) {
  return g.N >= kPairCells && g.n[0] >= 4 && fx == 2 && g.n[1] >= 4 && g.n[2] >= 4;
}

void launch_gs_pair(const MGLevel<float>& L, const MGLevel<float>* C, int first, double* p,
                    bool keep, cudaStream_t s) {
  // even shares of at most 30 pairs and kPairRows - 2 rows; as many runs of planes
  // as make the number of rounds (two CTAs per SM at a time) times the planes of a
  // run, halo included, least
  const int hx = L.geo.n[0] / 2, ny = L.geo.n[1], nz = L.geo.n[2];
  const int tx = (hx + 29) / 30, ty = (ny + kPairRows - 3) / (kPairRows - 2);
  PairTiles t;
  t.px = (hx + tx - 1) / tx;
  t.py = (ny + ty - 1) / ty;
  const long long tiles = (long long)tx * ty;
  long long best = 0;
  t.kz = nz;
  for (int runs = 1; 4 * runs <= nz; ++runs) {
    const int kz = (nz + runs - 1) / runs;
    const long long cost = (tiles * ((nz + kz - 1) / kz) + kPairCTAs * 152 - 1) / (kPairCTAs * 152) * (kz + 3);
    if (runs == 1 || cost < best) {
      best = cost;
      t.kz = kz;
    }
  }
  const dim3 gs(tx, ty, (nz + t.kz - 1) / t.kz);
  void (*k)(MGLevel<float>, MGLevel<float>, int, double*, int, PairTiles) =
      C ? (p ? k_gs_pair<true, true> : k_gs_pair<true, false>)
        : (p ? k_gs_pair<false, true> : k_gs_pair<false, false>);
  overlap_launch(k, gs, dim3(32 * kPairRows), 0, s, L, C ? *C : L, first, p, keep ? 1 : 0, t);
}

template <typename T>
void launch_gs_zero(const MGLevel<T>& L, int colour, cudaStream_t s) {
  const int hx = (L.geo.n[0] + 1) / 2;
  dim3 bs(32, 4, 2);
  dim3 gs((hx + 31) / 32, (L.geo.n[1] + 3) / 4, (L.geo.n[2] + 1) / 2);
  overlap_launch(k_gs_zero<T>, gs, bs, 0, s, L, colour);
}

void launch_gs_addp(const MGLevel<float>& L, int colour, double* p, bool store, cudaStream_t s) {
  const int hx = (L.geo.n[0] + 1) / 2;
  dim3 bs(32, 4, 2);
  dim3 gs((hx + 31) / 32, (L.geo.n[1] + 3) / 4, (L.geo.n[2] + 1) / 2);
  overlap_launch(k_gs_addp, gs, bs, 0, s, L, colour, p, store ? 1 : 0);
}

template <typename T>
void launch_gs_prolong(const MGLevel<T>& F, const MGLevel<T>& C, int colour, cudaStream_t s) {
  const int hx = (F.geo.n[0] + 1) / 2;
  dim3 bs(32, 4, 2);
  dim3 gs((hx + 31) / 32, (F.geo.n[1] + 3) / 4, (F.geo.n[2] + 1) / 2);
  overlap_launch(k_gs_prolong<T>, gs, bs, 0, s, F, C, colour);
}

template <typename T>
__global__ void k_beta_coarsen(MGLevel<T> F, MGLevel<T> C) {
  dependency_wait();
  long long cc = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (cc >= C.geo.N) return;
  int I, J, K;
  decode_lv(C.geo, cc, I, J, K);
  int base[3] = {I * F.f[0], J * F.f[1], K * F.f[2]};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    int cnt[3] = {F.f[0], F.f[1], F.f[2]};
    cnt[d] = 1;
    T acc = T(0);
    for (int dz = 0; dz < cnt[2]; ++dz)
      for (int dy = 0; dy < cnt[1]; ++dy)
        for (int dx = 0; dx < cnt[0]; ++dx)
          acc += F.beta[d][lin(F.geo, base[0] + dx, base[1] + dy, base[2] + dz)];
    C.beta[d][cc] = acc / (T)(cnt[0] * cnt[1] * cnt[2]);
  }
}

template <typename T>
void launch_beta_coarsen(const MGLevel<T>& F, const MGLevel<T>& C, cudaStream_t s) {
  overlap_launch(k_beta_coarsen<T>, grid1d(C.geo.N, 128), 128, 0, s, F, C);
}

// ---------------------------------------------------------------------------
// conjugate gradients on the coarsest level in one CTA: mean-free rhs,
// x0 = 0, stop at ||r|| <= rtol ||b|| or on breakdown, mean-free result.
// The vectors are double in both precisions.
template <typename T>
__device__ void coarse_cg_block(const MGLevel<T>& L, double* r,
                                double* dd, double* Ad, double rtol,
                                int maxit, double* sh) {
  const Geo& g = L.geo;
  const int N = (int)g.N;
  double acc = 0.0;
  for (int c = threadIdx.x; c < N; c += blockDim.x) acc += (double)L.b[c];
  double mean = block_sum_all(acc, sh) / (double)N;
  acc = 0.0;
  for (int c = threadIdx.x; c < N; c += blockDim.x) {
    double v = (double)L.b[c] - mean;
    r[c] = v;
    dd[c] = v;
    Ad[c] = 0.0;      // Ad doubles as the solution accumulator x until the end
    acc += v * v;
  }
  double rr = block_sum_all(acc, sh);
  double bn = sqrt(rr);
  double* x = Ad + N;
  for (int c = threadIdx.x; c < N; c += blockDim.x) x[c] = 0.0;
  if (bn != 0.0) {
    for (int it = 0; it < maxit; ++it) {
      if (sqrt(rr) <= rtol * bn) break;
      __syncthreads();
      acc = 0.0;
      for (int c = threadIdx.x; c < N; c += blockDim.x) {
        int i, j, k;
        decode_lv(g, c, i, j, k);
        OpNb<T> nb;
        neighbours(L, i, j, k, c, nb);
        double a = apply_L_at<T, double>(L, dd, c, nb);
        Ad[c] = a;
        acc += dd[c] * a;
      }
      double pAp = block_sum_all(acc, sh);
      if (!(pAp > 0.0)) break;   // breakdown (exhausted search direction or rounding)
      double a = rr / pAp;
      acc = 0.0;
      for (int c = threadIdx.x; c < N; c += blockDim.x) {
        x[c] = x[c] + a * dd[c];
        double rv = r[c] - a * Ad[c];
        r[c] = rv;
        acc += rv * rv;
      }
      double rr_new = block_sum_all(acc, sh);
      double beta = rr_new / rr;
      for (int c = threadIdx.x; c < N; c += blockDim.x) dd[c] = r[c] + beta * dd[c];
      rr = rr_new;
    }
  }
  __syncthreads();
  acc = 0.0;
  for (int c = threadIdx.x; c < N; c += blockDim.x) acc += x[c];
  double xm = block_sum_all(acc, sh) / (double)N;
  for (int c = threadIdx.x; c < N; c += blockDim.x) L.x[c] = (T)(x[c] - xm);
}

template <typename T>
__global__ void __launch_bounds__(1024) k_coarse_cg(MGLevel<T> L, double* r,
                                                    double* dd,
                                                    double* Ad, double rtol,
                                                    int maxit) {
  __shared__ double sh[33];
  coarse_cg_block(L, r, dd, Ad, rtol, maxit, sh);
}

template <typename T>
void launch_coarse_cg(const MGLevel<T>& L, double* r, double* d, double* Ad, double rtol,
                      int maxit, cudaStream_t s) {
  k_coarse_cg<T><<<1, 1024, 0, s>>>(L, r, d, Ad, rtol, maxit);
}

// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_residual_norm2(MGLevel<T> L, double* partial) {
  dependency_wait();
  __shared__ double sh[33];
  double acc = 0.0;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < L.geo.N;
       c += (long long)gridDim.x * blockDim.x) {
    int i, j, k;
    decode_lv(L.geo, c, i, j, k);
    OpNb<T> nb;
    neighbours(L, i, j, k, (int)c, nb);
    double r = (double)(L.b[c] - apply_L_at<T, T>(L, L.x, (int)c, nb));
    acc += r * r;
  }
  double s = block_sum_all(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

template <typename T>
void launch_residual_norm2(const MGLevel<T>& L, double* partial, double* out, cudaStream_t s) {
  overlap_launch(k_residual_norm2<T>, kRedBlocks, 256, 0, s, L, partial);
  launch_sum_partials(partial, kRedBlocks, out, s);
}

// float -> double for a finite beta >= 0 (normal or zero) with integer
// operations only: sign and mantissa move over, the exponent is rebiased
// (127 -> 1023).  GB300 issues FP64 work (conversions included) at a small
// fraction of the FP32 and integer rates, and this kernel is bound by it.
__device__ __forceinline__ double beta_to_double(float f) {
  const unsigned fb = __float_as_uint(f);
  const unsigned mag = fb & 0x7fffffffu;
  const unsigned hi = (fb & 0x80000000u) | (((mag >> 23) + 896u) << 20) | ((mag & 0x7fffffu) >> 3);
  const unsigned lo = fb << 29;
  return mag == 0u ? 0.0 : __hiloint2double((int)hi, (int)lo);
}

// With e32: the first Gauss-Seidel sweep of the next inner solve (colour 0
// from e = 0, the other colour 0) is taken here, from the float residual just
// stored, with the same arithmetic as k_gs_zero: the inner solve then starts
// at its second sweep.  w32: the finest level's float 1/h^2 per axis.
__global__ void k_residual64(Geo g, const double* p, const double* b,
                             const float* b0, const float* b1,
                             const float* b2, float* r32,
                             double* partial, float* e32, W3 w32,
                             double* rd, const int* gate) {
  dependency_wait();
  if (gate && !*gate) return;
  __shared__ double sh[33];
  const float* be[3] = {b0, b1, b2};
  const int st[3] = {1, g.n[0], g.n[0] * g.n[1]};
  const double wu = g.n[0] > 1 ? g.w[0] : (g.n[1] > 1 ? g.w[1] : g.w[2]);
  double acc = 0.0;
  for (long long cl = blockIdx.x * (long long)blockDim.x + threadIdx.x; cl < g.N;
       cl += (long long)gridDim.x * blockDim.x) {
    const int c = (int)cl;
    int i, j, k;
    decode_lv(g, c, i, j, k);
    const int idx[3] = {i, j, k};
    const double pc = p[c];
    float blo[3] = {0.f, 0.f, 0.f}, bhi[3] = {0.f, 0.f, 0.f};
    // the fine level has cubic cells: one weight 1/h^2 for every coupled axis
    double lsum = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int n = g.n[d];
      if (n == 1) continue;
      const int clo = idx[d] == 0 ? c + (n - 1) * st[d] : c - st[d];
      const int chi = idx[d] == n - 1 ? c - (n - 1) * st[d] : c + st[d];
      blo[d] = be[d][c];
      bhi[d] = (g.bc[d] == WALL && idx[d] == n - 1) ? 0.f : be[d][chi];
      lsum = fma(beta_to_double(blo[d]), pc - p[clo], lsum);
      lsum = fma(beta_to_double(bhi[d]), pc - p[chi], lsum);
    }
    const double r = fma(-wu, lsum, b[c]);
    const float rf = narrow<float>(r);
    r32[c] = rf;
    if (rd) rd[c] = r;
    if (e32) {
      const float z[3] = {0.f, 0.f, 0.f};
      e32[c] = ((i + j + k) & 1) == 0 ? gs_formula(g, w32.w, w32.w[0] != 0.f ? w32.w[0] : (w32.w[1] != 0.f ? w32.w[1] : w32.w[2]), rf,
                                                       blo, bhi, z, z)
                                          : 0.f;
    }
    acc += r * r;
  }
  double s = block_sum_all(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

void launch_residual64(const Geo& g, const double* p, const double* b, float* const* beta,
                       float* r32, double* partial, double* out, cudaStream_t s, float* e32,
                       const float* w32, double* rd, const int* gate) {
  W3 w = {{0.f, 0.f, 0.f}};
  if (w32)
    for (int d = 0; d < 3; ++d) w.w[d] = w32[d];
  overlap_launch(k_residual64, kRedBlocks, 256, 0, s, g, p, b, beta[0], beta[1], beta[2], r32, partial, e32, w,
                                          rd, gate);
  launch_sum_partials(partial, kRedBlocks, out, s, gate);
}

// ---------------------------------------------------------------------------
// The residual of the next refinement from the one before: after p += e,
// r -= L e.  The correction e and beta are float, so the differences of e
// and their products with beta are formed exactly as pairs of floats (Knuth's
// two-sum, the fused product error) and summed as such: 48 bits in float
// arithmetic, which the GPU does 64 times as fast as double.  Formed from p
// (k_residual64, 14 FP64 operations a cell) the pass is bound by the FP64
// pipe: 0.56 ms at 256^3 against 0.19 ms here.  Its error, 2^-48 beta |de| of a
// face, is that of rounding p itself (2^-53 beta |p|) once e varies over 32
// cells and more, and it does not grow: the solve forms the residual from p
// again before it stops, and goes on from that one if it is above the
// tolerance.  The rule (fvm_api.cu) takes this pass from 2^19 cells; below,
// the two launches more of a refinement cost what it saves.
struct FloatPair {
  float h, l;
};

__device__ __forceinline__ FloatPair face_product(float beta, float a, float b) {
  const float s = __fsub_rn(a, b);
  const float t = __fsub_rn(s, a);
  const float err = __fsub_rn(__fsub_rn(a, __fsub_rn(s, t)), __fadd_rn(b, t));
  FloatPair p;
  p.h = __fmul_rn(beta, s);
  p.l = __fmaf_rn(beta, err, __fmaf_rn(beta, s, -p.h));
  return p;
}

__device__ __forceinline__ void pair_add(FloatPair& s, float h, float l) {
  const float t = __fadd_rn(s.h, h);
  const float z = __fsub_rn(t, s.h);
  const float e = __fadd_rn(__fsub_rn(s.h, __fsub_rn(t, z)), __fsub_rn(h, z));
  s.h = t;
  s.l = __fadd_rn(s.l, __fadd_rn(e, l));
}

// A thread owns a column of cells and walks planes k0 .. k1-1 upward; the
// product of a z-face serves the cells on both of its sides.
__global__ void __launch_bounds__(256, 6)
    k_residual_update(MGLevel<float> L, double* rd, float* y,
                      double* partial, int tx, int ty, int chunks, int kz) {
  dependency_wait();
  __shared__ double sh[33];
  const Geo& g = L.geo;
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2], nxy = nx * ny;
  const float* e = L.x;
  const float *b0 = L.beta[0], *b1 = L.beta[1],
              *b2 = L.beta[2];
  const double w = (double)g.w[nx > 1 ? 0 : (ny > 1 ? 1 : 2)];
  double acc = 0.0;
  for (int t = blockIdx.x; t < tx * ty * chunks; t += gridDim.x) {
    const int q = t / tx, i = (t - q * tx) * 32 + (threadIdx.x & 31);
    const int ch = q / ty, j = (q - ch * ty) * 8 + (threadIdx.x >> 5);
    if (i >= nx || j >= ny) continue;
    const int k0 = ch * kz, k1 = min(k0 + kz, nz);
    const int col = j * nx + i;
    const int xm = i == 0 ? nx - 1 : -1, xp = i == nx - 1 ? 1 - nx : 1;
    const int ym = j == 0 ? (ny - 1) * nx : -nx, yp = j == ny - 1 ? (1 - ny) * nx : nx;
    const bool wx = i == nx - 1 && g.bc[0] == WALL, wy = j == ny - 1 && g.bc[1] == WALL;
    int c = k0 * nxy + col;
    float ec = e[c];
    float bz = b2[c];
    FloatPair zl = face_product(bz, ec, e[k0 == 0 ? (nz - 1) * nxy + col : c - nxy]);
    for (int k = k0; k < k1; ++k) {
      const int cn = k == nz - 1 ? col : c + nxy;
      const float en = e[cn], bzl = bz;
      bz = (k == nz - 1 && g.bc[2] == WALL) ? 0.f : b2[cn];
      const float xl = b0[c], xh = wx ? 0.f : b0[c + xp];
      const float yl = b1[c], yh = wy ? 0.f : b1[c + yp];
      FloatPair s = face_product(xl, ec, e[c + xm]);
      FloatPair f = face_product(xh, ec, e[c + xp]);
      pair_add(s, f.h, f.l);
      f = face_product(yl, ec, e[c + ym]);
      pair_add(s, f.h, f.l);
      f = face_product(yh, ec, e[c + yp]);
      pair_add(s, f.h, f.l);
      pair_add(s, zl.h, zl.l);
      f = face_product(bz, ec, en);
      pair_add(s, f.h, f.l);
      zl.h = -f.h;
      zl.l = -f.l;
      const double r = fma(-w, widen(s.l), fma(-w, widen(s.h), rd[c]));
      rd[c] = r;
      const float rf = (float)r;
      L.b[c] = rf;
      if (y) {
        // the next inner solve's first sweep: colour 0 from 0
        const float lo[3] = {xl, yl, bzl}, hi[3] = {xh, yh, bz}, z[3] = {0.f, 0.f, 0.f};
        y[c] = ((i + j + k) & 1) == 0 ? gs_formula(g, L.w, L.wu, rf, lo, hi, z, z) : 0.f;
      }
      acc = fma(r, r, acc);
      ec = en;
      c = cn;
    }
  }
  const double s = block_sum_all(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

void launch_residual_update(const MGLevel<float>& L, double* rd, float* y, double* partial,
                            double* out, cudaStream_t s) {
  const ColumnRuns r = column_runs(L.geo);
  overlap_launch(k_residual_update, r.blocks, 256, 0, s, L, rd, y, partial, r.tx, r.ty, r.chunks,
                 r.kz);
  launch_sum_partials(partial, r.blocks, out, s);
}

__global__ void k_add_correction(long long n, double* p, const float* e) {
  dependency_wait();
  long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c < n) p[c] = p[c] + (double)e[c];
}

void launch_add_correction(long long n, double* p, const float* e, cudaStream_t s) {
  overlap_launch(k_add_correction, grid1d(n, 256), 256, 0, s, n, p, e);
}

// ---------------------------------------------------------------------------
// device-side control of the pressure solve (one thread each)
__global__ void k_ctl_reset(SolveCtl* ctl) {
  dependency_wait();
  ctl->iters = 0;
  ctl->status = 0;
  ctl->zero = 0;
  ctl->verify = 0;
  ctl->rel = 0.0;
}

void launch_ctl_reset(SolveCtl* ctl, cudaStream_t s) { overlap_launch(k_ctl_reset, 1, 1, 0, s, ctl); }

// the stopping rule of the host loop, on the device: stop on a non-finite
// norm (EUNSTABLE), a zero right-hand side, after `fixed` cycles, at
// rel <= rtol, or at maxit cycles above rtol (ENOCONV)
__global__ void k_ctl_step(cudaGraphConditionalHandle h, SolveCtl* ctl, const double* bn2p,
                           const double* r2p, double rtol, int maxit, int fixed,
                           unsigned long long* runs_total) {
  dependency_wait();
  const double bn2 = *bn2p;
  unsigned go = 0;
  if (!isfinite(bn2)) {
    ctl->status = FVM_EUNSTABLE;
  } else if (bn2 == 0.0) {
    ctl->zero = 1;
    ctl->rel = 0.0;
  } else {
    const double rel = sqrt(*r2p) / sqrt(bn2);
    ctl->rel = rel;
    if (!isfinite(rel)) {
      ctl->status = FVM_EUNSTABLE;
    } else if (fixed > 0) {
      go = ctl->iters < fixed;
    } else {
      go = rel > rtol && ctl->iters < maxit;
      if (!go && rel > rtol) ctl->status = FVM_ENOCONV;
    }
  }
  if (go) {
    ctl->iters += 1;
    *runs_total += 1ull;
  }
  cudaGraphSetConditional(h, go);
}

void launch_ctl_step(cudaGraphConditionalHandle h, SolveCtl* ctl, const double* bn2,
                     const double* r2, double rtol, int maxit, int fixed,
                     unsigned long long* runs_total, cudaStream_t s) {
  overlap_launch(k_ctl_step, 1, 1, 0, s, h, ctl, bn2, r2, rtol, maxit, fixed, runs_total);
}

__global__ void k_ctl_check(SolveCtl* ctl, const double* bn2p, const double* r2p, double rtol,
                            int maxit, int fixed) {
  dependency_wait();
  const double rel = sqrt(*r2p) / sqrt(*bn2p);
  const bool go = isfinite(rel) && (fixed > 0 ? ctl->iters < fixed
                                              : (rel > rtol && ctl->iters < maxit));
  ctl->verify = go ? 0 : 1;
}

void launch_ctl_check(SolveCtl* ctl, const double* bn2, const double* r2, double rtol, int maxit,
                      int fixed, cudaStream_t s) {
  overlap_launch(k_ctl_check, 1, 1, 0, s, ctl, bn2, r2, rtol, maxit, fixed);
}

__global__ void k_zero_if_rhs_zero(const SolveCtl* ctl, double* p,
                                   long long n) {
  dependency_wait();
  if (!ctl->zero) return;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n;
       c += (long long)gridDim.x * blockDim.x)
    p[c] = 0.0;
}

void launch_zero_if_rhs_zero(const SolveCtl* ctl, double* p, long long n, cudaStream_t s) {
  overlap_launch(k_zero_if_rhs_zero, kRedBlocks, 256, 0, s, ctl, p, n);
}

__global__ void k_ctl_store(const SolveCtl* ctl, SolveCtl* rec, int* sticky) {
  dependency_wait();
  *rec = *ctl;
  if (ctl->status) atomicMax(sticky, ctl->status);
}

void launch_ctl_store(const SolveCtl* ctl, SolveCtl* rec, int* sticky, cudaStream_t s) {
  overlap_launch(k_ctl_store, 1, 1, 0, s, ctl, rec, sticky);
}

#define FVM_MG_INST(T)                                                                       \
  template void launch_sum_field<T>(const T*, long long, bool, double*, double*,             \
                                    cudaStream_t);                                           \
  template void launch_zero<T>(T*, long long, cudaStream_t);                                 \
  template void launch_gs<T>(const MGLevel<T>&, int, cudaStream_t, const int*, int, const T*); \
  template void launch_residual_restrict<T>(const MGLevel<T>&, const MGLevel<T>&, cudaStream_t, bool, \
                                            bool);                                           \
  template void launch_inv_diag<T>(const MGLevel<T>&, cudaStream_t);                         \
  template void launch_prolong<T>(const MGLevel<T>&, const MGLevel<T>&, cudaStream_t);       \
  template void launch_gs_prolong<T>(const MGLevel<T>&, const MGLevel<T>&, int, cudaStream_t); \
  template void launch_gs_zero<T>(const MGLevel<T>&, int, cudaStream_t);                      \
  template void launch_beta_coarsen<T>(const MGLevel<T>&, const MGLevel<T>&, cudaStream_t);  \
  template void launch_coarse_cg<T>(const MGLevel<T>&, double*, double*, double*, double,  \
                                    int, cudaStream_t);                                      \
  template void launch_residual_norm2<T>(const MGLevel<T>&, double*, double*, cudaStream_t);

FVM_MG_INST(double)
FVM_MG_INST(float)

}  // namespace fvm
