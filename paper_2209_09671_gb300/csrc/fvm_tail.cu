// The coarse levels of a V-cycle in one launch of one thread-block cluster.
//
// A coarse level is too small to fill the GPU: a colour sweep of 32^3 cells
// takes 2.6 us as a launch of its own (almost all of it launch and drain), and
// a V-cycle makes a dozen of them per level.  On one CTA the same levels
// are bound by that SM instead.  Here kTailCTAs CTAs of one cluster keep every
// level of the tail in their shared memory, each a run of rows of it; a sweep
// reads the rows of other CTAs through distributed shared memory and ends
// with a cluster barrier (475 clocks; a remote load is 240).  Levels small
// enough for one CTA run on CTA 0 between block barriers (44 clocks) while the
// others wait.
//
// Per cell a level holds x, b, the six face coefficients beta / h_d^2 and the
// reciprocal of their sum (7 numbers prepared once per solve by k_tail_pack,
// so that a sweep divides nothing), the coarsest level its coefficients and
// conjugate-gradient vectors in double.  A row is stored with its even
// columns first, then the odd ones: the cells of one colour are consecutive
// and their loads free of bank conflicts.
//
// Measured per V-cycle against the levels of at most 4096 cells on one CTA and
// the larger ones as launches: 256^3 float (32^3 cells and below) 51 against
// 134 + 45 us, 128^3 double 105 against 344 + 60 us, the 64^2 double drop 53
// against 156 us; bound by the barriers and the latencies between them.
#include "fvm_device.cuh"

namespace fvm {

namespace {

constexpr int kTailThreads = 512;

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
// address of the same shared-memory location in CTA `rank` of the cluster
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void ld_cl(unsigned a, float& v) {
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a));
}
__device__ __forceinline__ void ld_cl(unsigned a, double& v) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a));
}
__device__ __forceinline__ void st_cl(unsigned a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// what a CTA knows of one level
template <typename T>
struct View {
  const TailLevel<T>& L;
  char* sm;
  int rank, nrows;      // rows of this CTA
  __device__ View(const TailLevel<T>& l, char* s, int r) : L(l), sm(s), rank(r) {
    const int r0 = r * l.rpc;
    nrows = r0 >= l.rows ? 0 : (l.rows - r0 < l.rpc ? l.rows - r0 : l.rpc);
  }
  __device__ T* x() const { return reinterpret_cast<T*>(sm + L.ox); }
  __device__ T* b() const { return reinterpret_cast<T*>(sm + L.ob); }
  template <typename C>
  __device__ C* a() const { return reinterpret_cast<C*>(sm + L.oa); }
  __device__ int4* tab() const { return reinterpret_cast<int4*>(sm + L.otab); }
};

// quotient t / d for 0 <= t < 2^20 (id = 1 / d)
__device__ __forceinline__ int quot(int t, float id) { return (int)(((float)t + 0.5f) * id); }

// position of column i in a stored row: even columns, then odd ones
__device__ __forceinline__ int row_pos(int i, int hx) { return (i & 1) * hx + (i >> 1); }

// shared-cluster address of row R of an array at byte offset `off` (elements
// of `esize` bytes)
template <typename T>
__device__ __forceinline__ unsigned row_addr(const TailLevel<T>& L, unsigned base, int off, int R,
                                             int esize) {
  const int rk = quot(R, 1.0f / (float)L.rpc);
  return map_rank(base + off + (R - rk * L.rpc) * L.pitch * esize, rk);
}

// the six coefficients of cell (i, row R) and the reciprocal of their sum
template <typename T, typename C>
__device__ __forceinline__ C cell_coefs(const TailLevel<T>& L, int i, int R, C* a) {
  const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
  const int k = quot(R, 1.0f / (float)ny), j = R - k * ny;
  const int c = R * nx + i;
  const int idx[3] = {i, j, k}, st[3] = {1, nx, nx * ny};
  C den = C(0);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    a[2 * d] = a[2 * d + 1] = C(0);
    const int n = L.n[d];
    if (n == 1) continue;
    const bool last = idx[d] == n - 1;
    const int hi = last ? c - (n - 1) * st[d] : c + st[d];
    a[2 * d] = (C)L.beta[d][c] * (C)L.w[d];
    a[2 * d + 1] = (last && L.wall[d]) ? C(0) : (C)L.beta[d][hi] * (C)L.w[d];
    den += a[2 * d] + a[2 * d + 1];
  }
  return C(1) / den;
}

// fill the coefficient block of CTA `rank` (layout of shared memory and of
// the packed copy in global memory)
template <typename T>
__device__ void fill_coefs(const TailLevel<T>& L, bool coarsest, void* dst, int rank, int tid,
                           int nthr) {
  const int r0 = rank * L.rpc;
  const int nrows = max(0, min(L.rpc, L.rows - r0));
  for (int t = tid; t < nrows * L.pitch; t += nthr) {
    const int q = quot(t, 1.0f / (float)L.pitch), pos = t - q * L.pitch;
    const int i = pos < L.hx ? 2 * pos : 2 * (pos - L.hx) + 1;
    if (i >= L.n[0]) continue;
    if (coarsest) {
      double a[6];
      cell_coefs<T, double>(L, i, r0 + q, a);
      for (int m = 0; m < 6; ++m) ((double*)dst)[m * L.cap + t] = a[m];
    } else {
      T a[6];
      const T inv = cell_coefs<T, T>(L, i, r0 + q, a);
      for (int m = 0; m < 6; ++m) ((T*)dst)[m * L.cap + t] = a[m];
      ((T*)dst)[6 * L.cap + t] = inv;
    }
  }
}

// G = (L + s 1 1^T / N)^-1 on a coarsest level of N <= 32 cells, s the mean
// diagonal: Gauss-Jordan without pivoting (the matrix is symmetric and positive
// definite: L has the constants as its only null vectors), by one block
template <typename T>
__device__ void coarsest_inverse(const TailLevel<T>& L, double* G) {
  __shared__ double M[32][33];
  __shared__ double diag[32];
  const int N = L.rows * L.n[0], nx = L.n[0], ny = L.n[1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int r = w; r < N; r += nw)
    if (lane < N) M[r][lane] = 0.0;
  __syncthreads();
  if (w == 0 && lane < N) {
    const int R = lane / nx, i = lane - R * nx, k = R / ny, j = R - k * ny;
    double a[6], dg = 0.0;
    cell_coefs<T, double>(L, i, R, a);
    const int idx[3] = {i, j, k}, st[3] = {1, nx, nx * ny};
    for (int d = 0; d < 3; ++d) {
      const int n = L.n[d];
      if (n == 1) continue;
      const int lo = idx[d] == 0 ? lane + (n - 1) * st[d] : lane - st[d];
      const int hi = idx[d] == n - 1 ? lane - (n - 1) * st[d] : lane + st[d];
      M[lane][lo] -= a[2 * d];
      M[lane][hi] -= a[2 * d + 1];
      dg += a[2 * d] + a[2 * d + 1];
    }
    M[lane][lane] += dg;
    diag[lane] = dg;
  }
  __syncthreads();
  double s = 0.0;
  for (int q = 0; q < N; ++q) s += diag[q];
  s /= (double)N * (double)N;
  for (int r = w; r < N; r += nw)
    if (lane < N) M[r][lane] += s;
  __syncthreads();
  for (int p = 0; p < N; ++p) {
    const double ip = 1.0 / M[p][p];
    const double mp = lane < N ? M[p][lane] : 0.0;
    const double rp = lane == p ? ip : mp * ip;      // the scaled pivot row
    double f[4], v[4];
    for (int q = 0; q < 4; ++q) {
      const int r = w + q * nw;
      if (r < N && lane < N) {
        f[q] = M[r][p];
        v[q] = M[r][lane];
      }
    }
    __syncthreads();
    for (int q = 0; q < 4; ++q) {
      const int r = w + q * nw;
      if (r < N && lane < N) {
        if (r == p) M[r][lane] = rp;
        else M[r][lane] = lane == p ? -f[q] * ip : fma(-f[q], rp, v[q]);
      }
    }
    __syncthreads();
  }
  for (int r = w; r < N; r += nw)
    if (lane < N) G[r * N + lane] = M[r][lane];
}

// one Gauss-Seidel sweep of a colour over the CTA's rows
template <typename T>
__device__ __forceinline__ void sweep(const View<T>& V, int col) {
  const TailLevel<T>& L = V.L;
  T* x = V.x();
  const T* b = V.b();
  const T* a = V.template a<T>();
  const int hx = L.hx, nx = L.n[0], cap = L.cap;
  const float ihx = 1.0f / (float)hx;
  for (int t = threadIdx.x; t < V.nrows * hx; t += kTailThreads) {
    const int q = quot(t, ihx), i2 = t - q * hx;
    const int4 ra = V.tab()[2 * q];
    const int s = (col + V.tab()[2 * q + 1].y) & 1;
    const int i = 2 * i2 + s;
    if (i >= nx) continue;
    const int row = q * L.pitch, p = s * hx + i2, c = row + p;
    T ym, yp, zm, zp;
    const unsigned o = p * (unsigned)sizeof(T);
    ld_cl(ra.x + o, ym);
    ld_cl(ra.y + o, yp);
    ld_cl(ra.z + o, zm);
    ld_cl(ra.w + o, zp);
    const T xm = x[row + row_pos(i == 0 ? nx - 1 : i - 1, hx)];
    const T xp = x[row + row_pos(i == nx - 1 ? 0 : i + 1, hx)];
    T num = b[c];
    num += a[c] * xm + a[cap + c] * xp;
    num += a[2 * cap + c] * ym + a[3 * cap + c] * yp;
    num += a[4 * cap + c] * zm + a[5 * cap + c] * zp;
    x[c] = num * a[6 * cap + c];
  }
}

// r = b - L x over the CTA's rows; 0 at the cells of colour 1 when the last
// sweep was theirs (in double: see restrict_point)
template <typename T>
__device__ __forceinline__ void residual(const View<T>& V, T* r, bool half) {
  const TailLevel<T>& L = V.L;
  const T* x = V.x();
  const T* b = V.b();
  const T* a = V.template a<T>();
  const int hx = L.hx, nx = L.n[0], cap = L.cap;
  const float ip = 1.0f / (float)L.pitch;
  for (int t = threadIdx.x; t < V.nrows * L.pitch; t += kTailThreads) {
    const int q = quot(t, ip), p = t - q * L.pitch;
    const int i = p < hx ? 2 * p : 2 * (p - hx) + 1;
    if (i >= nx) continue;
    if (half && ((i + V.tab()[2 * q + 1].y) & 1)) {
      r[t] = T(0);
      continue;
    }
    const int4 ra = V.tab()[2 * q];
    const int row = q * L.pitch;
    T ym, yp, zm, zp;
    const unsigned o = p * (unsigned)sizeof(T);
    ld_cl(ra.x + o, ym);
    ld_cl(ra.y + o, yp);
    ld_cl(ra.z + o, zm);
    ld_cl(ra.w + o, zp);
    const T xc = x[t];
    const T xm = x[row + row_pos(i == 0 ? nx - 1 : i - 1, hx)];
    const T xp = x[row + row_pos(i == nx - 1 ? 0 : i + 1, hx)];
    T out = a[t] * (xc - xm) + a[cap + t] * (xc - xp);
    out += a[2 * cap + t] * (xc - ym) + a[3 * cap + t] * (xc - yp);
    out += a[4 * cap + t] * (xc - zm) + a[5 * cap + t] * (xc - zp);
    r[t] = b[t] - out;
  }
}

// x from a start of 0 with the first colour-0 sweep taken (it needs only b)
template <typename T>
__device__ __forceinline__ T first_x(const View<T>& V, int c, int i, int parity, T b, bool sweep0) {
  return sweep0 && ((i + parity) & 1) == 0 ? b * V.template a<T>()[6 * V.L.cap + c] : T(0);
}

// b of the coarse level = mean over the children of the fine residual
template <typename T>
__device__ __forceinline__ void restrict_rows(const View<T>& F, const View<T>& C, unsigned base,
                                              int oscr, bool coarsest, bool sweep0) {
  const TailLevel<T>& L = C.L;
  const int fx = F.L.f[0], fy = F.L.f[1], fz = F.L.f[2];
  const T scale = T(1) / (T)(fx * fy * fz);   // a power of two
  const float ip = 1.0f / (float)L.pitch, iny = 1.0f / (float)L.n[1];
  for (int t = threadIdx.x; t < C.nrows * L.pitch; t += kTailThreads) {
    const int q = quot(t, ip), p = t - q * L.pitch;
    const int I = p < L.hx ? 2 * p : 2 * (p - L.hx) + 1;
    if (I >= L.n[0]) continue;
    const int R = C.rank * L.rpc + q;
    const int K = quot(R, iny), J = R - K * L.n[1];
    T acc = T(0);
    for (int dz = 0; dz < fz; ++dz)
      for (int dy = 0; dy < fy; ++dy) {
        const unsigned ra = row_addr(F.L, base, oscr, (K * fz + dz) * F.L.n[1] + J * fy + dy,
                                     (int)sizeof(T));
        for (int dx = 0; dx < fx; ++dx) {
          T v;
          ld_cl(ra + row_pos(I * fx + dx, F.L.hx) * (unsigned)sizeof(T), v);
          acc += v;
        }
      }
    const T b = acc * scale;
    C.b()[t] = b;
    if (!coarsest) C.x()[t] = first_x(C, t, I, J + K, b, sweep0);
  }
}

// x += the coarse correction of the parent cell
template <typename T>
__device__ __forceinline__ void prolong_rows(const View<T>& F, const TailLevel<T>& C) {
  const TailLevel<T>& L = F.L;
  const int hx = L.hx;
  const float ip = 1.0f / (float)L.pitch;
  for (int t = threadIdx.x; t < F.nrows * L.pitch; t += kTailThreads) {
    const int q = quot(t, ip), p = t - q * L.pitch;
    const int i = p < hx ? 2 * p : 2 * (p - hx) + 1;
    if (i >= L.n[0]) continue;
    const unsigned pa = (unsigned)F.tab()[2 * q + 1].x;
    T v;
    ld_cl(pa + row_pos(L.f[0] == 2 ? i >> 1 : i, C.hx) * (unsigned)sizeof(T), v);
    F.x()[t] += v;
  }
}

// the sums of s and of t over the warp, in every lane (two chains at once: an
// FP64 addition takes 63 clocks from issue to result)
__device__ __forceinline__ void warp_sum2(double& s, double& t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    t += __shfl_xor_sync(0xffffffffu, t, o);
  }
}

// Sums over the cells of a level spread over `nact` CTAs (CTA 0 alone when nact
// is 1, else the whole cluster takes part), in a fixed order.  The first warp
// adds the threads' values from shared memory and works out the scalars of
// the iteration: the FP64 pipe of an SM does 2 lanes a clock, so shuffling,
// dividing or taking roots in every warp keeps it busy for thousands of clocks
// (25 x 25 cells: 1160 instead of 870 us per V-cycle).
struct Reduce {
  double* vals;     // 2 x kTailThreads
  double* slots;    // 2 sets of 2 x kTailCTAs, written by the other CTAs
  double* out;      // the scalar handed to every thread, and three for its user
  unsigned base_slots;
  int nact, rank, used;   // used: threads of this CTA with a value
  int phase;
  // the sums of v and u over all cells go through `f` in warp 0 (the same
  // numbers in every CTA); every thread gets f's value
  template <typename F>
  __device__ __forceinline__ double run2(double v, double u, F f) {
    const int tid = threadIdx.x;
    if (tid < used) {
      vals[tid] = v;
      vals[kTailThreads + tid] = u;
    }
    __syncthreads();
    double s = 0.0, t = 0.0;
    if (tid < 32) {
      for (int q = tid; q < used; q += 32) {
        s += vals[q];
        t += vals[kTailThreads + q];
      }
      warp_sum2(s, t);
    }
    if (nact > 1) {
      const int set = (phase++ & 1) * 2 * kTailCTAs;
      if (tid < kTailCTAs) {
        const unsigned to = map_rank(base_slots + (set + rank) * 8, tid);
        st_cl(to, s);
        st_cl(to + kTailCTAs * 8, t);
      }
      cluster_sync();
      if (tid < 32) {
        s = tid < nact ? slots[set + tid] : 0.0;
        t = tid < nact ? slots[set + kTailCTAs + tid] : 0.0;
        warp_sum2(s, t);
      }
    }
    if (tid < 32) {
      s = f(s, t);
      if (tid == 0) *out = s;
    }
    __syncthreads();
    return *out;   // (rewritten only after the next call's first barrier)
  }
  template <typename F>
  __device__ __forceinline__ double run(double v, F f) {
    return run2(v, 0.0, [&](double s, double) { return f(s); });
  }
};

// conjugate gradients on the coarsest level: mean-free right-hand side,
// x0 = 0, stop at ||r|| <= rtol ||b|| or on breakdown, mean-free result; the
// vectors are double in both precisions
template <typename T>
__device__ void coarsest_cg(const View<T>& V, const TailArgs<T>& A, Reduce& red) {
  const TailLevel<T>& L = V.L;
  const int cap = L.cap, hx = L.hx, nx = L.n[0];
  const double* a = V.template a<double>();
  double* d = reinterpret_cast<double*>(V.sm + A.ocg);
  double *r = d + cap, *x = r + cap, *Ad = x + cap;
  const int nc = V.nrows * L.pitch;
  const float ip = 1.0f / (float)L.pitch;
  const double N = (double)L.rows * nx;
  // columns beyond nx in a padded row hold 0 in every vector
  auto column = [&](int t) {
    const int q = quot(t, ip), p = t - q * L.pitch;
    return p < hx ? 2 * p : 2 * (p - hx) + 1;
  };
  double acc = 0.0;
  for (int t = threadIdx.x; t < nc; t += kTailThreads)
    if (column(t) < nx) acc += (double)V.b()[t];
  const double mean = red.run(acc, [&](double s) { return s / N; });
  acc = 0.0;
  for (int t = threadIdx.x; t < nc; t += kTailThreads) {
    const double v = column(t) < nx ? (double)V.b()[t] - mean : 0.0;
    r[t] = d[t] = v;
    x[t] = 0.0;
    acc += v * v;
  }
  // rr and the stopping threshold live in warp 0; (the barrier also publishes d)
  double rr = 0.0, stop = 0.0;   // ||r||^2 and its threshold
  double go = red.run(acc, [&](double s) {
    rr = s;
    stop = A.rtol * A.rtol * s;
    return s != 0.0 && !(s <= stop) ? 1.0 : 0.0;
  });
  for (int it = 0; it < A.maxit && go != 0.0; ++it) {
    acc = 0.0;
    for (int t = threadIdx.x; t < nc; t += kTailThreads) {
      const int q = quot(t, ip), p = t - q * L.pitch;
      const int i = p < hx ? 2 * p : 2 * (p - hx) + 1;
      if (i >= nx) continue;
      const int4 ra = V.tab()[2 * q];
      const int row = q * L.pitch;
      const unsigned o = p * 8u;
      const double dc = d[t];
      double v0, v1, v2, v3;
      ld_cl(ra.x + o, v0);
      ld_cl(ra.y + o, v1);
      ld_cl(ra.z + o, v2);
      ld_cl(ra.w + o, v3);
      // an axis of one cell has coefficients 0; three short chains, as an FP64
      // operation takes 63 clocks from issue to result
      double ox = a[t] * (dc - d[row + row_pos(i == 0 ? nx - 1 : i - 1, hx)]);
      double oy = a[2 * cap + t] * (dc - v0);
      double oz = 0.0;
      ox = fma(a[cap + t], dc - d[row + row_pos(i == nx - 1 ? 0 : i + 1, hx)], ox);
      oy = fma(a[3 * cap + t], dc - v1, oy);
      if (L.n[2] > 1) {
        oz = a[4 * cap + t] * (dc - v2);
        oz = fma(a[5 * cap + t], dc - v3, oz);
      }
      const double out = (ox + oy) + oz;
      Ad[t] = out;
      acc = fma(dc, out, acc);
    }
    // step length; 0 on breakdown (exhausted direction or rounding)
    const double al = red.run(acc, [&](double s) { return s > 0.0 ? rr / s : 0.0; });
    if (al == 0.0) break;
    acc = 0.0;
    for (int t = threadIdx.x; t < nc; t += kTailThreads) {
      if (column(t) >= nx) continue;
      x[t] = fma(al, d[t], x[t]);
      const double v = fma(-al, Ad[t], r[t]);
      r[t] = v;
      acc = fma(v, v, acc);
    }
    // direction update, negative when ||r|| has reached the threshold
    const double beta = red.run(acc, [&](double s) {
      const double q = s / rr;
      rr = s;
      return s <= stop ? -1.0 : q;
    });
    if (beta < 0.0) break;
    for (int t = threadIdx.x; t < nc; t += kTailThreads) d[t] = fma(beta, d[t], r[t]);
    if (red.nact > 1) cluster_sync();
    else __syncthreads();
  }
  acc = 0.0;
  for (int t = threadIdx.x; t < nc; t += kTailThreads) acc += x[t];
  const double xm = red.run(acc, [&](double s) { return s / N; });
  for (int t = threadIdx.x; t < nc; t += kTailThreads) V.x()[t] = (T)(x[t] - xm);
}

// The coarsest level by defect correction: dx = G r with the float inverse G
// of the level's operator (launch_tail_inverse, once per solve), r -= L dx in
// double, until ||r|| <= rtol ||b||: each step gains what the float inverse
// resolves (four to six digits), where conjugate gradients take 50 to 170
// iterations of two dependent sums each (5 us an iteration).  The whole tail
// per V-cycle: 25 x 25 coarsest cells 870 -> 65 us (to 1e-12), 11 x 18 x 5
// 364 -> 88 us (to 1e-6).  The result
// meets the same double residual; its mean is left as it comes (a constant
// is no correction).  Returns false when a step gains less than a factor
// of two (an operator too ill-conditioned for float, or not a number): the
// caller then runs conjugate gradients.
template <typename T>
__device__ bool coarsest_refine(const View<T>& V, const TailArgs<T>& A, Reduce& red) {
  const TailLevel<T>& L = V.L;
  const int cap = L.cap, hx = L.hx, nx = L.n[0], np = A.np;
  const double* a = V.template a<double>();
  double* d = reinterpret_cast<double*>(V.sm + A.ocg);
  double *r = d + cap, *x = r + cap;
  float* mine = reinterpret_cast<float*>(V.sm + A.ovec);   // own part of the scaled residual
  float* full = mine + (L.rpc * nx + 3) / 4 * 4;           // all of it
  const unsigned mine_a = smem_u32(mine);
  const int nc = V.nrows * L.pitch, own = V.nrows * nx, chunk = L.rpc * nx;
  const int ncell = L.rows * nx;
  const float ip = 1.0f / (float)L.pitch, ic = 1.0f / (float)chunk;
  const double N = (double)ncell;
  auto column = [&](int t) {
    const int q = quot(t, ip), p = t - q * L.pitch;
    return p < hx ? 2 * p : 2 * (p - hx) + 1;
  };
  double acc = 0.0, sq = 0.0;
  for (int t = threadIdx.x; t < nc; t += kTailThreads) {
    const double v = column(t) < nx ? (double)V.b()[t] : 0.0;
    acc += v;
    sq = fma(v, v, sq);
  }
  double rr = 0.0, stop = 0.0;   // ||r||^2 and its threshold, in warp 0
  // (the mean of a restricted residual is small beside its size, so that its
  // square is subtracted from the sum without cancellation)
  double mean = 0.0;
  double* bmean = red.out + 1;
  double sc = red.run2(acc, sq, [&](double s, double t) {
    mean = s / N;
    if (threadIdx.x == 0) *bmean = mean;
    rr = t - s * mean;
    stop = A.rtol * A.rtol * rr;
    return rr > stop ? 1.0 : 0.0;
  });
  mean = *bmean;
  for (int t = threadIdx.x; t < nc; t += kTailThreads) {
    r[t] = column(t) < nx ? (double)V.b()[t] - mean : 0.0;
    x[t] = 0.0;
  }
  bool ok = true;
  while (sc != 0.0) {
    // scale so that the residual's norm is of order one in float: half its
    // exponent, a power of two
    if (threadIdx.x == 0) {
      const int e = (int)((__double2hiint(rr) >> 20) & 0x7ff) - 1023;
      bmean[1] = __hiloint2double((1023 - (e >> 1)) << 20, 0);
      bmean[2] = 1.0 / (bmean[1] * (*A.gscale));
    }
    __syncthreads();
    const double scale = bmean[1], back = bmean[2];
    for (int t = threadIdx.x; t < nc; t += kTailThreads) {
      const int q = quot(t, ip), i = column(t);
      if (i < nx) mine[q * nx + i] = (float)(r[t] * scale);
    }
    if (red.nact > 1) cluster_sync();
    else __syncthreads();
    for (int c = threadIdx.x; c < np; c += kTailThreads) {
      float v = 0.f;
      if (c < ncell) {
        const int rk = quot(c, ic);
        ld_cl(map_rank(mine_a + (c - rk * chunk) * 4u, rk), v);
      }
      full[c] = v;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float4* f4 = reinterpret_cast<const float4*>(full);
    for (int r0 = w * 4; r0 < own; r0 += kTailThreads / 8) {
      float s[4] = {0.f, 0.f, 0.f, 0.f};
      for (int c = lane; c < np / 4; c += 32) {
        const float4 v = f4[c];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          if (r0 + m >= own) continue;
          const float4 g = reinterpret_cast<const float4*>(
              A.G + (size_t)(V.rank * chunk + r0 + m) * np)[c];
          s[m] += g.x * v.x + g.y * v.y + g.z * v.z + g.w * v.w;
        }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[m] += __shfl_xor_sync(0xffffffffu, s[m], o);
      if (lane < 4 && r0 + lane < own) {
        const float v = lane == 0 ? s[0] : (lane == 1 ? s[1] : (lane == 2 ? s[2] : s[3]));
        const int q = quot(r0 + lane, 1.0f / (float)nx);
        d[q * L.pitch + row_pos(r0 + lane - q * nx, hx)] = (double)v * back;
      }
    }
    if (red.nact > 1) cluster_sync();
    else __syncthreads();
    acc = 0.0;
    for (int t = threadIdx.x; t < nc; t += kTailThreads) {
      const int q = quot(t, ip), p = t - q * L.pitch;
      const int i = p < hx ? 2 * p : 2 * (p - hx) + 1;
      if (i >= nx) continue;
      const int4 ra = V.tab()[2 * q];
      const int row = q * L.pitch;
      const unsigned o = p * 8u;
      const double dc = d[t];
      double v0, v1, v2, v3;
      ld_cl(ra.x + o, v0);
      ld_cl(ra.y + o, v1);
      ld_cl(ra.z + o, v2);
      ld_cl(ra.w + o, v3);
      double ox = a[t] * (dc - d[row + row_pos(i == 0 ? nx - 1 : i - 1, hx)]);
      double oy = a[2 * cap + t] * (dc - v0);
      double oz = a[4 * cap + t] * (dc - v2);
      ox = fma(a[cap + t], dc - d[row + row_pos(i == nx - 1 ? 0 : i + 1, hx)], ox);
      oy = fma(a[3 * cap + t], dc - v1, oy);
      oz = fma(a[5 * cap + t], dc - v3, oz);
      const double rn = r[t] - ((ox + oy) + oz);
      r[t] = rn;
      x[t] += dc;
      acc = fma(rn, rn, acc);
    }
    // 0: done, 1: another step, 2: no gain (or not a number)
    sc = red.run(acc, [&](double s) {
      const double was = rr;
      rr = s;
      return s <= stop ? 0.0 : (s <= 0.25 * was ? 1.0 : 2.0);
    });
    if (sc == 2.0) {
      ok = false;
      break;
    }
  }
  if (ok)
    for (int t = threadIdx.x; t < nc; t += kTailThreads) V.x()[t] = (T)x[t];
  return ok;
}

// The coarsest level of at most 32 cells: x = G (b - mean b) with the inverse
// G of L + s 1 1^T / N formed once per solve (coarsest_inverse).  On mean-free
// right-hand sides that is the mean-free solution of L x = b to rounding,
// where conjugate gradients would run their iterations' dependent reductions,
// divisions and roots in every cycle.  One lane per cell.
template <typename T>
__device__ void coarsest_direct(const View<T>& V) {
  const TailLevel<T>& L = V.L;
  const int N = L.rows * L.n[0], lane = threadIdx.x;
  if (lane >= 32) return;
  const double* G = V.template a<double>();
  const int q = quot(lane, 1.0f / (float)L.n[0]), c = q * L.pitch + row_pos(lane - q * L.n[0], L.hx);
  double b = lane < N ? (double)V.b()[c] : 0.0;
  double bs = b, none = 0.0;
  warp_sum2(bs, none);
  const double mean = bs / (double)N;
  b = lane < N ? b - mean : 0.0;
  double s0 = 0.0, s1 = 0.0;
  for (int m = 0; m < N; m += 2) {
    const double b0 = __shfl_sync(0xffffffffu, b, m), b1 = __shfl_sync(0xffffffffu, b, (m + 1) & 31);
    if (lane < N) {
      s0 = fma(G[m * N + lane], b0, s0);
      if (m + 1 < N) s1 = fma(G[(m + 1) * N + lane], b1, s1);
    }
  }
  if (lane < N) V.x()[c] = (T)(s0 + s1);
}

// The whole solve of a grid whose finest level is in the tail: cycles until
// ||b - L x|| <= rtol ||b|| (or the fixed count, or the cap), with the stopping
// rule of k_ctl_step.  Warp 0 of every CTA works it out from the same sums.
template <typename T, typename F>
__device__ __forceinline__ void solve_loop(const View<T>& V, const TailArgs<T>& A, Reduce& red,
                                           F cycle) {
  const TailLevel<T>& L = V.L;
  const int hx = L.hx, nx = L.n[0], cap = L.cap;
  const float ip = 1.0f / (float)L.pitch;
  int iters = 0, status = 0, zero = 0;
  double rel = 0.0;
  const double bn2 = *A.bn2;
  for (;;) {
    const T* x = V.x();
    const T* b = V.b();
    const T* a = V.template a<T>();
    double acc = 0.0;
    for (int t = threadIdx.x; t < V.nrows * L.pitch; t += kTailThreads) {
      const int q = quot(t, ip), p = t - q * L.pitch;
      const int i = p < hx ? 2 * p : 2 * (p - hx) + 1;
      if (i >= nx) continue;
      const int4 ra = V.tab()[2 * q];
      const int row = q * L.pitch;
      T ym, yp, zm, zp;
      const unsigned o = p * (unsigned)sizeof(T);
      ld_cl(ra.x + o, ym);
      ld_cl(ra.y + o, yp);
      ld_cl(ra.z + o, zm);
      ld_cl(ra.w + o, zp);
      const T xc = x[t];
      const T xm = x[row + row_pos(i == 0 ? nx - 1 : i - 1, hx)];
      const T xp = x[row + row_pos(i == nx - 1 ? 0 : i + 1, hx)];
      const T ox = a[t] * (xc - xm) + a[cap + t] * (xc - xp);
      const T oy = a[2 * cap + t] * (xc - ym) + a[3 * cap + t] * (xc - yp);
      const T oz = L.n[2] > 1 ? a[4 * cap + t] * (xc - zm) + a[5 * cap + t] * (xc - zp) : T(0);
      const double r = (double)(b[t] - ((ox + oy) + oz));
      acc = fma(r, r, acc);
    }
    red.nact = L.nact;
    red.used = min(V.nrows * L.pitch, kTailThreads);
    const double go = red.run(acc, [&](double r2) {
      if (!isfinite(bn2)) {
        status = FVM_EUNSTABLE;
        return 0.0;
      }
      if (bn2 == 0.0) {
        zero = 1;
        return 0.0;
      }
      rel = sqrt(r2) / sqrt(bn2);
      if (!isfinite(rel)) {
        status = FVM_EUNSTABLE;
        return 0.0;
      }
      if (A.fixed > 0) return iters < A.fixed ? 1.0 : 0.0;
      if (rel <= A.tol) return 0.0;
      if (iters < A.maxcycles) return 1.0;
      status = FVM_ENOCONV;
      return 0.0;
    });
    if (go == 0.0) break;
    cycle(iters > 0 && A.pre0 > 0 && A.post0 > 0);
    ++iters;
  }
  if (V.rank == 0 && threadIdx.x == 0) {
    A.ctl->iters = iters;
    A.ctl->status = status;
    A.ctl->zero = zero;
    A.ctl->rel = rel;
  }
}

// row tables: addresses of the rows beside each own row (the array a sweep or
// the conjugate gradients read there), the parent row, the row's parity
template <typename T>
__device__ void fill_table(const TailArgs<T>& A, int l, char* sm, unsigned base, int rank) {
  const TailLevel<T>& L = A.L[l];
  const View<T> V(L, sm, rank);
  const bool cg = l == A.nl - 1;
  const int off = cg ? A.ocg : L.ox, es = cg ? 8 : (int)sizeof(T);
  const int ny = L.n[1], nz = L.n[2];
  for (int q = threadIdx.x; q < V.nrows; q += kTailThreads) {
    const int R = rank * L.rpc + q;
    const int k = quot(R, 1.0f / (float)ny), j = R - k * ny;
    int4 ra, rb;
    ra.x = (int)row_addr(L, base, off, k * ny + (j == 0 ? ny - 1 : j - 1), es);
    ra.y = (int)row_addr(L, base, off, k * ny + (j == ny - 1 ? 0 : j + 1), es);
    ra.z = (int)row_addr(L, base, off, (k == 0 ? nz - 1 : k - 1) * ny + j, es);
    ra.w = (int)row_addr(L, base, off, (k == nz - 1 ? 0 : k + 1) * ny + j, es);
    rb.x = rb.z = rb.w = 0;
    rb.y = (j + k) & 1;
    if (!cg) {
      const TailLevel<T>& C = A.L[l + 1];
      rb.x = (int)row_addr(C, base, C.ox, (L.f[2] == 2 ? k >> 1 : k) * C.n[1] + (L.f[1] == 2 ? j >> 1 : j),
                           (int)sizeof(T));
    }
    V.tab()[2 * q] = ra;
    V.tab()[2 * q + 1] = rb;
  }
}

}  // namespace

template <typename T>
__global__ void __launch_bounds__(kTailThreads) k_tail(const __grid_constant__ TailArgs<T> A) {
  extern __shared__ __align__(16) char sm[];
  dependency_wait();
  const int rank = (int)cluster_rank();
  const unsigned base = smem_u32(sm);
  const int last = A.nl - 1;
  // coefficients: the packed copy, or from the betas
  for (int l = 0; l <= last; ++l) {
    const TailLevel<T>& L = A.L[l];
    if (rank >= L.nact) continue;
    const int bytes = L.cb;
    if (A.pack) {
      const int4* src = reinterpret_cast<const int4*>((const char*)A.pack + L.opack + (size_t)rank * bytes);
      int4* dst = reinterpret_cast<int4*>(sm + L.oa);
      for (int t = threadIdx.x; t < bytes / 16; t += kTailThreads) dst[t] = src[t];
    } else {
      fill_coefs(L, l == last, sm + L.oa, rank, threadIdx.x, kTailThreads);
    }
    fill_table(A, l, sm, base, rank);
  }
  Reduce red;
  red.vals = reinterpret_cast<double*>(sm + A.ored);
  red.slots = red.vals + 2 * kTailThreads;
  red.out = red.slots + 4 * kTailCTAs;
  red.base_slots = base + A.ored + 2 * kTailThreads * 8;
  red.nact = red.used = 0;
  red.rank = rank;
  red.phase = 0;
  __syncthreads();
  int single = 0;   // first level that CTA 0 holds alone
  while (single <= last && A.L[single].nact > 1) ++single;
  auto sync = [&](int l) {
    if (l < single) cluster_sync();
    else __syncthreads();
  };
  {
    // the top level's right-hand side; x starts at 0, or from the caller's
    const View<T> V(A.L[0], sm, rank);
    const TailLevel<T>& L = V.L;
    const float ip = 1.0f / (float)L.pitch;
    for (int t = threadIdx.x; t < V.nrows * L.pitch; t += kTailThreads) {
      const int q = quot(t, ip), p = t - q * L.pitch;
      const int i = p < L.hx ? 2 * p : 2 * (p - L.hx) + 1;
      if (i >= L.n[0]) continue;
      const int c = (rank * L.rpc + q) * L.n[0] + i;
      const T b = L.b[c];
      V.b()[t] = b;
      if (A.ctl) V.x()[t] = L.x[c];
      else if (last > 0) V.x()[t] = first_x(V, t, i, V.tab()[2 * q + 1].y, b, A.pre > 0);
    }
  }
  cluster_sync();
  T* scr = reinterpret_cast<T*>(sm + A.oscr);
  // one V-cycle; swept: the top level's first half-sweep is taken (it came with
  // b, or would repeat the previous cycle's last one)
  auto cycle = [&](bool swept) {
    for (int l = 0; l < last; ++l) {
      if (l >= single && rank) break;
      const View<T> V(A.L[l], sm, rank);
      const int pre = l == 0 ? A.pre0 : A.pre;
      for (int h = l > 0 || swept ? 1 : 0; h < 2 * pre; ++h) {
        sweep(V, h & 1);
        sync(l);
      }
      residual(V, scr, pre > 0 && sizeof(T) == sizeof(double));
      sync(l);
      restrict_rows(V, View<T>(A.L[l + 1], sm, rank), base, A.oscr, l + 1 == last, A.pre > 0);
      sync(l);
    }
    if (last < single || rank == 0) {
      const View<T> V(A.L[last], sm, rank);
      red.nact = V.L.nact;
      red.used = min(V.nrows * V.L.pitch, kTailThreads);
      if (A.direct) coarsest_direct(V);
      else if (!A.G || !coarsest_refine(V, A, red)) coarsest_cg(V, A, red);
    }
    for (int l = last - 1; l >= 0; --l) {
      if (l >= single && rank) continue;
      const View<T> V(A.L[l], sm, rank);
      sync(l);
      prolong_rows(V, A.L[l + 1]);
      sync(l);
      const int post = l == 0 ? A.post0 : A.post;
      for (int h = 0; h < 2 * post; ++h) {
        sweep(V, 1 - (h & 1));
        sync(l);
      }
    }
  };
  if (!A.ctl) {
    cycle(A.pre0 > 0);
  } else if (single > 0 || rank == 0) {
    solve_loop(View<T>(A.L[0], sm, rank), A, red, cycle);
  }
  if (last == 0) __syncthreads();
  {
    const View<T> V(A.L[0], sm, rank);
    const TailLevel<T>& L = V.L;
    const float in = 1.0f / (float)L.n[0];
    for (int t = threadIdx.x; t < V.nrows * L.n[0]; t += kTailThreads) {
      const int q = quot(t, in), i = t - q * L.n[0];
      L.x[(rank * L.rpc) * L.n[0] + t] = V.x()[q * L.pitch + row_pos(i, L.hx)];
    }
  }
}

// the coefficient blocks of every level and CTA, once per solve
template <typename T>
__global__ void k_tail_pack(const __grid_constant__ TailArgs<T> A) {
  dependency_wait();
  const int l = blockIdx.y, rank = blockIdx.x;
  const TailLevel<T>& L = A.L[l];
  if (rank >= L.nact) return;
  const bool coarsest = l == A.nl - 1;
  char* dst = (char*)A.pack + L.opack + (size_t)rank * L.cb;
  if (coarsest && A.direct) {
    if (blockIdx.z == 0) coarsest_inverse(L, (double*)dst);
    return;
  }
  fill_coefs(L, coarsest, dst, rank, threadIdx.x + blockIdx.z * blockDim.x,
             blockDim.x * gridDim.z);
}

// ---------------------------------------------------------------------------
// The float inverse of the coarsest operator, (L + s 1 1^T / N) / s with s the
// mean diagonal, by block Gauss-Jordan elimination over the whole GPU: one
// launch per block of 32 pivots, from one matrix into the other (every tile
// of a step reads the pivot rows and columns of the step before).  Symmetric
// and positive definite, so no pivoting.  Rows beyond N hold the identity.
// 32 x 32 tiles, whose CTAs are more and each repeat the pivot block's
// inverse, took 17 us per block for 625 cells, 32 us for 990.
template <typename T>
__global__ void k_inv_init(const __grid_constant__ TailLevel<T> L, float* W, int np,
                           double* gscale) {
  __shared__ float part[8];
  const int nx = L.n[0], N = L.rows * nx;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float a[6], sum = 0.f;
  for (int c = threadIdx.x; c < N; c += 256) {
    const int R = c / nx;
    cell_coefs<T, float>(L, c - R * nx, R, a);
    sum += (a[0] + a[1]) + (a[2] + a[3]) + (a[4] + a[5]);
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) part[w] = sum;
  __syncthreads();
  sum = 0.f;
  for (int q = 0; q < 8; ++q) sum += part[q];
  const float s = sum / (float)N, is = 1.0f / s;
  if (blockIdx.x == 0 && threadIdx.x == 0) *gscale = (double)s;
  const int r = blockIdx.x * 8 + w;
  float* row = W + (size_t)r * np;
  if (r >= N) {
    for (int c = lane; c < np; c += 32) row[c] = c == r ? 1.f : 0.f;
    return;
  }
  for (int c = lane; c < np; c += 32) row[c] = c < N ? 1.0f / (float)N : 0.f;
  __syncwarp();
  if (lane == 0) {
    const int ny = L.n[1], R = r / nx, i = r - R * nx, k = R / ny, j = R - k * ny;
    cell_coefs<T, float>(L, i, R, a);
    const int idx[3] = {i, j, k}, st[3] = {1, nx, nx * ny};
    float dg = 0.f;
    for (int d = 0; d < 3; ++d) {
      const int n = L.n[d];
      if (n == 1) continue;
      row[idx[d] == 0 ? r + (n - 1) * st[d] : r - st[d]] -= a[2 * d] * is;
      row[idx[d] == n - 1 ? r - (n - 1) * st[d] : r + st[d]] -= a[2 * d + 1] * is;
      dg += a[2 * d] + a[2 * d + 1];
    }
    row[r] += dg * is;
  }
}

// one block of 32 pivots (rows and columns b * 32 ...) on a 64 x 64 tile: every
// CTA inverts the pivot block D itself (2 us; as a launch of its own it would
// cost the gap between launches as well), forms X = D^-1 A[pivots, tile] and
// subtracts A[tile, pivots] X
__global__ void __launch_bounds__(256) k_inv_step(const float* __restrict__ A,
                                                  float* __restrict__ B, int np, int b) {
  __shared__ float D[2][32][33];
  __shared__ __align__(16) float Ct[32][68], R[32][64], X[32][64];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int i0 = blockIdx.y * 64, j0 = blockIdx.x * 64, p0 = b * 32;
  const int tx = tid & 15, ty = tid >> 4;
  const bool pc = ((j0 + tx * 4) >> 5) == b;    // the thread's columns are pivots
  const bool pr = ((i0 + ty * 4) >> 5) == b;    // the thread's rows are pivots
  float4 t[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    t[q] = *reinterpret_cast<const float4*>(A + (size_t)(i0 + ty * 4 + q) * np + j0 + tx * 4);
#pragma unroll
  for (int q = 0; q < 4; ++q) D[0][w + 8 * q][lane] = A[(size_t)(p0 + w + 8 * q) * np + p0 + lane];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    Ct[lane][w + 8 * q] = A[(size_t)(i0 + w + 8 * q) * np + p0 + lane];
    R[w + 8 * (q >> 1)][lane + 32 * (q & 1)] =
        A[(size_t)(p0 + w + 8 * (q >> 1)) * np + j0 + lane + 32 * (q & 1)];
  }
  __syncthreads();
  // D <- D^-1, from one copy into the other
  for (int p = 0; p < 32; ++p) {
    const float(*S)[33] = D[p & 1];
    float(*O)[33] = D[(p & 1) ^ 1];
    const float ip = __fdividef(1.0f, S[p][p]);
    const float rp = lane == p ? ip : S[p][lane] * ip;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = w + 8 * q;
      const float f = S[r][p], v = S[r][lane];
      O[r][lane] = r == p ? rp : (lane == p ? -f * ip : v - f * rp);
    }
    __syncthreads();
  }
  {
    const float(*V)[33] = D[0];
    const int r = ty * 2;
    float4 x0 = {0.f, 0.f, 0.f, 0.f}, x1 = x0;
    if (pc) {
      const int c = (j0 + tx * 4) & 31;
      x0 = {V[r][c], V[r][c + 1], V[r][c + 2], V[r][c + 3]};
      x1 = {V[r + 1][c], V[r + 1][c + 1], V[r + 1][c + 2], V[r + 1][c + 3]};
    } else {
#pragma unroll 8
      for (int m = 0; m < 32; ++m) {
        const float4 v = *reinterpret_cast<const float4*>(&R[m][tx * 4]);
        const float d0 = V[r][m], d1 = V[r + 1][m];
        x0.x += d0 * v.x; x0.y += d0 * v.y; x0.z += d0 * v.z; x0.w += d0 * v.w;
        x1.x += d1 * v.x; x1.y += d1 * v.y; x1.z += d1 * v.z; x1.w += d1 * v.w;
      }
    }
    *reinterpret_cast<float4*>(&X[r][tx * 4]) = x0;
    *reinterpret_cast<float4*>(&X[r + 1][tx * 4]) = x1;
  }
  __syncthreads();
  if (pr) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      t[q] = *reinterpret_cast<const float4*>(&X[(i0 + ty * 4 + q) & 31][tx * 4]);
  } else {
    if (pc)
#pragma unroll
      for (int q = 0; q < 4; ++q) t[q] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
    for (int m = 0; m < 32; ++m) {
      const float4 v = *reinterpret_cast<const float4*>(&X[m][tx * 4]);
      const float4 c = *reinterpret_cast<const float4*>(&Ct[m][ty * 4]);
      const float cc[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        t[q].x -= cc[q] * v.x; t[q].y -= cc[q] * v.y; t[q].z -= cc[q] * v.z; t[q].w -= cc[q] * v.w;
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
    *reinterpret_cast<float4*>(B + (size_t)(i0 + ty * 4 + q) * np + j0 + tx * 4) = t[q];
}

template <typename T>
void launch_tail_inverse(const TailArgs<T>& A, float* W0, float* W1, double* gscale,
                         cudaStream_t s) {
  const int nb = inverse_blocks(A), nt = A.np / 64;
  k_inv_init<T><<<A.np / 8, 256, 0, s>>>(A.L[A.nl - 1], W0, A.np, gscale);
  for (int b = 0; b < nb; ++b)
    k_inv_step<<<dim3(nt, nt), 256, 0, s>>>(b & 1 ? W1 : W0, b & 1 ? W0 : W1, A.np, b);
}

// Layout of a tail that starts at level Ls[0] with nl levels; false when it
// does not fit.  The cells a CTA should have: enough that a sweep's work is
// no smaller than the barrier that ends it.
template <typename T>
bool tail_layout(const MGLevel<T>* Ls, int nl, bool inverse, TailArgs<T>& A, size_t* smem,
                 size_t* pack) {
  if (nl < 1 || nl > kTailLevels) return false;
  A.nl = nl;
  int off = 0;
  size_t po = 0;
  auto take = [&](size_t bytes) {
    const int o = off;
    off += (int)((bytes + 15) / 16 * 16);
    return o;
  };
  size_t scr = 0;
  for (int l = 0; l < nl; ++l) {
    const MGLevel<T>& M = Ls[l];
    TailLevel<T>& L = A.L[l];
    const bool coarsest = l == nl - 1;
    if (M.geo.N > kTailMaxCells) return false;
    for (int d = 0; d < 3; ++d) {
      L.n[d] = M.geo.n[d];
      L.wall[d] = M.geo.bc[d] == WALL;
      L.f[d] = M.f[d];
      L.w[d] = M.w[d];
      L.beta[d] = M.beta[d];
    }
    L.x = M.x;
    L.b = M.b;
    L.hx = (L.n[0] + 1) / 2;
    L.pitch = 2 * L.hx;
    L.rows = L.n[1] * L.n[2];
    // the float inverse is read by rows, from all CTAs at once
    const bool inv = coarsest && inverse && M.geo.N > 32;
    const int per = inv ? kTailInvCells
                        : (coarsest ? kTailCgCells : (sizeof(T) == 8 ? kTailCells64 : kTailCells32));
    int want = (int)((M.geo.N + per - 1) / per);
    if (coarsest && !inv && M.geo.N <= kTailCgSingle) want = 1;
    want = want > kTailCTAs ? kTailCTAs : want;
    if (l > 0 && want > A.L[l - 1].nact) want = A.L[l - 1].nact;
    L.rpc = (L.rows + want - 1) / want;
    L.nact = (L.rows + L.rpc - 1) / L.rpc;
    if (l > 0 && L.nact > A.L[l - 1].nact) return false;
    L.cap = (L.rpc * L.pitch + 3) / 4 * 4;
    size_t cb = (size_t)L.cap * (coarsest ? 6 * sizeof(double) : 7 * sizeof(T));
    if (coarsest && M.geo.N <= 32) cb = cb > M.geo.N * M.geo.N * 8 ? cb : (size_t)(M.geo.N * M.geo.N * 8 + 15) / 16 * 16;
    if (cb + 2 * L.cap * sizeof(T) > (size_t)kTailSmem) return false;
    L.cb = (int)cb;
    L.ox = take(L.cap * sizeof(T));
    L.ob = take(L.cap * sizeof(T));
    L.oa = take(cb);
    L.otab = take((size_t)L.rpc * 32);
    L.opack = po;
    po += cb * L.nact;
    if (coarsest) {
      A.ocg = take((size_t)L.cap * 4 * sizeof(double));
      A.np = inv ? (int)((M.geo.N + 63) / 64 * 64) : 0;
      A.ovec = take(inv ? ((size_t)(L.rpc * L.n[0] + 3) / 4 * 4 + A.np) * sizeof(float) : 0);
    }
    else if (L.cap * sizeof(T) > scr) scr = L.cap * sizeof(T);
    if (off > kTailSmem) return false;
  }
  A.oscr = take(scr);
  A.ored = take((2 * kTailThreads + 4 * kTailCTAs + 4) * sizeof(double));
  *smem = off;
  *pack = po;
  return off <= kTailSmem;
}

template <typename T>
void launch_tail_pack(const TailArgs<T>& A, cudaStream_t s) {
  overlap_launch(k_tail_pack<T>, dim3(kTailCTAs, A.nl, 2), 256, 0, s, A);
}

// The limits belong to the kernel, not to a launch, and contexts of other grids
// may launch it from other host threads: they are always set to the same values
// (with each grid's own size a thread could lower the limit between another
// one's setting and launch, and that launch was refused).
template <typename T>
void tail_config(size_t smem, cudaStream_t s, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at) {
  cudaFuncSetAttribute(k_tail<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTailSmem);
  cudaFuncSetAttribute(k_tail<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cfg = {};
  cfg.gridDim = dim3(kTailCTAs);
  cfg.blockDim = dim3(kTailThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kTailCTAs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

template <typename T>
void launch_tail(const TailArgs<T>& A, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[2];
  tail_config<T>(smem, s, cfg, at);
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  cudaLaunchKernelEx(&cfg, k_tail<T>, A);
}

// whether the current device (or the part of it that this process may use) can
// hold the cluster at all
template <typename T>
bool tail_schedulable() {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute at[1];
  tail_config<T>(kTailSmem, nullptr, cfg, at);
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k_tail<T>, &cfg) == cudaSuccess) return clusters > 0;
  cudaGetLastError();
  return false;
}

#define FVM_TAIL_INST(T)                                                                        \
  template bool tail_layout<T>(const MGLevel<T>*, int, bool, TailArgs<T>&, size_t*, size_t*);   \
  template void launch_tail_inverse<T>(const TailArgs<T>&, float*, float*, double*, cudaStream_t); \
  template void launch_tail_pack<T>(const TailArgs<T>&, cudaStream_t);                          \
  template void launch_tail<T>(const TailArgs<T>&, size_t, cudaStream_t);                       \
  template bool tail_schedulable<T>();

FVM_TAIL_INST(double)
FVM_TAIL_INST(float)

}  // namespace fvm
