// Periodic Gaussian-gamma Coulomb potential V = gamma b and the gradient of a^T gamma b
// by Ewald summation (SCC-DFTB screened Coulomb, SI Sec. D; GPU Ewald, Sec. "Scalability").
//
//   gamma_IJ = sum_L' [erfc(eta d) - erfc(a_IJ d)] / d
//            + (4 pi / V) sum_{k != 0} exp(-k^2/4eta^2)/k^2 cos(k.(R_J - R_I))
//            - pi / (eta^2 V) + delta_IJ (U_I - 2 eta / sqrt(pi)),
//   a_IJ = 1 / sqrt(2 (sigma_I^2 + sigma_J^2)),  sigma_I = 1 / (sqrt(pi) U_I).
//
// Reciprocal space uses separable phase tables: e^{ik.R} = X[m1] Y[m2] Z[m3] with
// X[m] = exp(2 pi i m x / L).  k-vectors are grouped in rows of fixed (m1, m2).  The structure factor runs a
// block over a few rows and a chunk of atoms, a thread per pair +-m3, with the products X Y of the rows and the
// Z phases of the atoms staged in shared memory; partial sums are reduced in FP64 in a fixed order.  The
// potential kernel keeps each atom's Z phases in shared memory and takes four k-rows at a time.  T = float for
// the mixed path (FP64 final sums), double for the plain path.
#include <cmath>
#include <mutex>
#include <vector>
#include "ewald.cuh"

namespace sedacs {

namespace {

template <typename T> struct C2;
template <> struct C2<float> { using t = float2; };
template <> struct C2<double> { using t = double2; };

// a b + c d with one rounding of c d: which product is rounded first is the same for a phase and its conjugate.
__device__ __forceinline__ float dot2(float a, float b, float c, float d) { return __fmaf_rn(a, b, __fmul_rn(c, d)); }
__device__ __forceinline__ double dot2(double a, double b, double c, double d) { return __fma_rn(a, b, __dmul_rn(c, d)); }

// Phase tables in FP64, stored as T: tab[(axis * (nmax + 1) + m) * N + J] = exp(2 pi i m u), u = x / L.
template <typename T>
__global__ void phase_table_kernel(const double* R, int N, EwaldGeom g, typename C2<T>::t* tab) {
  const int J = blockIdx.x * blockDim.x + threadIdx.x, a = blockIdx.y;
  if (J >= N) return;
  {
    const double u = R[3 * J + a] / g.box_b[a] / kBohrA * 1.0;   // x (A) -> bohr -> fraction
    double s, c;
    sincospi(2.0 * (u - floor(u)), &s, &c);
    double re = 1.0, im = 0.0;
    const int nm = g.nmax[a];
    typename C2<T>::t* col = tab + (long long)a * (g.nmax_all + 1) * N + J;
    for (int m = 0; m <= nm; ++m) {
      typename C2<T>::t v;
      v.x = (T)re;
      v.y = (T)im;
      col[(long long)m * N] = v;
      const double nr = re * c - im * s, ni = re * s + im * c;
      re = nr;
      im = ni;
    }
  }
}

// S(k) partial over an atom chunk.  A block takes the entries (two k-rows, m3 >= 0) of its table line, one thread
// each, which also covers -m3 (the conjugate phase); four sums per k-vector, over every fourth atom of the chunk,
// are added in a fixed order in FP64.  Per 64 atoms the block forms b X Y for its rows and stages the atoms' Z
// phases.  Five FP32 operations a k-vector and atom (the products that +-m3 share are formed once) bound it: a Z
// phase read from shared memory serves four k-vectors, a product b X Y two.
// Measured (GB300, 30,000 atoms): 0.43 ms; 0.59 ms with one row per thread (shared-memory reads bound), 2.95 ms
// with a block per row.
constexpr int kSfThreads = 128, kSfRows = 32, kSfAtoms = 64;

template <typename T> struct Pair2;              // two complex numbers, one shared-memory read in FP32
template <> struct __align__(16) Pair2<float> { float2 a, b; };
template <> struct __align__(16) Pair2<double> { double2 a, b; };

template <typename T>
__global__ void __launch_bounds__(kSfThreads) structure_factor_kernel(const SfBlock* blocks, const int2* entries,
                                                                      const KRow* rows, int nrows,
                                                                      const typename C2<T>::t* tab, const double* b,
                                                                      int N, int nmax_all, int m3max, int max_rows,
                                                                      int chunk, double* part, long long nk_total) {
  using CT = typename C2<T>::t;
  const SfBlock blk = blocks[blockIdx.x];
  const int a0 = blockIdx.y * chunk, a1 = min(N, a0 + chunk);
  constexpr int kPitch = kSfAtoms + 2;
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ int2 ms[kSfRows];                               // (m1, m2) of the rows
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)threadIdx.x < blk.n_rows)
    ms[threadIdx.x] = make_int2(rows[blk.row0 + threadIdx.x].m1, rows[blk.row0 + threadIdx.x].m2);
  CT* c12 = reinterpret_cast<CT*>(sm);                       // [row][kPitch]
  CT* zs = c12 + max_rows * kPitch;                          // [atom][zw]
  const int zw = (m3max + 1) | 1;
  const bool mine = (int)threadIdx.x < blk.n_entries;
  const int2 en = mine ? entries[blk.entry0 + threadIdx.x] : make_int2(blk.row0, 0);
  const int two = en.x + 1 < nrows ? 1 : 0;                  // the last row may stand alone
  const CT* c[2] = {c12 + (en.x - blk.row0) * kPitch, c12 + (en.x - blk.row0 + two) * kPitch};
  T pr[2][4], pi[2][4], nr[2][4], ni[2][4];                  // +m3 and -m3 of both rows
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int g = 0; g < 4; ++g) pr[r][g] = pi[r][g] = nr[r][g] = ni[r][g] = 0;
  for (int j0 = a0; j0 < a1; j0 += kSfAtoms) {
    const int n = min(kSfAtoms, a1 - j0);
    __syncthreads();
    // a warp stages a row, or one m3, of the 64 atoms, two per lane
    T q[2];
    bool in[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      in[h] = lane + 32 * h < n;
      q[h] = in[h] ? (T)b[j0 + lane + 32 * h] : (T)0;
    }
#pragma unroll 2
    for (int r = warp; r < blk.n_rows; r += kSfThreads / 32) {
      const int m1 = ms[r].x, m2 = ms[r].y;
      const CT* xp = tab + (long long)m1 * N + j0 + lane;
      const CT* yp = tab + ((long long)nmax_all + 1 + abs(m2)) * N + j0 + lane;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        CT x, y, v;
        x.x = x.y = y.x = y.y = 0;
        if (in[h]) {
          x = xp[32 * h];
          y = yp[32 * h];
        }
        if (m2 < 0) y.y = -y.y;
        v.x = q[h] * dot2(x.x, y.x, -x.y, y.y);
        v.y = q[h] * dot2(x.y, y.x, x.x, y.y);
        c12[r * kPitch + lane + 32 * h] = v;
      }
    }
#pragma unroll 4
    for (int m = warp; m <= m3max; m += kSfThreads / 32) {
      const CT* zp = tab + (2LL * (nmax_all + 1) + m) * N + j0 + lane;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (in[h]) zs[(lane + 32 * h) * zw + m] = zp[32 * h];
    }
    __syncthreads();
    if (!mine) continue;
    const CT* z = zs + en.y;
    auto add = [&](int r, int g, const CT cv, const CT zp) {
      pr[r][g] += dot2(cv.x, zp.x, -cv.y, zp.y);
      pi[r][g] += dot2(cv.x, zp.y, cv.y, zp.x);
      nr[r][g] += dot2(cv.x, zp.x, cv.y, zp.y);
      ni[r][g] += dot2(cv.x, -zp.y, cv.y, zp.x);
    };
    int j = 0;
    for (; j + 4 <= n; j += 4) {
#pragma unroll
      for (int h = 0; h < 4; h += 2) {
        const CT z0 = z[(j + h) * zw], z1 = z[(j + h + 1) * zw];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const Pair2<T> cc = *reinterpret_cast<const Pair2<T>*>(c[r] + j + h);
          add(r, h, cc.a, z0);
          add(r, h + 1, cc.b, z1);
        }
      }
    }
#pragma unroll
    for (int g = 0; g < 3; ++g)
      if (j + g < n)
#pragma unroll
        for (int r = 0; r < 2; ++r) add(r, g, c[r][j + g], z[(j + g) * zw]);
  }
  if (!mine) return;
  auto put = [&](const KRow kr, int m3, const T (&re4)[4], const T (&im4)[4]) {
    if (m3 < kr.m3lo || m3 > kr.m3hi) return;
    double re = 0.0, im = 0.0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      re += (double)re4[g];
      im += (double)im4[g];
    }
    const long long o = (long long)blockIdx.y * nk_total + kr.koff + (m3 - kr.m3lo);
    part[2 * o] = re;
    part[2 * o + 1] = im;
  };
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (r > two) break;
    const KRow kr = rows[en.x + r];
    put(kr, en.y, pr[r], pi[r]);
    if (en.y > 0) put(kr, -en.y, nr[r], ni[r]);
  }
}

// S(k) = sum over atom chunks (fixed order), times the k weight; stored as T complex.
template <typename T>
__global__ void sf_reduce_kernel(const double* part, int nchunk, long long nk, const double* wk,
                                 typename C2<T>::t* ws) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= nk) return;
  double re = 0.0, im = 0.0;
#pragma unroll 4
  for (int c = 0; c < nchunk; ++c) {
    const double2 p = reinterpret_cast<const double2*>(part)[c * nk + k];
    re += p.x;
    im += p.y;
  }
  ws[k].x = (T)(wk[k] * re);
  ws[k].y = (T)(wk[k] * im);
}

// Per atom I: sum_k w S(k) e^{-ik.R_I} -> Re (potential) and, for gradients, Im weighted by k.
// mode 0: out[I] = Re sum (nv = 1).  mode 1: g[I][c] = sum w k_c [a_I Im(S_b e^-ikR) + b_I Im(S_a e^-ikR)].
// A block takes blockDim atoms and one of gridDim.y chunks of the rows, four rows at a time: a Z phase read from
// shared memory serves four k-vectors, whose weighted structure factors (zero past a row's end, which adds
// nothing) sit beside each other for broadcast reads.  The sums over m3 are in T, those over rows in FP64.
// Measured (GB300, 30,000 atoms), potential: 0.51 ms; 0.76 ms while the X and Y phases lay atom by atom (a line per
// lane), 1.68 ms with one row at a time as well.  FP32 arithmetic (0.26 ms) and the FP64 row sums (0.17 ms) bound it.
template <typename T, int MODE>
__global__ void recip_atom_kernel(const KRow* rows, int nrows, const typename C2<T>::t* tab, const typename C2<T>::t* ws,
                                  long long nk, int N, int nmax_all, int m3max, EwaldGeom g, const double* av,
                                  const double* bv, double* out_part) {
  // block (atom chunk, row chunk): rows [r0, r1) of the k list, partial sums per row chunk
  const int rchunk = (nrows + gridDim.y - 1) / gridDim.y;
  const int r0 = blockIdx.y * rchunk, r1 = min(nrows, r0 + rchunk);
  double* out = out_part + (long long)blockIdx.y * (MODE == 0 ? N : 3 * N);
  using CT = typename C2<T>::t;
  constexpr int NV = MODE == 0 ? 1 : 2;        // structure factors: S_b, and S_a for the gradient
  extern __shared__ unsigned char sm[];
  CT* zt = reinterpret_cast<CT*>(sm);          // [m3max + 1][blockDim]
  CT* ss = zt + (m3max + 1) * blockDim.x;      // [2 m3max + 1][4 rows][NV]
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const int bd = blockDim.x;
  if (I < N)
    for (int m = 0; m <= m3max; ++m) zt[m * bd + threadIdx.x] = tab[(2LL * (nmax_all + 1) + m) * N + I];
  double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0;
  const double tpx = 2.0 * M_PI / g.box_b[0], tpy = 2.0 * M_PI / g.box_b[1], tpz = 2.0 * M_PI / g.box_b[2];
  const T aI = MODE == 1 && I < N ? (T)av[I] : (T)0, bI = MODE == 1 && I < N ? (T)bv[I] : (T)0;
  for (int rb = r0; rb < r1; rb += 4) {
    KRow kr[4];
    int lo = m3max, hi = -m3max;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      kr[q] = rows[min(rb + q, r1 - 1)];
      if (rb + q >= r1) { kr[q].m3lo = 1; kr[q].m3hi = 0; }
      else {
        lo = min(lo, kr[q].m3lo);
        hi = max(hi, kr[q].m3hi);
      }
    }
    __syncthreads();
    for (int q = threadIdx.x; q < (hi - lo + 1) * 4; q += blockDim.x) {
      const int t = q >> 2, r = q & 3, m3 = lo + t;
      const KRow k = rows[min(rb + r, r1 - 1)];
      const bool in = rb + r < r1 && m3 >= k.m3lo && m3 <= k.m3hi;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        CT x;
        x.x = x.y = 0;
        if (in) x = ws[v * nk + k.koff + (m3 - k.m3lo)];
        ss[(t * 4 + r) * NV + v] = x;
      }
    }
    __syncthreads();
    if (I >= N) continue;
    CT xy[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const CT x = tab[(long long)kr[q].m1 * N + I];
      CT y = tab[((long long)nmax_all + 1 + abs(kr[q].m2)) * N + I];
      if (kr[q].m2 < 0) y.y = -y.y;
      xy[q].x = dot2(x.x, y.x, -x.y, y.y);
      xy[q].y = -dot2(x.y, y.x, x.x, y.y);   // conj -> e^{-i(k1 x + k2 y)}
    }
    T s1[4], s3[4];                     // sums over m3: the real part, or the Im-combination weighted by 1 and by m3
#pragma unroll
    for (int q = 0; q < 4; ++q) s1[q] = s3[q] = 0;
    const CT* zp = zt + (lo < 0 ? -lo : lo) * bd + threadIdx.x;
    const CT* sp = ss;
    auto step = [&](const CT z, int m3) {       // z = conj(Z[m3])
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        CT e;
        e.x = dot2(xy[q].x, z.x, -xy[q].y, z.y);
        e.y = dot2(xy[q].x, z.y, xy[q].y, z.x);
        if (MODE == 0) {
          const CT sv = sp[q];
          s1[q] += dot2(sv.x, e.x, -sv.y, e.y);
        } else {
          // Im(S e^{-ikR}) for S_b (vector 0) and S_a (vector 1)
          const CT sb = sp[2 * q], sa = sp[2 * q + 1];
          const T imb = sb.x * e.y + sb.y * e.x;
          const T ima = sa.x * e.y + sa.y * e.x;
          const T comb = aI * imb + bI * ima;
          s1[q] += comb;
          s3[q] += comb * (T)m3;
        }
      }
      sp += 4 * NV;
    };
    int m3 = lo;
#pragma unroll 2
    for (; m3 < 0; ++m3, zp -= bd) step(*zp, m3);           // conj(Z[-m]) = Z[m]
#pragma unroll 2
    for (; m3 <= hi; ++m3, zp += bd) {
      CT z = *zp;
      z.y = -z.y;
      step(z, m3);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (rb + q >= r1) break;
      if (MODE == 0) {
        acc0 += (double)s1[q];
      } else {
        acc0 += (double)s1[q] * (tpx * kr[q].m1);
        acc1 += (double)s1[q] * (tpy * kr[q].m2);
        acc2 += (double)s3[q] * tpz;
      }
    }
  }
  if (I >= N) return;
  if (MODE == 0) {
    out[I] = acc0;
  } else {
    out[3 * I] = acc0;
    out[3 * I + 1] = acc1;
    out[3 * I + 2] = acc2;
  }
}

// Real-space part, one warp per atom I over images within rc.  mode 0: V_I += sum_J phi b_J;
// mode 1: dE/dR_I += -sum_J (a_I b_J + a_J b_I) phi'(d) d_hat.  Differences of positions are
// taken in FP64, the rest in T; lane sums are combined by a fixed shuffle tree.
template <typename T, int MODE>
__global__ void real_space_kernel(const double* R, const int* species, int N, EwaldGeom g, const int* cell_start,
                                  const int* cell_count, const int* cell_atoms, const int* cell_of, const double* av,
                                  const double* bv, double* out) {
  const int I = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (I >= N) return;
  const T rc2 = (T)(g.rc_b * g.rc_b);
  const T eta = (T)g.eta;
  const T sq = (T)1.1283791670955126;    // 2 / sqrt(pi)
  const T inv_b = (T)(1.0 / kBohrA);
  const T bx = (T)g.box_b[0], by = (T)g.box_b[1], bz = (T)g.box_b[2];
  const int si = species[I];
  double acc = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
  const double xi = R[3 * I], yi = R[3 * I + 1], zi = R[3 * I + 2];
  auto visit = [&](int J, T dx, T dy, T dz) {
    const T d2 = dx * dx + dy * dy + dz * dz;
    if (d2 >= rc2 || d2 == (T)0) return;
    const T d = sqrt(d2);
    const T aij = (T)g.a[si][species[J]];
    const T e1 = erfc(eta * d), e2 = erfc(aij * d);
    const T phi = (e1 - e2) / d;
    if (MODE == 0) {
      acc += (double)phi * bv[J];
    } else {
      const T dphi = (-sq * eta * exp(-(eta * d) * (eta * d)) + sq * aij * exp(-(aij * d) * (aij * d))) / d - phi / d;
      const double coef = (av[I] * bv[J] + av[J] * bv[I]) * (double)(dphi / d);
      gx -= coef * (double)dx;
      gy -= coef * (double)dy;
      gz -= coef * (double)dz;
    }
  };
  auto rel = [&](int J, T& dx, T& dy, T& dz) {
    dx = (T)(R[3 * J] - xi) * inv_b;
    dy = (T)(R[3 * J + 1] - yi) * inv_b;
    dz = (T)(R[3 * J + 2] - zi) * inv_b;
    dx -= bx * rint(dx / bx);
    dy -= by * rint(dy / by);
    dz -= bz * rint(dz / bz);
  };
  if (g.brute) {
    for (int J = lane; J < N; J += 32) {
      T dx, dy, dz;
      rel(J, dx, dy, dz);
      for (int ix = -g.nimg[0]; ix <= g.nimg[0]; ++ix)
        for (int iy = -g.nimg[1]; iy <= g.nimg[1]; ++iy)
          for (int iz = -g.nimg[2]; iz <= g.nimg[2]; ++iz) visit(J, dx + ix * bx, dy + iy * by, dz + iz * bz);
    }
  } else {
    const int cid = cell_of[I];
    const int cz = cid % g.nc[2], cy = (cid / g.nc[2]) % g.nc[1], cx = cid / (g.nc[2] * g.nc[1]);
    for (int ddx = -1; ddx <= 1; ++ddx)
      for (int ddy = -1; ddy <= 1; ++ddy)
        for (int ddz = -1; ddz <= 1; ++ddz) {
          const int x = (cx + ddx + g.nc[0]) % g.nc[0];
          const int y = (cy + ddy + g.nc[1]) % g.nc[1];
          const int z = (cz + ddz + g.nc[2]) % g.nc[2];
          const int c = (x * g.nc[1] + y) * g.nc[2] + z;
          for (int q = lane; q < cell_count[c]; q += 32) {
            const int J = cell_atoms[cell_start[c] + q];
            T dx, dy, dz;
            rel(J, dx, dy, dz);
            visit(J, dx, dy, dz);
          }
        }
  }
  if (MODE == 0) {
    acc = warp_sum(acc);
    if (lane == 0) out[I] = acc;
  } else {
    gx = warp_sum(gx);
    gy = warp_sum(gy);
    gz = warp_sum(gz);
    if (lane == 0) {
      out[3 * I] = gx;
      out[3 * I + 1] = gy;
      out[3 * I + 2] = gz;
    }
  }
}

// ---- cell path of the real-space sum (cells at least rc wide, 3 or more per axis) -------------
// Atoms are ordered by cell, and by index inside a cell (deterministic).  Each sorted entry
// keeps its coordinates relative to its cell's origin (bohr) and its species; the warp of atom
// I scans the 27 neighbour cells with coalesced loads, queues the pairs inside rc in shared
// memory (ballot + popc) and evaluates them 32 at a time, so the erfc/exp work runs with
// full warps.

template <typename T> struct Pos4;
template <> struct Pos4<float> { using t = float4; };
template <> struct Pos4<double> { using t = double4; };

__global__ void cell_count_kernel(const double* R, int N, EwaldGeom g, int* cell_of, int* cell_count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  int c[3];
  for (int a = 0; a < 3; ++a) {
    const double x = R[3 * i + a] / kBohrA;
    const double w = x - g.box_b[a] * floor(x / g.box_b[a]);
    c[a] = min(max((int)floor(w / (g.box_b[a] / g.nc[a])), 0), g.nc[a] - 1);
  }
  const int cid = (c[0] * g.nc[1] + c[1]) * g.nc[2] + c[2];
  cell_of[i] = cid;
  atomicAdd(&cell_count[cid], 1);
}

// exclusive scan of the cell counts (one block)
__global__ void cell_scan_kernel(const int* count, int ncell, int* start) {
  const int per = (ncell + blockDim.x - 1) / blockDim.x;
  const int b0 = threadIdx.x * per, b1 = min(ncell, b0 + per);
  int s = 0;
  for (int c = b0; c < b1; ++c) s += count[c];
  int total;
  int acc = scan1024(s, &total);
  if (threadIdx.x == 0) start[ncell] = total;
  for (int c = b0; c < b1; ++c) {
    start[c] = acc;
    acc += count[c];
  }
}

__global__ void cell_append_kernel(const int* cell_of, int N, const int* cell_start, int* cell_fill, int* cell_atoms) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int c = cell_of[i];
  cell_atoms[cell_start[c] + atomicAdd(&cell_fill[c], 1)] = i;
}

// Every atom's place in its cell is its rank by index among the cell's atoms (a few hundred, counted directly);
// blockDim atoms of a cell per block.
template <typename T>
__global__ void cell_rank_kernel(const double* R, const int* species, EwaldGeom g, const int* cell_start,
                                 const int* unsorted, int* sorted_atom, typename Pos4<T>::t* pos_s) {
  __shared__ int tile[256];
  const int c = blockIdx.x, s0 = cell_start[c], s1 = cell_start[c + 1];
  const int cz = c % g.nc[2], cy = (c / g.nc[2]) % g.nc[1], cx = c / (g.nc[2] * g.nc[1]);
  const double o[3] = {cx * (g.box_b[0] / g.nc[0]), cy * (g.box_b[1] / g.nc[1]), cz * (g.box_b[2] / g.nc[2])};
  for (int b0 = s0 + blockIdx.y * blockDim.x; b0 < s1; b0 += gridDim.y * blockDim.x) {
    const int q = b0 + threadIdx.x;
    const int i = q < s1 ? unsorted[q] : 0;
    int rank = 0;
    for (int t0 = s0; t0 < s1; t0 += blockDim.x) {
      const int n = min((int)blockDim.x, s1 - t0);
      __syncthreads();
      if ((int)threadIdx.x < n) tile[threadIdx.x] = unsorted[t0 + threadIdx.x];
      __syncthreads();
      for (int t = 0; t < n; ++t) rank += tile[t] < i;
    }
    if (q >= s1) continue;
    const int k = s0 + rank;
    sorted_atom[k] = i;
    typename Pos4<T>::t p;
    double r[3];
    for (int a = 0; a < 3; ++a) {
      const double x = R[3 * i + a] / kBohrA;
      r[a] = (x - g.box_b[a] * floor(x / g.box_b[a])) - o[a];
    }
    p.x = (T)r[0];
    p.y = (T)r[1];
    p.z = (T)r[2];
    p.w = (T)species[i];
    pos_s[k] = p;
  }
}

// A warp per atom: the 27 cells around it are tested 64 atoms at a time, pairs within the cutoff wait in a ring and
// are worked off 32 at a time in the order found, so that every lane has a pair.  Bound by instructions: the tests
// (9,100 candidates an atom for 1,400 pairs) and two erfc a pair.  Measured (GB300, 30,000 atoms): 0.74 ms, 0.79 ms
// with 32 tests at a time and the queue moved up after each use.
template <typename T, int MODE>
__global__ void real_cells_kernel(const typename Pos4<T>::t* pos_s, const int* sorted_atom, const int* cell_start,
                                  int N, EwaldGeom g, const double* av, const double* bv, double* out) {
  using PT = typename Pos4<T>::t;
  constexpr int kQ = 128;                          // ring: fewer than 32 waiting, 64 added at a time
  __shared__ int qj[4][kQ];
  __shared__ PT qd[4][kQ];                         // displacement and species
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * 4 + wib;              // sorted index of atom I
  if (k >= N) return;
  const int I = sorted_atom[k];
  const typename Pos4<T>::t pi = pos_s[k];
  const int si = (int)pi.w;
  // cell of k: the one whose range holds k
  int lo = 0, hi = g.nc[0] * g.nc[1] * g.nc[2];
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (cell_start[mid] <= k) lo = mid; else hi = mid;
  }
  const int c = lo;
  const int cz = c % g.nc[2], cy = (c / g.nc[2]) % g.nc[1], cx = c / (g.nc[2] * g.nc[1]);
  const T wx = (T)(g.box_b[0] / g.nc[0]), wy = (T)(g.box_b[1] / g.nc[1]), wz = (T)(g.box_b[2] / g.nc[2]);
  const T rc2 = (T)(g.rc_b * g.rc_b);
  const T eta = (T)g.eta;
  const T sq = (T)1.1283791670955126;    // 2 / sqrt(pi)
  const double aI = MODE == 1 ? av[I] : 0.0, bI = MODE == 1 ? bv[I] : 0.0;
  double acc = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
  int qn = 0, head = 0;
  auto flush = [&](int cnt) {
    // lanes < cnt take one queued pair each
    if (lane < cnt) {
      const int slot = (head + lane) & (kQ - 1);
      const int J = sorted_atom[qj[wib][slot]];
      const PT q = qd[wib][slot];
      const T dx = q.x, dy = q.y, dz = q.z;
      const T d2 = dx * dx + dy * dy + dz * dz;
      const T d = sqrt(d2);
      const int sj = (int)q.w;
      const T aij = (T)g.a[si][sj];
      const T e1 = erfc(eta * d), e2 = erfc(aij * d);
      const T phi = (e1 - e2) / d;
      if (MODE == 0) {
        acc += (double)phi * bv[J];
      } else {
        const T dphi = (-sq * eta * exp(-(eta * d) * (eta * d)) + sq * aij * exp(-(aij * d) * (aij * d))) / d - phi / d;
        const double coef = (aI * bv[J] + av[J] * bI) * (double)(dphi / d);
        gx -= coef * (double)dx;
        gy -= coef * (double)dy;
        gz -= coef * (double)dz;
      }
    }
  };
  for (int ddx = -1; ddx <= 1; ++ddx)
    for (int ddy = -1; ddy <= 1; ++ddy)
      for (int ddz = -1; ddz <= 1; ++ddz) {
        const int x = (cx + ddx + g.nc[0]) % g.nc[0];
        const int y = (cy + ddy + g.nc[1]) % g.nc[1];
        const int z = (cz + ddz + g.nc[2]) % g.nc[2];
        const int cn = (x * g.nc[1] + y) * g.nc[2] + z;
        const int j0 = cell_start[cn], j1 = cell_start[cn + 1];
        const T ox = (T)ddx * wx - pi.x, oy = (T)ddy * wy - pi.y, oz = (T)ddz * wz - pi.z;
        for (int jb = j0; jb < j1; jb += 64) {
          PT d[2];
          unsigned m[2];
          bool in[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int j = jb + 32 * h + lane;
            in[h] = false;
            if (j < j1) {
              d[h] = pos_s[j];
              d[h].x += ox;
              d[h].y += oy;
              d[h].z += oz;
              const T d2 = d[h].x * d[h].x + d[h].y * d[h].y + d[h].z * d[h].z;
              in[h] = d2 < rc2 && j != k;
            }
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) m[h] = __ballot_sync(0xffffffffu, in[h]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (in[h]) {
              const int slot = (head + qn + __popc(m[h] & ((1u << lane) - 1u))) & (kQ - 1);
              qj[wib][slot] = jb + 32 * h + lane;
              qd[wib][slot] = d[h];
            }
            qn += __popc(m[h]);
          }
          __syncwarp();
          while (qn >= 32) {
            flush(32);
            head += 32;
            qn -= 32;
          }
          __syncwarp();
        }
      }
  flush(qn);
  if (MODE == 0) {
    acc = warp_sum(acc);
    if (lane == 0) out[I] = acc;
  } else {
    gx = warp_sum(gx);
    gy = warp_sum(gy);
    gz = warp_sum(gz);
    if (lane == 0) {
      out[3 * I] = gx;
      out[3 * I + 1] = gy;
      out[3 * I + 2] = gz;
    }
  }
}

__global__ void chunk_reduce_kernel(const double* part, int nchunk, long long len, double* out) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= len) return;
  double s = 0.0;
  for (int c = 0; c < nchunk; ++c) s += part[c * len + t];
  out[t] = s;
}

// out = real + recip + self/background terms (potential) or real + recip (gradient, Ha/A).
__global__ void combine_pot_kernel(const double* real, const double* recip, const double* b, const int* species,
                                   EwaldGeom g, const double* bsum, double* V, int N) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= N) return;
  V[I] = real[I] + recip[I] - M_PI / (g.eta * g.eta * g.vol) * bsum[0] +
         (g.u[species[I]] - 2.0 * g.eta / sqrt(M_PI)) * b[I];
}

__global__ void combine_grad_kernel(const double* real, const double* recip, double* G, int N, double scale) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * N) return;
  G[i] = (real[i] + recip[i]) * scale;
}

__global__ void sum_kernel(const double* b, int N, double* out) {
  __shared__ double red[1024];
  double s = 0.0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) s += b[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0];
}

}  // namespace

// =================================================================================================
Ewald::~Ewald() { release(); }

void Ewald::release() {
  for (void* p : {(void*)rows_d, (void*)wk_d, (void*)tab, (void*)part, (void*)ws, (void*)real_buf, (void*)recip_buf,
                  (void*)cell_of, (void*)cell_count, (void*)cell_start, (void*)cell_atoms, (void*)cell_raw, (void*)scal,
                  (void*)rpart, (void*)sf_blocks, (void*)sf_entries, pos_s})
    if (p) cudaFree(p);
  rows_d = nullptr; wk_d = nullptr; tab = nullptr; part = nullptr; ws = nullptr; real_buf = nullptr;
  recip_buf = nullptr; rpart = nullptr; cell_of = cell_count = cell_start = cell_atoms = cell_raw = nullptr;
  sf_blocks = nullptr;
  sf_entries = nullptr; scal = nullptr;
  pos_s = nullptr;
  N_ = 0;
}

cudaError_t Ewald::setup(int N, const double box_A[3], const double hubbard_u[3], bool fp64, double tol) {
  release();
  N_ = N;
  fp64_ = fp64;
  const double x = sqrt(-log(tol));
  // Real-space cutoff: up to 15 A, and at most a third of the shortest box side so that the cell
  // path (3 or more cells per axis) applies; not below 9 A (small boxes use the image loop).
  // The k-space work falls as rc^-3 and the real-space work rises as rc^3; with the queued
  // real-space kernel the balance for condensed-phase densities lies near 15 A.
  const double lmin = std::min(box_A[0], std::min(box_A[1], box_A[2]));
  const double rc = std::min(15.0, std::max(9.0, lmin / 3.0 * (1.0 - 1e-6))) / kBohrA;
  g.rc_b = rc;
  g.eta = (x + 0.3) / rc;
  const double kmax = 2.0 * g.eta * x;
  g.vol = 1.0;
  for (int a = 0; a < 3; ++a) {
    g.box_b[a] = box_A[a] / kBohrA;
    g.vol *= g.box_b[a];
    g.nmax[a] = (int)floor(kmax * g.box_b[a] / (2.0 * M_PI));
    g.nimg[a] = (int)floor((rc + 0.5 * g.box_b[a]) / g.box_b[a]);
    g.nc[a] = (int)floor(g.box_b[a] / (rc * (1.0 + 1e-9)));
    g.u[a] = hubbard_u[a];
  }
  g.brute = (g.nc[0] < 3 || g.nc[1] < 3 || g.nc[2] < 3 || g.nimg[0] > 0 || g.nimg[1] > 0 || g.nimg[2] > 0) ? 1 : 0;
  for (int a = 0; a < 3; ++a) if (g.nc[a] < 1) g.nc[a] = 1;
  g.nmax_all = std::max(g.nmax[0], std::max(g.nmax[1], g.nmax[2]));
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      const double si = 1.0 / (sqrt(M_PI) * hubbard_u[i]), sj = 1.0 / (sqrt(M_PI) * hubbard_u[j]);
      g.a[i][j] = 1.0 / sqrt(2.0 * (si * si + sj * sj));
    }
  // k rows (half space)
  std::vector<KRow> rows;
  std::vector<double> wk;
  long long koff = 0;
  const double k2max = kmax * kmax;
  const double tp[3] = {2 * M_PI / g.box_b[0], 2 * M_PI / g.box_b[1], 2 * M_PI / g.box_b[2]};
  m3max_ = 0;
  for (int m1 = 0; m1 <= g.nmax[0]; ++m1)
    for (int m2 = -g.nmax[1]; m2 <= g.nmax[1]; ++m2) {
      if (m1 == 0 && m2 < 0) continue;
      const double k12 = (tp[0] * m1) * (tp[0] * m1) + (tp[1] * m2) * (tp[1] * m2);
      if (k12 > k2max) continue;
      int hi = (int)floor(sqrt((k2max - k12)) / tp[2]);
      hi = std::min(hi, g.nmax[2]);
      int lo = (m1 == 0 && m2 == 0) ? 1 : -hi;
      if (hi < lo) continue;
      KRow r;
      r.m1 = m1; r.m2 = m2; r.m3lo = lo; r.m3hi = hi; r.koff = koff;
      for (int m3 = lo; m3 <= hi; ++m3) {
        const double kz = tp[2] * m3;
        const double k2 = k12 + kz * kz;
        wk.push_back(k2 <= k2max ? 2.0 * (4.0 * M_PI / g.vol) * exp(-k2 / (4.0 * g.eta * g.eta)) / k2 : 0.0);
      }
      koff += hi - lo + 1;
      m3max_ = std::max(m3max_, hi);
      rows.push_back(r);
    }
  nrows_ = (int)rows.size();
  nk_ = koff;
  cudaError_t e;
  if ((e = cudaMalloc(&rows_d, sizeof(KRow) * std::max(1, nrows_)))) return e;
  if ((e = cudaMalloc(&wk_d, sizeof(double) * std::max(1LL, nk_)))) return e;
  cudaMemcpy(rows_d, rows.data(), sizeof(KRow) * nrows_, cudaMemcpyHostToDevice);
  cudaMemcpy(wk_d, wk.data(), sizeof(double) * nk_, cudaMemcpyHostToDevice);
  const size_t csz = fp64 ? sizeof(double2) : sizeof(float2);
  if ((e = cudaMalloc(&tab, csz * 3 * (size_t)N * (g.nmax_all + 1)))) return e;
  nchunk_ = (N + kChunk - 1) / kChunk;
  // structure-factor blocks: runs of at most kSfThreads entries (rows r and r + 1, m3 >= 0) and kSfRows rows
  std::vector<int2> entries;
  std::vector<SfBlock> blocks;
  for (int r = 0; r < nrows_; r += 2) {
    const KRow& k0 = rows[r];
    const KRow& k1 = rows[std::min(r + 1, nrows_ - 1)];
    for (int m3 = std::max(0, std::min(k0.m3lo, k1.m3lo)); m3 <= std::max(k0.m3hi, k1.m3hi); ++m3) {
      if (blocks.empty() || blocks.back().n_entries == kSfThreads || r + 1 - blocks.back().row0 >= kSfRows)
        blocks.push_back({(int)entries.size(), 0, r, 0});
      entries.push_back(make_int2(r, m3));
      blocks.back().n_entries += 1;
      blocks.back().n_rows = std::min(r + 2, nrows_) - blocks.back().row0;
    }
  }
  sf_rows_ = 0;
  for (const SfBlock& b : blocks) sf_rows_ = std::max(sf_rows_, b.n_rows);
  n_sf_ = (int)blocks.size();
  if ((e = cudaMalloc(&sf_blocks, sizeof(SfBlock) * std::max(1, n_sf_)))) return e;
  if ((e = cudaMalloc(&sf_entries, sizeof(int2) * std::max<size_t>(1, entries.size())))) return e;
  cudaMemcpy(sf_blocks, blocks.data(), sizeof(SfBlock) * blocks.size(), cudaMemcpyHostToDevice);
  cudaMemcpy(sf_entries, entries.data(), sizeof(int2) * entries.size(), cudaMemcpyHostToDevice);
  if ((e = cudaMalloc(&part, sizeof(double) * 2 * (size_t)std::max(1, nchunk_) * std::max(1LL, nk_)))) return e;
  if ((e = cudaMalloc(&ws, csz * 2 * (size_t)nk_))) return e;
  if ((e = cudaMalloc(&real_buf, sizeof(double) * 3 * N))) return e;
  if ((e = cudaMalloc(&recip_buf, sizeof(double) * 3 * N))) return e;
  if ((e = cudaMalloc(&rpart, sizeof(double) * 3 * (size_t)N * kRowChunks))) return e;
  if ((e = cudaMalloc(&scal, sizeof(double) * 4))) return e;
  const int ncell = g.nc[0] * g.nc[1] * g.nc[2];
  if ((e = cudaMalloc(&cell_of, sizeof(int) * N))) return e;
  if ((e = cudaMalloc(&cell_atoms, sizeof(int) * N))) return e;
  if ((e = cudaMalloc(&cell_raw, sizeof(int) * N))) return e;
  if ((e = cudaMalloc(&cell_count, sizeof(int) * ncell))) return e;
  if ((e = cudaMalloc(&cell_start, sizeof(int) * (ncell + 1)))) return e;
  if ((e = cudaMalloc(&pos_s, sizeof(double4) * N))) return e;
  return cudaSuccess;
}

// The dynamic shared-memory limit of a kernel is a process-wide attribute, while the size a
// launch needs depends on the context's k set: the limit only ever grows (largest request of
// any context so far), so a context never lowers it below what another one launches with.
static std::mutex g_smem_mutex;
static int g_smem[6] = {0, 0, 0, 0, 0, 0};

template <typename K>
static void raise_smem(K kernel, int slot, size_t bytes) {
  std::lock_guard<std::mutex> lock(g_smem_mutex);
  if ((int)bytes > g_smem[slot]) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    g_smem[slot] = (int)bytes;
  }
}

template <typename T>
static size_t sf_smem(int m3max, int rows) {
  return sizeof(typename C2<T>::t) * (rows * (kSfAtoms + 2) + (size_t)kSfAtoms * ((m3max + 1) | 1));
}
template <typename T>
static size_t recip_smem(int m3max, int tpb, int nv) {
  return sizeof(typename C2<T>::t) * ((size_t)(m3max + 1) * tpb + (size_t)(2 * m3max + 1) * 4 * nv);
}

cudaError_t Ewald::prepare(const double* dR, const int* dspecies, cudaStream_t s) {
  if (fp64_) {
    raise_smem(recip_atom_kernel<double, 0>, 0, recip_smem<double>(m3max_, 64, 1));
    raise_smem(recip_atom_kernel<double, 1>, 1, recip_smem<double>(m3max_, 64, 2));
    raise_smem(structure_factor_kernel<double>, 4, sf_smem<double>(m3max_, sf_rows_));
  } else {
    raise_smem(recip_atom_kernel<float, 0>, 2, recip_smem<float>(m3max_, 128, 1));
    raise_smem(recip_atom_kernel<float, 1>, 3, recip_smem<float>(m3max_, 128, 2));
    raise_smem(structure_factor_kernel<float>, 5, sf_smem<float>(m3max_, sf_rows_));
  }
  const int TB = 128, nb = (N_ + TB - 1) / TB;
  if (fp64_) phase_table_kernel<double><<<dim3(nb, 3), TB, 0, s>>>(dR, N_, g, reinterpret_cast<double2*>(tab));
  else phase_table_kernel<float><<<dim3(nb, 3), TB, 0, s>>>(dR, N_, g, reinterpret_cast<float2*>(tab));
  if (!g.brute) {
    // cell list on the device: counts, scan, stable fill with cell-relative coordinates
    const int ncell = g.nc[0] * g.nc[1] * g.nc[2];
    cudaMemsetAsync(cell_count, 0, sizeof(int) * ncell, s);
    cell_count_kernel<<<nb, TB, 0, s>>>(dR, N_, g, cell_of, cell_count);
    cell_scan_kernel<<<1, 1024, 0, s>>>(cell_count, ncell, cell_start);
    cudaMemsetAsync(cell_count, 0, sizeof(int) * ncell, s);
    cell_append_kernel<<<nb, TB, 0, s>>>(cell_of, N_, cell_start, cell_count, cell_raw);
    if (fp64_)
      cell_rank_kernel<double><<<dim3(ncell, 4), 256, 0, s>>>(dR, dspecies, g, cell_start, cell_raw, cell_atoms,
                                                              reinterpret_cast<double4*>(pos_s));
    else
      cell_rank_kernel<float><<<dim3(ncell, 4), 256, 0, s>>>(dR, dspecies, g, cell_start, cell_raw, cell_atoms,
                                                             reinterpret_cast<float4*>(pos_s));
  }
  sb_tag_ = 0;
  dR_ = dR;
  dspecies_ = dspecies;
  return cudaGetLastError();
}

// w S of the charges b into vector `vec` of ws
template <typename T>
static void run_sf(Ewald& E, const double* b, int vec, cudaStream_t s) {
  using CT = typename C2<T>::t;
  if (E.n_sf_ > 0)
    structure_factor_kernel<T><<<dim3(E.n_sf_, E.nchunk_), kSfThreads, sf_smem<T>(E.m3max_, E.sf_rows_), s>>>(
        E.sf_blocks, E.sf_entries, E.rows_d, E.nrows_, reinterpret_cast<const CT*>(E.tab), b, E.N_, E.g.nmax_all,
        E.m3max_, E.sf_rows_, Ewald::kChunk, E.part, E.nk_);
  sf_reduce_kernel<T><<<(int)((E.nk_ + 255) / 256), 256, 0, s>>>(E.part, E.nchunk_, E.nk_, E.wk_d,
                                                                 reinterpret_cast<CT*>(E.ws) + (size_t)vec * E.nk_);
}

template <typename T, int MODE>
static void run_real(Ewald& E, const double* a, const double* b, cudaStream_t s) {
  if (E.g.brute) {
    real_space_kernel<T, MODE><<<(32 * E.N_ + 127) / 128, 128, 0, s>>>(E.dR_, E.dspecies_, E.N_, E.g, E.cell_start,
                                                                      E.cell_count, E.cell_atoms, E.cell_of, a, b,
                                                                      E.real_buf);
  } else {
    real_cells_kernel<T, MODE><<<(E.N_ + 3) / 4, 128, 0, s>>>(
        reinterpret_cast<const typename Pos4<T>::t*>(E.pos_s), E.cell_atoms, E.cell_start, E.N_, E.g, a, b,
        E.real_buf);
  }
}

cudaError_t Ewald::potential(const double* b, double* V, cudaStream_t s, int tag) {
  const int TB = 128, nb = (N_ + TB - 1) / TB;
  if (fp64_) {
    run_sf<double>(*this, b, 0, s);
    run_real<double, 0>(*this, nullptr, b, s);
    const int tpb = 64;
    recip_atom_kernel<double, 0><<<dim3((N_ + tpb - 1) / tpb, kRowChunks), tpb, recip_smem<double>(m3max_, tpb, 1), s>>>(
        rows_d, nrows_, reinterpret_cast<const double2*>(tab), reinterpret_cast<const double2*>(ws), nk_, N_,
        g.nmax_all, m3max_, g, nullptr, nullptr, rpart);
    chunk_reduce_kernel<<<(N_ + 255) / 256, 256, 0, s>>>(rpart, kRowChunks, N_, recip_buf);
  } else {
    run_sf<float>(*this, b, 0, s);
    run_real<float, 0>(*this, nullptr, b, s);
    const int tpb = 128;
    recip_atom_kernel<float, 0><<<dim3((N_ + tpb - 1) / tpb, kRowChunks), tpb, recip_smem<float>(m3max_, tpb, 1), s>>>(
        rows_d, nrows_, reinterpret_cast<const float2*>(tab), reinterpret_cast<const float2*>(ws), nk_, N_,
        g.nmax_all, m3max_, g, nullptr, nullptr, rpart);
    chunk_reduce_kernel<<<(N_ + 255) / 256, 256, 0, s>>>(rpart, kRowChunks, N_, recip_buf);
  }
  sb_tag_ = tag;
  sum_kernel<<<1, 1024, 0, s>>>(b, N_, scal);
  combine_pot_kernel<<<nb, TB, 0, s>>>(real_buf, recip_buf, b, dspecies_, g, scal, V, N_);
  return cudaGetLastError();
}

cudaError_t Ewald::gradient(const double* a, const double* b, double* G, cudaStream_t s, int tag) {
  // vector 0 = b (S_b), vector 1 = a (S_a); S_b is kept from the potential call with the same
  // nonzero tag (same charges at the same geometry)
  const bool reuse = tag != 0 && tag == sb_tag_;
  if (fp64_) {
    if (!reuse) run_sf<double>(*this, b, 0, s);
    run_sf<double>(*this, a, 1, s);
    run_real<double, 1>(*this, a, b, s);
    const int tpb = 64;
    recip_atom_kernel<double, 1><<<dim3((N_ + tpb - 1) / tpb, kRowChunks), tpb, recip_smem<double>(m3max_, tpb, 2), s>>>(
        rows_d, nrows_, reinterpret_cast<const double2*>(tab), reinterpret_cast<const double2*>(ws), nk_, N_,
        g.nmax_all, m3max_, g, a, b, rpart);
    chunk_reduce_kernel<<<(3 * N_ + 255) / 256, 256, 0, s>>>(rpart, kRowChunks, 3LL * N_, recip_buf);
  } else {
    if (!reuse) run_sf<float>(*this, b, 0, s);
    run_sf<float>(*this, a, 1, s);
    run_real<float, 1>(*this, a, b, s);
    const int tpb = 128;
    recip_atom_kernel<float, 1><<<dim3((N_ + tpb - 1) / tpb, kRowChunks), tpb, recip_smem<float>(m3max_, tpb, 2), s>>>(
        rows_d, nrows_, reinterpret_cast<const float2*>(tab), reinterpret_cast<const float2*>(ws), nk_, N_,
        g.nmax_all, m3max_, g, a, b, rpart);
    chunk_reduce_kernel<<<(3 * N_ + 255) / 256, 256, 0, s>>>(rpart, kRowChunks, 3LL * N_, recip_buf);
  }
  combine_grad_kernel<<<(3 * N_ + 255) / 256, 256, 0, s>>>(real_buf, recip_buf, G, N_, 1.0 / kBohrA);
  return cudaGetLastError();
}

}  // namespace sedacs
