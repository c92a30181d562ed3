// Learned charge-response preconditioner on the GPU: a message-passing network on the atom
// graph, linear in the residual y, K_NN(y) = -c y + G(y):
//   h0_i = y_i e[s_i];  a_i = sum_j phi_l(r_ij) * h_j;  h_i <- h_i + A_l a_i + B_l h_i  (3 layers)
//   G(y)_i = w . h3_i;  phi_l(r) = sum_b C_l[b] exp(-((r - m_b)/0.7)^2) (cos(pi r/6) + 1)/2  (r < 6 A)
// 64 channels, FP32.  Forward, backward (parameter gradients with fixed-order reductions)
// and Adam are hand-written kernels; training pairs (x = J v, v) come from the Krylov kernel
// (SI Sec. B).  Parameter order: e[3][64], then per layer C[8][64], A[64][64], B[64][64], then w[64].
#include <cmath>
#include <vector>

#include "engine.cuh"

namespace sedacs {

namespace {

constexpr int W = 64, NB = 8, NL = 3;
constexpr int kParams = 3 * W + NL * (NB * W + 2 * W * W) + W;
constexpr int kPart = 2 * W * W + NB * W;           // gradient parts of one block and layer: dA, dB, dC
constexpr float kRcut = 6.0f, kSig = 0.7f;

__host__ __device__ inline int off_e() { return 0; }
__host__ __device__ inline int off_C(int l) { return 3 * W + l * (NB * W + 2 * W * W); }
__host__ __device__ inline int off_A(int l) { return off_C(l) + NB * W; }
__host__ __device__ inline int off_B(int l) { return off_A(l) + W * W; }
__host__ __device__ inline int off_w() { return 3 * W + NL * (NB * W + 2 * W * W); }

// per edge (CSR order): r and the 8 radial basis values with the cosine cutoff
__global__ void edge_basis_kernel(const double* R, const long long* row_ptr, const int* col, int N, double bx,
                                  double by, double bz, float* ebas) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= N) return;
  const double box[3] = {bx, by, bz};
  for (long long p = row_ptr[i] + lane; p < row_ptr[i + 1]; p += 32) {
    const int j = col[p];
    double d2 = 0.0;
    for (int a = 0; a < 3; ++a) {
      double d = R[3 * j + a] - R[3 * i + a];
      d -= box[a] * rint(d / box[a]);
      d2 += d * d;
    }
    const float r = (float)sqrt(d2);
    const float fc = r < kRcut ? 0.5f * (cosf(3.14159265358979f * r / kRcut) + 1.0f) : 0.0f;
    for (int b = 0; b < NB; ++b) {
      const float m = 0.8f + (6.0f - 0.8f) * b / (NB - 1);
      const float t = (r - m) / kSig;
      ebas[p * NB + b] = expf(-t * t) * fc;
    }
  }
}

__global__ void embed_kernel(const double* y, const int* species, const float* P, float* h0, int N) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)N * W) return;
  const int i = (int)(t / W), c = (int)(t % W);
  h0[t] = (float)y[i] * P[off_e() + species[i] * W + c];
}

// ---- layer kernels: a block takes kTile atoms, eight warps -----------------------------------------
// The per-atom work is a sum over about 30 edges with ten loads each (latency) and two 64 x 64 mixes, so a
// block gathers its atoms' sums warp by warp into shared memory and mixes them from there, with both
// matrices in shared memory: one launch and one pass over the activations per layer and direction.
// Measured (GB300, 9,000 atoms, 27 edges each), an application and a parameter gradient: 0.83 ms in all, against
// 2.44 ms with one kernel per step, of which 1.75 ms went to the filter gradient on 141 blocks of two warps and
// 0.35 ms to mixes that read the matrices by columns.
constexpr int kTile = 32, kWarps = 8;
constexpr int kPitch = W + 1;                       // transposed matrices: conflict-free on both sides

// Sum over the edges of atom i of phi(r) x[col][c], phi = sum_b e_b C[b][c], for two channels (lane, lane + 32).
// Four edges in flight.
__device__ __forceinline__ void edge_sum(const float* __restrict__ x, const long long* __restrict__ row_ptr,
                                         const int* __restrict__ col, const float* __restrict__ ebas, int i, int lane,
                                         const float (&c0)[NB], const float (&c1)[NB], float& s0, float& s1) {
  s0 = s1 = 0.f;
  const long long p1 = row_ptr[i + 1];
#pragma unroll 4
  for (long long p = row_ptr[i]; p < p1; ++p) {
    const float* xj = x + (long long)col[p] * W;
    const float4 e0 = *reinterpret_cast<const float4*>(ebas + p * NB), e1 = *reinterpret_cast<const float4*>(ebas + p * NB + 4);
    const float h0 = xj[lane], h1 = xj[lane + 32];
    const float e[NB] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
    float f0 = 0.f, f1 = 0.f;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      f0 = fmaf(e[b], c0[b], f0);
      f1 = fmaf(e[b], c1[b], f1);
    }
    s0 = fmaf(f0, h0, s0);
    s1 = fmaf(f1, h1, s1);
  }
}

// Sums over the edges of atom i of e_b x[col][c], two channels (lane, lane + 32) and all b.
__device__ __forceinline__ void edge_moments(const float* __restrict__ x, const long long* __restrict__ row_ptr,
                                             const int* __restrict__ col, const float* __restrict__ ebas, int i, int lane,
                                             float (&m)[NB], float (&n)[NB]) {
#pragma unroll
  for (int b = 0; b < NB; ++b) m[b] = n[b] = 0.f;
  const long long p1 = row_ptr[i + 1];
#pragma unroll 4
  for (long long p = row_ptr[i]; p < p1; ++p) {
    const float* xj = x + (long long)col[p] * W;
    const float4 e0 = *reinterpret_cast<const float4*>(ebas + p * NB), e1 = *reinterpret_cast<const float4*>(ebas + p * NB + 4);
    const float h0 = xj[lane], h1 = xj[lane + 32];
    const float e[NB] = {e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      m[b] = fmaf(e[b], h0, m[b]);
      n[b] = fmaf(e[b], h1, n[b]);
    }
  }
}

// dst[k][c] (pitch kPitch) = M[c][k] (trans 0) or M[k][c] (trans 1)
__device__ __forceinline__ void load_matrix(float* dst, const float* M, int trans) {
  for (int t = threadIdx.x; t < W * W; t += blockDim.x) {
    const int r = t / W, q = t % W;
    dst[trans ? r * kPitch + q : q * kPitch + r] = M[t];
  }
}

// acc[q] += sum_k M[k][c] x[8 g + q][k] for this thread's channel c = tid % 64 and atoms 8 g .. (g = tid / 64)
__device__ __forceinline__ void mix8(const float* M, const float* x, float (&acc)[8]) {
  const int c = threadIdx.x & 63, g = threadIdx.x >> 6;
#pragma unroll 4
  for (int k = 0; k < W; k += 4) {
    const float m0 = M[k * kPitch + c], m1 = M[(k + 1) * kPitch + c], m2 = M[(k + 2) * kPitch + c],
                m3 = M[(k + 3) * kPitch + c];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(x + (8 * g + q) * W + k);
      acc[q] = fmaf(m0, v.x, fmaf(m1, v.y, fmaf(m2, v.z, fmaf(m3, v.w, acc[q]))));
    }
  }
}

// One layer: a_i = sum_j phi(r_ij) * h_j (kept for the backward pass), out = h + A a + B h.  The two mixes are summed
// from zero and h comes last: they are a tenth of h, and 128 sums on top of h would round at its size each.
__global__ void __launch_bounds__(256) layer_fwd_kernel(const float* h, const float* P, int l, const long long* row_ptr,
                                                        const int* col, const float* ebas, int N, float* a, float* out) {
  extern __shared__ float sm[];
  float *sA = sm, *sB = sA + W * kPitch, *sa = sB + W * kPitch, *sh = sa + kTile * W;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, i0 = blockIdx.x * kTile;
  load_matrix(sA, P + off_A(l), 0);
  load_matrix(sB, P + off_B(l), 0);
  const float* C = P + off_C(l);
  float c0[NB], c1[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) { c0[b] = C[b * W + lane]; c1[b] = C[b * W + lane + 32]; }
  for (int q = warp; q < kTile; q += kWarps) {
    const int i = i0 + q;
    float s0 = 0.f, s1 = 0.f, h0 = 0.f, h1 = 0.f;
    if (i < N) {
      edge_sum(h, row_ptr, col, ebas, i, lane, c0, c1, s0, s1);
      h0 = h[(long long)i * W + lane];
      h1 = h[(long long)i * W + lane + 32];
      a[(long long)i * W + lane] = s0;
      a[(long long)i * W + lane + 32] = s1;
    }
    sa[q * W + lane] = s0;
    sa[q * W + lane + 32] = s1;
    sh[q * W + lane] = h0;
    sh[q * W + lane + 32] = h1;
  }
  __syncthreads();
  const int c = threadIdx.x & 63, g = threadIdx.x >> 6;
  float ma[8], mb[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) ma[q] = mb[q] = 0.f;
  mix8(sA, sa, ma);
  mix8(sB, sh, mb);
  for (int q = 0; q < 8; ++q)
    if (i0 + 8 * g + q < N) out[(long long)(i0 + 8 * g + q) * W + c] = sh[(8 * g + q) * W + c] + (ma[q] + mb[q]);
}

// Backward through the mixes of a layer: ga = A^T gh, base = gh + B^T gh (gh last, as h above), and this block's part of
// dA = sum gh a^T, dB = sum gh h^T (part[blk][0 .. W W) and [W W .. 2 W W)).
__global__ void __launch_bounds__(256) mix_bwd_kernel(const float* gh, const float* a, const float* h, const float* P, int l,
                                                      int N, float* ga, float* base, float* part) {
  extern __shared__ float sm[];
  float *sA = sm, *sB = sA + W * kPitch, *sg = sB + W * kPitch, *sa = sg + kTile * W, *sh = sa + kTile * W;
  const int i0 = blockIdx.x * kTile, n = min(kTile, N - i0);
  load_matrix(sA, P + off_A(l), 1);
  load_matrix(sB, P + off_B(l), 1);
  for (int t = threadIdx.x; t < kTile * W; t += blockDim.x) {
    const bool in = t < n * W;
    const long long at = (long long)i0 * W + t;
    sg[t] = in ? gh[at] : 0.f;
    sa[t] = in ? a[at] : 0.f;
    sh[t] = in ? h[at] : 0.f;
  }
  __syncthreads();
  const int c = threadIdx.x & 63, g = threadIdx.x >> 6;
  float acc[8], bas[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) acc[q] = bas[q] = 0.f;
  mix8(sA, sg, acc);
  mix8(sB, sg, bas);
  for (int q = 0; q < 8; ++q)
    if (8 * g + q < n) {
      ga[(long long)(i0 + 8 * g + q) * W + c] = acc[q];
      base[(long long)(i0 + 8 * g + q) * W + c] = sg[(8 * g + q) * W + c] + bas[q];
    }
  // outer products: thread (row block of four channels, column block of four) over both matrices
  const int r4 = (threadIdx.x >> 4) * 4, k4 = (threadIdx.x & 15) * 4;
  float oa[4][4] = {}, ob[4][4] = {};
  for (int q = 0; q < n; ++q) {
    const float4 x = *reinterpret_cast<const float4*>(sg + q * W + r4);
    const float4 y = *reinterpret_cast<const float4*>(sa + q * W + k4), z = *reinterpret_cast<const float4*>(sh + q * W + k4);
    const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w}, zv[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        oa[u][v] = fmaf(xv[u], yv[v], oa[u][v]);
        ob[u][v] = fmaf(xv[u], zv[v], ob[u][v]);
      }
  }
  float* pb = part + (long long)blockIdx.x * kPart;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    *reinterpret_cast<float4*>(pb + (r4 + u) * W + k4) = make_float4(oa[u][0], oa[u][1], oa[u][2], oa[u][3]);
    *reinterpret_cast<float4*>(pb + W * W + (r4 + u) * W + k4) = make_float4(ob[u][0], ob[u][1], ob[u][2], ob[u][3]);
  }
}

// Backward through the aggregation: gout_i = base_i + sum_j phi(r_ij) * ga_j (the graph and the filter are
// symmetric, so its transpose is itself), and this block's part of dC[b][c] = sum_i ga_i[c] sum_j e_b h_j[c]
// (part[blk][2 W W ..)).
__global__ void __launch_bounds__(256) aggregate_bwd_kernel(const float* ga, const float* h, const float* base, const float* P,
                                                            int l, const long long* row_ptr, const int* col,
                                                            const float* ebas, int N, float* gout, float* part) {
  __shared__ float red[kWarps][NB * W];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, i0 = blockIdx.x * kTile;
  const float* C = P + off_C(l);
  float c0[NB], c1[NB], d0[NB], d1[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    c0[b] = C[b * W + lane];
    c1[b] = C[b * W + lane + 32];
    d0[b] = d1[b] = 0.f;
  }
  for (int q = warp; q < kTile; q += kWarps) {
    const int i = i0 + q;
    if (i >= N) break;
    float m[NB], n[NB], s0, s1;
    edge_sum(ga, row_ptr, col, ebas, i, lane, c0, c1, s0, s1);
    const long long at = (long long)i * W + lane;
    gout[at] = base[at] + s0;
    gout[at + 32] = base[at + 32] + s1;
    edge_moments(h, row_ptr, col, ebas, i, lane, m, n);
    const float g0 = ga[at], g1 = ga[at + 32];
#pragma unroll
    for (int b = 0; b < NB; ++b) { d0[b] = fmaf(g0, m[b], d0[b]); d1[b] = fmaf(g1, n[b], d1[b]); }
  }
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    red[warp][b * W + lane] = d0[b];
    red[warp][b * W + lane + 32] = d1[b];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < NB * W; t += blockDim.x) {
    float s = 0.f;
    for (int w = 0; w < kWarps; ++w) s += red[w][t];
    part[(long long)blockIdx.x * kPart + 2 * W * W + t] = s;
  }
}

__global__ void output_kernel(const double* y, const float* h3, const float* P, double c_k0, int N, double* u) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= N) return;
  const float* w = P + off_w();
  float s = h3[(long long)i * W + lane] * w[lane] + h3[(long long)i * W + lane + 32] * w[lane + 32];
  s = warp_sumf(s);
  if (lane == 0) u[i] = -c_k0 * y[i] + (double)s;
}

// gh3_i[c] = gu_i w_c
__global__ void out_bwd_kernel(const double* gu, const float* P, int N, float* gh) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= (long long)N * W) return;
  gh[t] = (float)gu[t / W] * P[off_w() + (int)(t % W)];
}

// part[blk][c] = sum_i g_i gu_i * h_i[c] ... generic: part[blk][c] = sum_i x_i[c] * s_i (s optional -> 1)
__global__ void vec_partial_kernel(const float* x, const double* s, int N, int chunk, float* part) {
  const int i0 = blockIdx.x * chunk, i1 = min(N, i0 + chunk);
  const int c = threadIdx.x;
  float acc = 0.f;
  for (int i = i0; i < i1; ++i) acc += x[(long long)i * W + c] * (s ? (float)s[i] : 1.f);
  part[blockIdx.x * W + c] = acc;
}

// species embedding gradient partials: part[blk][s*W + c] = sum_{i in chunk, s_i = s} gh0_i[c] y_i
__global__ void embed_bwd_partial_kernel(const float* gh, const double* y, const int* species, int N, int chunk,
                                         float* part) {
  const int i0 = blockIdx.x * chunk, i1 = min(N, i0 + chunk);
  const int c = threadIdx.x;
  float acc[3] = {0.f, 0.f, 0.f};
  for (int i = i0; i < i1; ++i) acc[species[i]] += gh[(long long)i * W + c] * (float)y[i];
  for (int s = 0; s < 3; ++s) part[blockIdx.x * 3 * W + s * W + c] = acc[s];
}

// out[e] += sum over blocks of part[blk][e], e < len, row length pitch: a block takes 32 elements, its eight warps
// every eighth row, in FP64; the warps' sums are added in a fixed order.  The elements of one layer (dA, dB, dC) go to
// their places in the gradient through off[0 .. 2] (segments of W W, W W and the rest), other sums to off[0].
struct GradOff {
  int o[3];
};
__global__ void __launch_bounds__(256) reduce_parts_kernel(const float* part, int nblk, int len, int pitch, float* grad,
                                                           GradOff off) {
  __shared__ double red[kWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, e = blockIdx.x * 32 + lane;
  double s = 0.0;
  if (e < len) {
#pragma unroll 8
    for (int b = warp; b < nblk; b += kWarps) s += (double)part[(long long)b * pitch + e];
  }
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && e < len) {
    for (int w = 1; w < kWarps; ++w) s += red[w][lane];
    const int seg = len > 2 * W * W ? min(e / (W * W), 2) : 0;
    grad[off.o[seg] + e - seg * (W * W)] += (float)s;
  }
}

__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int n, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  m[t] = b1 * m[t] + (1.f - b1) * g[t];
  v[t] = b2 * v[t] + (1.f - b2) * g[t] * g[t];
  p[t] -= lr * (m[t] / c1) / (sqrtf(v[t] / c2) + eps);
}

__global__ void residual_kernel(const double* u, const double* v, int N, double scale, double* gu, double* acc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) gu[i] = scale * (u[i] - v[i]);
  (void)acc;
}

__global__ void f2d_kernel(const float* x, double* y, long long n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < n) y[t] = (double)x[t];
}
__global__ void d2f_kernel(const double* x, float* y, long long n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < n) y[t] = (float)x[t];
}

inline int nb(long long n, int tb) { return (int)((n + tb - 1) / tb); }

}  // namespace

int gnn_num_params() { return kParams; }
void dev_dot_into(sedacs_ctx* ctx, const double* a, const double* b, double* out);

// Parameter, moment and activation buffers (allocated once).
cudaError_t gnn_prepare_params(sedacs_ctx* ctx) {
  GnnState& G = ctx->gnn;
  cudaError_t e;
  const int N = ctx->N;
  if (!G.P) {
    if ((e = cudaMalloc(&G.P, sizeof(float) * kParams))) return e;
    if ((e = cudaMalloc(&G.grad, sizeof(float) * kParams))) return e;
    if ((e = cudaMalloc(&G.m, sizeof(float) * kParams))) return e;
    if ((e = cudaMalloc(&G.v, sizeof(float) * kParams))) return e;
    cudaMemset(G.P, 0, sizeof(float) * kParams);
    cudaMemset(G.m, 0, sizeof(float) * kParams);
    cudaMemset(G.v, 0, sizeof(float) * kParams);
    if ((e = cudaMalloc(&G.act, sizeof(float) * (size_t)N * W * (2 * NL + 4)))) return e;
    G.nchunk = (N + kTile - 1) / kTile;
    if ((e = cudaMalloc(&G.part, sizeof(float) * (size_t)G.nchunk * kPart))) return e;
    if ((e = cudaMalloc(&G.p64, sizeof(double) * kParams))) return e;
    if ((e = cudaMalloc(&G.gu, sizeof(double) * N))) return e;
    if ((e = cudaMalloc(&G.u, sizeof(double) * N))) return e;
  }
  return cudaSuccess;
}

// Edge basis of the current graph (and the buffers above).
cudaError_t gnn_prepare(sedacs_ctx* ctx) {
  GnnState& G = ctx->gnn;
  cudaError_t e;
  const int N = ctx->N;
  if ((e = gnn_prepare_params(ctx))) return e;
  if (ctx->nnz * NB > G.ebas_cap) {
    if (G.ebas) cudaFree(G.ebas);
    G.ebas_cap = ctx->nnz * NB + ctx->nnz * NB / 4 + 1024;
    if ((e = cudaMalloc(&G.ebas, sizeof(float) * G.ebas_cap))) return e;
  }
  edge_basis_kernel<<<nb(32LL * N, 128), 128, 0, ctx->stream>>>(ctx->d_R, ctx->d_row_ptr, ctx->d_col, N, ctx->box[0],
                                                                ctx->box[1], ctx->box[2], G.ebas);
  ctx->launches += 1;
  return cudaGetLastError();
}

// activations layout: h[0..NL] then a[0..NL-1], then two gradient buffers
static float* act(sedacs_ctx* ctx, int k) { return ctx->gnn.act + (size_t)k * ctx->N * W; }

// dynamic shared memory: two padded matrices and two (forward) or three (backward) tiles of activations
constexpr int kFwdSmem = (2 * W * kPitch + 2 * kTile * W) * 4, kBwdSmem = (2 * W * kPitch + 3 * kTile * W) * 4;

void gnn_forward(sedacs_ctx* ctx, const double* y, double* u) {
  const int N = ctx->N;
  cudaStream_t s = ctx->stream;
  GnnState& G = ctx->gnn;
  cudaFuncSetAttribute(layer_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem);
  embed_kernel<<<nb((long long)N * W, 256), 256, 0, s>>>(y, ctx->d_species, G.P, act(ctx, 0), N);
  for (int l = 0; l < NL; ++l)
    layer_fwd_kernel<<<G.nchunk, 256, kFwdSmem, s>>>(act(ctx, l), G.P, l, ctx->d_row_ptr, ctx->d_col, G.ebas, N,
                                                     act(ctx, NL + 1 + l), act(ctx, l + 1));
  output_kernel<<<nb(32LL * N, 128), 128, 0, s>>>(y, act(ctx, NL), G.P, ctx->prm.c_k0, N, u);
  ctx->launches += 2 + NL;
}

// grad += d/dP sum_i gu_i K_NN(y)_i  (forward activations must be current)
void gnn_backward(sedacs_ctx* ctx, const double* y, const double* gu) {
  const int N = ctx->N;
  cudaStream_t s = ctx->stream;
  GnnState& G = ctx->gnn;
  cudaFuncSetAttribute(mix_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBwdSmem);
  float* gh = act(ctx, 2 * NL + 1);
  float* tmp = act(ctx, 2 * NL + 2);
  float* base = act(ctx, 2 * NL + 3);
  out_bwd_kernel<<<nb((long long)N * W, 256), 256, 0, s>>>(gu, G.P, N, gh);
  vec_partial_kernel<<<G.nchunk, W, 0, s>>>(act(ctx, NL), gu, N, kTile, G.part);
  reduce_parts_kernel<<<nb(W, 32), 256, 0, s>>>(G.part, G.nchunk, W, W, G.grad, GradOff{{off_w(), 0, 0}});
  for (int l = NL - 1; l >= 0; --l) {
    float* h = act(ctx, l);
    mix_bwd_kernel<<<G.nchunk, 256, kBwdSmem, s>>>(gh, act(ctx, NL + 1 + l), h, G.P, l, N, tmp, base, G.part);
    aggregate_bwd_kernel<<<G.nchunk, 256, 0, s>>>(tmp, h, base, G.P, l, ctx->d_row_ptr, ctx->d_col, G.ebas, N, gh, G.part);
    reduce_parts_kernel<<<nb(kPart, 32), 256, 0, s>>>(G.part, G.nchunk, kPart, kPart, G.grad,
                                                      GradOff{{off_A(l), off_B(l), off_C(l)}});
  }
  embed_bwd_partial_kernel<<<G.nchunk, W, 0, s>>>(gh, y, ctx->d_species, N, kTile, G.part);
  reduce_parts_kernel<<<nb(3 * W, 32), 256, 0, s>>>(G.part, G.nchunk, 3 * W, 3 * W, G.grad, GradOff{{off_e(), 0, 0}});
  ctx->launches += 5 + 3 * NL;
}

void gnn_adam(sedacs_ctx* ctx, float lr) {
  GnnState& G = ctx->gnn;
  G.t += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  adam_kernel<<<nb(kParams, 256), 256, 0, ctx->stream>>>(G.P, G.grad, G.m, G.v, kParams, lr, b1, b2, 1e-8f,
                                                        1.f - powf(b1, (float)G.t), 1.f - powf(b2, (float)G.t));
  ctx->launches += 1;
}

void gnn_zero_grad(sedacs_ctx* ctx) { cudaMemsetAsync(ctx->gnn.grad, 0, sizeof(float) * kParams, ctx->stream); }

void gnn_set_params_f64(sedacs_ctx* ctx, const double* d_p) {
  d2f_kernel<<<nb(kParams, 256), 256, 0, ctx->stream>>>(d_p, ctx->gnn.P, kParams);
}
void gnn_get_params_f64(sedacs_ctx* ctx, double* d_p, bool grad) {
  f2d_kernel<<<nb(kParams, 256), 256, 0, ctx->stream>>>(grad ? ctx->gnn.grad : ctx->gnn.P, d_p, kParams);
}

// one Adam step on the mean squared error over n pairs (x_k, v_k), each an N-vector in device
// memory; the loss is read back (one sync per pair) only when want_loss
double gnn_train_step(sedacs_ctx* ctx, const double* X, const double* V, int n, float lr, bool want_loss) {
  const int N = ctx->N;
  cudaStream_t s = ctx->stream;
  GnnState& G = ctx->gnn;
  gnn_zero_grad(ctx);
  std::vector<double> losses(n);
  double* lbuf = ctx->d_scal + 12;
  double loss = 0.0;
  for (int k = 0; k < n; ++k) {
    const double* x = X + (size_t)k * N;
    const double* v = V + (size_t)k * N;
    gnn_forward(ctx, x, G.u);
    residual_kernel<<<nb(N, 256), 256, 0, s>>>(G.u, v, N, 2.0 / n, G.gu, nullptr);
    gnn_backward(ctx, x, G.gu);
    if (!want_loss) continue;
    // loss: sum (u - v)^2 / n  = sum gu^2 * n / 4
    dev_dot_into(ctx, G.gu, G.gu, lbuf);
    double l = 0.0;
    cudaMemcpyAsync(&l, lbuf, sizeof(double), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    loss += l * n / 4.0;
  }
  gnn_adam(ctx, lr);
  return loss / n;
}

}  // namespace sedacs
