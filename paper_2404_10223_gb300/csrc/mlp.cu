// Rotation-proposal network (include/tnqe_mlp.h): forward, backward and Adam
// kernels in FP32 on CUDA cores.  The network is small (tens of thousands of
// parameters, batches of a few thousand rows): a gradient is 0.3 GFLOP at batch 512,
// 4 us of the FP32 rate, so launches and latency bound it.  Seven launches: the GELU
// and its derivative, the loss and the bias gradients are in the epilogues and
// operand loads of the products, the three weight gradients are one launch, cut along
// the batch until the GPU is filled, and one launch adds the cuts in a fixed order.
// (Separate kernels with 16 x 16 tiles, uncut weight gradients and one thread per bias
// sum: 17 launches.)  Adam step of 74-256-66, copies and host included: 149 -> 90 us at
// batch 16, 296 -> 112 at 512, 1421 -> 250 at 4096; at 512 the kernels are 45 us of it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <stdexcept>
#include <string>
#include <vector>

#include "../../include/tnqe_mlp.h"

namespace {

constexpr int GT = 32;         // GEMM tile edge
constexpr int GK = 32;         // depth of a staged slab
constexpr int GS = GT + 4;     // row stride in shared memory (16-byte rows)
constexpr int GTHREADS = 128;  // a thread computes 2 x 4 entries
constexpr int GST = 4;         // slabs in flight

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

struct Tile {
  float As[GST][GK][GS], Bs[GST][GK][GS];
};

// Entry i of a thread's share of a slab: row r and depth k.  Along k a warp takes 8 depths of 4 rows (whole
// sectors of memory, and 32 banks with the stride of 36 words); along the rows 32 rows of one depth.
__device__ __forceinline__ void slab_entry(int i, bool kmajor, int& r, int& k) {
  const int lane = threadIdx.x & 31, w = (threadIdx.x >> 5) + i * (GTHREADS / 32);
  r = kmajor ? (lane >> 3) + 4 * (w >> 2) : lane;
  k = kmajor ? (lane & 7) + 8 * (w & 3) : w;
}
// Copies one slab of an operand, asynchronously: entries (row r0 + r, k0 + k), r, k < 32, of a matrix with
// unit stride along k (kmajor) or along the rows; zero outside rows x kend.  Words of 4 bytes: the
// layouts have no alignment beyond that, and the slab is transposed on the way.
__device__ __forceinline__ void copy_slab(float (*S)[GS], const float* __restrict__ P, int ld, bool kmajor, int rows,
                                          int r0, int k0, int kend) {
#pragma unroll
  for (int i = 0; i < GT * GK / GTHREADS; ++i) {
    int r, k;
    slab_entry(i, kmajor, r, k);
    const bool in = r0 + r < rows && k0 + k < kend;
    const float* src = !in ? P : (kmajor ? P + (long long)(r0 + r) * ld + k0 + k : P + (long long)(k0 + k) * ld + r0 + r);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(&S[k][r])),
                 "l"(src), "r"(in ? 4 : 0) : "memory");
  }
}

// acc[i][j] = sum over k in [k0, k1) of A(m, k) B(n, k) for the thread's rows m0 + 2 ty + i and columns
// n0 + 4 tx + j; colsum[i] (if wanted) the sum of A(m, k).  32 x 32 tiles: the products of a
// batch of 512 are 40 to 128 tiles, which a larger tile would leave on a fraction of the
// SMs.  With one warp per scheduler the chain of slab loads is the time, so three are in
// flight while one is multiplied.
__device__ __forceinline__ void tile_product(Tile& S, const float* A, int lda, bool ak, int M, const float* B, int ldb,
                                             bool bk, int N, int m0, int n0, int k0, int k1, float (&acc)[2][4],
                                             float (&colsum)[2]) {
  const int tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    colsum[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  }
  auto copy = [&](int buf, int k) {                // one group per slab, empty beyond the last
    if (k < k1) {
      copy_slab(S.As[buf], A, lda, ak, M, m0, k, k1);
      copy_slab(S.Bs[buf], B, ldb, bk, N, n0, k, k1);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < GST - 1; ++s) copy(s, k0 + s * GK);
  int buf = 0;
  for (int k = k0; k < k1; k += GK, buf = (buf + 1) % GST) {
    asm volatile("cp.async.wait_group %0;" ::"n"(GST - 2) : "memory");
    __syncthreads();                               // the slab has arrived, and the one before is read
    copy((buf + GST - 1) % GST, k + (GST - 1) * GK);
#pragma unroll 8
    for (int kk = 0; kk < GK; ++kk) {
      const float2 a = *reinterpret_cast<const float2*>(&S.As[buf][kk][2 * ty]);
      const float4 b = *reinterpret_cast<const float4*>(&S.Bs[buf][kk][4 * tx]);
      const float av[2] = {a.x, a.y}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        colsum[i] += av[i];
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
      }
    }
  }
}

// One layer: Z = A W^T + bias (A: B x K, W: N x K).  LAST 0: Z and gelu(Z) are written; 1: Z alone;
// 2: Z, dZ = 2 w (Z - T) / (N sum w), and the block's share of the loss in lossp.
template <int LAST>
__global__ void __launch_bounds__(GTHREADS) layer_kernel(const float* __restrict__ A, const float* __restrict__ W,
                                                         const float* __restrict__ bias, float* __restrict__ Z,
                                                         float* __restrict__ G, int B, int N, int K,
                                                         const float* __restrict__ T, const float* __restrict__ w,
                                                         float* __restrict__ lossp) {
  __shared__ Tile S;
  __shared__ float red[GTHREADS / 32];
  const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT, tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  float acc[2][4], cs[2];
  tile_product(S, A, K, true, B, W, K, true, N, m0, n0, 0, K, acc, cs);
  float scale = 0.f, loss = 0.f;
  if (LAST == 2) {                                 // every block sums the weights (in the same order)
    float s = 0.f;
    for (int i = threadIdx.x; i < B; i += GTHREADS) s += w ? w[i] : 1.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    s = 0.f;
#pragma unroll
    for (int i = 0; i < GTHREADS / 32; ++i) s += red[i];
    __syncthreads();
    scale = 1.f / (s * (float)N);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = m0 + 2 * ty + i;
    if (m >= B) continue;
    const float wb = LAST == 2 ? (w ? w[m] : 1.f) : 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n >= N) continue;
      const long long x = (long long)m * N + n;
      const float z = acc[i][j] + bias[n];
      Z[x] = z;
      if (LAST == 0) G[x] = gelu_f(z);
      if (LAST == 2) {
        const float r = z - T[x];
        G[x] = 2.f * wb * r * scale;
        loss += wb * r * r;
      }
    }
  }
  if (LAST == 2) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
      float s = 0.f;
      for (int i = 0; i < GTHREADS / 32; ++i) s += red[i];
      lossp[blockIdx.y * gridDim.x + blockIdx.x] = s * scale;
    }
  }
}

// dZ_prev = (dZ W) gelu'(Z_prev) (dZ: B x K, W: K x N)
__global__ void __launch_bounds__(GTHREADS) back_kernel(const float* __restrict__ dZ, const float* __restrict__ W,
                                                        const float* __restrict__ Z, float* __restrict__ out, int B,
                                                        int N, int K) {
  __shared__ Tile S;
  const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT, tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  float acc[2][4], cs[2];
  tile_product(S, dZ, K, true, B, W, N, false, N, m0, n0, 0, K, acc, cs);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = m0 + 2 * ty + i;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (m < B && n < N) out[(long long)m * N + n] = acc[i][j] * gelu_grad(Z[(long long)m * N + n]);
    }
  }
}

// (Three launches of 16 x 16 tiles, each over the whole batch, and three of bias sums took 40-46 us and 31 us
// each at batch 512; this one and the reduction take 11 + 4.)
// Weight and bias gradients of the three layers, cut number blockIdx.y of the batch: dW = dZ^T A (M x N), db
// the column sums of dZ, into slice blockIdx.y of the partial gradients.
struct GradLayer {
  const float* dZ;
  const float* A;
  long long oW, ob;
  int M, N, tiles_n, first;      // first tile of the layer in blockIdx.x
};
struct GradLayers {
  GradLayer l[3];
};
__global__ void __launch_bounds__(GTHREADS) grad_kernel(const GradLayers L, int B, int cut, long long count,
                                                        float* __restrict__ part) {
  __shared__ Tile S;
  int q = 2;
  while (q > 0 && (int)blockIdx.x < L.l[q].first) --q;
  const GradLayer& l = L.l[q];
  const int t = blockIdx.x - l.first, m0 = (t / l.tiles_n) * GT, n0 = (t % l.tiles_n) * GT;
  const int k0 = blockIdx.y * cut, k1 = min(B, k0 + cut), tx = threadIdx.x & 7, ty = threadIdx.x >> 3;
  float acc[2][4], cs[2];
  tile_product(S, l.dZ, l.M, false, l.M, l.A, l.N, false, l.N, m0, n0, k0, k1, acc, cs);
  float* out = part + (long long)blockIdx.y * count;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = m0 + 2 * ty + i;
    if (m >= l.M) continue;
    if (n0 == 0 && tx == 0) out[l.ob + m] = cs[i];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + 4 * tx + j;
      if (n < l.N) out[l.oW + (long long)m * l.N + n] = acc[i][j];
    }
  }
}
// g = the sum of the slices in order; block 0 also adds the loss shares
__global__ void reduce_kernel(const float* __restrict__ part, long long count, int slices, float* __restrict__ g,
                              const float* __restrict__ lossp, int nloss, float* __restrict__ loss) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) {
    float s = 0.f;
    for (int k = 0; k < slices; ++k) s += part[k * count + i];
    g[i] = s;
  }
  if (blockIdx.x == 0) {
    __shared__ float red[256];
    float s = 0.f;
    for (int k = threadIdx.x; k < nloss; k += blockDim.x) s += lossp[k];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
      if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = red[0];
  }
}
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long long n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace

struct tnqe_mlp {
  int n_in = 0, n_h = 0, n_out = 0, max_batch = 0;
  long long count = 0;
  long long oW1 = 0, ob1 = 0, oW2 = 0, ob2 = 0, oW3 = 0, ob3 = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  float *P = nullptr, *G = nullptr, *Mo = nullptr, *Vo = nullptr;
  float *X = nullptr, *Z1 = nullptr, *A1 = nullptr, *Z2 = nullptr, *A2 = nullptr, *Y = nullptr;
  float *T = nullptr, *w = nullptr, *dY = nullptr, *dA = nullptr, *dZ = nullptr, *rowloss = nullptr, *scal = nullptr;
  float* part = nullptr;         // partial gradients, one slice per cut of the batch
  long long step = 0;
  int launches = 0;
  std::string err;
};

namespace {

struct MlpError : std::runtime_error {
  tnqe_status st;
  MlpError(tnqe_status s, const std::string& m) : std::runtime_error(m), st(s) {}
};
void ck(cudaError_t e, const char* what) {
  if (e != cudaSuccess)
    throw MlpError(e == cudaErrorMemoryAllocation ? TNQE_ERR_NOMEM : TNQE_ERR_CUDA,
                   std::string(what) + ": " + cudaGetErrorString(e));
}
void launched(tnqe_mlp* n) {
  ++n->launches;
  ck(cudaGetLastError(), "kernel launch");
}
int tiles(int x) { return (x + GT - 1) / GT; }
unsigned blocks(long long x) { return (unsigned)((x + 255) / 256); }

void check_batch(tnqe_mlp* n, const void* X, int batch) {
  if (!X || batch < 1 || batch > n->max_batch) throw MlpError(TNQE_ERR_ARG, "batch must be in [1, max_batch]");
}

// Cuts of the batch in the weight gradients: enough blocks for two per SM of a GB300 (five fit; a cut more
// adds a slice to write and read back), at least 64 rows each (below that a cut is two slabs
// deep, and the prologue costs as much as the product).
int grad_tiles(const tnqe_mlp* n) {
  return tiles(n->n_h) * tiles(n->n_in) + tiles(n->n_h) * tiles(n->n_h) + tiles(n->n_out) * tiles(n->n_h);
}
int grad_slices(const tnqe_mlp* n, int B) {
  return std::max(1, std::min((304 + grad_tiles(n) - 1) / grad_tiles(n), (B + 63) / 64));
}

// mode 1: the outputs alone; 2: the loss and its derivative too
void forward(tnqe_mlp* n, int B, int mode, bool weighted) {
  const int I = n->n_in, H = n->n_h, O = n->n_out;
  layer_kernel<0><<<dim3(tiles(H), tiles(B)), GTHREADS, 0, n->stream>>>(n->X, n->P + n->oW1, n->P + n->ob1, n->Z1,
                                                                       n->A1, B, H, I, nullptr, nullptr, nullptr);
  launched(n);
  layer_kernel<0><<<dim3(tiles(H), tiles(B)), GTHREADS, 0, n->stream>>>(n->A1, n->P + n->oW2, n->P + n->ob2, n->Z2,
                                                                       n->A2, B, H, H, nullptr, nullptr, nullptr);
  launched(n);
  const dim3 g(tiles(O), tiles(B));
  if (mode == 1)
    layer_kernel<1><<<g, GTHREADS, 0, n->stream>>>(n->A2, n->P + n->oW3, n->P + n->ob3, n->Y, nullptr, B, O, H, nullptr,
                                                   nullptr, nullptr);
  else
    layer_kernel<2><<<g, GTHREADS, 0, n->stream>>>(n->A2, n->P + n->oW3, n->P + n->ob3, n->Y, n->dY, B, O, H, n->T,
                                                   weighted ? n->w : nullptr, n->rowloss);
  launched(n);
}

// loss into scal[1], gradient into G (after forward in mode 2)
void backward(tnqe_mlp* n, int B) {
  const int I = n->n_in, H = n->n_h, O = n->n_out;
  back_kernel<<<dim3(tiles(H), tiles(B)), GTHREADS, 0, n->stream>>>(n->dY, n->P + n->oW3, n->Z2, n->dZ, B, H, O);
  launched(n);
  back_kernel<<<dim3(tiles(H), tiles(B)), GTHREADS, 0, n->stream>>>(n->dZ, n->P + n->oW2, n->Z1, n->dA, B, H, H);
  launched(n);
  const int S = grad_slices(n, B), cut = ((B + S - 1) / S + GK - 1) / GK * GK;
  GradLayers L;
  L.l[0] = GradLayer{n->dA, n->X, n->oW1, n->ob1, H, I, tiles(I), 0};
  L.l[1] = GradLayer{n->dZ, n->A1, n->oW2, n->ob2, H, H, tiles(H), tiles(H) * tiles(I)};
  L.l[2] = GradLayer{n->dY, n->A2, n->oW3, n->ob3, O, H, tiles(H), tiles(H) * tiles(I) + tiles(H) * tiles(H)};
  const int slices = (B + cut - 1) / cut;
  grad_kernel<<<dim3(grad_tiles(n), slices), GTHREADS, 0, n->stream>>>(L, B, cut, n->count, n->part);
  launched(n);
  reduce_kernel<<<blocks(n->count), 256, 0, n->stream>>>(n->part, n->count, slices, n->G, n->rowloss,
                                                         tiles(O) * tiles(B), n->scal + 1);
  launched(n);
}

void upload_batch(tnqe_mlp* n, const float* X, const float* T, const float* w, int B) {
  ck(cudaMemcpyAsync(n->X, X, sizeof(float) * B * n->n_in, cudaMemcpyHostToDevice, n->stream), "copy X");
  if (T) ck(cudaMemcpyAsync(n->T, T, sizeof(float) * B * n->n_out, cudaMemcpyHostToDevice, n->stream), "copy T");
  if (w) {
    for (int i = 0; i < B; ++i)
      if (!(w[i] >= 0.f) || !std::isfinite(w[i])) throw MlpError(TNQE_ERR_ARG, "row weights must be finite and >= 0");
    ck(cudaMemcpyAsync(n->w, w, sizeof(float) * B, cudaMemcpyHostToDevice, n->stream), "copy w");
  }
}

tnqe_status mlp_fail(tnqe_mlp* n, const MlpError& e) {
  if (n) n->err = e.what();
  return e.st;
}

}  // namespace

extern "C" {

tnqe_status tnqe_mlp_create(int n_in, int n_hidden, int n_out, int max_batch, void* stream, tnqe_mlp** out) {
  if (!out) return TNQE_ERR_ARG;
  *out = nullptr;
  if (n_in < 1 || n_hidden < 1 || n_out < 1 || n_in > 4096 || n_hidden > 4096 || n_out > 4096 || max_batch < 1 ||
      max_batch > 65536)
    return TNQE_ERR_ARG;
  tnqe_mlp* n = new tnqe_mlp();
  try {
    n->n_in = n_in;
    n->n_h = n_hidden;
    n->n_out = n_out;
    n->max_batch = max_batch;
    const long long I = n_in, H = n_hidden, O = n_out;
    n->oW1 = 0;
    n->ob1 = H * I;
    n->oW2 = n->ob1 + H;
    n->ob2 = n->oW2 + H * H;
    n->oW3 = n->ob2 + H;
    n->ob3 = n->oW3 + O * H;
    n->count = n->ob3 + O;
    if (stream) {
      n->stream = (cudaStream_t)stream;
    } else {
      ck(cudaStreamCreateWithFlags(&n->stream, cudaStreamNonBlocking), "stream");
      n->own_stream = true;
    }
    auto alloc = [&](float** p, long long cnt) {
      ck(cudaMalloc(p, sizeof(float) * (size_t)std::max(1LL, cnt)), "cudaMalloc");
      ck(cudaMemset(*p, 0, sizeof(float) * (size_t)std::max(1LL, cnt)), "cudaMemset");
    };
    const long long B = max_batch;
    alloc(&n->P, n->count);
    alloc(&n->G, n->count);
    alloc(&n->Mo, n->count);
    alloc(&n->Vo, n->count);
    alloc(&n->X, B * I);
    alloc(&n->Z1, B * H);
    alloc(&n->A1, B * H);
    alloc(&n->Z2, B * H);
    alloc(&n->A2, B * H);
    alloc(&n->Y, B * O);
    alloc(&n->T, B * O);
    alloc(&n->w, B);
    alloc(&n->dY, B * O);
    alloc(&n->dA, B * H);
    alloc(&n->dZ, B * H);
    alloc(&n->rowloss, (long long)tiles((int)B) * tiles(n_out));   // loss shares of the last layer's tiles
    alloc(&n->part, n->count * grad_slices(n, max_batch));
    alloc(&n->scal, 4);
    *out = n;
    return TNQE_OK;
  } catch (const MlpError& e) {
    tnqe_mlp_destroy(n);
    return e.st;
  }
}

long long tnqe_mlp_param_count(const tnqe_mlp* n) { return n ? n->count : 0; }

tnqe_status tnqe_mlp_set_params(tnqe_mlp* n, const float* params) {
  if (!n || !params) return TNQE_ERR_ARG;
  try {
    std::vector<float> h(params, params + n->count);
    for (float x : h)
      if (!std::isfinite(x)) throw MlpError(TNQE_ERR_ARG, "non-finite parameter");
    ck(cudaMemcpyAsync(n->P, h.data(), sizeof(float) * n->count, cudaMemcpyHostToDevice, n->stream), "copy params");
    ck(cudaMemsetAsync(n->Mo, 0, sizeof(float) * n->count, n->stream), "clear m");
    ck(cudaMemsetAsync(n->Vo, 0, sizeof(float) * n->count, n->stream), "clear v");
    ck(cudaStreamSynchronize(n->stream), "sync");
    n->step = 0;
    return TNQE_OK;
  } catch (const MlpError& e) {
    return mlp_fail(n, e);
  }
}

tnqe_status tnqe_mlp_get_params(const tnqe_mlp* n, float* params) {
  if (!n || !params) return TNQE_ERR_ARG;
  if (cudaStreamSynchronize(n->stream) != cudaSuccess) return TNQE_ERR_CUDA;
  if (cudaMemcpy(params, n->P, sizeof(float) * n->count, cudaMemcpyDeviceToHost) != cudaSuccess) return TNQE_ERR_CUDA;
  return TNQE_OK;
}

tnqe_status tnqe_mlp_forward(tnqe_mlp* n, const float* X, int batch, float* Y) {
  if (!n || !Y) return TNQE_ERR_ARG;
  try {
    check_batch(n, X, batch);
    n->launches = 0;
    upload_batch(n, X, nullptr, nullptr, batch);
    forward(n, batch, 1, false);
    ck(cudaMemcpyAsync(Y, n->Y, sizeof(float) * batch * n->n_out, cudaMemcpyDeviceToHost, n->stream), "copy Y");
    ck(cudaStreamSynchronize(n->stream), "sync");
    return TNQE_OK;
  } catch (const MlpError& e) {
    return mlp_fail(n, e);
  }
}

tnqe_status tnqe_mlp_gradient(tnqe_mlp* n, const float* X, const float* T, const float* w, int batch, float* loss,
                              float* grad) {
  if (!n || !T) return TNQE_ERR_ARG;
  try {
    check_batch(n, X, batch);
    n->launches = 0;
    upload_batch(n, X, T, w, batch);
    forward(n, batch, 2, w != nullptr);
    backward(n, batch);
    float l = 0.f;
    ck(cudaMemcpyAsync(&l, n->scal + 1, sizeof(float), cudaMemcpyDeviceToHost, n->stream), "copy loss");
    if (grad) ck(cudaMemcpyAsync(grad, n->G, sizeof(float) * n->count, cudaMemcpyDeviceToHost, n->stream), "copy grad");
    ck(cudaStreamSynchronize(n->stream), "sync");
    if (loss) *loss = l;
    return TNQE_OK;
  } catch (const MlpError& e) {
    return mlp_fail(n, e);
  }
}

tnqe_status tnqe_mlp_adam_step(tnqe_mlp* n, const float* X, const float* T, const float* w, int batch, float lr,
                               float beta1, float beta2, float eps, float* loss) {
  if (!n || !T) return TNQE_ERR_ARG;
  try {
    check_batch(n, X, batch);
    if (!(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
      throw MlpError(TNQE_ERR_ARG, "bad Adam hyper-parameters");
    n->launches = 0;
    upload_batch(n, X, T, w, batch);
    forward(n, batch, 2, w != nullptr);
    backward(n, batch);
    ++n->step;
    const float c1 = 1.f - std::pow(beta1, (float)n->step), c2 = 1.f - std::pow(beta2, (float)n->step);
    adam_kernel<<<blocks(n->count), 256, 0, n->stream>>>(n->P, n->G, n->Mo, n->Vo, n->count, lr, beta1, beta2, eps, c1,
                                                         c2);
    launched(n);
    float l = 0.f;
    ck(cudaMemcpyAsync(&l, n->scal + 1, sizeof(float), cudaMemcpyDeviceToHost, n->stream), "copy loss");
    ck(cudaStreamSynchronize(n->stream), "sync");
    if (loss) *loss = l;
    return TNQE_OK;
  } catch (const MlpError& e) {
    return mlp_fail(n, e);
  }
}

int tnqe_mlp_last_launches(const tnqe_mlp* n) { return n ? n->launches : 0; }

const char* tnqe_mlp_last_error(const tnqe_mlp* n) { return n ? n->err.c_str() : "null network"; }

void tnqe_mlp_destroy(tnqe_mlp* n) {
  if (!n) return;
  if (n->stream) cudaStreamSynchronize(n->stream);
  float* bufs[] = {n->P, n->G, n->Mo, n->Vo, n->X, n->Z1, n->A1, n->Z2, n->A2,
                   n->Y, n->T, n->w, n->dY, n->dA, n->dZ, n->rowloss, n->scal, n->part};
  for (float* p : bufs)
    if (p) cudaFree(p);
  if (n->own_stream && n->stream) cudaStreamDestroy(n->stream);
  delete n;
}

}  // extern "C"
