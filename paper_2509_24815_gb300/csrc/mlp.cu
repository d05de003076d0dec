// Per-query parameter model (an addition; the paper tunes alpha_q / cut and
// heap_factor globally, Section 5.3): MLP 64 -> 128 -> 64 -> 2 with ReLU,
// fp32 weights and bf16 activations.  Outputs map to
//   cut = clamp(round(3 + 27 * sigmoid(o0)), 3, 30)
//   heap_factor = 0.5 + 0.5 * sigmoid(o1)
// Training: loss = mean over rows of sum_j (sigmoid(o_j) - t_j)^2, Adam.
#include <cuda_bf16.h>

#include "search_impl.h"

namespace seismic {

namespace {

constexpr int IN = SEISMIC_MLP_IN, H1 = SEISMIC_MLP_H1, H2 = SEISMIC_MLP_H2, OUT = 2;
constexpr int OW1 = 0, OB1 = OW1 + H1 * IN, OW2 = OB1 + H1, OB2 = OW2 + H2 * H1, OW3 = OB2 + H2, OB3 = OW3 + OUT * H2;
static_assert(OB3 + OUT == SEISMIC_MLP_PARAMS, "parameter packing");
constexpr int kRows = 32;  // rows per CTA
constexpr int kNT = 512;
static_assert(IN == 64 && H1 == 128 && H2 == 64 && OUT == 2 && kRows == 32 && kNT == 512, "the tiles below");
// Shared-memory row strides of a multiple of 4 floats that is 4 mod 32: eight
// lanes on eight consecutive rows read float4s from 32 different banks.
constexpr int S1 = IN + 4, S2 = H1 + 4;

__device__ __forceinline__ float bfr(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + __expf(-x)); }
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

struct MlpSmem {  // read as float4s
  alignas(16) float w1[H1 * S1];
  alignas(16) float w2[H2 * S2];
  alignas(16) float w3[OUT * H2];
  alignas(16) float a0[kRows * S1];
  alignas(16) float z1[kRows * S2];  // pre-activation
  alignas(16) float a1[kRows * S2];  // bf16-rounded ReLU
  alignas(16) float z2[kRows * S1];
  alignas(16) float a2[kRows * S1];
  float b1[H1], b2[H2], b3[OUT], o[kRows * OUT];
};
static_assert(IN == H2, "rows of a0, z2 and a2 share a stride");

__device__ void mlp_load(MlpSmem &s, const float *w) {
  for (int i = threadIdx.x; i < SEISMIC_MLP_PARAMS; i += kNT) {
    const float x = w[i];
    if (i < OB1) s.w1[(i - OW1) / IN * S1 + (i - OW1) % IN] = x;
    else if (i < OW2) s.b1[i - OB1] = x;
    else if (i < OB2) s.w2[(i - OW2) / H1 * S2 + (i - OW2) % H1] = x;
    else if (i < OW3) s.b2[i - OB2] = x;
    else if (i < OB3) s.w3[i - OW3] = x;
    else s.b3[i - OB3] = x;
  }
  __syncthreads();
}

// Outputs of one layer, 4 rows by J columns per thread (rows 4 rg .., columns
// c0 + 32 j): z = bias + the products in input order, so each is the same chain
// of fused multiply-adds whatever the tile.
template <int N, int J>
__device__ __forceinline__ void mlp_tile(const float *w, int sw, const float *bias, const float *in, int si, int rg, int c0,
                                         float z[4][J]) {
#pragma unroll
  for (int j = 0; j < J; j++)
#pragma unroll
    for (int r = 0; r < 4; r++) z[r][j] = bias[c0 + 32 * j];
#pragma unroll 4
  for (int f = 0; f < N; f += 4) {
    float4 x[4];
#pragma unroll
    for (int r = 0; r < 4; r++) x[r] = ld4(in + (4 * rg + r) * si + f);
#pragma unroll
    for (int j = 0; j < J; j++) {
      const float4 y = ld4(w + (c0 + 32 * j) * sw + f);
#pragma unroll
      for (int r = 0; r < 4; r++) {
        z[r][j] = fmaf(y.x, x[r].x, z[r][j]);
        z[r][j] = fmaf(y.y, x[r].y, z[r][j]);
        z[r][j] = fmaf(y.z, x[r].z, z[r][j]);
        z[r][j] = fmaf(y.w, x[r].w, z[r][j]);
      }
    }
  }
}

// forward for rows [r0, r0 + nr) held in shared memory
__device__ void mlp_fwd(MlpSmem &s, const float *feat, uint64_t r0, int nr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rg = warp & 7, half = warp >> 3;
  for (int i = tid; i < kRows * IN; i += kNT) {
    const int r = i / IN, f = i % IN;
    s.a0[r * S1 + f] = r < nr ? bfr(feat[(r0 + r) * IN + f]) : 0.0f;
  }
  __syncthreads();
  {
    float z[4][2];
    mlp_tile<IN, 2>(s.w1, S1, s.b1, s.a0, S1, rg, 64 * half + lane, z);
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const int at = (4 * rg + r) * S2 + 64 * half + lane + 32 * j;
        s.z1[at] = z[r][j];
        s.a1[at] = bfr(fmaxf(z[r][j], 0.0f));
      }
  }
  __syncthreads();
  {
    float z[4][1];
    mlp_tile<H1, 1>(s.w2, S2, s.b2, s.a1, S2, rg, 32 * half + lane, z);
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int at = (4 * rg + r) * S1 + 32 * half + lane;
      s.z2[at] = z[r][0];
      s.a2[at] = bfr(fmaxf(z[r][0], 0.0f));
    }
  }
  __syncthreads();
  if (tid < kRows * OUT) {
    const int r = tid / OUT, j = tid % OUT;
    float z = s.b3[j];
    for (int f = 0; f < H2; f += 4) {
      const float4 x = ld4(s.a2 + r * S1 + f), y = ld4(s.w3 + j * H2 + f);
      z = fmaf(y.x, x.x, z);
      z = fmaf(y.y, x.y, z);
      z = fmaf(y.z, x.z, z);
      z = fmaf(y.w, x.w, z);
    }
    s.o[tid] = z;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kNT) k_mlp_forward(const float *__restrict__ w, const float *__restrict__ feat,
                                                      uint64_t n, float *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char smraw[];
  MlpSmem &s = *reinterpret_cast<MlpSmem *>(smraw);
  mlp_load(s, w);
  for (uint64_t r0 = (uint64_t)blockIdx.x * kRows; r0 < n; r0 += (uint64_t)gridDim.x * kRows) {
    int nr = (int)((n - r0) < (uint64_t)kRows ? (n - r0) : (uint64_t)kRows);
    mlp_fwd(s, feat, r0, nr);
    for (int i = threadIdx.x; i < nr * OUT; i += kNT) out[r0 * OUT + i] = s.o[i];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kNT) k_mlp_params(const float *__restrict__ w, const float *__restrict__ feat,
                                                     uint64_t n, uint32_t cut_fb, float hf_fb,
                                                     uint32_t *__restrict__ q_cut, float *__restrict__ q_hf) {
  extern __shared__ __align__(16) unsigned char smraw[];
  MlpSmem &s = *reinterpret_cast<MlpSmem *>(smraw);
  mlp_load(s, w);
  for (uint64_t r0 = (uint64_t)blockIdx.x * kRows; r0 < n; r0 += (uint64_t)gridDim.x * kRows) {
    int nr = (int)((n - r0) < (uint64_t)kRows ? (n - r0) : (uint64_t)kRows);
    mlp_fwd(s, feat, r0, nr);
    for (int r = threadIdx.x; r < nr; r += kNT) {
      float o0 = s.o[r * OUT], o1 = s.o[r * OUT + 1];
      uint32_t c = cut_fb;
      float h = hf_fb;
      if (isfinite(o0) && isfinite(o1)) {  // fixed parameters are the fallback
        c = (uint32_t)min(30.0f, max(3.0f, rintf(3.0f + 27.0f * sigm(o0))));
        h = 0.5f + 0.5f * sigm(o1);
      }
      q_cut[r0 + r] = c;
      q_hf[r0 + r] = h;
    }
    __syncthreads();
  }
}

struct MlpGradSmem {
  MlpSmem f;
  alignas(16) float dz1[kRows * S2];
  alignas(16) float dz2[kRows * S1];
  float dzo[kRows * OUT], loss;
};

// Adds four consecutive floats to g (16-byte aligned).
__device__ __forceinline__ void red4(float *g, float x, float y, float z, float w) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(g), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

// forward + backward; each thread keeps a 4 x 4 tile of both weight gradients
// (and the first threads the small ones) in registers over the CTA's rows and
// adds them to g (zeroed by the caller) once at the end, four at a time.
// Bound by shared-memory reads: every operand tile is read as float4s from
// conflict-free rows (weights read at a stride of 64 or 128 floats, 32 lanes on
// one bank, and scalar reads took the whole step of 4096 rows, its four launches
// included, to 108 us; now 40 us).
__global__ void __launch_bounds__(kNT) k_mlp_grad(const float *__restrict__ w, const float *__restrict__ feat,
                                                   const float *__restrict__ tgt, uint64_t n, float *__restrict__ g,
                                                   float *__restrict__ loss) {
  extern __shared__ __align__(16) unsigned char smraw[];
  MlpGradSmem &sg = *reinterpret_cast<MlpGradSmem *>(smraw);
  MlpSmem &s = sg.f;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) sg.loss = 0.0f;
  mlp_load(s, w);
  const float inv_n = 1.0f / (float)n;
  // tiles: rows m of W1 4 (tid / 16) .. and its columns 4 (tid % 16) ..; rows of W2 4 (tid / 32) .., columns 4 (tid % 32) ..
  const int m1 = tid / 16 * 4, f1 = tid % 16 * 4, m2 = warp * 4, f2 = lane * 4;
  float g1[4][4] = {}, g2[4][4] = {}, gs = 0.0f;  // gs: a bias or an output weight
  for (uint64_t r0 = (uint64_t)blockIdx.x * kRows; r0 < n; r0 += (uint64_t)gridDim.x * kRows) {
    const int nr = (int)((n - r0) < (uint64_t)kRows ? (n - r0) : (uint64_t)kRows);
    mlp_fwd(s, feat, r0, nr);
    if (tid < kRows * OUT) {
      const int r = tid / OUT, j = tid % OUT;
      float d = 0.0f;
      if (r < nr) {
        const float sgm = sigm(s.o[tid]), e = sgm - tgt[(r0 + r) * OUT + j];
        atomicAdd(&sg.loss, e * e * inv_n);
        d = 2.0f * e * sgm * (1.0f - sgm) * inv_n;
      }
      sg.dzo[tid] = d;
    }
    __syncthreads();
    for (int i = tid; i < kRows * H2; i += kNT) {
      const int r = i / H2, m = i % H2;
      float d = 0.0f;
#pragma unroll
      for (int j = 0; j < OUT; j++) d = fmaf(s.w3[j * H2 + m], sg.dzo[r * OUT + j], d);
      sg.dz2[r * S1 + m] = s.z2[r * S1 + m] > 0.0f ? d : 0.0f;
    }
    __syncthreads();
    {  // dz1: rows 2 warp, 2 warp + 1, columns 4 lane ..
      float d[2][4] = {};
#pragma unroll 4
      for (int j = 0; j < H2; j += 4) {
        const float4 x0 = ld4(sg.dz2 + (2 * warp) * S1 + j), x1 = ld4(sg.dz2 + (2 * warp + 1) * S1 + j);
        const float xa[2][4] = {{x0.x, x0.y, x0.z, x0.w}, {x1.x, x1.y, x1.z, x1.w}};
#pragma unroll
        for (int jj = 0; jj < 4; jj++) {
          const float4 y = ld4(s.w2 + (j + jj) * S2 + 4 * lane);
#pragma unroll
          for (int r = 0; r < 2; r++) {
            d[r][0] = fmaf(y.x, xa[r][jj], d[r][0]);
            d[r][1] = fmaf(y.y, xa[r][jj], d[r][1]);
            d[r][2] = fmaf(y.z, xa[r][jj], d[r][2]);
            d[r][3] = fmaf(y.w, xa[r][jj], d[r][3]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 2; r++) {
        const int at = (2 * warp + r) * S2 + 4 * lane;
        const float4 z = ld4(s.z1 + at);
        *reinterpret_cast<float4 *>(sg.dz1 + at) = make_float4(z.x > 0.0f ? d[r][0] : 0.0f, z.y > 0.0f ? d[r][1] : 0.0f,
                                                               z.z > 0.0f ? d[r][2] : 0.0f, z.w > 0.0f ? d[r][3] : 0.0f);
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int r = 0; r < nr; r++) {
      const float4 d = ld4(sg.dz1 + r * S2 + m1), x = ld4(s.a0 + r * S1 + f1);
      const float da[4] = {d.x, d.y, d.z, d.w}, xa[4] = {x.x, x.y, x.z, x.w};
      const float4 e = ld4(sg.dz2 + r * S1 + m2), y = ld4(s.a1 + r * S2 + f2);
      const float ea[4] = {e.x, e.y, e.z, e.w}, ya[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
          g1[i][j] = fmaf(da[i], xa[j], g1[i][j]);
          g2[i][j] = fmaf(ea[i], ya[j], g2[i][j]);
        }
    }
    for (int r = 0; r < nr; r++) {
      if (tid < H1) gs += sg.dz1[r * S2 + tid];
      else if (tid < H1 + H2) gs += sg.dz2[r * S1 + tid - H1];
      else if (tid < H1 + H2 + OUT * H2) gs = fmaf(sg.dzo[r * OUT + (tid - H1 - H2) / H2], s.a2[r * S1 + (tid - H1 - H2) % H2], gs);
      else if (tid < H1 + H2 + OUT * H2 + OUT) gs += sg.dzo[r * OUT + tid - H1 - H2 - OUT * H2];
    }
    __syncthreads();
  }
  // the gradient may start at any 4-byte boundary
  const bool al = (reinterpret_cast<uintptr_t>(g) & 15u) == 0;
#pragma unroll
  for (int i = 0; i < 4; i++) {
    float *p1 = g + OW1 + (m1 + i) * IN + f1, *p2 = g + OW2 + (m2 + i) * H1 + f2;
    if (al) {
      red4(p1, g1[i][0], g1[i][1], g1[i][2], g1[i][3]);
      red4(p2, g2[i][0], g2[i][1], g2[i][2], g2[i][3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; j++) {
        atomicAdd(p1 + j, g1[i][j]);
        atomicAdd(p2 + j, g2[i][j]);
      }
    }
  }
  if (tid < H1) atomicAdd(g + OB1 + tid, gs);
  else if (tid < H1 + H2) atomicAdd(g + OB2 + tid - H1, gs);
  else if (tid < H1 + H2 + OUT * H2 + OUT) atomicAdd(g + OW3 + tid - H1 - H2, gs);
  if (tid == 0) atomicAdd(loss, sg.loss);
}
static_assert(OW1 % 4 == 0 && OW2 % 4 == 0 && OB3 == OW3 + OUT * H2, "vector additions and the small gradients' order");

__global__ void k_adam(float *w, const float *g, float *m, float *v, float lr, float b1c, float b2c) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < SEISMIC_MLP_PARAMS; i += gridDim.x * blockDim.x) {
    float gi = g[i];
    float mi = b1 * m[i] + (1.0f - b1) * gi;
    float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / b1c) / (sqrtf(vi / b2c) + eps);
  }
}

// features: one warp per query
__global__ void k_features(const uint64_t *__restrict__ ip, const uint16_t *__restrict__ terms,
                           const float *__restrict__ vals, uint32_t nq, const uint32_t *__restrict__ list_ptr,
                           const uint32_t *__restrict__ blk_ptr, uint32_t dim, float *__restrict__ feat) {
  const int lane = threadIdx.x & 31;
  const uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (q >= nq) return;
  const uint64_t b = ip[q], e = ip[q + 1];
  float *f = feat + (size_t)q * IN;
  for (int i = lane; i < IN; i += 32) f[i] = 0.0f;
  __syncwarp();
  uint32_t nz = 0;
  float l1 = 0.0f, l2 = 0.0f;
  for (uint64_t p = b + lane; p < e; p += 32) {
    float v = vals[p];
    if (v == 0.0f) continue;
    nz++;
    l1 += fabsf(v);
    l2 = fmaf(v, v, l2);
    const uint16_t t = terms[p];
    uint32_t r = 0;  // rank by (value desc, term asc) among nonzeros
    for (uint64_t j = b; j < e; j++) {
      float vj = vals[j];
      if (vj == 0.0f) continue;
      r += (vj > v || (vj == v && terms[j] < t)) ? 1u : 0u;
    }
    if (r < 16 && t < dim) {
      f[1 + r] = v;
      f[17 + r] = __logf(1.0f + (float)(list_ptr[t + 1] - list_ptr[t]));
      f[33 + r] = __logf(1.0f + (float)(blk_ptr[t + 1] - blk_ptr[t]));
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    nz += __shfl_xor_sync(0xffffffffu, nz, o);
    l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    l2 += __shfl_xor_sync(0xffffffffu, l2, o);
  }
  if (lane == 0) {
    f[0] = __logf(1.0f + (float)nz);
    f[49] = l1;
    f[50] = sqrtf(l2);
  }
}

size_t mlp_smem(bool grad) { return grad ? sizeof(MlpGradSmem) : sizeof(MlpSmem); }

int set_attr(const void *fn, size_t smem) {
  SZ_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  return SEISMIC_OK;
}

}  // namespace

int launch_features(const uint64_t *ip, const uint16_t *t, const float *v, uint32_t nq, const uint32_t *list_ptr,
                    const uint32_t *blk_ptr, uint32_t dim, float *feat, cudaStream_t st) {
  if (!nq) return SEISMIC_OK;
  const uint32_t warps_per_block = 8;
  k_features<<<(nq + warps_per_block - 1) / warps_per_block, warps_per_block * 32, 0, st>>>(ip, t, v, nq, list_ptr,
                                                                                           blk_ptr, dim, feat);
  SZ_CUDA(cudaGetLastError());
  return SEISMIC_OK;
}

int launch_mlp_params(const float *w, const float *feat, uint32_t n, uint32_t cut_fb, float hf_fb, uint32_t *q_cut,
                      float *q_hf, cudaStream_t st) {
  if (!n) return SEISMIC_OK;
  size_t sm = mlp_smem(false);
  int rc = set_attr((const void *)k_mlp_params, sm);
  if (rc) return rc;
  uint32_t grid = std::min<uint32_t>((n + kRows - 1) / kRows, 1024);
  k_mlp_params<<<grid, kNT, sm, st>>>(w, feat, n, cut_fb, hf_fb, q_cut, q_hf);
  SZ_CUDA(cudaGetLastError());
  return SEISMIC_OK;
}

int mlp_forward_impl(const float *w, const float *feat, uint64_t n, float *out, cudaStream_t st) {
  if (!w || !feat || !out) return fail(SEISMIC_EINVAL, "NULL argument");
  if (!n) return SEISMIC_OK;
  size_t sm = mlp_smem(false);
  int rc = set_attr((const void *)k_mlp_forward, sm);
  if (rc) return rc;
  uint32_t grid = (uint32_t)std::min<uint64_t>((n + kRows - 1) / kRows, 1024);
  k_mlp_forward<<<grid, kNT, sm, st>>>(w, feat, n, out);
  SZ_CUDA(cudaGetLastError());
  return SEISMIC_OK;
}

int mlp_train_step_impl(float *w, float *g, float *m, float *v, const float *feat, const float *tgt, uint64_t n,
                        float lr, uint32_t step, float *loss, cudaStream_t st) {
  if (!w || !g || !m || !v || !feat || !tgt || !loss) return fail(SEISMIC_EINVAL, "NULL argument");
  if (!n || step == 0) return fail(SEISMIC_EINVAL, "n and step must be >= 1");
  size_t sm = mlp_smem(true);
  int rc = set_attr((const void *)k_mlp_grad, sm);
  if (rc) return rc;
  SZ_CUDA(cudaMemsetAsync(g, 0, SEISMIC_MLP_PARAMS * 4, st));
  SZ_CUDA(cudaMemsetAsync(loss, 0, 4, st));
  uint32_t grid = (uint32_t)std::min<uint64_t>((n + kRows - 1) / kRows, 304);
  k_mlp_grad<<<grid, kNT, sm, st>>>(w, feat, tgt, n, g, loss);
  SZ_CUDA(cudaGetLastError());
  float b1c = 1.0f - powf(0.9f, (float)step), b2c = 1.0f - powf(0.999f, (float)step);
  k_adam<<<(SEISMIC_MLP_PARAMS + 255) / 256, 256, 0, st>>>(w, g, m, v, lr, b1c, b2c);
  SZ_CUDA(cudaGetLastError());
  return SEISMIC_OK;
}

}  // namespace seismic

using namespace seismic;

extern "C" {

int seismic_set_mlp(seismic_index *ix, const float *weights, uint64_t n_floats) {
  if (!ix || !weights) return fail(SEISMIC_EINVAL, "NULL argument");
  if (n_floats != SEISMIC_MLP_PARAMS) return fail(SEISMIC_EINVAL, "MLP weights: wrong count");
  for (uint64_t i = 0; i < n_floats; i++)
    if (!std::isfinite(weights[i])) return fail(SEISMIC_EINVAL, "MLP weights: non-finite value");
  SZ_CUDA(cudaSetDevice(ix->device));
  int rc = ix->mlp.alloc(n_floats * 4);
  if (rc) return rc;
  SZ_CUDA(cudaMemcpy(ix->mlp.p, weights, n_floats * 4, cudaMemcpyHostToDevice));
  ix->has_mlp = 1;
  return SEISMIC_OK;
}

int seismic_query_features(seismic_index *ix, const seismic_csr *queries, float *features, int32_t on_device,
                           void *stream) {
  if (!ix || !queries || !features) return fail(SEISMIC_EINVAL, "NULL argument");
  if (queries->n_rows == 0) return SEISMIC_OK;
  if (queries->dim != ix->dim) return fail(SEISMIC_EINVAL, "queries: dim differs from the index");
  SZ_CUDA(cudaSetDevice(ix->device));
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const uint64_t nq = queries->n_rows;
  const uint64_t *ip = queries->indptr;
  const uint16_t *t = queries->terms;
  const float *v = queries->vals;
  DevBuf stage;
  if (!queries->on_device) {
    int rc = validate_host_csr(queries, "queries", ix->dim);
    if (rc) return rc;
    uint64_t nnz = queries->indptr[nq];
    size_t b_ip = (nq + 1) * 8, b_t = ((nnz * 2 + 15) / 16) * 16;
    if ((rc = stage.alloc(b_ip + b_t + nnz * 4 + 16))) return rc;
    uint8_t *base = stage.as<uint8_t>();
    SZ_CUDA(cudaMemcpyAsync(base, queries->indptr, b_ip, cudaMemcpyHostToDevice, st));
    if (nnz) {
      SZ_CUDA(cudaMemcpyAsync(base + b_ip, queries->terms, nnz * 2, cudaMemcpyHostToDevice, st));
      SZ_CUDA(cudaMemcpyAsync(base + b_ip + b_t, queries->vals, nnz * 4, cudaMemcpyHostToDevice, st));
    }
    ip = reinterpret_cast<const uint64_t *>(base);
    t = reinterpret_cast<const uint16_t *>(base + b_ip);
    v = reinterpret_cast<const float *>(base + b_ip + b_t);
  }
  float *dfeat = features;
  DevBuf fo;
  if (!on_device) {
    int rc = fo.alloc(nq * SEISMIC_MLP_IN * 4);
    if (rc) return rc;
    dfeat = fo.as<float>();
  }
  int rc = launch_features(ip, t, v, (uint32_t)nq, ix->list_ptr.as<uint32_t>(), ix->blk_ptr.as<uint32_t>(), ix->dim,
                           dfeat, st);
  if (rc) return rc;
  if (!on_device) {
    SZ_CUDA(cudaMemcpyAsync(features, dfeat, nq * SEISMIC_MLP_IN * 4, cudaMemcpyDeviceToHost, st));
  }
  SZ_CUDA(cudaStreamSynchronize(st));
  return SEISMIC_OK;
}

int seismic_mlp_forward(const float *weights, const float *features, uint64_t n, float *out, void *stream) {
  return mlp_forward_impl(weights, features, n, out, reinterpret_cast<cudaStream_t>(stream));
}

int seismic_mlp_train_step(float *weights, float *grads, float *adam_m, float *adam_v, const float *features,
                           const float *targets, uint64_t n, float lr, uint32_t step, float *loss_out, void *stream) {
  return mlp_train_step_impl(weights, grads, adam_m, adam_v, features, targets, n, lr, step, loss_out,
                             reinterpret_cast<cudaStream_t>(stream));
}

}  // extern "C"
