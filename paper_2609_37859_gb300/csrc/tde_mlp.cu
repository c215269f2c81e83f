// tde_mlp.cu -- the learned EOS guess: a 2 -> 64 -> 64 -> 2 SiLU network that maps
// normalised (log10 rho, log10 e) to normalised (log10 T, log10 P).  The paper
// has no learned component; the network only chooses the temperature cell in
// which one Newton step on the interpolated log e column is taken, and
// table bisection stays both the fallback and the judge (Sec. 4.2 runtime map).
//
//  * Training: FP32 forward/backward kernels on BF16-rounded weights (the
//    weights inference uses), gradients reduced per CTA in shared memory, then
//    Adam on FP32 master weights.  Samples are drawn on the device from the
//    table itself with a counter-based generator (SplitMix64).
//  * Inference: per CTA tile of 128 cells, layer 1 and the SiLU in FP32 CUDA
//    cores, the 64 x 64 layer on the 5th-generation tensor cores
//    (tcgen05.mma kind::f16, BF16 operands from shared memory, FP32 accumulator
//    in tensor memory, read back with tcgen05.ld), layer 3 in FP32, then the
//    Newton step (64-bit fixed point, as the bisection's) with its fallback.
#include <cuda_bf16.h>
#include <math.h>
#include <string.h>

#include <vector>

#include "tde_internal.h"

namespace tde {

constexpr int H = 64;
constexpr int NPARAM = 2 * H + H + H * H + H + 2 * H + 2;   // 4482
// parameter offsets (same layout as the oracle's)
constexpr int OW1 = 0, OB1 = 2 * H, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + 2 * H;

struct MLPNorm {
  float cr, sr, ce, se, cT, sT, cP, sP;   // x_norm = (x - c) / s
  float isr, ise;                         // 1 / sr, 1 / se
  float idlt;                             // 1 / (log10 T cell width)
};

__device__ __forceinline__ float silu_f(float a) { return a / (1.0f + __expf(-a)); }
// Pairs of FP32 values for the packed FMA (one instruction for two)
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_pack(float a, float b) {
  f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ void f2_split(f2 v, float &a, float &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// SiLU for inference of two values from half their pre-activations, with one MUFU
// operation each: a sigmoid(a) = (a / 2)(1 + tanh(a / 2))
__device__ __forceinline__ f2 silu2_half(f2 z) {
  float a, b, ta, tb;
  f2_split(z, a, b);
  asm("tanh.approx.f32 %0, %1;" : "=f"(ta) : "f"(a));
  asm("tanh.approx.f32 %0, %1;" : "=f"(tb) : "f"(b));
  return f2_fma(z, f2_pack(ta, tb), z);
}
__device__ __forceinline__ float dsilu_f(float a) {
  const float s = 1.0f / (1.0f + __expf(-a));
  return s * (1.0f + a * (1.0f - s));
}

// ---------------------------------------------------------------- SplitMix64
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
__device__ __forceinline__ double u01(unsigned long long seed, unsigned long long ctr) {
  return (double)(splitmix64(seed ^ splitmix64(ctr)) >> 11) * (1.0 / 9007199254740992.0);
}

// training samples: (log rho, log T) uniform over the table -> inputs
// (log rho, log e) and targets (log T, log P), normalised
__global__ void k_mlp_samples(DTable t, MLPNorm nm, long long n, unsigned long long seed, float *x,
                              float *y) {
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n;
       s += (long long)gridDim.x * blockDim.x) {
    const double a = u01(seed, 2 * s), c = u01(seed, 2 * s + 1);
    const double xr = a * (t.nr - 1), yt = c * (t.nt - 1);
    int i = (int)floor(xr), j = (int)floor(yt);
    if (i > t.nr - 2) i = t.nr - 2;
    if (j > t.nt - 2) j = t.nt - 2;
    const double w = xr - i, u = yt - j;
    const double lr = t.lr0 + xr / t.inv_dlr;
    const double lT = t.lt0 + yt * t.dlt;
    const double le = bilin(t.le, t.nt, i, w, j, u);
    const double lp = bilin(t.lp, t.nt, i, w, j, u);
    // second input: position of log10 e inside the interpolated column at this density
    const double glo = (1.0 - w) * t.le[(size_t)i * t.nt] + w * t.le[(size_t)(i + 1) * t.nt];
    const double ghi = (1.0 - w) * t.le[(size_t)i * t.nt + t.nt - 1] + w * t.le[(size_t)(i + 1) * t.nt + t.nt - 1];
    x[2 * s] = (float)((lr - nm.cr) / nm.sr);
    x[2 * s + 1] = (float)(((le - glo) / (ghi - glo) - nm.ce) / nm.se);
    y[2 * s] = (float)((lT - nm.cT) / nm.sT);
    y[2 * s + 1] = (float)((lp - nm.cP) / nm.sP);
  }
}

// ------------------------------------------------------------------ training

constexpr int TRAIN_ALIGN = 128;   // a training batch is a multiple of this many samples
constexpr int GS = 32;             // samples per CTA in the gradient kernel
constexpr int GT = 512;            // its threads
constexpr int HP = H + 4;          // padded row of a [..][H] tile (16-byte rows on distinct banks)

// one Adam step after the gradient (in the CTA that finishes last)
struct AdamArgs {
  float *w, *m, *v;         // FP32 master weights and moments
  __nv_bfloat16 *wb;        // their BF16 rounding
  unsigned *done;           // CTAs finished (zero between launches); null: gradient only
  float lr, b1, b2, eps, bc1, bc2;
};

__device__ __forceinline__ void red4(float *p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// loss and gradient of L = (1/n) sum_s sum_o (y - target)^2 over samples
// [s0, s0 + count) with the BF16-rounded weights wb; gradient and loss are
// accumulated into g (NPARAM floats) and *loss.
//
// A batch is little work (4096 samples: 0.11 GFLOP), so what bounds a step is the
// depth of its dependent sums and the number of SMs it reaches: a CTA takes 32
// samples (a batch of 4096 fills 128 SMs) with 16 warps, every layer's products
// are register tiles of 4 or 8 outputs a thread (operands read as float4), and the
// CTA that finishes last applies Adam instead of a second launch.  One training
// step of 4096: 17 us (79 with a thread per sample and 128 samples a CTA).
__global__ void __launch_bounds__(GT) k_mlp_grad(const __nv_bfloat16 *wb_in,
                                                 const float *x,
                                                 const float *tg, long long s0,
                                                 long long count, float inv_n, float *g,
                                                 float *loss, AdamArgs ad) {
  pdl_begin();
  extern __shared__ __align__(16) float sh[];
  float *W2 = sh;                  // [H][HP]
  float *sh1 = W2 + H * HP;        // [GS][HP] hidden 1
  float *sh2 = sh1 + GS * HP;      // [GS][HP] hidden 2
  float *sg2 = sh2 + GS * HP;      // [GS][HP] gradient of pre-activation 2
  float *sg1 = sg2 + GS * HP;      // [GS][HP] gradient of pre-activation 1
  float *sw = sg1 + GS * HP;       // W1, b1, b2, W3, b3
  float *W1 = sw, *b1 = W1 + 2 * H, *b2 = b1 + H, *W3 = b2 + H, *b3 = W3 + 2 * H;
  float *sx = b3 + 4;              // [GS][2]
  float *sgy = sx + 2 * GS;        // [GS][2]
  __shared__ int s_last;
  const int tid = threadIdx.x;
  const bool vec = (reinterpret_cast<uintptr_t>(g + OW2) & 15) == 0;   // a caller's g may start on any float
  const long long first = s0 + blockIdx.x * (long long)GS;
  {   // eight weights of a row per thread (OW2 is a multiple of eight)
    static_assert(H * H / 8 == GT && OW2 % 8 == 0, "weight rows");
    const uint4 v = *reinterpret_cast<const uint4 *>(wb_in + OW2 + 8 * tid);
    float *d = W2 + (tid / (H / 8)) * HP + 8 * (tid % (H / 8));
    const unsigned u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {   // a BF16 is the high half of its FP32
      d[2 * q] = __uint_as_float(u[q] << 16);
      d[2 * q + 1] = __uint_as_float(u[q] & 0xffff0000u);
    }
  }
  if (tid < 2 * H) {
    W1[tid] = __bfloat162float(wb_in[OW1 + tid]);
    W3[tid] = __bfloat162float(wb_in[OW3 + tid]);
  }
  if (tid < H) {
    b1[tid] = __bfloat162float(wb_in[OB1 + tid]);
    b2[tid] = __bfloat162float(wb_in[OB2 + tid]);
  }
  if (tid < 2) b3[tid] = __bfloat162float(wb_in[OB3 + tid]);
  if (tid < 2 * GS) sx[tid] = first + tid / 2 < s0 + count ? x[2 * first + tid] : 0.f;
  const bool live = first + (tid >> 4) < s0 + count;
  const float t0 = live ? tg[2 * (first + (tid >> 4))] : 0.f, t1 = live ? tg[2 * (first + (tid >> 4)) + 1] : 0.f;
  __syncthreads();
  // layer 1
  for (int q = tid; q < GS * H; q += GT) {
    const int k = q / H, o = q % H;
    sh1[k * HP + o] = silu_f(W1[2 * o] * sx[2 * k] + W1[2 * o + 1] * sx[2 * k + 1] + b1[o]);
  }
  __syncthreads();
  // layer 2: sample sg and outputs og + 16 j
  const int og = tid & 15, sg = tid >> 4;
  float a2[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) a2[j] = b2[og + 16 * j];
  {
    const float *h0 = sh1 + sg * HP;
#pragma unroll 4
    for (int i = 0; i < H; i += 4) {
      const float4 p = *reinterpret_cast<const float4 *>(h0 + i);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 w = *reinterpret_cast<const float4 *>(W2 + (og + 16 * j) * HP + i);
        a2[j] += w.x * p.x; a2[j] += w.y * p.y; a2[j] += w.z * p.z; a2[j] += w.w * p.w;
      }
    }
  }
  // layer 3 (a sample's outputs over the 16 lanes of its group), loss, backward
  float l = 0.f, gy0, gy1;
  {
    float y0 = 0.f, y1 = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int o = og + 16 * j;
      const float h = silu_f(a2[j]);
      sh2[sg * HP + o] = h;
      y0 += W3[o] * h;
      y1 += W3[H + o] * h;
    }
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) {
      y0 += __shfl_xor_sync(0xffffffffu, y0, d);
      y1 += __shfl_xor_sync(0xffffffffu, y1, d);
    }
    const float r0 = live ? y0 + b3[0] - t0 : 0.f, r1 = live ? y1 + b3[1] - t1 : 0.f;
    gy0 = 2.f * r0 * inv_n;
    gy1 = 2.f * r1 * inv_n;
    if (og == 0) {
      sgy[2 * sg] = gy0;
      sgy[2 * sg + 1] = gy1;
      l = r0 * r0 + r1 * r1;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int o = og + 16 * j;
      sg2[sg * HP + o] = (W3[o] * gy0 + W3[H + o] * gy1) * dsilu_f(a2[j]);
    }
  }
  l += __shfl_xor_sync(0xffffffffu, l, 16);   // the warp's two samples
  if ((tid & 31) == 0) atomicAdd(loss, l * inv_n);
  __syncthreads();
  // gradient of hidden 1: sample sg and inputs 4 og .. 4 og + 3
  {
    float gh[4] = {0.f, 0.f, 0.f, 0.f};
    const float *g0 = sg2 + sg * HP;
#pragma unroll 4
    for (int o = 0; o < H; o += 4) {
      const float4 p = *reinterpret_cast<const float4 *>(g0 + o);
      const float pa[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 w = *reinterpret_cast<const float4 *>(W2 + (o + j) * HP + 4 * og);
        gh[0] += w.x * pa[j]; gh[1] += w.y * pa[j]; gh[2] += w.z * pa[j]; gh[3] += w.w * pa[j];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = 4 * og + u;
      const float a1 = W1[2 * i] * sx[2 * sg] + W1[2 * i + 1] * sx[2 * sg + 1] + b1[i];
      sg1[sg * HP + i] = gh[u] * dsilu_f(a1);
    }
  }
  // dW2[o][i] = sum_s ga2[s][o] h1[s][i]: outputs 2 sg, 2 sg + 1, inputs 4 og .. 4 og + 3
  {
    float d[2][4] = {};
#pragma unroll 8
    for (int k = 0; k < GS; ++k) {
      const float4 h = *reinterpret_cast<const float4 *>(sh1 + k * HP + 4 * og);
      const float2 q = *reinterpret_cast<const float2 *>(sg2 + k * HP + 2 * sg);
      d[0][0] += q.x * h.x; d[0][1] += q.x * h.y; d[0][2] += q.x * h.z; d[0][3] += q.x * h.w;
      d[1][0] += q.y * h.x; d[1][1] += q.y * h.y; d[1][2] += q.y * h.z; d[1][3] += q.y * h.w;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float *p = g + OW2 + (2 * sg + j) * H + 4 * og;
      if (vec) red4(p, d[j][0], d[j][1], d[j][2], d[j][3]);
      else
        for (int u = 0; u < 4; ++u) atomicAdd(p + u, d[j][u]);
    }
  }
  __syncthreads();
  // the small gradients: two warps per sum over the samples
  {
    const int o = tid & (H - 1), part = tid / H;
    if (part < 6) {
      const float *c = part == 0 ? sg2 : (part < 3 ? sh2 : sg1);
      const float *f = part == 1 || part == 2 ? sgy + part - 1 : sx + (part == 5 ? 1 : 0);
      const bool plain = part == 0 || part == 3;
      float d = 0.f;
#pragma unroll 8
      for (int k = 0; k < GS; ++k) d += plain ? c[k * HP + o] : c[k * HP + o] * f[2 * k];
      const int at = part == 0 ? OB2 + o : part == 1 ? OW3 + o : part == 2 ? OW3 + H + o : part == 3 ? OB1 + o
                                         : part == 4 ? OW1 + 2 * o : OW1 + 2 * o + 1;
      atomicAdd(g + at, d);
    } else if (part == 6 && o < 2) {
      float d = 0.f;
      for (int k = 0; k < GS; ++k) d += sgy[2 * k + o];
      atomicAdd(g + OB3 + o, d);
    }
  }
  if (!ad.done) return;
  // Adam in the CTA that finishes last: its additions are ordered before the count,
  // and the count before its reads
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(ad.done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // (all of a thread's loads before its arithmetic: one round of memory latency)
  constexpr int NQ = (NPARAM + GT - 1) / GT;
  float gq[NQ], mq[NQ], vq[NQ], wq[NQ];
#pragma unroll
  for (int u = 0; u < NQ; ++u) {
    const int q = tid + u * GT;
    if (q < NPARAM) {
      gq[u] = __ldcg(g + q);
      mq[u] = ad.m[q];
      vq[u] = ad.v[q];
      wq[u] = ad.w[q];
    }
  }
#pragma unroll
  for (int u = 0; u < NQ; ++u) {
    const int q = tid + u * GT;
    if (q < NPARAM) {
      const float m = ad.b1 * mq[u] + (1.f - ad.b1) * gq[u];
      const float v = ad.b2 * vq[u] + (1.f - ad.b2) * gq[u] * gq[u];
      const float w = wq[u] - ad.lr * (m / ad.bc1) / (sqrtf(v / ad.bc2) + ad.eps);
      ad.m[q] = m;
      ad.v[q] = v;
      ad.w[q] = w;
      ad.wb[q] = __float2bfloat16_rn(w);
      g[q] = 0.f;
    }
  }
  if (tid == 0) *ad.done = 0;
}

__global__ void k_round_bf16(const float *w, __nv_bfloat16 *wb, int n) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x)
    wb[q] = __float2bfloat16_rn(w[q]);
}

// ---------------------------------------------------------------- inference

// tcgen05 shared-memory matrix descriptor: K-major, no swizzle ("interleaved"
// core matrices of 8 rows x 16 bytes), leading-dimension byte offset = distance
// between core matrices along K, stride byte offset = distance between 8-row
// groups, descriptor version 1 (bits 46-47).
__device__ __forceinline__ unsigned long long smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (unsigned long long)((saddr & 0x3FFFFu) >> 4) | ((unsigned long long)(lbo >> 4) << 16) |
         ((unsigned long long)(sbo >> 4) << 32) | (1ull << 46);
}

// instruction descriptor, kind::f16: D = F32 (bits 4-5 = 1), A = B = BF16
// (bits 7-9 and 10-12 = 1), both K-major, N >> 3 in bits 17-22, M >> 4 in 24-28
constexpr uint32_t IDESC_BF16_M128_N64 = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) |
                                         ((128u >> 4) << 24);

// byte offset of element (row r, k) of a [rows][64] BF16 tile in the core-matrix layout
__device__ __forceinline__ uint32_t core_off(int r, int k) {
  return (uint32_t)((r >> 3) * 1024 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

constexpr int IT = 128;   // cells per tile = threads per CTA

// Wait until the mbarrier's phase of the given parity completes, for at most one
// second of the global nanosecond timer (try_wait may suspend the thread for a
// while, so the limit is on time, not on polls); false if it expired.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar_addr, uint32_t parity) {
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar_addr), "r"(parity));
    if (done) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > 1000000000ull) return false;
  }
}

struct SurrogateArgs {
  DTable t;
  MLPNorm nm;
  const __nv_bfloat16 *wb;
  long long n;
  const double *rho, *e;
  double *T, *P, *cs2;
  float *yout;        // raw network outputs [n][2] (normalised; NEWTON = 0)
  const float *xin;   // the network's inputs [n][2] (NEWTON = 0)
  Counters *cnt;
  int *status;        // set to 1 if a bounded wait expired
  int skip_mma;       // failure-detection test: issue no MMA, so the wait expires
  CellMap cm;         // which cells: plain arrays (cm.blocks null) or cells of blocks
  // the fused Newton step (k_eos_surrogate<1>): results of accepted cells, the
  // closure's clamped energy (eu, or null), the queue of cells left for
  // bisection and its length
  double *eu;
  long long *queue;
  unsigned long long *qcount;
  // the hydro form (k_eos_surrogate<2, DUAL>): the cells' conserved state and primitives
  Phys p;
  const double *U;
  double *W;
  long long ntot;
};

// Cells of a cell map: block position bp's cell count, and the array index of
// its cell `local` (plain arrays: one "block" of n cells, index = local).
__device__ __forceinline__ long long cm_cells(const CellMap &cm, long long n, int bp) {
  if (!cm.blocks) return n;
  const DevBlock &B = cm.blocks[cm.ids[bp]];
  return cm.padded ? (long long)B.p[0] * B.p[1] * B.p[2] : (long long)B.n[0] * B.n[1] * B.n[2];
}
__device__ __forceinline__ long long cm_flat(const CellMap &cm, int bp, long long local) {
  if (!cm.blocks) return cm.list ? (long long)cm.list[local] : local;
  const DevBlock &B = cm.blocks[cm.ids[bp]];
  if (cm.padded) return B.off + local;
  // 32-bit division only (a block has < 2^31 cells; 64-bit division would
  // take the FP64 pipe)
  const unsigned l = (unsigned)local, nx = (unsigned)B.n[0], ny = (unsigned)B.n[1];
  const unsigned r = l / nx;
  const int i = (int)(l - r * nx), k = (int)(r / ny), j = (int)(r - (unsigned)k * ny);
  return B.off + ((long long)(k + cm.g[2]) * B.p[1] + (j + cm.g[1])) * B.p[0] + (i + cm.g[0]);
}

// Split a tile or chunk index of a cell map into (block position, first cell),
// per = tiles or chunks per block, size = cells per tile or chunk; 32-bit
// division (counts < 2^31), none for plain arrays.
__device__ __forceinline__ void cm_split(const CellMap &cm, long long t, long long per, int size, int &bp,
                                         long long &first) {
  if (!cm.blocks) {
    bp = 0;
    first = t * size;
    return;
  }
  const unsigned q = (unsigned)t / (unsigned)per;
  bp = (int)q;
  first = (long long)((unsigned)t - q * (unsigned)per) * size;
}

// One Newton step from the guessed log10 T, judged by the table bracket.
// The column g is linear inside a temperature cell, so the step from the
// guess's cell j lands on x = j + (y - g_j) / (g_{j+1} - g_j); if the root is in
// cell j that is the root itself, otherwise x lies in the cell j' the linear
// extension points to (FP32 decides which), and the root is taken there when j'
// brackets it.  An accepted cell is the one bisection finds (g_j <= y < g_{j+1}
// is unique) and the state is evaluated with the same formulas (eos_at), so the
// result is the bisection result bit for bit.  Returns false for the cells left
// to bisection (clamped inputs, a step that misses).  FX: on the prepared table; else the
// step is taken in FP64 and the results in the form that the cell's entries call for, as
// eos_invert_views does (log e within 1e-12 of a node, where the two forms may see it in
// different cells, is left to it).
template <int FX>
__device__ __forceinline__ bool newton_cell(const DTable &t, double rho_c, double e, float lTg, float idlt,
                                            double &P, double &cs2, double *T) {
  if (!dgt0(e)) return false;
  const int nt = t.nt;
  if (!FX) {
    int i;
    double w;
    if (rho_cell(t, rho_c, i, w)) return false;
    const double y = tlog10(t, e);
    const double *__restrict__ ra = t.le + (size_t)i * nt;
    const double *__restrict__ rb = ra + nt;
    const float xg = (lTg - (float)t.lt0) * idlt;
    int j = (int)floorf(fminf(fmaxf(xg, 0.f), (float)(nt - 2)));
    j = min(max(j, 0), nt - 2);
    double g0 = lerp_rn(w, __ldg(ra + j), __ldg(rb + j)), g1 = lerp_rn(w, __ldg(ra + j + 1), __ldg(rb + j + 1));
    double s = cell_solve(y, g0, g1);
    if (!(dle(g0, y) && dlt(y, g1))) {
      const double xn = __dadd_rn(dint(j), s);   // the Newton result, in cell units
      if (!(xn >= 0.0 && xn < (double)(nt - 1))) return false;
      j = (int)xn;
      g0 = lerp_rn(w, __ldg(ra + j), __ldg(rb + j));
      g1 = lerp_rn(w, __ldg(ra + j + 1), __ldg(rb + j + 1));
      if (!(dle(g0, y) && dlt(y, g1))) return false;
      s = cell_solve(y, g0, g1);
    }
    if (!(y - g0 > 1e-12 && g1 - y > 1e-12)) return false;
    double ev;
    if (t.fa.valid) {
      int ix;
      ufx wx;
      bool cl = false, out;
      if (fx_rho_cell(t.fm, t.fa, t.nr, rho_c, ix, wx)) return false;
      if (fx_cell_views<true>(t, ix, wx, fx_log2(t.fm, e), j, cl, out, e, P, cs2, ev, T)) return !cl;
      if (!out) return false;
    }
    fp64_cell<true>(t, i, w, j, s, false, e, P, cs2, ev, T);
    return true;
  }
  int i;
  ufx w;
  if (fx_rho_cell(t.fm, t.fa, t.nr, rho_c, i, w)) return false;
  const fx y = fx_log2(t.fm, e);
  const longlong2 *__restrict__ row = t.node + (size_t)i * nt * 3;
  const float xg = (lTg - (float)t.lt0) * idlt;
  int j = (int)floorf(fminf(fmaxf(xg, 0.f), (float)(nt - 2)));
  j = min(max(j, 0), nt - 2);
  fx g0 = fx_pair(row + 3 * j, w), g1 = fx_pair(row + 3 * j + 3, w);
  bool in = g0 <= y && y < g1;
  if (!in) {
    // (the top 32 bits are enough to choose a cell)
    const float xn = (float)j + __fdividef((float)(int)((y - g0) >> 32), (float)max((int)((g1 - g0) >> 32), 1));
    if (xn >= 0.f && xn < (float)(nt - 1)) {
      j = (int)xn;
      g0 = fx_pair(row + 3 * j, w);
      g1 = fx_pair(row + 3 * j + 3, w);
      in = g0 <= y && y < g1;
    }
  }
  // at the coldest node bisection clamps (y <= g_0): leave that to it
  if (!(in && (j > 0 || g0 < y))) return false;
  double ev;
  eos_at<true>(t, row + 3 * j, w, j, fx_frac(y - g0, g1 - g0), false, e, P, cs2, ev, T);
  return true;
}

// The learned guess.
// NEWTON = 0: the network alone (raw outputs);
// NEWTON = 1: the guess goes straight into the Newton step in the same
// thread (newton_cell), accepted cells are written and the rest queued for
// k_eos_fallback (one atomic per tile reserves the tile's queue slots; the
// accepted count is added once per CTA);
// NEWTON = 2 (hydro): as 1, with the table inputs formed from the cell's conserved
// state and the primitives of accepted cells written, so the FP64 work of the
// conversion runs beside the network's integer and MUFU work and the state is read by
// one kernel; the queued cells are converted by k_fallback_c2p.  A step of 8.4 M cells:
// 14.3 -> 13.2 ms against separate kernels for inputs, inversion and conversion.
// What bounds it is instruction issue (two thirds of its slots): the layers go two
// units at a time through the packed FP32 FMA, and the output the inversion does not
// use is left out (5.9 M cells 780 -> 728 us; one 16-byte record of weights per unit
// instead of an array per weight was slower, 868 us: a third more shared reads).
// FX: the table has the prepared form (newton_cell).
template <int NEWTON, int DUAL = 0, int FX = 1>
__global__ void __launch_bounds__(IT, FX ? 8 : 6) k_eos_surrogate(const SurrogateArgs a) {
  pdl_begin();
  __shared__ __align__(1024) unsigned char sA[IT * H * 2];   // h1, BF16, core-matrix layout
  __shared__ __align__(1024) unsigned char sB[H * H * 2];    // W2, BF16, core-matrix layout
  // layer 1's weights and the hidden biases, halved for silu2_half; read four at a time
  __shared__ __align__(16) float sW1[2][H], sb1[H], sb2[H], sW3[2][H];
  __shared__ float sb3[2];
  __shared__ __align__(8) unsigned long long mbar;
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort;
  __shared__ unsigned s_wc[IT / 32];
  __shared__ unsigned long long s_base;
  __shared__ unsigned s_acc;
  unsigned n_acc = 0;
  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t sA_addr = (uint32_t)__cvta_generic_to_shared(sA);
  const uint32_t sB_addr = (uint32_t)__cvta_generic_to_shared(sB);
  const uint32_t mbar_addr = (uint32_t)__cvta_generic_to_shared(&mbar);
  if (warp == 0) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&tmem_base);
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst), "r"(64));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  for (int q = tid; q < H * H; q += IT) {
    const int o = q / H, i = q % H;
    *reinterpret_cast<__nv_bfloat16 *>(sB + core_off(o, i)) = a.wb[OW2 + q];
  }
  if (tid < H) {
    sW1[0][tid] = 0.5f * __bfloat162float(a.wb[OW1 + 2 * tid]);
    sW1[1][tid] = 0.5f * __bfloat162float(a.wb[OW1 + 2 * tid + 1]);
    sb1[tid] = 0.5f * __bfloat162float(a.wb[OB1 + tid]);
    sb2[tid] = 0.5f * __bfloat162float(a.wb[OB2 + tid]);
    sW3[0][tid] = __bfloat162float(a.wb[OW3 + tid]);
    sW3[1][tid] = __bfloat162float(a.wb[OW3 + H + tid]);
  }
  if (tid < 2) sb3[tid] = __bfloat162float(a.wb[OB3 + tid]);
  if (tid == 0) {
    s_abort = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_addr), "r"(1));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tbase = tmem_base;
  uint32_t phase = 0;
  // tiles of IT cells, tpb per block (a.n = the largest block's cell count)
  const long long tpb = (a.n + IT - 1) / IT;
  const long long ntiles = tpb * (a.cm.blocks ? a.cm.nblk : 1);
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    int bp;
    long long first;
    cm_split(a.cm, tile, tpb, IT, bp, first);
    const long long ncell = cm_cells(a.cm, a.n, bp);
    if (first >= ncell) continue;   // the whole tile (uniform)
    const long long local = first + tid;
    const bool live = local < ncell;
    const long long c = live ? cm_flat(a.cm, bp, local) : 0;
    // after an expired wait (s_abort, uniform) the network is skipped: the
    // Newton kernel queues the remaining cells for bisection, the plain one stops
    float y0 = 0.f;
    double rho_c = 1.0, e_c = 0.0;   // the table's inputs
    if (NEWTON == 2 && live) {
      double u[6], vx, vy, vz, Ue, rho;
#pragma unroll
      for (int v = 0; v < 5 + DUAL; ++v) u[v] = a.U[v * a.ntot + c];
      c2p_energy<DUAL>(a.p, u, rho, vx, vy, vz, Ue, nullptr);
      eos_inputs(a.p, rho, Ue, rho_c, e_c);
    }
    if (!s_abort) {
      // ---- inputs and layer 1, FP32 only: the network needs log10 rho and the
      // position z of log10 e in its column to FP32 accuracy (the exact work of
      // the inversion is newton_cell's)
      float x0 = 0.f, x1 = 0.f;
      if (live) {
        if (!NEWTON) {
          x0 = a.xin[2 * c];
          x1 = a.xin[2 * c + 1];
        } else {
          const DTable &t = a.t;
          const float lr = __log2f((float)(NEWTON == 1 ? a.rho[c] : rho_c)) * 0.30102999566f;
          const float ly = __log2f((float)(NEWTON == 1 ? a.e[c] : e_c)) * 0.30102999566f;
          const float xr = fminf(fmaxf((lr - (float)t.lr0) * (float)t.inv_dlr, 0.f), (float)(t.nr - 1));
          const int ti = min((int)xr, t.nr - 2);
          const float w32 = xr - (float)ti;
          const float *__restrict__ ra = t.le32 + (size_t)ti * t.nt;
          const float *__restrict__ rb = ra + t.nt;
          const float glo = fmaf(w32, __ldg(rb) - __ldg(ra), __ldg(ra));
          const float ghi = fmaf(w32, __ldg(rb + t.nt - 1) - __ldg(ra + t.nt - 1), __ldg(ra + t.nt - 1));
          x0 = fminf(fmaxf((lr - a.nm.cr) * a.nm.isr, -2.f), 2.f);
          const float z = __fdividef(ly - glo, ghi - glo);
          x1 = (fminf(fmaxf(z, -1.f), 2.f) - a.nm.ce) * a.nm.ise;
        }
      }
      const f2 xx0 = f2_pack(x0, x0), xx1 = f2_pack(x1, x1);
#pragma unroll
      for (int k8 = 0; k8 < H / 8; ++k8) {
        __align__(16) __nv_bfloat162 hv[4];
#pragma unroll
        for (int u = 0; u < 8; u += 4) {
          const int o = 8 * k8 + u;
          const ulonglong2 w0 = *reinterpret_cast<const ulonglong2 *>(&sW1[0][o]);
          const ulonglong2 w1 = *reinterpret_cast<const ulonglong2 *>(&sW1[1][o]);
          const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(&sb1[o]);
          float h0, h1;
          f2_split(silu2_half(f2_fma(w0.x, xx0, f2_fma(w1.x, xx1, b.x))), h0, h1);
          hv[u / 2] = __floats2bfloat162_rn(h0, h1);
          f2_split(silu2_half(f2_fma(w0.y, xx0, f2_fma(w1.y, xx1, b.y))), h0, h1);
          hv[u / 2 + 1] = __floats2bfloat162_rn(h0, h1);
        }
        *reinterpret_cast<uint4 *>(sA + core_off(tid, 8 * k8)) = *reinterpret_cast<uint4 *>(hv);
      }
      // make the generic-proxy shared stores visible to the tensor core
      asm volatile("fence.proxy.async.shared::cta;");
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncthreads();
      // ---- layer 2 on the tensor core: D[128 x 64] = h1[128 x 64] * W2^T
      if (tid == 0 && !a.skip_mma) {
        asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
        for (int ks = 0; ks < H / 16; ++ks) {
          const unsigned long long ad = smem_desc(sA_addr + ks * 256, 128, 1024);
          const unsigned long long bd = smem_desc(sB_addr + ks * 256, 128, 1024);
          const uint32_t acc = ks > 0 ? 1u : 0u;
          asm volatile(
              "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tbase),
              "l"(ad), "l"(bd), "r"(IDESC_BF16_M128_N64), "r"(acc));
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            mbar_addr));
      }
      // bounded wait for the MMAs (one second of the global timer at most)
      if (!mbar_wait_bounded(mbar_addr, phase)) s_abort = 1;
      phase ^= 1u;
      __syncthreads();
      if (!s_abort) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        // ---- read the accumulator row of this thread (warp w owns TMEM lanes
        // 32w..32w+31) in two halves of 32 columns, and apply layer 3 (FP32)
        // (two units at a time; the second output, log P, is not the inversion's)
        const f2 half2 = f2_pack(0.5f, 0.5f);
        f2 yy0 = f2_pack(sb3[0], 0.f), yy1 = f2_pack(sb3[1], 0.f);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t r[32];
          const uint32_t taddr = tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)(32 * hf);
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
              "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
              : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
                "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
                "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
                "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
              : "r"(taddr));
          asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
          for (int q = 0; q < 32; q += 4) {
            const int o = 32 * hf + q;
            const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(&sb2[o]);
            const ulonglong2 w0 = *reinterpret_cast<const ulonglong2 *>(&sW3[0][o]);
            const ulonglong2 w1 = *reinterpret_cast<const ulonglong2 *>(&sW3[1][o]);
            const f2 p = silu2_half(f2_fma(f2_pack(__uint_as_float(r[q]), __uint_as_float(r[q + 1])), half2, b.x));
            yy0 = f2_fma(w0.x, p, yy0);
            if (!NEWTON) yy1 = f2_fma(w1.x, p, yy1);
            const f2 v = silu2_half(f2_fma(f2_pack(__uint_as_float(r[q + 2]), __uint_as_float(r[q + 3])), half2, b.y));
            yy0 = f2_fma(w0.y, v, yy0);
            if (!NEWTON) yy1 = f2_fma(w1.y, v, yy1);
          }
        }
        float y0a, y0b;
        f2_split(yy0, y0a, y0b);
        y0 = y0a + y0b;
        if (!NEWTON && live) {
          float y1a, y1b;
          f2_split(yy1, y1a, y1b);
          a.yout[2 * c] = y0;
          a.yout[2 * c + 1] = y1a + y1b;
        }
      }
      // every thread has its row in registers: the next tile may reuse sA and TMEM
      asm volatile("tcgen05.fence::before_thread_sync;");
    }
    const bool have = !s_abort;   // uniform: set before the last barrier
    if (!NEWTON && !have) break;
    if (NEWTON) {
      // the Newton step from this thread's guess; misses are queued
      double Pv, cv, Tv;
      if (NEWTON == 1 && live) {   // (read again: not held in registers through the network)
        rho_c = a.rho[c];
        e_c = a.e[c];
      }
      const bool ok = live ? (have && newton_cell<FX>(a.t, rho_c, e_c, a.nm.cT + a.nm.sT * y0, a.nm.idlt, Pv, cv,
                                                      NEWTON == 1 && a.T ? &Tv : nullptr))
                           : true;
      if (NEWTON == 1 && live && ok) {
        if (a.P) a.P[c] = Pv;
        if (a.cs2) a.cs2[c] = cv;
        if (a.T) a.T[c] = Tv;
        if (a.eu) a.eu[c] = 0.0;   // inside the table
      }
      if (NEWTON == 2 && live && ok) {
        double u[6], w[8], vx, vy, vz, Ue, rho;
#pragma unroll
        for (int v = 0; v < 5 + DUAL; ++v) u[v] = a.U[v * a.ntot + c];
        c2p_energy<DUAL>(a.p, u, rho, vx, vy, vz, Ue, a.cnt);
        c2p_prims<EOS_TABLE, DUAL>(a.p, DUAL ? u[5] : 0.0, rho, vx, vy, vz, Pv * a.p.inv_unit_p, cv * a.p.inv_unit_e,
                                   Ue, w, a.cnt);
#pragma unroll
        for (int v = 0; v < 7 + DUAL; ++v) a.W[v * a.ntot + c] = w[v];
      }
      n_acc += (live && ok) ? 1u : 0u;
      const int lane = tid & 31;
      const unsigned rm = __ballot_sync(0xffffffffu, !ok);
      if (lane == 0) s_wc[warp] = __popc(rm);
      __syncthreads();
      if (tid == 0) {
        unsigned tot = 0;
        for (int q = 0; q < IT / 32; ++q) {
          const unsigned v = s_wc[q];
          s_wc[q] = tot;   // exclusive prefix over the warps
          tot += v;
        }
        s_base = tot ? atomicAdd(a.qcount, (unsigned long long)tot) : 0ull;
      }
      __syncthreads();
      if (!ok) a.queue[s_base + s_wc[warp] + __popc(rm & ((1u << lane) - 1u))] = c;
    }
    __syncthreads();
  }
  if (NEWTON) {   // accepted cells: one atomic per CTA
    for (int o = 16; o > 0; o >>= 1) n_acc += __shfl_xor_sync(0xffffffffu, n_acc, o);
    if (tid == 0) s_acc = 0;
    __syncthreads();
    if ((tid & 31) == 0) atomicAdd(&s_acc, n_acc);
    __syncthreads();
    if (tid == 0 && a.cnt && s_acc) atomicAdd(&a.cnt->surrogate_accepted, (unsigned long long)s_acc);
  }
  if (s_abort && tid == 0) atomicExch(a.status, 1);
  // wait (bounded) for any MMA still in flight before freeing tensor memory
  if (s_abort) mbar_wait_bounded(mbar_addr, phase ^ 1u);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(64));
}

// Table bisection for the cells the Newton step left (their indices in queue).
// With eu (the hydro closure's buffers) the clamped table energy is returned
// (0 inside the table) and the closure counts clamps; without, they are counted here.
// PREP: the table has its prepared form.
template <int PREP>
__global__ void __launch_bounds__(256) k_eos_fallback(DTable t, const long long *queue,
                                                      const unsigned long long *qcount,
                                                      const double *rho,
                                                      const double *e, double *T, double *P,
                                                      double *cs2, double *eu, Counters *cnt) {
  pdl_begin();
  const long long nq = (long long)*qcount;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nq;
       q += (long long)gridDim.x * blockDim.x) {
    const long long c = queue[q];
    double Pv, cv, euv, Tv;
    const bool cl = PREP ? eos_invert_node(t, rho[c], e[c], Pv, cv, euv, &Tv) : eos_invert(t, rho[c], e[c], Pv, cv, euv, &Tv);
    if (cl && !eu) count(&cnt->table_clamp);
    if (T) T[c] = Tv;
    if (P) P[c] = Pv;
    if (cs2) cs2[c] = cv;
    if (eu) eu[c] = cl ? euv : 0.0;
  }
}

// the primitives of the cells the hydro form left (their indices in queue)
template <int DUAL, int PREP>
__global__ void __launch_bounds__(256) k_fallback_c2p(Phys p, const long long *queue, const unsigned long long *qcount,
                                                      const double *U, double *W, long long ntot, Counters *cnt) {
  pdl_begin();
  const long long nq = (long long)*qcount;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nq;
       q += (long long)gridDim.x * blockDim.x) {
    const long long c = queue[q];
    double u[6], w[8];
#pragma unroll
    for (int v = 0; v < 5 + DUAL; ++v) u[v] = U[v * ntot + c];
    cons_to_prim<EOS_TABLE, DUAL, PREP ? 2 : 0>(p, u, w, cnt);
#pragma unroll
    for (int v = 0; v < 7 + DUAL; ++v) W[v * ntot + c] = w[v];
  }
}

}  // namespace tde

// ================================================================ host side

#include <random>

using namespace tde;

namespace {

int mlp_fail(tde_ctx *c, int code, const char *msg) {
  c->err = msg;
  return code;
}

#define MCK(ctx, call)                                                   \
  do {                                                                   \
    cudaError_t _e = (call);                                             \
    if (_e != cudaSuccess) {                                             \
      (ctx)->err = std::string(#call) + ": " + cudaGetErrorString(_e);   \
      return TDE_ECUDA;                                                  \
    }                                                                    \
  } while (0)

// d_w: the weights, Adam's m and v (NPARAM floats each), the gradient (from OG, so
// that its W2 part starts on 16 bytes) and the count of finished CTAs
constexpr int OG = (3 * NPARAM + OW2 + 3) / 4 * 4 - OW2, WBUF = OG + NPARAM + 2;
static_assert((OG + OW2) % 4 == 0 && OG >= 3 * NPARAM, "gradient alignment");

MLPNorm norm_of(const tde_eos *e) {
  MLPNorm n;
  n.cr = (float)e->norm[0]; n.sr = (float)e->norm[1];
  n.ce = (float)e->norm[2]; n.se = (float)e->norm[3];
  n.cT = (float)e->norm[4]; n.sT = (float)e->norm[5];
  n.cP = (float)e->norm[6]; n.sP = (float)e->norm[7];
  n.isr = (float)(1.0 / e->norm[1]);
  n.ise = (float)(1.0 / e->norm[3]);
  n.idlt = (float)(1.0 / e->tab.dlt);
  return n;
}

int ensure_net_buffers(tde_eos *e) {
  tde_ctx *c = e->ctx;
  if (!e->d_w) {
    MCK(c, cudaMalloc(&e->d_w, sizeof(float) * WBUF));
    MCK(c, cudaMemset(e->d_w, 0, sizeof(float) * WBUF));
  }
  if (!e->d_wb) MCK(c, cudaMalloc(&e->d_wb, sizeof(__nv_bfloat16) * NPARAM));
  if (!e->d_status) {
    MCK(c, cudaMalloc(&e->d_status, sizeof(int)));
    MCK(c, cudaMemset(e->d_status, 0, sizeof(int)));
  }
  return TDE_OK;
}

int upload_weights(tde_eos *e, const float *w) {
  tde_ctx *c = e->ctx;
  MCK(c, cudaMemcpyAsync(e->d_w, w, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, c->stream));
  MCK(c, cudaMemsetAsync(e->d_w + NPARAM, 0, sizeof(float) * (WBUF - NPARAM), c->stream));   // m, v, g, count
  k_round_bf16<<<(NPARAM + 255) / 256, 256, 0, c->stream>>>(e->d_w, (__nv_bfloat16 *)e->d_wb, NPARAM);
  MCK(c, cudaGetLastError());
  MCK(c, cudaStreamSynchronize(c->stream));
  e->has_net = true;
  return TDE_OK;
}

size_t grad_smem() { return sizeof(float) * ((H + 4 * GS) * HP + 2 * H + H + H + 2 * H + 4 + 4 * GS); }

cudaError_t launch_grad(tde_eos *e, const float *x, const float *tg, long long s0, long long count,
                        float inv_n, float *g, float *loss, const AdamArgs &ad, cudaStream_t s) {
  cudaError_t err = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)grad_smem());
  if (err != cudaSuccess) return err;
  const unsigned grid = (unsigned)((count + GS - 1) / GS);
  pdl_launch(k_mlp_grad, grid, GT, grad_smem(), s, (const __nv_bfloat16 *)e->d_wb, x, tg, s0, count, inv_n, g,
                                           loss, ad);
  return cudaGetLastError();
}

// the network alone on n normalised inputs xin
cudaError_t launch_surrogate_kernel(tde_eos *e, long long n, const float *xin, float *yout, cudaStream_t s) {
  SurrogateArgs a{};
  a.t = e->tab;
  a.nm = norm_of(e);
  a.wb = (const __nv_bfloat16 *)e->d_wb;
  a.n = n;
  a.yout = yout;
  a.xin = xin;
  a.cnt = e->d_cnt;
  a.status = e->d_status;
  a.skip_mma = e->inject_wait_expiry;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, e->ctx->device);
  // one wave of resident CTAs: registers (64 x 128 threads) and shared memory
  // (27 KB, largest carveout) admit 8 per SM, and 8 x 64 TMEM columns fill the
  // SM's 512 exactly
  cudaFuncSetAttribute(k_eos_surrogate<0>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       (int)cudaSharedmemCarveoutMaxShared);
  const int per_sm = 8;
  const long long tiles = (n + IT - 1) / IT;
  const unsigned grid = (unsigned)std::min<long long>(tiles, (long long)sms * per_sm);
  pdl_launch(k_eos_surrogate<0>, grid, IT, 0, s, a);
  return cudaGetLastError();
}

// the network and the Newton step in one pass (k_eos_surrogate<1>): 8 CTAs per
// SM (64 registers), 8 x 64 TMEM columns fill the SM's 512 (six CTAs with the FP64
// Newton step)
cudaError_t launch_surrogate_newton(tde_eos *e, const CellMap &cm, long long n, const double *rho,
                                    const double *en, double *T, double *P, double *cs2, double *eu,
                                    long long *queue, unsigned long long *qcount, Counters *cnt,
                                    cudaStream_t s, const tde_mesh *hy = nullptr, const double *hyU = nullptr) {
  SurrogateArgs a{};
  a.t = e->tab;
  a.nm = norm_of(e);
  a.wb = (const __nv_bfloat16 *)e->d_wb;
  a.n = n;
  a.rho = rho;
  a.e = en;
  a.T = T;
  a.P = P;
  a.cs2 = cs2;
  a.cnt = cnt;
  a.status = e->d_status;
  a.skip_mma = e->inject_wait_expiry;
  a.cm = cm;
  a.eu = eu;
  a.queue = queue;
  a.qcount = qcount;
  const bool fx = e->tab.node != nullptr;
  auto k = fx ? k_eos_surrogate<1> : k_eos_surrogate<1, 0, 0>;
  if (hy) {
    a.p = hy->phys;
    a.U = hyU;
    a.W = hy->d_W;
    a.ntot = (long long)hy->ntot;
    if (fx) k = hy->phys.dual ? k_eos_surrogate<2, 1> : k_eos_surrogate<2, 0>;
    else k = hy->phys.dual ? k_eos_surrogate<2, 1, 0> : k_eos_surrogate<2, 0, 0>;
  }
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, e->ctx->device);
  cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  const int per_sm = fx ? 8 : 6;
  const long long tiles = (n + IT - 1) / IT * (cm.blocks ? cm.nblk : 1);
  const unsigned grid = (unsigned)std::min<long long>(tiles, (long long)sms * per_sm);
  pdl_launch(k, grid, IT, 0, s, a);
  return cudaGetLastError();
}

// The learned-guess inversion of the cells of cm (n = largest block's cell
// count, or the array length): guess, Newton step with queueing, bisection of
// the queue.  The same inputs give the bisection results bit for bit.
cudaError_t surrogate_run(tde_eos *e, const CellMap &cm, long long n, const double *rho,
                          const double *en, double *T, double *P, double *cs2, double *eu,
                          long long *queue, unsigned long long *qcount, Counters *cnt, cudaStream_t s) {
  cudaError_t r = cudaMemsetAsync(qcount, 0, sizeof(unsigned long long), s);
  if (r != cudaSuccess) return r;
  r = launch_surrogate_newton(e, cm, n, rho, en, T, P, cs2, eu, queue, qcount, cnt, s);
  if (r != cudaSuccess) return r;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, e->ctx->device);
  const long long ncell = n * (cm.blocks ? cm.nblk : 1);
  const unsigned gf = (unsigned)std::min<long long>((ncell + 255) / 256, (long long)sms * 8);
  pdl_launch(e->tab.node ? k_eos_fallback<1> : k_eos_fallback<0>, gf, 256, 0, s, e->tab, queue, qcount, rho, en, T, P, cs2, eu, cnt);
  return cudaGetLastError();
}

}  // namespace

namespace tde {
cudaError_t launch_eos_surrogate(tde_eos *e, int64_t n, const double *rho, const double *en,
                                 double *T, double *P, double *cs2, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (e->queue_cap < n) {
    cudaFree(e->d_queue);
    e->d_queue = nullptr;
    e->queue_cap = 0;
    cudaError_t r = cudaMalloc(&e->d_queue, sizeof(long long) * (size_t)n);
    if (r != cudaSuccess) return r;
    e->queue_cap = n;
  }
  if (!e->d_qcount) {
    cudaError_t r = cudaMalloc(&e->d_qcount, sizeof(unsigned long long));
    if (r != cudaSuccess) return r;
  }
  ProfScope ps(e->ctx, TDE_K_EOS);
  e->ctx->launches[TDE_K_EOS] += 1;   // the guess with its Newton step, then the bisection of the misses
  return surrogate_run(e, CellMap{}, n, rho, en, T, P, cs2, nullptr, e->d_queue,
                       e->d_qcount, e->d_cnt, s);
}

// the interior cells of cm from the state U to the mesh's primitives: guess, Newton
// step and conversion in one kernel, then the queued cells
cudaError_t launch_surrogate_c2p(tde_mesh *m, const CellMap &cm, int64_t nmax, const double *U, cudaStream_t s) {
  tde_eos *e = m->eos;
  const SurrogateBuf &sb = m->sb;
  cudaError_t r = cudaMemsetAsync(sb.qcount, 0, sizeof(unsigned long long), s);
  if (r != cudaSuccess) return r;
  r = launch_surrogate_newton(e, cm, nmax, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, sb.queue, sb.qcount,
                              m->d_cnt, s, m, U);
  if (r != cudaSuccess) return r;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, e->ctx->device);
  const unsigned gf = (unsigned)std::min<long long>((nmax * cm.nblk + 255) / 256, (long long)sms * 8);
  auto k = m->phys.dual ? k_fallback_c2p<1, 0> : k_fallback_c2p<0, 0>;
  if (e->tab.node) k = m->phys.dual ? k_fallback_c2p<1, 1> : k_fallback_c2p<0, 1>;
  return pdl_launch(k, gf, 256, 0, s, m->phys, sb.queue, sb.qcount, U, m->d_W, (long long)m->ntot, m->d_cnt);
}

cudaError_t launch_eos_surrogate_cells(tde_eos *e, const CellMap &cm, int64_t nmax,
                                       const SurrogateBuf &sb, Counters *cnt, cudaStream_t s) {
  if (nmax <= 0 || cm.nblk <= 0) return cudaSuccess;
  return surrogate_run(e, cm, nmax, sb.rho, sb.e, nullptr, sb.P, sb.cs2, sb.eu, sb.queue,
                       sb.qcount, cnt, s);
}
}  // namespace tde

extern "C" int tde_eos_surrogate_set_weights(tde_eos *e, const float *w, size_t n) {
  if (!e) return TDE_EINVAL;
  if (!w || n != (size_t)NPARAM) return mlp_fail(e->ctx, TDE_EINVAL, "tde_eos_surrogate_set_weights: need 4482 floats");
  int r = ensure_net_buffers(e);
  if (r) return r;
  return upload_weights(e, w);
}

extern "C" int tde_eos_surrogate_get_weights(tde_eos *e, float *w, size_t n) {
  if (!e) return TDE_EINVAL;
  if (!w || n != (size_t)NPARAM || !e->has_net) return mlp_fail(e->ctx, TDE_EINVAL, "tde_eos_surrogate_get_weights: no weights or size");
  MCK(e->ctx, cudaMemcpyAsync(w, e->d_w, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, e->ctx->stream));
  MCK(e->ctx, cudaStreamSynchronize(e->ctx->stream));
  return TDE_OK;
}

extern "C" int tde_eos_surrogate_reset(tde_eos *e) {
  if (!e) return TDE_EINVAL;
  e->has_net = false;
  return TDE_OK;
}

extern "C" int tde_eos_inject_wait_expiry(tde_eos *e, int on) {
  if (!e) return TDE_EINVAL;
  e->inject_wait_expiry = on ? 1 : 0;
  return TDE_OK;
}

extern "C" int tde_eos_check(tde_eos *e) {
  if (!e) return TDE_EINVAL;
  tde_ctx *c = e->ctx;
  MCK(c, cudaStreamSynchronize(c->stream));
  if (!e->d_status) return TDE_OK;
  int st = 0;
  MCK(c, cudaMemcpy(&st, e->d_status, sizeof(int), cudaMemcpyDeviceToHost));
  if (!st) return TDE_OK;
  MCK(c, cudaMemset(e->d_status, 0, sizeof(int)));
  return mlp_fail(c, TDE_ETIMEOUT,
                  "learned-guess inference: a bounded wait for the tensor-core results expired (the cells "
                  "took the bisection fallback)");
}

extern "C" int tde_eos_surrogate_norm(const tde_eos *e, double *out8) {
  if (!e || !out8) return TDE_EINVAL;
  memcpy(out8, e->norm, sizeof(e->norm));
  return TDE_OK;
}

extern "C" int tde_eos_surrogate_grad(tde_eos *e, int64_t n, const float *x, const float *target,
                                      float *grad, float *loss) {
  if (!e) return TDE_EINVAL;
  tde_ctx *c = e->ctx;
  if (n <= 0 || !x || !target || !grad || !loss || !e->has_net)
    return mlp_fail(c, TDE_EINVAL, "tde_eos_surrogate_grad: arguments or no weights");
  MCK(c, cudaMemsetAsync(grad, 0, sizeof(float) * NPARAM, c->stream));
  MCK(c, cudaMemsetAsync(loss, 0, sizeof(float), c->stream));
  ProfScope ps(c, TDE_K_EOS);
  MCK(c, launch_grad(e, x, target, 0, n, 1.0f / (float)n, grad, loss, AdamArgs{}, c->stream));
  return TDE_OK;
}

extern "C" int tde_eos_surrogate_forward(tde_eos *e, int64_t n, const float *x, float *y) {
  if (!e) return TDE_EINVAL;
  tde_ctx *c = e->ctx;
  if (n <= 0 || !x || !y || !e->has_net) return mlp_fail(c, TDE_EINVAL, "tde_eos_surrogate_forward: arguments or no weights");
  ProfScope ps(c, TDE_K_EOS);
  MCK(c, launch_surrogate_kernel(e, n, x, y, c->stream));
  return TDE_OK;
}

extern "C" int tde_eos_surrogate_train(tde_eos *e, uint64_t seed, int n_samples, int epochs, int batch,
                                       double lr, tde_train_report *rep) {
  if (!e) return TDE_EINVAL;
  tde_ctx *c = e->ctx;
  if (n_samples < TRAIN_ALIGN || epochs < 1 || batch < TRAIN_ALIGN || batch % TRAIN_ALIGN || !(lr > 0.0))
    return mlp_fail(c, TDE_EINVAL, "tde_eos_surrogate_train: sizes (batch a multiple of 128)");
  int r = ensure_net_buffers(e);
  if (r) return r;
  if (!e->has_net) {   // seeded Glorot-normal initialisation, zero biases
    std::vector<float> w(NPARAM, 0.f);
    std::mt19937_64 rng(seed ^ 0x5eedull);
    auto fill = [&](int off, int fan_out, int fan_in) {
      std::normal_distribution<float> nd(0.f, std::sqrt(2.f / (fan_in + fan_out)));
      for (int q = 0; q < fan_out * fan_in; ++q) w[off + q] = nd(rng);
    };
    fill(OW1, H, 2);
    fill(OW2, H, H);
    fill(OW3, 2, H);
    r = upload_weights(e, w.data());
    if (r) return r;
  }
  const int nb_per_epoch = n_samples / batch;
  const int nbt = nb_per_epoch * epochs;
  cudaStream_t s = c->stream;
  // samples, targets and losses in one allocation, given back below.  A stream-ordered one
  // maps its memory anew after every synchronisation (0.1 ms), a small ordinary one comes
  // out of a block that is mapped already, a large one does not: a training of one batch of
  // 4096 samples (64 KB) takes 156 and 53 us, one of 2^15 (512 KB) 262 and 309.
  float *d_x = nullptr;
  const size_t bytes = sizeof(float) * (4 * (size_t)n_samples + nbt);
  const bool ordered = bytes > 128 * 1024;
  MCK(c, ordered ? cudaMallocAsync((void **)&d_x, bytes, s) : cudaMalloc((void **)&d_x, bytes));
  float *d_y = d_x + 2 * (size_t)n_samples, *d_loss = d_y + 2 * (size_t)n_samples;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaEventRecord(e0, s);
  cudaMemsetAsync(d_loss, 0, sizeof(float) * nbt, s);
  k_mlp_samples<<<1024, 256, 0, s>>>(e->tab, norm_of(e), n_samples, seed, d_x, d_y);
  AdamArgs ad;
  ad.w = e->d_w;
  ad.m = ad.w + NPARAM;
  ad.v = ad.m + NPARAM;
  ad.wb = (__nv_bfloat16 *)e->d_wb;
  ad.b1 = 0.9f;
  ad.b2 = 0.999f;
  ad.eps = 1e-8f;
  float *g = e->d_w + OG;
  ad.done = reinterpret_cast<unsigned *>(g + NPARAM);
  int step = 0;
  cudaError_t err = cudaGetLastError();
  for (int ep = 0; ep < epochs && err == cudaSuccess; ++ep) {
    for (int bi = 0; bi < nb_per_epoch && err == cudaSuccess; ++bi, ++step) {
      const double prog = (double)step / (double)nbt;
      ad.lr = (float)(lr * (0.05 + 0.95 * 0.5 * (1.0 + cos(3.141592653589793 * prog))));
      ad.bc1 = 1.f - powf(ad.b1, (float)(step + 1));
      ad.bc2 = 1.f - powf(ad.b2, (float)(step + 1));
      err = launch_grad(e, d_x, d_y, (long long)bi * batch, batch, 1.0f / batch, g, d_loss + step, ad, s);
    }
  }
  cudaEventRecord(e1, s);
  std::vector<float> losses(nbt);
  if (err == cudaSuccess) err = cudaMemcpyAsync(losses.data(), d_loss, sizeof(float) * nbt, cudaMemcpyDeviceToHost, s);
  if (err == cudaSuccess) err = cudaStreamSynchronize(s);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (ordered) cudaFreeAsync(d_x, s);
  else cudaFree(d_x);
  if (err != cudaSuccess) {
    c->err = std::string("tde_eos_surrogate_train: ") + cudaGetErrorString(err);
    return TDE_ECUDA;
  }
  c->launches[TDE_K_EOS] += (uint64_t)nbt + 1;
  if (rep) {
    rep->loss_first = nbt ? losses.front() : 0.0;   // (fewer samples than a batch: nothing to train on)
    rep->loss_last = nbt ? losses.back() : 0.0;
    rep->epochs = epochs;
    rep->samples = n_samples;
    rep->batches = nbt;
    rep->ms = ms;
  }
  return TDE_OK;
}
