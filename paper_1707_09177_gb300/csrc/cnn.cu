// Learned initial guess for BiCGSTAB: a four-layer bias-free 3x3x3 CNN with
// periodic padding, channels 1 -> 32 -> 32 -> 32 -> 1, ReLU after the first
// three layers, applied to u_bar / sigma (sigma = RMS of u_bar) with residual
// output u0 = u_bar + sigma * y. The paper has no learned component; the
// network supplies the starting point of Algorithm 4.
//
// Activations are bfloat16, channels-last: H[b][p][32], p = (z*Y + y)*X + x.
// The 32 -> 32 layers are implicit GEMMs on the tensor cores (bf16 inputs,
// float32 accumulation): for an x-segment of 32 points per warp, the product
// over K = 27 taps x 32 input channels into N = 32 output channels; the 32 -> 1
// last layer sums over channels first (27 GEMM columns, one per tap), then over taps. The 1 -> 32 first
// layer runs on the CUDA cores in float32, so the small differences it forms
// from u_bar are not lost to bfloat16 rounding. The
// output is scaled by the fixed factor A = (delta/h)^2 = 1/(pi gamma)^2, the
// grid-unit weight of the Laplacian in G^{-1} = I - delta^2 Laplacian (Eq. df):
// u0 = u_bar + sigma * A * y. Training keeps float32 master
// weights and Adam moments; the loss is the relative mean-square error
// ||u0 - u_true||^2 / ||u_true||^2 averaged over the samples of a batch.
//
// Weight layout of the float32 master array (kCnnWeights floats):
//   W1 [27][32]        tap, out channel       (layer 1, in channel 1)
//   W2 [27][32][32]    tap, in, out
//   W3 [27][32][32]    tap, in, out
//   W4 [27][32]        tap, in channel        (layer 4, out channel 1)
// tap = (a*3 + b)*3 + c multiplies x at (z + a - 1, y + b - 1, x + c - 1).

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "cnn.h"

namespace gad {

namespace {

constexpr int C = 32;
constexpr int TAPS = 27;

__device__ __forceinline__ int wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, const uint32_t* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ void ldsm_x4(uint32_t* r, const void* p) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(p));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(s));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t* r, const void* p) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(p));
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(s));
}

// a * b + c of both halves of a pair in one instruction, each rounded as fmaf.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*reinterpret_cast<const uint64_t*>(&a)), "l"(*reinterpret_cast<const uint64_t*>(&b)),
        "l"(*reinterpret_cast<const uint64_t*>(&c)));
  return *reinterpret_cast<float2*>(&d);
}

// Row of a shared-memory point tile: 32 bf16 channels (64 bytes) + 16 bytes of
// padding, so the 8-row ldmatrix phases hit distinct banks.
constexpr int ROWB = 80;

// Copies the x-segment [x0 - 1, x0 + TX + 1) (periodic) of the `nr` activation
// rows y - 1 .. y + nr - 2 of z offset a into `dst` (rows of TX + 2 points, ROWB
// bytes per point): 16-byte cp.async copies, committed as one group.
__device__ __forceinline__ void stage_rows_async(unsigned char* dst, const __nv_bfloat16* H, long long base, int z,
                                                 int y, int a, int nr, int X, int Y, int Z, int x0, int TX, int tid,
                                                 int nthr) {
  const int n16 = (TX + 2) * 4;
  for (int bb = 0; bb < nr; ++bb) {
    const long long rowbase = base + ((long long)wrap(z + a - 1, Z) * Y + (y + bb - 1 + Y) % Y) * X;
    unsigned char* row = dst + bb * (TX + 2) * ROWB;
    for (int i = tid; i < n16; i += nthr) {
      const int pt = i >> 2, q = i & 3;
      const int x = wrap(x0 - 1 + pt, X);
      const unsigned sa = static_cast<unsigned>(__cvta_generic_to_shared(row + pt * ROWB + q * 16));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(H + (rowbase + x) * C + q * 8)
                   : "memory");
    }
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

}  // namespace

// ---------------------------------------------------------------------------
// 32 -> 32 convolution on the tensor cores (mma.sync). A block computes four
// rows y0 .. y0+3 of a TX-point x-segment; one warp computes 32 consecutive x
// points (two m16 tiles) x 32 output channels (four n8 tiles) of two of them,
// so a weight fragment feeds four mma. The six neighbour rows of a z offset
// are staged in shared memory (periodic) while those of the previous offset
// are in use. Weights come in mma B-fragment order (see k_pack_frag) from
// global memory (L1-resident). Bound by the mma.sync rate and the fragment
// reads (1.5 shared-memory or L1 wavefronts per mma). One row per block and
// one per warp: 64^3 x 8 375 -> 298 us.
// mode 0: out = bf16(relu(acc));  mode 1: out = bf16(acc * (mask > 0)).
constexpr int CONV_TY = 4;
__global__ void __launch_bounds__(128, 3) k_conv_mma(const __nv_bfloat16* __restrict__ Hin,
                                                     const uint2* __restrict__ Wf, __nv_bfloat16* __restrict__ Hout,
                                                     const __nv_bfloat16* __restrict__ Hmask, int X, int Y, int Z,
                                                     int TX, int mode) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31;
  const int segs = X / TX, ytiles = (Y + CONV_TY - 1) / CONV_TY;
  int r = blockIdx.x;
  const int seg = r % segs;
  r /= segs;
  const int y0 = (r % ytiles) * CONV_TY, z = r / ytiles;
  const int b = blockIdx.y;
  const int x0 = seg * TX, wx = (warp % (TX >> 5)) * 32, wy = 2 * (warp / (TX >> 5));
  const long long P = (long long)X * Y * Z;
  const long long base = (long long)b * P;
  float acc[2][2][4][4];                     // row, m tile, n tile
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[j][m][n][e] = 0.f;
  // ldmatrix lane address: matrix mi = lane/8, row i = lane%8 -> point row
  // i + 8*(mi & 1), channel offset 8*(mi >> 1)
  const int mi = lane >> 3, li = lane & 7;
  const int prow = li + 8 * (mi & 1), coff = 16 * (mi >> 1);
  // the rows of z offset a + 1 are copied (cp.async) into the other half of
  // shared memory while the taps of offset a run on the tensor cores
  const int rstride = (TX + 2) * ROWB, hstride = (CONV_TY + 2) * rstride;
  stage_rows_async(sm, Hin, base, z, y0, 0, CONV_TY + 2, X, Y, Z, x0, TX, tid, nthr);
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    if (a < 2) {
      stage_rows_async(sm + ((a + 1) & 1) * hstride, Hin, base, z, y0, a + 1, CONV_TY + 2, X, Y, Z, x0, TX, tid, nthr);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
#pragma unroll 1
    for (int bb = 0; bb < 3; ++bb) {
      const unsigned char* rowt = sm + (a & 1) * hstride + (wy + bb) * rstride + (wx + prow) * ROWB + coff;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int tap = (a * 3 + bb) * 3 + c;
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          uint32_t af[2][2][4];
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int m = 0; m < 2; ++m)        // row (x + c - 1) in the staged segment
              ldsm_x4(af[j][m], rowt + j * rstride + (m * 16 + c) * ROWB + ks * 32);
#pragma unroll
          for (int n = 0; n < 4; ++n) {
            const uint2 bw = __ldg(Wf + ((tap * 2 + ks) * 4 + n) * 32 + lane);
            const uint32_t bf[2] = {bw.x, bw.y};
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              mma_bf16(acc[j][0][n], af[j][0], bf);
              mma_bf16(acc[j][1][n], af[j][1], bf);
            }
          }
        }
      }
    }
    __syncthreads();  // this half is refilled next
  }
  // epilogue: C fragment (row g / g+8, cols 2t, 2t+1)
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (y0 + wy + j >= Y) break;
    const long long rowp = base + ((long long)z * Y + y0 + wy + j) * X + x0 + wx;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long long p = rowp + m * 16 + g + 8 * h;
#pragma unroll
        for (int n = 0; n < 4; ++n) {
          const int co = n * 8 + 2 * t;
          float v0 = acc[j][m][n][2 * h], v1 = acc[j][m][n][2 * h + 1];
          if (mode == 0) {
            v0 = fmaxf(v0, 0.f);
            v1 = fmaxf(v1, 0.f);
          } else {
            const __nv_bfloat162 mk = *reinterpret_cast<const __nv_bfloat162*>(Hmask + p * C + co);
            v0 = __bfloat162float(mk.x) > 0.f ? v0 : 0.f;
            v1 = __bfloat162float(mk.y) > 0.f ? v1 : 0.f;
          }
          *reinterpret_cast<uint32_t*>(Hout + p * C + co) = pack_bf16(v0, v1);
        }
      }
  }
}

// Weight gradient of a 32 -> 32 layer: dW[tap][ci][co] = sum_p Hin[p + off(tap)][ci] * dZ[p][co].
// Eighteen warps per block: warp (a, b, m) owns the three taps (a, b, c) and
// half m of the input channels (48 accumulators). The rows
// (b, z, x-segment, y) are split evenly and contiguously over the blocks; a
// block marches along y: per row it stages the three z planes' rows y + 1 and
// the dZ row y (cp.async, two rows ahead) into rings of five and three slots,
// so a row of Hin is fetched three times (once per z plane), not nine, and its
// latency overlaps two rows of mma. A block writes kWgradParts float32 partials
// per tap, ci and co, each over a part of its rows, so that the tensor cores'
// float32 sums stay short (k_reduce_parts adds the partials in float64). Bound
// by the mma.sync rate and the ldmatrix reads. Nine rows fetched synchronously
// per output row: 64^3 x 8 1310 -> 394 us.
constexpr int WG_H = 5, WG_Z = 3;          // ring slots
__global__ void __launch_bounds__(576) k_wgrad_mma(const __nv_bfloat16* __restrict__ Hin,
                                                   const __nv_bfloat16* __restrict__ dZ, float* __restrict__ part,
                                                   int X, int Y, int Z, int B, int TX) {
  extern __shared__ __align__(16) unsigned char sm[];
  const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31;
  const int segs = X / TX;
  const int rstride = (TX + 2) * ROWB;
  unsigned char* dzr = sm + WG_H * 3 * rstride;
  float acc[3][4][4];
  const long long P = (long long)X * Y * Z;
  const int mi = lane >> 3, li = lane & 7;
  const int wt = warp % 9, wm = warp / 9, wa = wt / 3, wb = wt - 3 * wa;
  const long long nrows = (long long)B * Z * segs * Y;
  auto copy16 = [](unsigned char* dst, const __nv_bfloat16* src) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
  };
  for (int part_i = blockIdx.x * kWgradParts; part_i < (int)(blockIdx.x + 1) * kWgradParts; ++part_i) {
    long long r = nrows * part_i / (gridDim.x * kWgradParts);
    const long long rend = nrows * (part_i + 1) / (gridDim.x * kWgradParts);
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[c][n][e] = 0.f;
    while (r < rend) {
      // a run of consecutive y of one (b, z, segment)
      const int y0 = (int)(r % Y), n = (int)min(rend - r, (long long)(Y - y0));
      long long col = r / Y;
      const int x0 = (int)(col % segs) * TX;
      col /= segs;
      const int z = (int)(col % Z);
      const long long base = (col / Z) * P;
      // Hin rows y0 + i (i = -1 .. n) of the three planes, slot (i + 1) % WG_H
      auto stage_h = [&](int i) {
        const int y = (y0 + i + Y) % Y;
        unsigned char* slot = sm + ((i + 1) % WG_H) * 3 * rstride;
        for (int q = tid; q < 3 * (TX + 2) * 4; q += nthr) {
          const int a = q / ((TX + 2) * 4), k = q - a * ((TX + 2) * 4), pt = k >> 2, ch = k & 3;
          copy16(slot + a * rstride + pt * ROWB + ch * 16,
                 Hin + (base + ((long long)wrap(z + a - 1, Z) * Y + y) * X + wrap(x0 - 1 + pt, X)) * C + ch * 8);
        }
      };
      auto stage_z = [&](int i) {
        unsigned char* slot = dzr + (i % WG_Z) * TX * ROWB;
        for (int q = tid; q < TX * 4; q += nthr)
          copy16(slot + (q >> 2) * ROWB + (q & 3) * 16,
                 dZ + (base + ((long long)z * Y + y0 + i) * X + x0 + (q >> 2)) * C + (q & 3) * 8);
      };
      __syncthreads();                         // the previous run's rows are no longer read
      stage_h(-1);
      stage_h(0);
      for (int i = 0; i < 2; ++i) {            // groups 0, 1: rows i + 1 and dZ row i
        if (i < n) {
          stage_h(i + 1);
          stage_z(i);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
      }
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        cp_async_wait<1>();
        __syncthreads();                       // row i is staged; row i - 1 is no longer read
        if (i + 2 < n) {
          stage_h(i + 3);
          stage_z(i + 2);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        const unsigned char* rowt = sm + ((i + wb) % WG_H) * 3 * rstride + wa * rstride;   // row i + wb - 1
        const unsigned char* dzt = dzr + (i % WG_Z) * TX * ROWB;
#pragma unroll 1
        for (int k0 = 0; k0 < TX; k0 += 16) {
          // B fragments (k = points, n = co) from dZ: transposed 8x8 loads.
          // matrices: mi&1 selects k half (points k0..7 / 8..15), mi>>1 selects n tile pair
          uint32_t bfr[4][2];
#pragma unroll
          for (int np = 0; np < 2; ++np) {
            uint32_t rgs[4];
            // lane address: rows = points k0 + li + 8*(mi & 1), channels 16*np + 8*(mi >> 1)
            ldsm_x4_t(rgs, dzt + (k0 + li + 8 * (mi & 1)) * ROWB + (16 * np + 8 * (mi >> 1)) * 2);
            bfr[2 * np + 0][0] = rgs[0];
            bfr[2 * np + 0][1] = rgs[1];
            bfr[2 * np + 1][0] = rgs[2];
            bfr[2 * np + 1][1] = rgs[3];
          }
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            // A fragments (m = ci, k = points) from the shifted input row, transposed loads:
            // matrices 0: ci 0-7, k 0-7; 1: ci 8-15, k 0-7; 2: ci 0-7, k 8-15; 3: ci 8-15, k 8-15
            uint32_t af[4];
            ldsm_x4_t(af, rowt + (k0 + li + 8 * (mi >> 1) + c) * ROWB + (wm * 16 + 8 * (mi & 1)) * 2);
#pragma unroll
            for (int n4 = 0; n4 < 4; ++n4) mma_bf16(acc[c][n4], af, bfr[n4]);
          }
        }
      }
      cp_async_wait<0>();
      r += n;
    }
    const int g = lane >> 2, t = lane & 3;
    float* pb = part + (long long)part_i * TAPS * C * C;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int tap = wt * 3 + c;
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int ci = wm * 16 + g + 8 * (e >> 1), co = n * 8 + 2 * t + (e & 1);
          pb[(tap * C + ci) * C + co] = acc[c][n][e];
        }
    }
  }
}

// ---------------------------------------------------------------------------
// CUDA-core layers and helpers.

// Packs float32 weights W[tap][ci][co] into mma B fragments:
// Wf[((tap*2 + ks)*4 + n)*32 + lane] = {B(2t, g), B(2t+1, g)}, {B(2t+8, g), B(2t+9, g)}
// with k = 16 ks + row, n8 tile n, g = lane/4, t = lane%4, B(k, j) = W[tap][k][8n + j];
// transposed: B(k, j) = W[26 - tap][8n + j][k] (backward data: flipped taps, swapped channels).
__global__ void k_pack_frag(const float* __restrict__ W, uint2* __restrict__ Wf, int transposed) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= TAPS * 2 * 4 * 32) return;
  const int lane = i & 31, n = (i >> 5) & 3, ks = (i >> 7) & 1, tap = i >> 8;
  const int g = lane >> 2, t = lane & 3;
  auto Bv = [&](int k, int j) {
    const int kk = ks * 16 + k, jj = n * 8 + j;
    return transposed ? W[((TAPS - 1 - tap) * C + jj) * C + kk] : W[(tap * C + kk) * C + jj];
  };
  Wf[i] = make_uint2(pack_bf16(Bv(2 * t, g), Bv(2 * t + 1, g)), pack_bf16(Bv(2 * t + 8, g), Bv(2 * t + 9, g)));
}

// Packs the layer-4 weights W4[tap][ci] as the B fragments of a GEMM whose 32
// columns are the taps (27..31 zero), for k_conv_out. Its A fragments come
// straight from global memory, lane t of a quad holding channels 8t .. 8t+7 of
// a point, so row k of k-step ks stands for channel 8 (k/2 mod 4) + 4 ks +
// 2 (k/8) + k mod 2:
// Wf[(ks*4 + n)*32 + lane] = {W4[8n+g][8t+4ks .. +1]}, {W4[8n+g][8t+4ks+2 .. +3]}.
__global__ void k_pack_frag4(const float* __restrict__ W4, uint2* __restrict__ Wf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * 4 * 32) return;
  const int lane = i & 31, n = (i >> 5) & 3, ks = i >> 7;
  const int tap = 8 * n + (lane >> 2), ci = 8 * (lane & 3) + 4 * ks;
  auto w = [&](int k) { return tap < TAPS ? W4[tap * C + ci + k] : 0.f; };
  Wf[i] = make_uint2(pack_bf16(w(0), w(1)), pack_bf16(w(2), w(3)));
}

// Packs the layer-4 weights for k_conv_out_mma: the B fragments of row offset d
// = -1 .. 8 (relative to the first of eight output rows), column j holding the
// weights of the tap dy = d - j (zero unless -1 <= dy <= 1):
// Wf[(((a*10 + d+1)*3 + c)*2 + ks)*32 + lane] = {B(2t, g), B(2t+1, g)}, {B(2t+8, g), B(2t+9, g)},
// B(k, j) = W4[(a, d - j + 1, c)][16 ks + k].
__global__ void k_pack_frag4t(const float* __restrict__ W4, uint2* __restrict__ Wf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * 10 * 3 * 2 * 32) return;
  const int lane = i & 31, ks = (i >> 5) & 1, adc = i >> 6, c = adc % 3, d = adc / 3 % 10, a = adc / 30;
  const int g = lane >> 2, t = lane & 3, bb = d - g;
  auto Bv = [&](int k) { return bb >= 0 && bb < 3 ? W4[((a * 3 + bb) * 3 + c) * C + ks * 16 + k] : 0.f; };
  Wf[i] = make_uint2(pack_bf16(Bv(2 * t), Bv(2 * t + 1)), pack_bf16(Bv(2 * t + 8), Bv(2 * t + 9)));
}

// sum of squares of each sample (float64 partials per block, then per sample)
__global__ void k_sumsq(const float* __restrict__ u, long long P, double* __restrict__ out) {
  const int b = blockIdx.y;
  double s = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P; i += (long long)gridDim.x * blockDim.x) {
    const double v = u[(long long)b * P + i];
    s += v * v;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    atomicAdd(out + b, t);
  }
}

// The bf16 pair v where the pair m is positive, zero elsewhere.
__device__ __forceinline__ uint32_t relu_mask(uint32_t v, uint32_t m) {
  const __nv_bfloat162 m2 = *reinterpret_cast<const __nv_bfloat162*>(&m);
  return (__bfloat162float(m2.x) > 0.f ? v & 0xffffu : 0u) | (__bfloat162float(m2.y) > 0.f ? v & 0xffff0000u : 0u);
}

// The 1 -> 32 convolutions in float32 on the CUDA cores:
//   first layer:              H1[p][co] = relu(sum_tap W1[tap][co] x0[p + off(tap)]), x0 = u_bar / sigma
//   layer-4 backward (BWD):   dZ3[p][ci] = (H3[p][ci] > 0) sum_tap W4[tap][ci] g[p - off(tap)]
// Bound by the float32 pipe (864 multiply-adds per point). A thread computes
// four consecutive x points, eight channels at a time as four packed pairs
// (fma.rn.f32x2: two multiply-adds per issue, each rounded as fmaf): the six
// values of each of the 9 neighbour rows are held doubled, and a 16-byte
// broadcast read of four weights feeds eight packed multiply-adds (the
// load/store unit moves 8 bytes of a broadcast per cycle, so the weights are
// not the ones to be doubled). The results go through shared memory so that a
// store covers 512 consecutive bytes (16 bytes at a 128-256 byte stride cost as
// many cycles of the load/store unit as the weight reads). Two points per
// thread, scalar multiply-adds and strided stores:
// 256^3 x 3 2.29 -> 1.57 ms, 64^3 x 8 backward 139 -> 100 us.
template <bool BWD>
__global__ void __launch_bounds__(128, 3) k_conv_1ch(const float* __restrict__ S, const double* __restrict__ sumsq,
                                                     const float* __restrict__ W, const __nv_bfloat16* __restrict__ mask,
                                                     __nv_bfloat16* __restrict__ out, int X, int Y, int Z) {
  const long long P = (long long)X * Y * Z;
  const int xg = X >> 2;                             // point groups of a row (X is a multiple of 32)
  const int b = blockIdx.y, lane = threadIdx.x & 31;
  __shared__ __align__(16) float w[TAPS * C];
  extern __shared__ __align__(16) unsigned char sm[];
  // this warp's 128 results, point 4 l + i (lane l) at i PLANE + l ROWB: written
  // and read back without bank conflicts
  constexpr int PLANE = 32 * ROWB + 64;
  unsigned char* stage = sm + (threadIdx.x >> 5) * (4 * PLANE);
  for (int i = threadIdx.x; i < TAPS * C; i += blockDim.x) w[i] = W[i];
  __syncthreads();
  const float scale = BWD ? 1.f : (float)(1.0 / sqrt(fmax(sumsq[b] / (double)P, 1e-300)));
  const long long groups = P >> 2;                   // not always a multiple of 32: the last warp's lanes are guarded
  for (long long pg0 = blockIdx.x * (long long)blockDim.x + threadIdx.x - lane; pg0 < groups;
       pg0 += (long long)gridDim.x * blockDim.x) {
    const long long pg = min(pg0 + lane, groups - 1);
    if (BWD)                                         // the mask rows of the epilogue, on their way to L2 meanwhile
      for (int j = 0; j < 2; ++j)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(mask + ((long long)b * P + 4 * pg + 2 * j) * C));
    const long long row0 = pg / xg;
    const int x = 4 * (int)(pg - row0 * xg);
    const int z = (int)(row0 / Y), y = (int)(row0 - (long long)z * Y);
    float2 v[9][6];                                  // row (a, b): x-1 .. x+4, doubled
#pragma unroll
    for (int r = 0; r < 9; ++r) {
      const long long row = (long long)b * P + ((long long)wrap(z + r / 3 - 1, Z) * Y + wrap(y + r % 3 - 1, Y)) * X;
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        float e = S[row + (c == 0 ? (x ? x - 1 : X - 1) : c == 5 ? (x + 4 == X ? 0 : x + 4) : x + c - 1)];
        if (!BWD) e *= scale;
        v[r][c] = make_float2(e, e);
      }
    }
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {                    // output channels 8q .. 8q + 7
      float2 s[4][4];                                // point x + i, channel pair
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) s[i][k] = make_float2(0.f, 0.f);
#pragma unroll
      for (int t = 0; t < TAPS; ++t) {
        const int u = BWD ? TAPS - 1 - t : t;        // p - off(t) = p + off(26 - t)
        const float4* wt = reinterpret_cast<const float4*>(w + t * C + 8 * q);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const float4 w4 = wt[k];
          const float2 wa = make_float2(w4.x, w4.y), wb = make_float2(w4.z, w4.w);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            s[i][2 * k] = fma2(wa, v[u / 3][u % 3 + i], s[i][2 * k]);
            s[i][2 * k + 1] = fma2(wb, v[u / 3][u % 3 + i], s[i][2 * k + 1]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {                  // point x + i
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 f = s[i][k];
          o[k] = BWD ? pack_bf16(f.x, f.y) : pack_bf16(fmaxf(f.x, 0.f), fmaxf(f.y, 0.f));
        }
        *reinterpret_cast<uint4*>(stage + i * PLANE + lane * ROWB + 16 * q) = make_uint4(o[0], o[1], o[2], o[3]);
      }
    }
    __syncwarp();
    // 16 bytes per lane in address order: 8 points of 64 bytes per store
    const long long p0 = (long long)b * P + 4 * pg0;
#pragma unroll 4
    for (int j = 0; j < 16; ++j) {
      const int pt = 8 * j + (lane >> 2), c16 = lane & 3;
      if (pg0 + (pt >> 2) < groups) {
        uint4 v = *reinterpret_cast<const uint4*>(stage + (pt & 3) * PLANE + (pt >> 2) * ROWB + 16 * c16);
        if (BWD) {
          const uint4 m = *reinterpret_cast<const uint4*>(mask + (p0 + pt) * C + 8 * c16);
          v.x = relu_mask(v.x, m.x);
          v.y = relu_mask(v.y, m.y);
          v.z = relu_mask(v.z, m.z);
          v.w = relu_mask(v.w, m.w);
        }
        *reinterpret_cast<uint4*>(out + (p0 + pt) * C + 8 * c16) = v;
      }
    }
    __syncwarp();
  }
}
constexpr size_t kConv1Smem = 4 * 4 * (32 * ROWB + 64);

// sum_tap, ci W4[tap][ci] H3[p + off(tap)][ci] of one point, weights rounded to
// bfloat16 as in the matrix products.
__device__ __noinline__ float out_point(const __nv_bfloat16* H3, const float* W4, long long base, int x, int y, int z,
                                        int X, int Y, int Z) {
  float s = 0.f;
  for (int tap = 0; tap < TAPS; ++tap) {
    const long long q = base + ((long long)wrap(z + tap / 9 - 1, Z) * Y + wrap(y + tap / 3 % 3 - 1, Y)) * X +
                        wrap(x + tap % 3 - 1, X);
    for (int ci = 0; ci < C; ++ci)
      s = fmaf(__bfloat162float(__float2bfloat16_rn(W4[tap * C + ci])), __bfloat162float(H3[q * C + ci]), s);
  }
  return s;
}

// Layer 4 of a training step, with the loss and its gradient: the implicit GEMM
// of k_conv_mma with one n8 tile whose eight columns are eight output rows y0 ..
// y0+7. A staged row d (relative to y0) is multiplied once by the fragment
// whose column j holds the taps dy = d - j, so the ten rows of a z offset serve
// eight output rows: 180 ldmatrix and mma per 16 x 8 outputs, where one useful
// column per output row took 432. Every output still adds its 27 taps x two
// halves of 16 channels in that order (the zero columns add nothing), which
// the loss gradient, proportional to the small difference u0 - u_true, is
// sensitive to. Where a staged activation is not finite its products with the
// zero columns are not zero; a sum that is not finite is therefore formed again
// from the output's own taps (out_point). A block owns a TX-point x-segment, a
// warp 16 of its points. 64^3 x 8: 402 -> 225 us.
// It writes u0, g = sigma * A * 2 (u0 - u_true) / ||u_true||^2 / B and
// accumulates sum (u0 - u_true)^2 / ||u_true||^2 / B into loss.
__global__ void __launch_bounds__(128) k_conv_out_mma(const __nv_bfloat16* __restrict__ H3,
                                                      const uint2* __restrict__ Wf, const float* __restrict__ W4,
                                                      const float* __restrict__ ubar,
                                                      const double* __restrict__ sumsq, float* __restrict__ u0,
                                                      const float* __restrict__ utrue,
                                                      const double* __restrict__ tsumsq, float* __restrict__ gout,
                                                      double* __restrict__ loss, int X, int Y, int Z, int B, int TX,
                                                      double ascale) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ double red[4];
  const int tid = threadIdx.x, nthr = blockDim.x, warp = tid >> 5, lane = tid & 31;
  const int segs = X / TX, ytiles = (Y + 7) / 8;
  int r = blockIdx.x;
  const int x0 = (r % segs) * TX;
  r /= segs;
  const int y0 = (r % ytiles) * 8, z = r / ytiles;
  const int b = blockIdx.y;
  const long long P = (long long)X * Y * Z;
  const long long base = (long long)b * P;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  const int mi = lane >> 3, li = lane & 7, g = lane >> 2, t = lane & 3;
  const int prow = warp * 16 + li + 8 * (mi & 1), coff = 16 * (mi >> 1);
  const int rstride = (TX + 2) * ROWB;
#pragma unroll 1
  for (int a = 0; a < 3; ++a) {
    stage_rows_async(sm, H3, base, z, y0, a, 10, X, Y, Z, x0, TX, tid, nthr);
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll 2
    for (int d = 0; d < 10; ++d)
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) {
          uint32_t af[4];
          ldsm_x4(af, sm + d * rstride + (prow + c) * ROWB + ks * 32 + coff);
          const uint2 bw = __ldg(Wf + (((a * 10 + d) * 3 + c) * 2 + ks) * 32 + lane);
          const uint32_t bf[2] = {bw.x, bw.y};
          mma_bf16(acc, af, bf);
        }
    __syncthreads();                         // the rows are replaced next
  }
  const double sigma = sqrt(fmax(sumsq[b] / (double)P, 1e-300)) * ascale;   // sigma * A
  const double inv = 1.0 / (tsumsq[b] * (double)B);
  double lsum = 0.0;
#pragma unroll
  for (int e = 0; e < 4; ++e) {              // point g + 8 (e / 2), row 2t + e % 2
    const int y = y0 + 2 * t + (e & 1);
    if (y < Y) {
      const int x = x0 + warp * 16 + g + 8 * (e >> 1);
      const long long gi = base + ((long long)z * Y + y) * X + x;
      const float o = isfinite(acc[e]) ? acc[e] : out_point(H3, W4, base, x, y, z, X, Y, Z);
      const float uo = ubar[gi] + (float)sigma * o;
      u0[gi] = uo;
      const double df = (double)uo - (double)utrue[gi];
      lsum += df * df * inv;
      gout[gi] = (float)(sigma * 2.0 * df * inv);
    }
  }
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0) red[warp] = lsum;
  __syncthreads();
  if (tid == 0) {
    double tt = 0.0;
    for (int w2 = 0; w2 < (nthr >> 5); ++w2) tt += red[w2];
    atomicAdd(loss, tt);
  }
}

// Layer 4 (32 -> 1) on the tensor cores and the residual output:
//   u0 = u_bar + sigma * A * sum_{tap, ci} W4[tap][ci] H3[p + off][ci].
// The sum over channels comes first: per input point q one row of the GEMM
// T[q][tap] = sum_ci H3[q][ci] W4[tap][ci] (K = 32, N = 27 taps of 32), then
// out[p] = sum_tap T[p + off(tap)][tap] adds 27 float32 values. Each point's
// channels are read and multiplied once (2 x 4 mma per 16 points), where an
// implicit GEMM over 27 taps x 32 channels with one useful column of eight
// takes 54 ldmatrix and 54 mma per 16 points.
// A block owns TX x 8 columns and marches along z over `zc` output planes: the
// (TX+2) x 10 points of a plane go to shared memory tap-major (row stride 4 mod
// 32: the fragment stores and the x-contiguous reads are conflict free), and
// each thread adds the plane's nine values per z tap to the running sums of
// the three output planes it touches. Bound by reading H3 (halo 1.16-1.3x,
// mostly from L2) and by shared memory (about 2 wavefronts per output).
// 256^3 x 3: 6.10 -> 1.16 ms.
// Inference only: the loss gradient is proportional to u0 - u_true, a small
// difference in which the order of these sums shows (weight gradients move by
// 2e-5), so training steps keep k_conv_out_mma's order.
constexpr int OUT_TY = 8;
template <int TX> struct OutTile {
  static constexpr int PTS = (TX + 2) * (OUT_TY + 2);
  static constexpr int NT = (PTS + 15) / 16;                  // m16 tiles of a plane
  static constexpr int LD = (NT * 16 + 31) / 32 * 32 + 4;     // floats per tap row
  static constexpr size_t smem = sizeof(float) * TAPS * LD;
};

template <int TX>
__global__ void __launch_bounds__(256, 3) k_conv_out(const __nv_bfloat16* __restrict__ H3,
                                                     const uint2* __restrict__ Wf, const float* __restrict__ ubar,
                                                     const double* __restrict__ sumsq, float* __restrict__ u0,
                                                     int X, int Y, int Z, int zc, double ascale) {
  using OT = OutTile<TX>;
  extern __shared__ __align__(16) float tsm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int segs = X / TX, ytiles = (Y + OUT_TY - 1) / OUT_TY;
  int r = blockIdx.x;
  const int x0 = (r % segs) * TX;
  r /= segs;
  const int y0 = (r % ytiles) * OUT_TY, z0 = (r / ytiles) * zc, z1 = min(z0 + zc, Z);
  const int b = blockIdx.y;
  const long long plane = (long long)X * Y, base = (long long)b * plane * Z;
  uint2 wf[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) wf[i] = Wf[i * 32 + lane];
  // the plane offsets (points) of this lane's rows g, g + 8 of each of its tiles
  constexpr int TPW = (OT::NT + 7) / 8;
  int off[TPW][2];
#pragma unroll
  for (int k = 0; k < TPW; ++k)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = min((warp + 8 * k) * 16 + g + 8 * h, OT::PTS - 1);
      const int yy = (y0 + i / (TX + 2) + Y - 1) % Y;
      off[k][h] = yy * X + wrap(x0 - 1 + i % (TX + 2), X);
    }
  const float sig = (float)(sqrt(fmax(sumsq[b] / (double)(plane * Z), 1e-300)) * ascale);   // sigma * A
  constexpr int NO = TX * OUT_TY / 256;                       // outputs per thread and plane
  const int ox = tid % TX, oy = tid / TX;
  float s0[NO], s1[NO];                                       // sums of planes zi - 1, zi
#pragma unroll
  for (int o = 0; o < NO; ++o) s0[o] = s1[o] = 0.f;
  // three tiles' loads in flight per lane; those of a plane's first three are
  // issued before the previous plane's sums
  uint4 a[3][2];
  auto load3 = [&](int zi, int k0) {
    const uint4* hp = reinterpret_cast<const uint4*>(H3 + (base + wrap(zi, Z) * plane) * C) + t;
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (k0 + k < TPW && warp + 8 * (k0 + k) < OT::NT) {
        a[k][0] = hp[4ll * off[k0 + k][0]];
        a[k][1] = hp[4ll * off[k0 + k][1]];
      }
  };
  load3(z0 - 1, 0);
  for (int zi = z0 - 1; zi <= z1; ++zi) {
#pragma unroll
    for (int k0 = 0; k0 < TPW; k0 += 3) {
      if (k0) load3(zi, k0);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k0 + k < TPW && warp + 8 * (k0 + k) < OT::NT) {
          float* dst = tsm + (warp + 8 * (k0 + k)) * 16 + g;
          const uint32_t a0[4] = {a[k][0].x, a[k][1].x, a[k][0].y, a[k][1].y};
          const uint32_t a1[4] = {a[k][0].z, a[k][1].z, a[k][0].w, a[k][1].w};
#pragma unroll
          for (int n = 0; n < 4; ++n) {
            float d[4] = {0.f, 0.f, 0.f, 0.f};
            const uint32_t b0[2] = {wf[n].x, wf[n].y}, b1[2] = {wf[4 + n].x, wf[4 + n].y};
            mma_bf16(d, a0, b0);
            mma_bf16(d, a1, b1);
            const int tap = 8 * n + 2 * t;
            if (tap < TAPS) {
              dst[tap * OT::LD] = d[0];
              dst[tap * OT::LD + 8] = d[2];
            }
            if (tap + 1 < TAPS) {
              dst[(tap + 1) * OT::LD] = d[1];
              dst[(tap + 1) * OT::LD + 8] = d[3];
            }
          }
        }
    }
    if (zi < z1) load3(zi + 1, 0);
    __syncthreads();
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const int yl = oy + o * (256 / TX);
      const float* sp = tsm + yl * (TX + 2) + ox;
      float p[3] = {0.f, s1[o], s0[o]};                       // tap a adds to output plane zi + 1 - a
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int bc = 0; bc < 9; ++bc) p[a] += sp[(a * 9 + bc) * OT::LD + (bc / 3) * (TX + 2) + bc % 3];
      s1[o] = p[0];
      s0[o] = p[1];
      if (zi > z0 && y0 + yl < Y) {
        const long long gi = base + (zi - 1) * plane + (long long)(y0 + yl) * X + x0 + ox;
        u0[gi] = ubar[gi] + sig * p[2];
      }
    }
    __syncthreads();
  }
}

template <int TX>
static cudaError_t launch_conv_out(const CnnBuffers& w, const float* ubar, float* u0, int X, int Y, int Z, int B,
                                   double ascale, cudaStream_t s) {
  const long long cols = (long long)(X / TX) * ((Y + OUT_TY - 1) / OUT_TY);
  const int zc = out_planes(cols * B, Z);
  const cudaError_t e =
      cudaFuncSetAttribute(k_conv_out<TX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OutTile<TX>::smem);
  if (e != cudaSuccess) return e;
  k_conv_out<TX><<<dim3((unsigned)(cols * ((Z + zc - 1) / zc)), B), 256, OutTile<TX>::smem, s>>>(
      w.H3, w.frag4, ubar, w.sumsq, u0, X, Y, Z, zc, ascale);
  return cudaGetLastError();
}

// Weight gradients of the 1-channel layers, as one correlation of a scalar
// field S with a 32-channel field V:
//   acc[tap][ch] = sum_p S[p + off(tap)] * scale_b * V[p][ch]
//   first (layer 1): S = u_bar, scale_b = 1/sigma_b, V = dZ1 -> dW1[tap][co]
//   last  (layer 4): S = g, scale_b = 1, V = H3; dW4[tap][ci] = sum_p H3[p + off(tap)][ci] g[p]
//                    = sum_q H3[q][ci] g[q - off(tap)], stored at the mirrored tap 26 - tap.
// A block walks segments (b, z, y, x0..x0+TW) of its share; the 3x3 neighbour
// rows of S over [x0 - 1, x0 + TW + 1) are staged in shared memory with
// cp.async one segment ahead (double buffer). Warp w owns TW/8 consecutive
// points and lane = channel: the three x taps of consecutive points share a
// sliding register window, so each point costs 9 shared loads, one 64-byte
// coalesced load of V and 27 FMAs per lane. The warps' sums are added in the
// block (fixed order) and written as one float32 partial of 27 x 32 per block.
// 1/sigma_b takes a float64 root and divide, which every thread computed per
// segment before (first layer, 64^3 x 8: 480 -> 288 us).
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// Stages the 9 neighbour rows of S for segment r (see k_wgrad_1ch).
__device__ __forceinline__ void stage_1ch(float* dst, const float* __restrict__ S, long long r, int segs, int X,
                                          int Y, int Z, int TW, long long P) {
  const int seg = (int)(r % segs);
  long long q = r / segs;
  const int y = (int)(q % Y);
  q /= Y;
  const int z = (int)(q % Z), b = (int)(q / Z);
  const int x0 = seg * TW, ld = TW + 2;
  for (int i = threadIdx.x; i < 9 * ld; i += blockDim.x) {
    const int rr = i / ld, j = i - rr * ld;
    const long long src = (long long)b * P + ((long long)wrap(z + rr / 3 - 1, Z) * Y + wrap(y + rr % 3 - 1, Y)) * X +
                          wrap(x0 - 1 + j, X);
    cp_async4(dst + i, S + src);
  }
}

__global__ void __launch_bounds__(256, 3) k_wgrad_1ch(const float* __restrict__ S, const double* __restrict__ sumsq,
                                                   const __nv_bfloat16* __restrict__ V, float* __restrict__ part,
                                                   int X, int Y, int Z, int B, int TW, int mirror) {
  extern __shared__ __align__(16) float sw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long P = (long long)X * Y * Z;
  const int segs = X / TW, ld = TW + 2, nst = 9 * ld;
  const long long nrows = (long long)B * Z * Y * segs;
  float acc[TAPS];
#pragma unroll
  for (int t = 0; t < TAPS; ++t) acc[t] = 0.f;
  const int npw = TW / 8, xs = warp * npw;
  int sb_of = -1;
  float scale = 1.f;
  long long r = blockIdx.x;
  if (r < nrows) stage_1ch(sw, S, r, segs, X, Y, Z, TW, P);
  cp_async_commit();
  for (int it = 0; r < nrows; ++it, r += gridDim.x) {
    if (r + gridDim.x < nrows) stage_1ch(sw + ((it + 1) & 1) * nst, S, r + gridDim.x, segs, X, Y, Z, TW, P);
    cp_async_commit();
    cp_async_wait1();
    __syncthreads();
    const float* sb = sw + (it & 1) * nst;
    const int seg = (int)(r % segs);
    const long long q = r / segs;                   // (b, z, y) row index
    const int b = (int)(q / ((long long)Z * Y));
    if (sumsq && b != sb_of) {                      // float64 divide and root only where the sample changes
      scale = (float)(1.0 / sqrt(fmax(sumsq[b] / (double)P, 1e-300)));
      sb_of = b;
    }
    const __nv_bfloat16* vrow = V + (q * X + seg * TW + xs) * C + lane;
    float win[9][3];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      win[k][0] = sb[k * ld + xs];
      win[k][1] = sb[k * ld + xs + 1];
    }
#pragma unroll 4
    for (int i = 0; i < npw; ++i) {
      const float v = __bfloat162float(vrow[(long long)i * C]) * scale;
#pragma unroll
      for (int k = 0; k < 9; ++k) {
        win[k][2] = sb[k * ld + xs + i + 2];
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[k * 3 + c] = fmaf(win[k][c], v, acc[k * 3 + c]);
        win[k][0] = win[k][1];
        win[k][1] = win[k][2];
      }
    }
    __syncthreads();
  }
  // block sum of the warps' partials, fixed order
  float* red = sw;
#pragma unroll
  for (int t = 0; t < TAPS; ++t) red[(warp * TAPS + t) * C + lane] = acc[t];
  __syncthreads();
  const int nw = blockDim.x >> 5;
  for (int i = tid; i < TAPS * C; i += blockDim.x) {
    float s = 0.f;
    for (int w = 0; w < nw; ++w) s += red[w * TAPS * C + i];
    const int tap = i / C, ch = i - tap * C;
    part[(long long)blockIdx.x * TAPS * C + (mirror ? TAPS - 1 - tap : tap) * C + ch] = s;
  }
}

// out[i] = sum_j part[j][i] (fixed order), j < nparts, i < n, n a multiple of
// 32. A block owns 32 columns: warp w sums the parts j = w, w + 8, .. of its
// columns (coalesced rows of 128 bytes, four in flight), then the eight warps'
// float64 sums are added in order. One thread per column over all the parts
// left 4 blocks on a chain of 456 dependent loads (864 columns: 73 -> 15 us).
__global__ void __launch_bounds__(256) k_reduce_parts(const float* __restrict__ part, int nparts, int n,
                                                      float* __restrict__ out) {
  __shared__ double red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
  double s = 0.0;
#pragma unroll 4
  for (int j = w; j < nparts; j += 8) s += part[(long long)j * n + i];
  red[w][lane] = s;
  __syncthreads();
  if (w == 0) {
    for (int q = 1; q < 8; ++q) s += red[q][lane];
    out[i] = (float)s;
  }
}

// Adam on the float32 master weights.
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ grad, int n, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = grad[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---------------------------------------------------------------------------
// Host drivers (called by the C ABI in api.cu).

int cnn_tile(int X) { return X % 64 == 0 ? 64 : 32; }

// One 32 -> 32 layer on the warp-level tensor-core kernel.
static cudaError_t launch_conv_mma(const __nv_bfloat16* in, const uint2* frag, __nv_bfloat16* out,
                                   const __nv_bfloat16* mask, int X, int Y, int Z, int B, int mode, cudaStream_t s) {
  const int TX = cnn_tile(X);
  auto smem = [](int tx) { return (size_t)2 * (CONV_TY + 2) * (tx + 2) * ROWB; };   // two z offsets' rows
  const size_t sm = smem(TX);
  // the limit of the widest tile: the attribute is shared by every thread that launches
  const cudaError_t e = cudaFuncSetAttribute(k_conv_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem(64));
  if (e != cudaSuccess) return e;
  const dim3 g((unsigned)((X / TX) * ((Y + CONV_TY - 1) / CONV_TY)) * Z, B);
  k_conv_mma<<<g, TX / 32 * 64, sm, s>>>(in, frag, out, mask, X, Y, Z, TX, mode);
  return cudaGetLastError();
}

bool cnn_shape_ok(int X, int Y, int Z) { return X % 32 == 0 && Y >= 3 && Z >= 3; }

cudaError_t cnn_forward(const CnnBuffers& w, const float* ubar, float* u0, const float* utrue, int X, int Y, int Z,
                        int B, double ascale, cudaStream_t s) {
  const long long P = (long long)X * Y * Z;
  const int TX = cnn_tile(X);
  cudaError_t e = cudaMemsetAsync(w.sumsq, 0, sizeof(double) * 2 * B + sizeof(double), s);
  if (e != cudaSuccess) return e;
  const dim3 gp((unsigned)((P + 255) / 256 < 2048 ? (P + 255) / 256 : 2048), B);
  k_sumsq<<<gp, 256, 0, s>>>(ubar, P, w.sumsq);
  if (utrue) k_sumsq<<<gp, 256, 0, s>>>(utrue, P, w.sumsq + B);
  const dim3 g1((unsigned)(P / 512 < 4096 ? (P + 511) / 512 : 4096), B);
  k_conv_1ch<false><<<g1, 128, kConv1Smem, s>>>(ubar, w.sumsq, w.master, nullptr, w.H1, X, Y, Z);
  if (w.umma2 && conv_tc_shape_ok(X, Y, Z)) {
    if ((e = conv_tc_forward(w.H1, w.umma2, w.H2, nullptr, X, Y, Z, B, 0, w.flag, w.wait_ns, s)) != cudaSuccess ||
        (e = conv_tc_forward(w.H2, w.umma3, w.H3, nullptr, X, Y, Z, B, 0, w.flag, w.wait_ns, s)) != cudaSuccess)
      return e;
  } else {
    if ((e = launch_conv_mma(w.H1, w.frag2, w.H2, nullptr, X, Y, Z, B, 0, s)) != cudaSuccess ||
        (e = launch_conv_mma(w.H2, w.frag3, w.H3, nullptr, X, Y, Z, B, 0, s)) != cudaSuccess)
      return e;
  }
  if (!utrue)
    return X % 64 == 0 ? launch_conv_out<64>(w, ubar, u0, X, Y, Z, B, ascale, s)
                       : launch_conv_out<32>(w, ubar, u0, X, Y, Z, B, ascale, s);
  const size_t sm = (size_t)10 * (TX + 2) * ROWB;
  e = cudaFuncSetAttribute(k_conv_out_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, 10 * (64 + 2) * ROWB);
  if (e != cudaSuccess) return e;
  const dim3 gc((unsigned)((X / TX) * ((Y + 7) / 8)) * Z, B);
  k_conv_out_mma<<<gc, 2 * TX, sm, s>>>(w.H3, w.frag4t, w.master + kW4, ubar, w.sumsq, u0, utrue, w.sumsq + B, w.g,
                                        w.sumsq + 2 * B, X, Y, Z, B, TX, ascale);
  return cudaGetLastError();
}

// One forward 32 -> 32 layer, H2 = ReLU(conv(H1, W2)), in the launch shape of
// inference (the tensor-core path when the grid allows it); for timing.
cudaError_t cnn_conv_layer(const CnnBuffers& w, int X, int Y, int Z, int B, cudaStream_t s, bool* tensor_cores) {
  const bool tc = w.umma2 && conv_tc_shape_ok(X, Y, Z);
  if (tensor_cores) *tensor_cores = tc;
  if (tc) return conv_tc_forward(w.H1, w.umma2, w.H2, nullptr, X, Y, Z, B, 0, w.flag, w.wait_ns, s);
  return launch_conv_mma(w.H1, w.frag2, w.H2, nullptr, X, Y, Z, B, 0, s);
}

cudaError_t cnn_pack(const CnnBuffers& w, bool training, cudaStream_t s) {
  const int n = TAPS * 2 * 4 * 32;
  k_pack_frag<<<(n + 255) / 256, 256, 0, s>>>(w.master + kW2, w.frag2, 0);
  k_pack_frag<<<(n + 255) / 256, 256, 0, s>>>(w.master + kW3, w.frag3, 0);
  k_pack_frag<<<(n + 255) / 256, 256, 0, s>>>(w.master + kW2, w.frag2t, 1);
  k_pack_frag<<<(n + 255) / 256, 256, 0, s>>>(w.master + kW3, w.frag3t, 1);
  if (training)
    k_pack_frag4t<<<(180 * 32 + 255) / 256, 256, 0, s>>>(w.master + kW4, w.frag4t);
  else
    k_pack_frag4<<<1, 256, 0, s>>>(w.master + kW4, w.frag4);
  if (w.umma2) {
    cudaError_t e;
    if ((e = conv_tc_pack(w.master + kW2, w.umma2, 0, s)) != cudaSuccess ||
        (e = conv_tc_pack(w.master + kW3, w.umma3, 0, s)) != cudaSuccess ||
        (e = conv_tc_pack(w.master + kW2, w.umma2t, 1, s)) != cudaSuccess ||
        (e = conv_tc_pack(w.master + kW3, w.umma3t, 1, s)) != cudaSuccess)
      return e;
  }
  return cudaGetLastError();
}

// x-segment of the 1-channel weight-gradient kernel: X itself up to 256 points,
// else the largest multiple of 32 up to 256 that divides X (X is a multiple of 32)
static int wgrad_1ch_tile(int X) {
  if (X <= 256) return X;
  for (int t = 256; t > 32; t -= 32)
    if (X % t == 0) return t;
  return 32;
}
static size_t wgrad_1ch_smem(int TW) {
  const size_t stage = sizeof(float) * 2 * 9 * (TW + 2), red = sizeof(float) * 8 * TAPS * C;
  return stage > red ? stage : red;
}

cudaError_t cnn_backward(const CnnBuffers& w, const float* ubar, int X, int Y, int Z, int B, cudaStream_t s) {
  const long long P = (long long)X * Y * Z;
  const int TX = cnn_tile(X);
  // layer 4
  const dim3 g1((unsigned)(P / 512 < 4096 ? (P + 511) / 512 : 4096), B);
  k_conv_1ch<true><<<g1, 128, kConv1Smem, s>>>(w.g, nullptr, w.master + kW4, w.H3, w.dA, X, Y, Z);
  const int TW = wgrad_1ch_tile(X);
  const size_t sm1 = wgrad_1ch_smem(TW);
  k_wgrad_1ch<<<kSmallBlocks, 256, sm1, s>>>(w.g, nullptr, w.H3, w.part, X, Y, Z, B, TW, 1);
  k_reduce_parts<<<TAPS * C / 32, 256, 0, s>>>(w.part, kSmallBlocks, TAPS * C, w.grad + kW4);
  // layer 3: dW3 from (H2, dZ3); dZ2 = conv^T(dZ3, W3) masked by H2
  const size_t smw = (size_t)(WG_H * 3 * (TX + 2) + WG_Z * TX) * ROWB;
  cudaError_t e = cudaFuncSetAttribute(k_wgrad_mma, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (WG_H * 3 * (64 + 2) + WG_Z * 64) * ROWB);
  if (e != cudaSuccess) return e;
  k_wgrad_mma<<<kWgradBlocks, 576, smw, s>>>(w.H2, w.dA, w.part, X, Y, Z, B, TX);
  k_reduce_parts<<<TAPS * C * C / 32, 256, 0, s>>>(w.part, kWgradBlocks * kWgradParts, TAPS * C * C, w.grad + kW3);
  const bool tc = w.umma2 && conv_tc_shape_ok(X, Y, Z);
  if (tc) {
    if ((e = conv_tc_forward(w.dA, w.umma3t, w.dB, w.H2, X, Y, Z, B, 1, w.flag, w.wait_ns, s)) != cudaSuccess) return e;
  } else {
    if ((e = launch_conv_mma(w.dA, w.frag3t, w.dB, w.H2, X, Y, Z, B, 1, s)) != cudaSuccess) return e;
  }
  // layer 2: dW2 from (H1, dZ2); dZ1 = conv^T(dZ2, W2) masked by H1
  k_wgrad_mma<<<kWgradBlocks, 576, smw, s>>>(w.H1, w.dB, w.part, X, Y, Z, B, TX);
  k_reduce_parts<<<TAPS * C * C / 32, 256, 0, s>>>(w.part, kWgradBlocks * kWgradParts, TAPS * C * C, w.grad + kW2);
  if (tc) {
    if ((e = conv_tc_forward(w.dB, w.umma2t, w.dA, w.H1, X, Y, Z, B, 1, w.flag, w.wait_ns, s)) != cudaSuccess) return e;
  } else {
    if ((e = launch_conv_mma(w.dB, w.frag2t, w.dA, w.H1, X, Y, Z, B, 1, s)) != cudaSuccess) return e;
  }
  // layer 1
  k_wgrad_1ch<<<kSmallBlocks, 256, sm1, s>>>(ubar, w.sumsq, w.dA, w.part, X, Y, Z, B, TW, 0);
  k_reduce_parts<<<TAPS * C / 32, 256, 0, s>>>(w.part, kSmallBlocks, TAPS * C, w.grad + kW1);
  return cudaGetLastError();
}

cudaError_t cnn_adam(const CnnBuffers& w, int step, float lr, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  k_adam<<<(kCnnWeights + 255) / 256, 256, 0, s>>>(w.master, w.m, w.v, w.grad, kCnnWeights, lr, b1, b2, 1e-8f, c1, c2);
  return cudaGetLastError();
}

}  // namespace gad
