// FP32 GEMM of the per-edge MLPs on the tensor cores (precision mode 0):
// C[M][N] = alpha * A[M][K] * B[K][N] with A and C FP32 and the fused element-wise epilogues
// of the FP32 path.
//
// How.  Each operand is split into three bf16 slices, a = a1 + a2 + a3, on a fixed-point grid
// per row and 32-element K-chunk (row of B^T: output column).  With 2^e <= max|a| < 2^(e+1)
// over the chunk:  a1 = a rounded to a multiple of 2^(e-7), a2 = the rest rounded to a multiple
// of 2^(e-16) (both at most 256 units, so exact in bf16), a3 = what is left, at most 2^(e-17),
// rounded to bf16 with an error of at most 2^(e-26).  Of the nine products of slices the six
// larger ones are kept; with f the exponent of B's chunk, a2 b3 and a3 b2 are at most 2^(e+f-25)
// and a3 b3 2^(e+f-34):
//     main  = sum a1 b1      integers in units of 2^(e+f-14).  As long as the units of the chunks
//                            agree and the sum stays below 2^24 of them, the tensor core's FP32
//                            accumulation, which truncates, is exact
//     cross = sum a1 b2 + a2 b1 + a2 b2 + a1 b3 + a3 b1      2^-8 of main: its truncation
//                            errors are 2^-31 of the result
// in two tensor-memory accumulators, added once, rounded to nearest, in the epilogue.  The
// splitting of a dot product into exactly accumulated slices follows Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012) 95.
//
// Accuracy.  The error is relative to the largest magnitudes of the chunks:
//     |error| <= (2^-23 + (K / 16 + 3) 2^-22) sum_k max|a| max|b|
// (slices; truncation of the accumulators where the chunks' units differ, as in [x | T] or
// [dE/dz | dE/dw]).  On rows of normal draws it is below a chain of FP32 products and sums:
// 5.6e-8 against 3.4e-7 at K = 352 (2-norm).  An element 2^p below the largest of its chunk keeps
// some p - 3 bits fewer than in FP32: with A's columns spread over a factor of 2^10 and B's rows
// over its inverse, so that all terms count alike, 1.6e-5 against 3.4e-7.  The weights here are
// uniform draws, whose rows are alike, and the forces gain (figures below).
// tests/test_gpu_arithmetic.py measures both and holds the bound.
//
// One persistent CTA per SM walks the (128-row tile, column slice of at most 128) tiles
// blockIdx.x, + gridDim.x, ...:
//   warps 0-7    two epilogue groups of 4 warps; group g drains tiles j = g mod 2 (its own
//                main and cross accumulators), so the next tile's products overlap it
//   warps 8-15   two splitting groups of 4 warps, on alternate 128 x 32 chunks of A: two chunks
//                in flight in registers (64 floats a thread), split and stored 64-byte swizzled
//   warp 16      TMA producer of the pre-split weight chunks (3 x slice x 32 bf16)
//   warp 17      MMA issuer: 6 products of M=128, N=slice, K=16 per step
// The ring holds 3 or 4 chunks (48 KB each at a 128-column slice): with two chunks of 64
// elements, the weight loads and the splitting of a stage could not start before the products
// of the one before had ended.
//
// What bounds it.  The six products take 64 us of the latent layer's 149 us (110,000 rows,
// K = 352, N = 256: 0.13 PFLOP/s of FP32 products, 3.3 TB/s of HBM; 64 us is what the issue
// of the products alone measures, 107 us everything but the epilogue); the rest is latency of
// the splitting and of the epilogue at 18 warps an SM.  The CUDA-core kernel that this one
// replaced ran at 0.6 of the FP32 FMA peak: all 16 launches of an evaluation took 12.47 ms at
// 358,000 edges and 67.2 ms at 1.97 million, now 4.35 and 22.7 ms; at 5,500 edges and widths
// of 16 to 64, 0.170 and now 0.128 ms, so it serves every size.  Against 64 bits the forces
// of those evaluations are off by 6.4e-7 and 1.4e-6 (relative, 2-norm), with FP32 FMAs by
// 7.2e-7 and 1.5e-6.
#include "sigmoid.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int FS_EW = 8;                       // epilogue warps
constexpr int FS_CW = 8;                       // splitting warps
constexpr int FS_THREADS = 32 * (FS_EW + FS_CW + 2);
constexpr int FS_TK = 32;                      // K elements of a chunk (64-byte rows)
constexpr uint32_t FS_ASLICE = TM * FS_TK * 2;   // bytes of one slice of an A chunk

// Epilogue-input streams of a mode: the residual (SILU_RES, HEAD), the pre-activations (DSILU),
// or both the residual gradient and the pre-activations of the layer below (RES_DS).
template <int MODE>
__host__ __device__ constexpr int fs_naux() {
  return MODE == EPI_RES_DS                                                   ? 2
         : (MODE == EPI_SILU_RES || MODE == EPI_HEAD || MODE == EPI_DSILU) ? 1
                                                                              : 0;
}
// Column groups of input a warp has room for (2 KB each and stream), and ring stages, within
// the 227 KB of a CTA.
template <int MODE>
__host__ __device__ constexpr int fs_auxn() { return MODE == EPI_RES_DS ? 2 : 4; }
template <int MODE>
__host__ __device__ constexpr int fs_stages() { return fs_naux<MODE>() ? 3 : 4; }

// A CTA's walk over its tiles: row tile and column slice of tile blockIdx.x + k * gridDim.x,
// advanced without a division per step.
struct FsWalk {
  int t, row, sl, step, drow, dsl, nsl;
  __device__ __forceinline__ FsWalk(int t0, int step_, int nslices)
      : t(t0), row(t0 / nslices), sl(t0 % nslices), step(step_), drow(step_ / nslices),
        dsl(step_ % nslices), nsl(nslices) {}
  __device__ __forceinline__ void next() {
    t += step;
    row += drow;
    sl += dsl;
    if (sl >= nsl) {
      sl -= nsl;
      ++row;
    }
  }
};

// Shared-memory matrix descriptor: K-major operand, 64-byte swizzle, rows of 64 B, 8-row core
// groups 512 B apart; start address encoded in 16-byte units.
__device__ __forceinline__ uint64_t smem_desc64(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;              // leading byte offset (not used by swizzled K-major)
  d |= (uint64_t)(512 >> 4) << 32;     // stride byte offset
  d |= (uint64_t)1 << 46;              // descriptor version
  d |= (uint64_t)4 << 61;              // 64-byte swizzle
  return d;
}

__device__ __forceinline__ void fs_cp16(uint32_t dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ float silu_nr(float z) { return z * sigm_nr(z); }
__device__ __forceinline__ float dsilu_nr(float z) {
  const float sg = sigm_nr(z);
  return sg * (1.f + z * (1.f - sg));
}

// Rounding constants of the splitting for a chunk whose largest magnitude is m: adding and
// subtracting c rounds to a multiple of 2^-23 of c's leading bit.  Magnitudes above 2^111 are
// clamped (they lose digits, not finiteness); a non-finite element makes the result
// non-finite.
__device__ __forceinline__ void split_consts(float m, float& c1, float& c2) {
  unsigned e = __float_as_uint(m) & 0x7f800000u;
  e = min(e, 238u << 23);
  c1 = __uint_as_float((e + (16u << 23)) | 0x400000u);
  c2 = __uint_as_float((e + (7u << 23)) | 0x400000u);
}
__device__ __forceinline__ void split3(float a, float c1, float c2, float& a1, float& a2,
                                       float& a3) {
  a1 = __fsub_rn(__fadd_rn(a, c1), c1);
  const float r = __fsub_rn(a, a1);            // exact
  a2 = __fsub_rn(__fadd_rn(r, c2), c2);
  a3 = __fsub_rn(r, a2);                       // exact; rounded to bf16 when packed
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// 16 columns of both accumulators (at taddr and taddr + 128) for a warp's 32 lanes; the wait
// is in the same statement, so nothing reads the registers before it
__device__ __forceinline__ void tmem_ld16x2(uint32_t taddr, uint32_t (&v)[16],
                                            uint32_t (&x)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
      "%13, %14, %15}, [%32];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, "
      "%26, %27, %28, %29, %30, %31}, [%33];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]),
        "=r"(x[5]), "=r"(x[6]), "=r"(x[7]), "=r"(x[8]), "=r"(x[9]), "=r"(x[10]), "=r"(x[11]),
        "=r"(x[12]), "=r"(x[13]), "=r"(x[14]), "=r"(x[15])
      : "r"(taddr), "r"(taddr + 128)
      : "memory");
}

// 32 consecutive bytes (32-byte aligned) in one load
__device__ __forceinline__ void ld8(const float* p, float (&v)[8]) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]),
                 "=f"(v[6]), "=f"(v[7])
               : "l"(p));
}

// Weights B^T = [W1 | 0 | scale W2], W1 [N][K1] and W2 [N][K2] FP32 (K2 = 0: W1 alone), the
// first part padded to a multiple of a chunk where there is a second -> three slices
// [3][N][ktot] bf16; one warp per row and chunk.  Run once per weight matrix, at creation.
__global__ void k_split_weights(const float* __restrict__ W1, const float* __restrict__ W2, int N,
                                int K1, int K2, int k1p, double scale,
                                __nv_bfloat16* __restrict__ out) {
  ff_pdl();
  const int K = k1p + K2, nk = (K + FS_TK - 1) / FS_TK;
  const long long t = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (t >= (long long)N * nk) return;
  const int n = (int)(t / nk), k = (int)(t % nk) * FS_TK + (threadIdx.x & 31);
  const size_t i = (size_t)n * K + k, sl = (size_t)N * K;
  float w = 0.f;
  if (k < K1) w = W1[(size_t)n * K1 + k];
  else if (k >= k1p && k < K) w = (float)(scale * (double)W2[(size_t)n * K2 + (k - k1p)]);
  float m = fabsf(w), c1, c2, a1, a2, a3;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  split_consts(m, c1, c2);
  if (k >= K) return;
  split3(w, c1, c2, a1, a2, a3);
  out[i] = __float2bfloat16_rn(a1);
  out[i + sl] = __float2bfloat16_rn(a2);
  out[i + 2 * sl] = __float2bfloat16_rn(a3);
}

// Stream u of a mode's epilogue inputs at row r, column col.
template <int MODE>
__device__ __forceinline__ const float* fs_aux(const EpiParams& ep, int u, size_t r, int col) {
  if (MODE == EPI_DSILU) return ep.z + r * ep.ldz + col;
  if (u == 1) return ep.z + r * ep.ldz + col;
  return ep.res + r * ep.ldr + col;
}

template <int MODE>
__global__ void __launch_bounds__(FS_THREADS, 1)
k_gemm_fs(const __grid_constant__ CUtensorMap tmB, const float* __restrict__ A, int lda,
          const float* __restrict__ A2, int lda2, int M, int N, int K1, int K2, int nslices,
          int nbw, EpiParams ep, int* __restrict__ err) {
  constexpr int S = fs_stages<MODE>();
  constexpr int NAUX = fs_naux<MODE>(), AUXN = fs_auxn<MODE>();
  constexpr int SLOT = NAUX * 2048;                               // bytes of a column group
  constexpr bool AUX = NAUX > 0;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t b_slice = (uint32_t)nbw * FS_TK * 2;
  const uint32_t st_bytes = 3 * FS_ASLICE + 3 * b_slice;
  float* tiles = reinterpret_cast<float*>(smem + S * st_bytes);   // FS_EW x 2 KB
  uint8_t* auxs = (uint8_t*)(tiles + FS_EW * 32 * 16);            // FS_EW x AUXN x SLOT
  uint64_t* bars = (uint64_t*)(auxs + FS_EW * AUXN * SLOT);
  uint64_t* fulla = bars;           // stage: slices of A stored (4 arrivals)
  uint64_t* fullb = fulla + S;      // stage: slices of B landed
  uint64_t* empty = fullb + S;      // stage: products that read it complete
  uint64_t* accf = empty + S;       // accumulators of group g complete
  uint64_t* acce = accf + 2;        // ... drained (4 arrivals)
  uint64_t* fin = acce + 2;
  uint32_t* tslot = (uint32_t*)(fin + 1);
  __shared__ int s_fail;
  __shared__ volatile int s_abort;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntiles = ff_cdiv(M, TM) * nslices;
  // K-chunks of A, then those of A2 (K2 = 0: none)
  const int k1c = (K1 + FS_TK - 1) / FS_TK, nk = k1c + (K2 + FS_TK - 1) / FS_TK;

  if (threadIdx.x == 0) {
    s_fail = 0;
    s_abort = 0;
    for (int q = 0; q < S; ++q) {
      mbar_init(smem_u32(&fulla[q]), 4);
      mbar_init(smem_u32(&fullb[q]), 1);
      mbar_init(smem_u32(&empty[q]), 1);
    }
    for (int g = 0; g < 2; ++g) {
      mbar_init(smem_u32(&accf[g]), 1);
      mbar_init(smem_u32(&acce[g]), 4);
    }
    mbar_init(smem_u32(fin), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == FS_EW + FS_CW + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = *tslot;
  ff_pdl();   // (the set-up above ran while the kernel ahead finished)

  if (warp >= FS_EW && warp < FS_EW + FS_CW) {
    // ---- splitting group g: chunks q = g mod 2 of this CTA's (tile, K-chunk) sequence; two
    // of them are in flight in registers.  (A group's wait for a stage tells one phase from the
    // next only because its chunk before, q - 2, has seen chunk q - 2 - S done, which is no
    // earlier than the stage's phase before last: S >= 2.)
    static_assert(S >= 2, "a stage per splitting group");
    const int g = (warp - FS_EW) >> 2, w = warp & 3;
    const int j = lane & 3, rsub = lane >> 2;
    float v[2][4][8];
    FsWalk it(blockIdx.x, gridDim.x, nslices);   // position (it, kc) of the next chunk to load
    int kc = g;
    bool more[2];
    auto load = [&](float (&d)[4][8], bool& have) {
      while (kc >= nk) {
        kc -= nk;
        it.next();
      }
      have = it.t < ntiles;
      if (have) {
        const int m0 = it.row * TM + w * 32 + rsub;
        const bool second = kc >= k1c;
        const int k = (second ? kc - k1c : kc) * FS_TK + 8 * j;
        const bool kok = k < (second ? K2 : K1);
        const float* src = second ? A2 : A;
        const int ld = second ? lda2 : lda;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = m0 + 8 * i;
          if (r < M && kok) {
            ld8(src + (size_t)r * ld + k, d[i]);
          } else {
#pragma unroll
            for (int x = 0; x < 8; ++x) d[i][x] = 0.f;
          }
        }
        kc += 2;
      }
    };
    uint32_t q = g;               // sequence number of the chunk being stored
    bool good = true;
    auto store = [&](const float (&d)[4][8]) {
      const uint32_t st = q % S;
      if (q >= S && !__all_sync(0xffffffffu, mbar_wait_ab(smem_u32(&empty[st]),
                                                          (q / S - 1) & 1, &s_abort)))
        return false;
      uint8_t* sa = smem + (size_t)st * st_bytes;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float m = 0.f;
#pragma unroll
        for (int x = 0; x < 8; ++x) m = fmaxf(m, fabsf(d[i][x]));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        float c1, c2;
        split_consts(m, c1, c2);
        const float2 k1 = make_float2(c1, c1), n1 = make_float2(-c1, -c1);
        const float2 k2 = make_float2(c2, c2), n2 = make_float2(-c2, -c2);
        const float2 m1 = make_float2(-1.f, -1.f);
        uint32_t p1[4], p2[4], p3[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          // split3 of two elements in packed instructions
          const float2 a = make_float2(d[i][2 * x], d[i][2 * x + 1]);
          const float2 s1 = __fadd2_rn(__fadd2_rn(a, k1), n1);
          const float2 r = __ffma2_rn(s1, m1, a);
          const float2 s2 = __fadd2_rn(__fadd2_rn(r, k2), n2);
          const float2 s3 = __ffma2_rn(s2, m1, r);
          p1[x] = pack2(s1.x, s1.y);
          p2[x] = pack2(s2.x, s2.y);
          p3[x] = pack2(s3.x, s3.y);
        }
        const int r = w * 32 + 8 * i + rsub;
        uint8_t* dst = sa + r * 64 + ((j ^ ((r >> 1) & 3)) << 4);
        *reinterpret_cast<uint4*>(dst) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
        *reinterpret_cast<uint4*>(dst + FS_ASLICE) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
        *reinterpret_cast<uint4*>(dst + 2 * FS_ASLICE) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&fulla[st]));
      q += 2;
      return true;
    };
    load(v[0], more[0]);
    load(v[1], more[1]);
    while (good && more[0]) {
      good = store(v[0]);
      load(v[0], more[0]);
      if (!good || !more[1]) break;
      good = store(v[1]);
      load(v[1], more[1]);
    }
    if (!good && lane == 0) {
      s_fail = 1;
      s_abort = 1;
    }
  } else if (warp == FS_EW + FS_CW) {
    // ---- TMA producer of the weight slices
    if (lane == 0) {
      uint32_t q = 0;
      bool good = true;
      for (int t = blockIdx.x; t < ntiles && good; t += gridDim.x) {
        const int n0 = (t % nslices) * nbw;
        for (int kc = 0; kc < nk; ++kc, ++q) {
          const uint32_t st = q % S;
          if (q >= S && !mbar_wait_ab(smem_u32(&empty[st]), (q / S - 1) & 1, &s_abort)) {
            good = false;
            break;
          }
          uint8_t* sb = smem + (size_t)st * st_bytes + 3 * FS_ASLICE;
          mbar_expect_tx(smem_u32(&fullb[st]), 3 * b_slice);
          for (int sl = 0; sl < 3; ++sl)
            tma_load_2d(smem_u32(sb + sl * b_slice), &tmB, kc * FS_TK, sl * N + n0,
                        smem_u32(&fullb[st]));
        }
      }
      if (!good) {
        s_fail = 1;
        s_abort = 1;
      }
      // the loads issued last land before the CTA may exit
      for (uint32_t k = 0; k < S && k < q; ++k) {
        const uint32_t p = q - 1 - k;
        mbar_wait(smem_u32(&fullb[p % S]), (p / S) & 1);
      }
    }
  } else if (warp == FS_EW + FS_CW + 1) {
    // ---- MMA issuer
    if (lane == 0) {
      uint32_t q = 0;
      bool good = true;
      int jt = 0;
      for (int t = blockIdx.x; t < ntiles && good; t += gridDim.x, ++jt) {
        const int g = jt & 1;
        if (jt >= 2 &&
            !mbar_wait_ab(smem_u32(&acce[g]), (uint32_t)(((jt >> 1) - 1) & 1), &s_abort)) {
          good = false;
          break;
        }
        fence_after();
        const int ncur = min(nbw, N - (t % nslices) * nbw);
        const uint32_t idesc = instr_desc(TM, ncur);
        const uint32_t dmain = tbase + (uint32_t)(g * 256), dcross = dmain + 128;
        for (int kc = 0; kc < nk; ++kc, ++q) {
          const uint32_t st = q % S, par = (q / S) & 1;
          if (!mbar_wait_ab(smem_u32(&fullb[st]), par, &s_abort) ||
              !mbar_wait_ab(smem_u32(&fulla[st]), par, &s_abort)) {
            good = false;
            break;
          }
          fence_after();
          const uint8_t* sa = smem + (size_t)st * st_bytes;
          const uint8_t* sb = sa + 3 * FS_ASLICE;
          uint64_t da[3], db[3];
          for (int sl = 0; sl < 3; ++sl) {
            da[sl] = smem_desc64(smem_u32(sa + sl * FS_ASLICE));
            db[sl] = smem_desc64(smem_u32(sb + sl * b_slice));
          }
          const int nkk =
              min(FS_TK / 16, (kc < k1c ? K1 - kc * FS_TK : K2 - (kc - k1c) * FS_TK) / 16);
          for (int kk = 0; kk < nkk; ++kk) {
            const uint64_t o = (uint64_t)(kk * 2);
            const uint32_t acc = (kc > 0 || kk > 0) ? 1u : 0u;
            mma_bf16(dmain, da[0] + o, db[0] + o, idesc, acc);
            mma_bf16(dcross, da[0] + o, db[1] + o, idesc, acc);
            mma_bf16(dcross, da[0] + o, db[2] + o, idesc, 1u);
            mma_bf16(dcross, da[1] + o, db[0] + o, idesc, 1u);
            mma_bf16(dcross, da[1] + o, db[1] + o, idesc, 1u);
            mma_bf16(dcross, da[2] + o, db[0] + o, idesc, 1u);
          }
          mma_commit(smem_u32(&empty[st]));
        }
        // (test hook: the first tile's accumulators are never signalled, so its epilogue group's
        // bounded wait runs out and every role leaves through the abort path)
        if (good && !(ep.test_stall && jt == 0)) mma_commit(smem_u32(&accf[g]));
      }
      if (!good) {
        s_fail = 1;
        s_abort = 1;
      }
      // every MMA issued above has completed before the tensor memory is released
      mma_commit(smem_u32(fin));
      mbar_wait(smem_u32(fin), 0);
    }
  } else {
    // ---- epilogue group g, lane quadrant warp & 3: 16 columns of the warp's 32 rows at a
    // time go through its shared tile (float4 groups XOR-swizzled, conflict-free both ways)
    // and leave as 64-byte row segments; a lane then owns 4 columns of rows rsub + 8 i.  Every
    // lane copies the epilogue inputs that it will read itself into its own slots, AUXN - 1
    // column groups ahead and across tile boundaries (48 KB in flight per SM: with one
    // group ahead in registers the residual modes ran at a third of the copy bandwidth).
    const int g = warp >> 2, quad = warp & 3;
    const int gq = lane & 3, rsub = lane >> 2;
    float* tile = tiles + warp * 32 * 16;
    uint8_t* my_aux = auxs + (size_t)warp * (AUXN * SLOT) + lane * 16;
    FsWalk at(blockIdx.x + g * gridDim.x, 2 * gridDim.x, nslices);   // next columns to fetch:
    int ac = 0;                                                      // tile, first column
    uint32_t an = 0;                                                 // column groups fetched
    auto fetch = [&]() {
      if (at.t < ntiles) {
        const int n0 = at.sl * nbw, mq = at.row * TM + quad * 32 + rsub;
#pragma unroll
        for (int u = 0; u < NAUX; ++u)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (mq + 8 * i < M)
              fs_cp16(smem_u32(my_aux + (an % AUXN) * SLOT + u * 2048 + i * 512),
                      fs_aux<MODE>(ep, u, (size_t)(mq + 8 * i), n0 + ac + 4 * gq));
        ac += 16;
        if (ac >= min(nbw, N - n0)) {
          ac = 0;
          at.next();
        }
      }
      ++an;
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    uint32_t un = 0;                               // column groups used
    if (AUX)
      for (int k = 0; k < AUXN - 1; ++k) fetch();
    bool good = true;
    int jt = g;
    FsWalk it(blockIdx.x + g * gridDim.x, 2 * gridDim.x, nslices);
    for (; it.t < ntiles; it.next(), jt += 2) {
      const int m0 = it.row * TM + quad * 32 + rsub;
      const int n0 = it.sl * nbw;
      const int ncur = min(nbw, N - n0);
      float fr[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        fr[i] = 0.f;
        if ((MODE == EPI_SILU_F || MODE == EPI_SILU_RES || MODE == EPI_HEAD ||
             MODE == EPI_RES_DS) && m0 + 8 * i < M)
          fr[i] = ep.f[(size_t)(m0 + 8 * i) * ep.ldf];
      }
      good = __all_sync(
          0xffffffffu, mbar_wait_ab(smem_u32(&accf[g]), (uint32_t)((jt >> 1) & 1), &s_abort,
                                    ep.test_stall ? kTestWaitLimit : kWaitLimit));
      if (!good) break;
      fence_after();
      float racc[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) racc[i][0] = racc[i][1] = 0.f;
      for (int c0 = 0; c0 < ncur; c0 += 16) {
        if (AUX) fetch();
        {
          uint32_t v[16], x[16];
          tmem_ld16x2(tbase + ((uint32_t)(quad * 32) << 16) + (uint32_t)(g * 256 + c0), v, x);
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            float s4[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
              s4[k] = __uint_as_float(v[4 * q4 + k]) + __uint_as_float(x[4 * q4 + k]);
            *reinterpret_cast<float4*>(&tile[lane * 16 + 4 * (q4 ^ ((lane >> 1) & 3))]) =
                make_float4(s4[0], s4[1], s4[2], s4[3]);
          }
        }
        __syncwarp();
        const int col = n0 + c0 + 4 * gq;
        if (AUX) asm volatile("cp.async.wait_group %0;" ::"n"(AUXN - 1) : "memory");
        const uint8_t* ax = my_aux + (un++ % AUXN) * SLOT;
        float4 w4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (MODE == EPI_HEAD) w4 = *reinterpret_cast<const float4*>(ep.wv + col);
        const float wv[4] = {w4.x, w4.y, w4.z, w4.w};
        // the arithmetic runs for all rows, so that the 16 chains of a lane interleave (under a
        // branch per row they ran four at a time); only the stores look at the row count
        float pre[4][4], o[4][4];   // RES_DS: pre = dE/dz of the layer below
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int rl = 8 * i + rsub;
          const float4 acc =
              *reinterpret_cast<const float4*>(&tile[rl * 16 + 4 * (gq ^ ((rl >> 1) & 3))]);
          float4 a = make_float4(0.f, 0.f, 0.f, 0.f), z = a;
          if (AUX) a = *reinterpret_cast<const float4*>(ax + i * 512);
          if (NAUX == 2) z = *reinterpret_cast<const float4*>(ax + 2048 + i * 512);
          const float v[4] = {ep.alpha * acc.x, ep.alpha * acc.y, ep.alpha * acc.z,
                              ep.alpha * acc.w};
          const float a4[4] = {a.x, a.y, a.z, a.w}, z4[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            pre[i][k] = v[k];
            if (MODE == EPI_HEAD || MODE == EPI_RES_DS) {
              // HEAD: sums of w a and w silu(v), dE/dz = beta f w silu'(v).  RES_DS: dE/dx, its
              // sum with silu(z), and dE/dz of the layer below.
              const float zk = MODE == EPI_HEAD ? v[k] : z4[k];
              const float sg = sigm_nr(zk), sv = zk * sg;
              const float ds = sg + sv * (1.f - sg);
              if (MODE == EPI_HEAD) {
                racc[i][0] += wv[k] * a4[k];
                racc[i][1] += wv[k] * sv;
                o[i][k] = ep.beta * fr[i] * wv[k] * ds;
              } else {
                o[i][k] = v[k] + ep.beta * a4[k];
                racc[i][0] += o[i][k] * sv;
                pre[i][k] = ep.alpha2 * fr[i] * o[i][k] * ds;
              }
              continue;
            }
            if (MODE == EPI_STORE) o[i][k] = v[k];
            else if (MODE == EPI_SILU) o[i][k] = silu_nr(v[k]);
            else if (MODE == EPI_SILU_F) o[i][k] = fr[i] * silu_nr(v[k]);
            else if (MODE == EPI_SILU_RES) o[i][k] = ep.beta * (a4[k] + fr[i] * silu_nr(v[k]));
            else o[i][k] = v[k] * dsilu_nr(a4[k]);   // DSILU
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (m0 + 8 * i >= M) continue;
          const size_t r = (size_t)(m0 + 8 * i);
          if (MODE == EPI_SILU || MODE == EPI_SILU_F || MODE == EPI_SILU_RES ||
              MODE == EPI_RES_DS)
            *reinterpret_cast<float4*>(ep.pre + r * ep.ldp + col) =
                make_float4(pre[i][0], pre[i][1], pre[i][2], pre[i][3]);
          if (MODE != EPI_RES_DS || ep.out)
            *reinterpret_cast<float4*>(ep.out + r * ep.ldo + col) =
                make_float4(o[i][0], o[i][1], o[i][2], o[i][3]);
        }
        __syncwarp();   // the shared tile is free again
      }
      if (MODE == EPI_HEAD || MODE == EPI_RES_DS) {
        // row sums over this slice's columns (the 4 lanes of a row), into the slice's own slot
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
          for (int q = 0; q < (MODE == EPI_HEAD ? 2 : 1); ++q) {
            racc[i][q] += __shfl_xor_sync(0xffffffffu, racc[i][q], 1);
            racc[i][q] += __shfl_xor_sync(0xffffffffu, racc[i][q], 2);
          }
          if (gq == 0 && m0 + 8 * i < M) {
            const size_t at_ = (size_t)it.sl * ep.gfp_ld + m0 + 8 * i;
            if (MODE == EPI_HEAD) {
              ep.eout[at_] = ep.beta * (racc[i][0] + fr[i] * racc[i][1]);
              ep.gfp[at_] = ep.beta * racc[i][1];
            } else {
              ep.gfp[at_] = ep.alpha2 * racc[i][0];
            }
          }
        }
      }
      // the accumulators are free again
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&acce[g]));
    }
    if (AUX) asm volatile("cp.async.wait_all;" ::: "memory");
    if (!good && lane == 0) {
      s_fail = 1;
      s_abort = 1;
    }
  }
  fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && s_fail) atomicOr(err, FF_FLAG_TIMEOUT);
  if (warp == FS_EW + FS_CW + 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(512)
                 : "memory");
}

template <int MODE>
bool launch_fs(const CUtensorMap& tb, const float* A, int lda, const float* A2, int lda2, int M,
               int N, int K1, int K2, int nslices, int nbw, const EpiParams& ep, int* err,
               cudaStream_t s) {
  static PerDevice<bool> limit;   // of dynamic shared memory, set on this device
  const FfDevice* dev = ff_device();
  if (!dev || !limit.get(dev->id, [](bool& set) {
        set = cudaFuncSetAttribute(k_gemm_fs<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   226 * 1024) == cudaSuccess;
        if (!set) cudaGetLastError();
        return set;
      }))
    return false;
  // ring, tiles, epilogue inputs, alignment, barriers
  const size_t bytes = fs_stages<MODE>() * (3 * (size_t)FS_ASLICE + 3 * (size_t)nbw * FS_TK * 2) +
                       FS_EW * 32 * 16 * 4 + FS_EW * fs_auxn<MODE>() * fs_naux<MODE>() * 2048 +
                       1024 + 256;
  const int ntiles = ff_cdiv(M, TM) * nslices;
  const int grid = ntiles < dev->n_sm ? ntiles : dev->n_sm;
  ff_launch_work(ntiles, k_gemm_fs<MODE>, grid, FS_THREADS, bytes, s, tb, A, lda, A2, lda2, M, N,
                 K1, K2, nslices, nbw, ep, err);
  return true;
}

using FsFn = bool (*)(const CUtensorMap&, const float*, int, const float*, int, int, int, int, int,
                      int, int, const EpiParams&, int*, cudaStream_t);
// indexed by epilogue mode
const FsFn kFs[] = {launch_fs<EPI_STORE>,    launch_fs<EPI_SILU>,  launch_fs<EPI_SILU_F>,
                    launch_fs<EPI_SILU_RES>, launch_fs<EPI_DSILU>, nullptr,   // (no EPI_RES)
                    launch_fs<EPI_HEAD>,     launch_fs<EPI_RES_DS>};

}  // namespace

int split_ld(int K1, int K2) {
  return K2 > 0 ? (K1 + FS_TK - 1) / FS_TK * FS_TK + K2 : K1;
}

void launch_split_weights(const float* W1, int N, int K1, const float* W2, int K2, double scale,
                          __nv_bfloat16* out, cudaStream_t s) {
  const int ld = split_ld(K1, K2);
  const long long n = (long long)N * ((ld + FS_TK - 1) / FS_TK);
  ff_launch(k_split_weights, ff_cdiv(n, 8), 256, 0, s, W1, W2, N, K1, K2, ld - K2, scale, out);
  ff_count_launch(1);
}

bool launch_gemm_f32(int mode, int M, int N, int K, const float* A, int lda,
                     const __nv_bfloat16* Bs, int ldb, const EpiParams& ep, int* err,
                     cudaStream_t s, const float* A2, int K2, int lda2) {
  ProfScope ps_(PC_GEMM_F32, s);
  if (M <= 0) return true;
  if (mode < EPI_STORE || mode > EPI_RES_DS || !kFs[mode]) return false;
  if (N % 16 != 0 || K % 16 != 0 || lda % 8 != 0 || ((uintptr_t)A & 31)) return false;
  if (A2 && (K2 <= 0 || K2 % 16 != 0 || lda2 % 8 != 0 || ((uintptr_t)A2 & 31))) return false;
  const int ktot = split_ld(K, A2 ? K2 : 0);
  if (ldb < ktot || ldb % 8 != 0) return false;
  const int nslices = (N + 127) / 128;
  const int nbw = nslices == 1 ? N : 128;
  CUtensorMap tb;
  if (!make_map(&tb, Bs, 3LL * N, ktot, ldb, nbw, FS_TK)) return false;
  if (!kFs[mode](tb, A, lda, A2, lda2, M, N, K, A2 ? K2 : 0, nslices, nbw, ep, err, s))
    return false;
  ff_count_launch(1);
  return true;
}
