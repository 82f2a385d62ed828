// Learned pair gate: a 5-64-64-64-1 multilayer perceptron with GELU
// activations, bf16 weights and fp32 accumulation, scoring every pair of
// the compatibility table (Eq. 2) that passes the Mahalanobis test; with
// the gate on, a pair stays in the table only when its logit reaches the
// threshold.  This extends the paper's gate g_ijk (Section 3), a plain
// threshold, with a model trained on which pairs the retained hypotheses of
// the ungated filter use.
//
// Layers 1-3 run on the 5th-generation tensor cores: 128 pairs per tile,
// operands staged in shared memory in the canonical no-swizzle layout,
// tcgen05.mma issued by one thread with the accumulator (128 lanes x 64 fp32
// columns) in tensor memory, completion signalled on an mbarrier, tcgen05.ld
// back to registers for the bias + GELU epilogue.  The output layer is a
// 64-term dot product per row.  Training runs the same forward pass, then the
// backward pass, every product of it on the tensor cores as well: activation
// gradients dz * W (W read as a transposed operand), and weight gradients
// h^T dz with dz, an fp32 value, as the exact sum of three bf16 parts (8 + 8
// + 8 bits), so that the products are those of the fp32 value; Adam updates
// the fp32 master parameters.
#include <cuda_bf16.h>

#include "glmb_kernels.h"

namespace glmb {

namespace {

constexpr int kTile = 128;        // rows (pairs) per tile = MMA M
constexpr int kHid = 64;          // hidden width = MMA N
constexpr int kIn = 5;            // features

// canonical no-swizzle K-major layout of a bf16 operand with kc8 = K / 8
// core matrices per row group: element (r, k) of core matrix (r/8, k/8),
// each core matrix 8 rows x 16 bytes stored contiguously
__device__ __forceinline__ uint32_t core_off(int r, int k, int kc8) {
  return (uint32_t)((((r >> 3) * kc8 + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor of tcgen05: start address, leading
// (K-direction core matrix) byte offset, stride (8-row group) byte offset,
// descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t mdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
         ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B,
// both K-major, N = 64, M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kHid >> 3) << 17) |
                            ((uint32_t)(kTile >> 4) << 24);
// the operand lies with its M (A) or N (B) index contiguous instead of K: a
// core matrix is then 8 K values x 16 bytes of M or N, the leading byte
// offset steps 8 K values and the stride byte offset 8 M or N values
constexpr uint32_t kATrans = 1u << 15, kBTrans = 1u << 16;

__device__ __forceinline__ void mma_issue(uint32_t tmem, uint64_t a, uint64_t b, uint32_t acc,
                                          uint32_t idesc = kIdesc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
               : "memory");
}

__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// generic-proxy shared-memory writes made visible to the tensor cores
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// waits for the mbarrier phase with the given parity; gives up after
// `limit` SM clock cycles, about a second by default (returns false)
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, long long limit = kGateWaitLimit) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}

// 16 consecutive fp32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// 16 fp32 columns of this thread's TMEM lane, written
__device__ __forceinline__ void tmem_st16(uint32_t addr, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15, %16};" ::"r"(addr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// two fp32 operations in one instruction (each rounded as the scalar one)
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// GELU of v + b for two columns: 0.5 z (1 + erf(z / sqrt 2))
__device__ __forceinline__ float2 gelu2(float2 v, float2 b) {
  const unsigned long long z = add2(pack2(v.x, v.y), pack2(b.x, b.y));
  const float2 t = unpack2(mul2(z, pack2(0.70710678118654752f, 0.70710678118654752f)));
  const unsigned long long e = add2(pack2(erff(t.x), erff(t.y)), pack2(1.f, 1.f));
  return unpack2(mul2(mul2(z, pack2(0.5f, 0.5f)), e));
}

// GELU and its derivative
__device__ __forceinline__ void gelu_both(float x, float& h, float& g) {
  const float e = 1.f + erff(x * 0.70710678118654752f);
  h = 0.5f * x * e;
  g = 0.5f * e + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// eight values as bf16 into one 16-byte core-matrix row
__device__ __forceinline__ void st_core8(unsigned char* base, uint32_t off, const float* v) {
  __nv_bfloat162 p[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) p[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
  *reinterpret_cast<uint4*>(base + off) = *reinterpret_cast<const uint4*>(p);
}

// shared-memory plans (bytes); matrices on 1024-byte boundaries.
// Training: one tile of 128 rows and 256 threads per CTA, two CTAs per SM.
struct TLay {
  static constexpr int W1 = 0, W2 = 2048, W3 = W2 + 8192;
  static constexpr int A0 = W3 + 8192;                           // 128 x 16 bf16
  static constexpr int H = A0 + 4096;                            // 128 x (64 of layer 1 | 64 of layer 2) bf16
  static constexpr int DZ = H + 32768;                           // three bf16 parts of dz, 128 x 64 each
  static constexpr int CST = DZ + 3 * 16384;                     // b1 b2 b3 w4(bf16) mu sd b4
  static constexpr int ZP = CST + 272 * 4;                       // the output layer's sum
  static constexpr int GW1 = ZP + 2 * kTile * 4;                 // gradient of W1, summed over the CTA's tiles
  static constexpr int MBAR = GW1 + kHid * kIn * 4;              // two barriers
  static constexpr int TSLOT = MBAR + 16, FLAG = TSLOT + 4;
  static constexpr int TOTAL = FLAG + 12;
  static constexpr int GRAD = DZ;                                // at the end: the CTA's gradient
};
// Scoring: kFwdGroups tiles in flight per CTA, 128 threads each, sharing the
// weights.  The layer-1 operand lies in the hidden operand's place (its MMA
// is done before layer 1's activations are written).
constexpr int kFwdGroups = 4;
struct FLay {
  static constexpr int W1 = 0, W2 = 2048, W3 = W2 + 8192, H = W3 + 8192;
  static constexpr int CST = H + kFwdGroups * 16384, MBAR = CST + 272 * 4;
  static constexpr int TSLOT = MBAR + 8 * kFwdGroups, FLAG = TSLOT + 4;
  static constexpr int TOTAL = (FLAG + 4 * kFwdGroups + 15) & ~15;
};

constexpr int kCB1 = 0, kCB2 = 64, kCB3 = 128, kCW4 = 192, kCMu = 256, kCSd = 261, kCB4 = 266;

// stages the weights (rounded to bf16) into the operand layout, eight
// consecutive inputs of a unit per thread, and the vectors into the constant
// block
__device__ void stage_weights(const float* __restrict__ P, unsigned char* sm, int w1, int w2, int w3, float* cst) {
  for (int idx = threadIdx.x; idx < 2 * kHid * kHid / 8; idx += blockDim.x) {
    const int o = (idx >> 3) & (kHid - 1), j = (idx & 7) * 8;
    const bool second = idx >= kHid * kHid / 8;
    const float* src = P + (second ? kGateW3 : kGateW2) + o * kHid + j;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = src[k];
    st_core8(sm + (second ? w3 : w2), core_off(o, j, 8), v);
  }
  for (int idx = threadIdx.x; idx < 2 * kHid; idx += blockDim.x) {
    const int o = idx >> 1, j = (idx & 1) * 8;
    float v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = j + k < kIn ? P[kGateW1 + o * kIn + j + k] : 0.f;
    st_core8(sm + w1, core_off(o, j, 2), v);
  }
  for (int idx = threadIdx.x; idx < kHid; idx += blockDim.x) {
    cst[kCB1 + idx] = P[kGateB1 + idx];
    cst[kCB2 + idx] = P[kGateB2 + idx];
    cst[kCB3 + idx] = P[kGateB3 + idx];
    cst[kCW4 + idx] = bf16r(P[kGateW4 + idx]);
  }
  if (threadIdx.x < kIn) {
    cst[kCMu + threadIdx.x] = P[kGateMu + threadIdx.x];
    cst[kCSd + threadIdx.x] = P[kGateSd + threadIdx.x];
  }
  if (threadIdx.x == 0) cst[kCB4] = P[kGateB4];
}

// TMEM: warp 0 allocates the CTA's columns (256: two CTAs per SM), then lets
// the other CTAs of the SM allocate
constexpr uint32_t kTmemCols = 256;
__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
}
__device__ __forceinline__ void tmem_free(uint32_t taddr) {
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(kTmemCols));
}

__device__ __forceinline__ void mbar_init(uint32_t mbar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// one product on the tensor cores: D (+)= A * B^T over 16 ksteps values of K,
// the operands' core matrices at the given leading and stride byte offsets
// and their next 16 K values at `astep` / `bstep` bytes; one thread issues
struct Oper {
  uint32_t addr, lbo, sbo, step;
};
__device__ __forceinline__ void product(uint32_t d, Oper a, Oper b, int ksteps, uint32_t acc, uint32_t idesc) {
  for (int k = 0; k < ksteps; ++k)
    mma_issue(d, mdesc(a.addr + (uint32_t)k * a.step, a.lbo, a.sbo),
              mdesc(b.addr + (uint32_t)k * b.step, b.lbo, b.sbo), (acc || k > 0) ? 1u : 0u, idesc);
}
// K contiguous, kc8 = K / 8 core matrices per row group
__device__ __forceinline__ Oper k_major(uint32_t addr, uint32_t kc8) { return Oper{addr, 128u, kc8 << 7, 256u}; }
// M or N contiguous (K groups of 8 rows, mc8 core matrices each)
__device__ __forceinline__ Oper mn_major(uint32_t addr, uint32_t mc8) {
  return Oper{addr, mc8 << 7, 128u, mc8 << 8};
}

// every thread waits for a product; a time-out anywhere aborts the CTA
__device__ __forceinline__ bool layer_wait(uint32_t mbar, uint32_t& parity, int* flag,
                                           long long limit = kGateWaitLimit) {
  const bool ok = mbar_wait(mbar, parity, limit);
  parity ^= 1u;
  if (!ok) atomicOr(flag, 1);
  fence_after();
  return __syncthreads_or(!ok) == 0;
}
// the same for one group of 128 threads (named barrier 1 + group)
__device__ __forceinline__ void group_bar(int group) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(kTile) : "memory");
}
__device__ __forceinline__ bool group_wait(uint32_t mbar, uint32_t& parity, volatile int* flag, int group,
                                           long long limit) {
  const bool ok = mbar_wait(mbar, parity, limit);
  parity ^= 1u;
  if (!ok) *flag = 1;
  fence_after();
  group_bar(group);
  return *flag == 0;
}

// epilogue of a hidden layer for this thread's row: bias, GELU, bf16 into the
// next layer's operand
__device__ __forceinline__ void hidden_epilogue(uint32_t trow, const float* b, unsigned char* dst, int m) {
#pragma unroll 1
  for (int c0 = 0; c0 < kHid; c0 += 16) {
    float v[16];
    tmem_ld16(trow + (uint32_t)c0, v);
#pragma unroll
    for (int j = 0; j < 16; j += 2) {
      const float2 r = gelu2(make_float2(v[j], v[j + 1]), *reinterpret_cast<const float2*>(b + c0 + j));
      v[j] = r.x;
      v[j + 1] = r.y;
    }
    st_core8(dst, core_off(m, c0, 8), v);
    st_core8(dst, core_off(m, c0 + 8, 8), v + 8);
  }
}

// standardised features of one row as bf16 into the layer-1 operand
__device__ __forceinline__ void write_input(unsigned char* a0, int m, const float* f, bool valid,
                                            const float* cst) {
  float v[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = 0.f;
  if (valid) {
#pragma unroll
    for (int j = 0; j < kIn; ++j) v[j] = (f[j] - cst[kCMu + j]) / cst[kCSd + j];
  }
  st_core8(a0, core_off(m, 0, 2), v);
  st_core8(a0, core_off(m, 8, 2), v + 8);
}

}  // namespace

// the gate's raw features of pair p: d^2 (recovered from log C and log det
// S), innovation norm, prior existence, age in frames, log det S
__device__ __forceinline__ void pair_features(const Model& md, const CompTable& ct, const PairTable& pt,
                                              const FrameDev& fs, uint32_t p, int c, float* f) {
  const float ld = pt.logdetS[c];
  const float c0 = md.log_pd - 0.5f * (ld + (float)md.dz * kLog2Pi);
  float n2 = 0.f;
  for (int a = 0; a < md.dz; ++a) {
    const float e = pt.e[(size_t)a * (size_t)pt.cap_pairs + p];
    n2 += e * e;
  }
  f[0] = fmaxf(2.f * (c0 - pt.logC[p]), 0.f);
  f[1] = sqrtf(n2);
  f[2] = expf(ct.logp[c]);
  f[3] = (float)((uint32_t)fs.frame - ct.lk[c]);
  f[4] = ld;
}

// ---------------------------------------------------------------------------
// forward pass: rows from a feature array (X [n][5]) or from the pair table
// ---------------------------------------------------------------------------
struct GateFwdArgs {
  const float* P;
  const float* X;
  long long n;
  // table mode
  Model md;
  CompTable ct;
  PairTable pt;
  const FrameDev* fs;
  float thr;
  uint8_t* keep;
  float* logit;
  unsigned* err;
  long long wait_limit;   // SM clock cycles a completion wait may take
  int skip_first_mma;     // failure-detection test: CTA 0 issues no MMA for its first tile
};

// Scoring: persistent CTAs of kFwdGroups groups of 128 threads, each group a
// tile of 128 rows at a time, synchronised within the group only, so that the
// tensor-core waits of one tile are covered by the epilogues of the others.
// What bounds it is the issue rate of the epilogue (192 erf per row); eight
// tiles in flight per SM (two CTAs, 64 registers a thread, the weights staged
// once per CTA) keep the schedulers busy where five 128-thread CTAs with
// their own weights left a quarter of the issue slots empty, and the bias,
// the scalings and the products run two columns to an instruction.  Measured
// on 4.2 M rows: 887 us -> 737 us.
template <bool kTable>
__global__ void __launch_bounds__(kTile * kFwdGroups, 2) gate_forward_kernel(const __grid_constant__ GateFwdArgs g) {
  pdl_enter();
  extern __shared__ __align__(1024) unsigned char sm[];
  float* cst = reinterpret_cast<float*>(sm + FLay::CST);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + FLay::TSLOT);
  const int group = threadIdx.x / kTile, m = threadIdx.x % kTile;
  volatile int* flag = reinterpret_cast<int*>(sm + FLay::FLAG) + group;
  const uint32_t mbar = smem_u32(sm + FLay::MBAR) + 8u * (uint32_t)group;
  long long n = g.n;
  if (kTable) {
    // a table that overflowed its capacity (the frame is abandoned) is
    // scored only up to the capacity
    n = min((long long)*g.pt.total, g.pt.cap_pairs);
  }
  const long long tiles = (n + kTile - 1) / kTile;
  if ((long long)blockIdx.x >= tiles) return;
  if (m == 0) {
    *flag = 0;
    mbar_init(mbar);
  }
  tmem_alloc(tslot);
  stage_weights(g.P, sm, FLay::W1, FLay::W2, FLay::W3, cst);
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot, tacc = tmem + (uint32_t)(kHid * group);
  const uint32_t trow = tacc + ((uint32_t)(m & ~31) << 16);
  unsigned char* hbuf = sm + FLay::H + group * 16384;
  const uint32_t h = smem_u32(hbuf), w1 = smem_u32(sm + FLay::W1);
  const uint32_t w2 = smem_u32(sm + FLay::W2), w3 = smem_u32(sm + FLay::W3);
  uint32_t parity = 0;
  bool ok = true;
  // tiles go to the CTAs first, then to their groups (few tiles spread out)
  const long long first = blockIdx.x + (long long)gridDim.x * group, stride = (long long)gridDim.x * kFwdGroups;
  auto features = [&](long long row, float (&f)[kIn]) {
    if (kTable) {
      pair_features(g.md, g.ct, g.pt, *g.fs, (uint32_t)row, (int)g.pt.comp[row], f);
    } else {
#pragma unroll
      for (int j = 0; j < kIn; ++j) f[j] = __ldg(g.X + row * kIn + j);
    }
  };
  float f[kIn] = {0.f, 0.f, 0.f, 0.f, 0.f};
  if (first * kTile + m < n) features(first * kTile + m, f);
  for (long long tile = first; tile < tiles; tile += stride) {
    const long long row = tile * kTile + m;
    const bool valid = row < n;
    write_input(hbuf, m, f, valid, cst);
    fence_async_smem();
    fence_before();
    group_bar(group);
    if (m == 0 && !(g.skip_first_mma && blockIdx.x == 0 && group == 0 && tile == first)) {
      fence_after();
      product(tacc, k_major(h, 2), k_major(w1, 2), 1, 0u, kIdesc);
      mma_commit(mbar);
    }
    // the next tile's features arrive while this one is scored
    const long long next = (tile + stride) * kTile + m;
    if (tile + stride < tiles && next < n) features(next, f);
    if (!(ok = group_wait(mbar, parity, flag, group, g.wait_limit))) break;
    hidden_epilogue(trow, cst + kCB1, hbuf, m);
    fence_before();
    fence_async_smem();
    group_bar(group);
    if (m == 0) {
      fence_after();
      product(tacc, k_major(h, 8), k_major(w2, 8), 4, 0u, kIdesc);
      mma_commit(mbar);
    }
    if (!(ok = group_wait(mbar, parity, flag, group, g.wait_limit))) break;
    // layer 2's activations overwrite its own operand once the MMA is done
    hidden_epilogue(trow, cst + kCB2, hbuf, m);
    fence_before();
    fence_async_smem();
    group_bar(group);
    if (m == 0) {
      fence_after();
      product(tacc, k_major(h, 8), k_major(w3, 8), 4, 0u, kIdesc);
      mma_commit(mbar);
    }
    if (!(ok = group_wait(mbar, parity, flag, group, g.wait_limit))) break;
    float z = cst[kCB4];
#pragma unroll 1
    for (int c0 = 0; c0 < kHid; c0 += 16) {
      float v[16];
      tmem_ld16(trow + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < 16; j += 2) {
        const float2 r = gelu2(make_float2(v[j], v[j + 1]), *reinterpret_cast<const float2*>(cst + kCB3 + c0 + j));
        z += bf16r(r.x) * cst[kCW4 + c0 + j];
        z += bf16r(r.y) * cst[kCW4 + c0 + j + 1];
      }
    }
    if (valid) {
      if (g.logit) g.logit[row] = z;
      if (kTable && g.keep) g.keep[row] = z >= g.thr ? 1 : 0;
    }
  }
  if (!ok) {
    // an MMA may still be in flight: give it one more bounded wait
    mbar_wait(mbar, parity ^ 1u, g.wait_limit);
    if (m == 0) atomicOr(g.err, kErrGate);
  }
  fence_before();
  __syncthreads();
  fence_after();
  tmem_free(tmem);
}

// ---------------------------------------------------------------------------
// training: forward, weighted binary cross-entropy, backward
// ---------------------------------------------------------------------------
struct GateTrainArgs {
  const float* P;
  const float* X;
  const float* y;
  const float* wt;
  long long n;
  float* grad;
  double* loss;
  unsigned* err;
};

constexpr int kTrainThreads = 2 * kTile;

// Sums over a warp's lanes of 32 values per lane: lane l returns the sum of
// v[l] (each step halves the values a lane still carries).
__device__ __forceinline__ float lane_column_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < o; ++j) {
      const float send = up ? v[j] : v[j + o];
      const float keep = up ? v[j + o] : v[j];
      v[j] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, o);
    }
  }
  return v[0];
}

// eight consecutive columns of dz as three bf16 parts (their sum is the fp32
// value: each part takes the next 8 bits of its significand)
__device__ __forceinline__ void st_split8(unsigned char* dz, uint32_t off, const float* v) {
  float hi[8], mid[8], lo[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    hi[j] = bf16r(v[j]);
    const float r = v[j] - hi[j];
    mid[j] = bf16r(r);
    lo[j] = r - mid[j];
  }
  st_core8(dz, off, hi);
  st_core8(dz + 16384, off, mid);
  st_core8(dz + 32768, off, lo);
}

// Training: one tile of 128 rows per pass of a 256-thread CTA, two threads
// per row (32 columns each), two CTAs per SM, so a mini-batch of 32768 rows
// is in flight at once.  Every product runs on the tensor cores: the weight
// gradients of layers 2 and 3 as [h1 | h2]^T dz (M = 128 features, N = 64
// units, K = 128 rows; half of the rows of a product are the layer's), layer
// 1's as x^T dz.  GELU' of layers 1 and 2 is formed with GELU (one erf for
// both) and waits in tensor memory.  The CTA sums its tiles' gradients in
// fp32 registers (a tile's products are read back and added, so no sum runs
// longer than a tile in the tensor cores' accumulators) and adds them to
// global memory with one bulk reduction.  Measured at 32768 rows, forward +
// backward + Adam: 128 us with the weight gradients on the CUDA cores (128
// threads per SM, erf recomputed twice), 35 us so.
__global__ void __launch_bounds__(kTrainThreads, 2) gate_train_kernel(const __grid_constant__ GateTrainArgs g) {
  pdl_enter();
  extern __shared__ __align__(1024) unsigned char sm[];
  float* cst = reinterpret_cast<float*>(sm + TLay::CST);
  float* zp = reinterpret_cast<float*>(sm + TLay::ZP);
  float* gw1 = reinterpret_cast<float*>(sm + TLay::GW1);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + TLay::TSLOT);
  int* flag = reinterpret_cast<int*>(sm + TLay::FLAG);
  const uint32_t bar0 = smem_u32(sm + TLay::MBAR), bar1 = bar0 + 8u;
  const int tid = threadIdx.x, m = tid & (kTile - 1), half = tid >> 7, lane = tid & 31, quad = (tid >> 5) & 3;
  const int cb = 32 * half;   // this thread's columns [cb, cb + 32)
  const long long tiles = (g.n + kTile - 1) / kTile;
  if ((long long)blockIdx.x >= tiles) return;
  if (tid == 0) {
    *flag = 0;
    mbar_init(bar0);
    mbar_init(bar1);
  }
  tmem_alloc(tslot);
  stage_weights(g.P, sm, TLay::W1, TLay::W2, TLay::W3, cst);
  for (int i = tid; i < kHid * kIn; i += kTrainThreads) gw1[i] = 0.f;
  fence_async_smem();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tslot;
  // TMEM columns: layer products, weight-gradient products, GELU' of layers 1 and 2
  const uint32_t tl = (uint32_t)(quad * 32) << 16;
  const uint32_t DH = tmem, DW = tmem + 64u, G1 = tmem + 128u + tl, G2 = tmem + 192u + tl;
  const uint32_t a0 = smem_u32(sm + TLay::A0), hh = smem_u32(sm + TLay::H), dz = smem_u32(sm + TLay::DZ);
  const uint32_t w1 = smem_u32(sm + TLay::W1), w2 = smem_u32(sm + TLay::W2), w3 = smem_u32(sm + TLay::W3);
  float gW[32];   // layer 2 (lanes of features 0-63) or 3: unit cb + k, input m & 63
#pragma unroll
  for (int k = 0; k < 32; ++k) gW[k] = 0.f;
  float gB1 = 0.f, gB2 = 0.f, gB3 = 0.f, gW4 = 0.f, gB4 = 0.f;   // column cb + lane (gB4: rows)
  double loss = 0.0;
  uint32_t p0 = 0, p1 = 0;
  bool ok = true, pending1 = false;
  // forward layer: activations into column block `lc` of H, GELU' to TMEM
  auto hidden = [&](const float* b, uint32_t gt, int lc) {
#pragma unroll 1
    for (int c0 = cb; c0 < cb + 32; c0 += 16) {
      float v[16], gr[16];
      tmem_ld16(DH + tl + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < 16; ++j) gelu_both(v[j] + b[c0 + j], v[j], gr[j]);
      tmem_st16(gt + (uint32_t)c0, gr);
      st_core8(sm + TLay::H, core_off(m, lc + c0, 16), v);
      st_core8(sm + TLay::H, core_off(m, lc + c0 + 8, 16), v + 8);
    }
    fence_before();
    fence_async_smem();
    __syncthreads();
  };
  // dz of a layer: bias gradient, three parts into DZ
  auto put_dz = [&](float (&d)[32], float& gb) {
#pragma unroll
    for (int k = 0; k < 32; k += 8) st_split8(sm + TLay::DZ, core_off(m, cb + k, 8), d + k);
    fence_before();
    fence_async_smem();
    __syncthreads();
    gb += lane_column_sum(d, lane);
  };
  // activation gradient dz W (into DH) and weight gradient [h1 | h2]^T dz
  // (into DW), the small parts first
  auto backward = [&](uint32_t w) {
    if (tid == 0) {
      fence_after();
      product(DH, k_major(dz, 8), mn_major(w, 8), 4, 0u, kIdesc | kBTrans);
      mma_commit(bar0);
      for (int s = 2; s >= 0; --s)
        product(DW, mn_major(hh, 16), mn_major(dz + 16384u * (uint32_t)s, 8), 8, s < 2 ? 1u : 0u,
                kIdesc | kATrans | kBTrans);
      mma_commit(bar1);
    }
    pending1 = true;
  };
  auto add_dw = [&](bool mine) {
    pending1 = false;
    if (!(ok = layer_wait(bar1, p1, flag))) return;
    if (mine)
#pragma unroll
      for (int c = 0; c < 32; c += 16) {
        float v[16];
        tmem_ld16(DW + tl + (uint32_t)(cb + c), v);
#pragma unroll
        for (int k = 0; k < 16; ++k) gW[c + k] += v[k];
      }
  };
  auto act_grad = [&](uint32_t gt, float (&d)[32]) {
#pragma unroll
    for (int c = 0; c < 32; c += 16) {
      float v[16], gr[16];
      tmem_ld16(DH + tl + (uint32_t)(cb + c), v);
      tmem_ld16(gt + (uint32_t)(cb + c), gr);
#pragma unroll
      for (int k = 0; k < 16; ++k) d[c + k] = v[k] * gr[k];
    }
  };
  for (long long tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
    const long long row = tile * kTile + m;
    const bool valid = row < g.n;
    if (half == 0) {
      float f[kIn] = {0.f, 0.f, 0.f, 0.f, 0.f};
      if (valid) {
#pragma unroll
        for (int j = 0; j < kIn; ++j) f[j] = g.X[row * kIn + j];
      }
      write_input(sm + TLay::A0, m, f, valid, cst);
    }
    const float yy = valid ? g.y[row] : 0.f, wt = valid ? g.wt[row] : 0.f;
    fence_before();
    fence_async_smem();
    __syncthreads();
    // ---- forward ----
    if (tid == 0) {
      fence_after();
      product(DH, k_major(a0, 2), k_major(w1, 2), 1, 0u, kIdesc);
      mma_commit(bar0);
    }
    if (!(ok = layer_wait(bar0, p0, flag))) break;
    hidden(cst + kCB1, G1, 0);
    if (tid == 0) {
      fence_after();
      product(DH, k_major(hh, 16), k_major(w2, 8), 4, 0u, kIdesc);
      mma_commit(bar0);
    }
    if (!(ok = layer_wait(bar0, p0, flag))) break;
    hidden(cst + kCB2, G2, kHid);
    if (tid == 0) {
      fence_after();
      product(DH, k_major(hh + 8u * 128u, 16), k_major(w3, 8), 4, 0u, kIdesc);
      mma_commit(bar0);
    }
    if (!(ok = layer_wait(bar0, p0, flag))) break;
    float h3[32], d[32];
#pragma unroll
    for (int c = 0; c < 32; c += 16) {
      float v[16];
      tmem_ld16(DH + tl + (uint32_t)(cb + c), v);
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        float hv;
        gelu_both(v[k] + cst[kCB3 + cb + c + k], hv, d[c + k]);   // d: GELU' for now
        h3[c + k] = bf16r(hv);
      }
    }
    // the output layer's sum runs over the 64 units in order, as in scoring:
    // the row's first thread hands it to the second
    float z = cst[kCB4];
    if (half == 0) {
#pragma unroll
      for (int k = 0; k < 32; ++k) z += h3[k] * cst[kCW4 + k];
      zp[m] = z;
    }
    __syncthreads();
    if (half == 1) {
      z = zp[m];
#pragma unroll
      for (int k = 0; k < 32; ++k) z += h3[k] * cst[kCW4 + 32 + k];
      zp[kTile + m] = z;
    }
    __syncthreads();
    z = zp[kTile + m];
    // ---- loss and output gradient ----
    float dl = 0.f;
    if (valid) {
      if (half == 0) {
        const float sp = fmaxf(z, 0.f) + log1pf(expf(-fabsf(z)));
        loss += (double)wt * (double)(sp - yy * z);
      }
      dl = wt * (1.f / (1.f + expf(-z)) - yy);
    }
    if (half == 0) gB4 += dl;
    // ---- layer 3: dz3 = dl w4 GELU'(z3) ----
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      d[k] = dl * cst[kCW4 + cb + k] * d[k];
      h3[k] *= dl;
    }
    put_dz(d, gB3);
    backward(w3);
    gW4 += lane_column_sum(h3, lane);
    // ---- layer 2: dz2 = (dz3 W3) GELU'(z2) ----
    if (!(ok = layer_wait(bar0, p0, flag))) break;
    act_grad(G2, d);
    add_dw(quad >= 2);   // h2^T dz3
    if (!ok) break;
    put_dz(d, gB2);
    backward(w2);
    // ---- layer 1: dz1 = (dz2 W2) GELU'(z1) ----
    if (!(ok = layer_wait(bar0, p0, flag))) break;
    act_grad(G1, d);
    add_dw(quad < 2);    // h1^T dz2
    if (!ok) break;
    put_dz(d, gB1);
    if (tid == 0) {
      // x^T dz1: features beyond the operand's 16 read what follows it; their
      // rows of the product are not used
      fence_after();
      for (int s = 2; s >= 0; --s)
        product(DW, mn_major(a0, 2), mn_major(dz + 16384u * (uint32_t)s, 8), 8, s < 2 ? 1u : 0u,
                kIdesc | kATrans | kBTrans);
      mma_commit(bar0);
    }
    if (!(ok = layer_wait(bar0, p0, flag))) break;
    if (quad == 0) {
#pragma unroll 1
      for (int c = 0; c < 32; c += 16) {
        float v[16];
        tmem_ld16(DW + tl + (uint32_t)(cb + c), v);
        if (lane < kIn)
#pragma unroll
          for (int k = 0; k < 16; ++k) gw1[(cb + c + k) * kIn + lane] += v[k];
      }
    }
  }
  if (!ok) {
    mbar_wait(bar0, p0 ^ 1u);
    mbar_wait(bar1, pending1 ? p1 : p1 ^ 1u);
    if (tid == 0) atomicOr(g.err, kErrGate);
  } else {
    // the CTA's gradient in parameter order (DZ's place: its products are
    // done), then one reduction into global memory
    float* gs = reinterpret_cast<float*>(sm + TLay::GRAD);
    const int base = quad >= 2 ? kGateW3 : kGateW2;
#pragma unroll
    for (int k = 0; k < 32; ++k) gs[base + (cb + k) * kHid + (m & 63)] = gW[k];
    if (tid < kHid) gs[kGateB1 + tid] = gs[kGateB2 + tid] = gs[kGateB3 + tid] = gs[kGateW4 + tid] = 0.f;
    __syncthreads();   // also: every tile's gw1
    for (int i = tid; i < kHid * kIn; i += kTrainThreads) gs[kGateW1 + i] = gw1[i];
    atomicAdd(&gs[kGateB1 + cb + lane], gB1);
    atomicAdd(&gs[kGateB2 + cb + lane], gB2);
    atomicAdd(&gs[kGateB3 + cb + lane], gB3);
    atomicAdd(&gs[kGateW4 + cb + lane], gW4);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      gB4 += __shfl_xor_sync(0xFFFFFFFFu, gB4, o);
      loss += __shfl_xor_sync(0xFFFFFFFFu, loss, o);
    }
    if (lane == 0 && half == 0) {
      atomicAdd(g.grad + kGateB4, gB4);
      atomicAdd(g.loss, loss);
    }
    constexpr uint32_t kBytes = kGateB4 * 4u;   // all but b4: a multiple of 16
    static_assert(kBytes % 16 == 0, "bulk reduction size");
    if ((reinterpret_cast<uintptr_t>(g.grad) & 15) == 0) {
      fence_async_smem();
      __syncthreads();
      if (tid == 0) {
        asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(g.grad),
                     "r"(smem_u32(gs)), "r"(kBytes)
                     : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
      }
    } else {   // a gradient buffer the bulk copy cannot address
      __syncthreads();
      for (int i = tid; i < kGateB4; i += kTrainThreads) atomicAdd(g.grad + i, gs[i]);
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  tmem_free(tmem);
}

// the gradient and the loss start at zero
__global__ void gate_zero_kernel(float* __restrict__ grad, double* __restrict__ loss) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kGateNParam) grad[i] = 0.f;
  if (i == 0) *loss = 0.0;
}

// Adam (Kingma and Ba 2015) on the trained parameters, bias-corrected
__global__ void gate_adam_kernel(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ mo,
                                 float* __restrict__ ve, int t, float lr, float b1, float b2, float eps) {
  pdl_enter();
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < kGateNTrain; i += gridDim.x * blockDim.x) {
    const float gi = G[i];
    const float mi = b1 * mo[i] + (1.f - b1) * gi;
    const float vi = b2 * ve[i] + (1.f - b2) * gi * gi;
    mo[i] = mi;
    ve[i] = vi;
    P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// raw features of every pair of the table (rows for training)
__global__ void gate_features_kernel(Model md, CompTable ct, PairTable pt, const FrameDev* __restrict__ fs,
                                     float* __restrict__ X, long long cap) {
  pdl_enter();
  const long long n = min((long long)*pt.total, cap);
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n;
       p += (long long)gridDim.x * blockDim.x) {
    float f[kIn];
    pair_features(md, ct, pt, *fs, (uint32_t)p, (int)pt.comp[p], f);
    for (int j = 0; j < kIn; ++j) X[p * kIn + j] = f[j];
  }
}

// stable compaction of the kept pairs into the gated table (a warp per
// component counts its kept pairs, takes their place and copies them), and
// the death probability (reading R2) over the pairs that remain
__global__ void gate_compact_kernel(Model md, CompTable ct, PairTable full, const uint8_t* __restrict__ keep,
                                    PairTable gated, const FrameDev* __restrict__ fs) {
  pdl_enter();
  const int T = fs->T, lane = threadIdx.x & 31, dz = md.dz;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  const size_t cf = (size_t)full.cap_pairs, cg = (size_t)gated.cap_pairs;
  for (int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < T; c += nw) {
    const uint32_t lo = min(full.ptr[c], (uint32_t)cf), hi = min(lo + full.cnt[c], (uint32_t)cf);
    unsigned kept = 0;
    for (uint32_t j = lo + lane; j < hi; j += 32) kept += keep[j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xFFFFFFFFu, kept, o);
    uint32_t out = 0;
    if (lane == 0) {
      out = kept ? atomicAdd(gated.total, kept) : 0u;
      gated.cnt[c] = kept;
      gated.ptr[c] = out;
    }
    out = __shfl_sync(0xFFFFFFFFu, out, 0);
    float lm = -INFINITY, ls = 0.f;
    bool any = false;
    for (uint32_t j0 = lo; j0 < hi; j0 += 32) {
      const uint32_t j = j0 + lane;
      const bool k = j < hi && keep[j];
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, k);
      const uint32_t q = out + __popc(bal & ((1u << lane) - 1u));
      if (k && q < cg) {
        const float lc = full.logC[j];
        gated.meas[q] = full.meas[j];
        gated.comp[q] = (uint32_t)c;
        gated.logC[q] = lc;
        gated.q[q] = full.q[j];
        for (int a = 0; a < dz; ++a) gated.e[a * cg + q] = full.e[a * cf + j];
        any = true;
        if (!md.kappa_zero) lse_push(lm, ls, lc - md.log_kappa);
      }
      out += __popc(bal);
    }
    lse_warp(lm, ls);
    const bool any_w = __any_sync(0xFFFFFFFFu, any);
    if (lane == 0) death_prob(md, ct.logp[c], ct.log1mp[c], lm, ls, any_w, gated.dprob[c], gated.dthr[c]);
  }
}

// Which pairs of the last update's table the retained hypotheses use (the
// gate's training labels), and which retained hypotheses use a pair whose
// logit is below the threshold.  One block per retained hypothesis: its new
// tracks are its parent's surviving slots in slot order, so walking both
// lists by label recovers each track's predicted component; theta then names
// the pair (component, detection), found by binary search in the component's
// slice (detections ascend within it).
__global__ void gate_usage_kernel(HypTable par, HypTable out, CompTable A, CompTable B,
                                  const long long* __restrict__ surv, int H_new, int h_up, int M,
                                  PairTable pt, const FrameDev* __restrict__ fs, const float* __restrict__ logit,
                                  float thr, uint8_t* __restrict__ used, uint8_t* __restrict__ hflag, int capT) {
  pdl_enter();
  extern __shared__ int kc[];
  const int n_comp = fs->n_comp, nb = fs->nb;
  for (int j = blockIdx.x; j < H_new; j += gridDim.x) {
    if (threadIdx.x == 0) {
      const int p = (int)(surv[j] / h_up);
      const uint32_t plo = par.ptr[p];
      const int Tp = (int)(par.ptr[p + 1] - plo), Ts = Tp + nb;
      const uint32_t lo = out.ptr[j], hi = out.ptr[j + 1];
      int s = 0;
      for (uint32_t e = lo; e < hi && (int)(e - lo) < capT; ++e) {
        const uint32_t ca = out.comp[e];
        const uint32_t lk = A.lk[ca], lb = A.lb[ca];
        int c = -1;
        while (s < Ts) {
          const int cs = s < Tp ? (int)par.comp[plo + s] : n_comp + (s - Tp);
          ++s;
          if (B.lk[cs] == lk && B.lb[cs] == lb) {
            c = cs;
            break;
          }
        }
        kc[e - lo] = c;
      }
    }
    __syncthreads();
    const int nt = min((int)(out.ptr[j + 1] - out.ptr[j]), capT);
    int bad = 0;
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
      const int t = out.theta[(size_t)j * M + i];
      if (t == 0 || t > nt) continue;
      const int c = kc[t - 1];
      if (c < 0) continue;
      uint32_t lo = pt.ptr[c], hi = lo + pt.cnt[c];
      const uint32_t end = hi;
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (pt.meas[mid] < (uint32_t)i) lo = mid + 1;
        else hi = mid;
      }
      if (lo < end && pt.meas[lo] == (uint32_t)i) {
        if (used) used[lo] = 1;
        if (logit && logit[lo] < thr) bad = 1;
      }
    }
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0 && hflag) hflag[j] = (uint8_t)bad;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int gate_forward_smem() { return FLay::TOTAL; }
int gate_train_smem() { return TLay::TOTAL; }

static bool gate_attrs_set = false;
static void gate_attrs() {
  if (gate_attrs_set) return;
  cudaFuncSetAttribute(gate_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TLay::TOTAL);
  cudaFuncSetAttribute(gate_forward_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FLay::TOTAL);
  cudaFuncSetAttribute(gate_forward_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FLay::TOTAL);
  gate_attrs_set = true;
}

void launch_gate_forward_rows(const float* P, const float* X, long long n, float* logit, unsigned* err, int grid,
                              cudaStream_t s) {
  gate_attrs();
  GateFwdArgs g{};
  g.P = P;
  g.X = X;
  g.n = n;
  g.logit = logit;
  g.err = err;
  const WaitTest wt = wait_test();
  g.wait_limit = wt.mode == kWaitTestGate ? wt.limit : kGateWaitLimit;
  g.skip_first_mma = wt.mode == kWaitTestGate ? 1 : 0;
  launch_k(gate_forward_kernel<false>, grid, kTile * kFwdGroups, FLay::TOTAL, s, g);
}

void launch_gate_forward_table(const float* P, float thr, const Model& md, const CompTable& ct,
                               const PairTable& full, const FrameDev* fs, float* logit, uint8_t* keep,
                               unsigned* err, int grid, cudaStream_t s) {
  gate_attrs();
  GateFwdArgs g{};
  g.P = P;
  g.md = md;
  g.ct = ct;
  g.pt = full;
  g.fs = fs;
  g.thr = thr;
  g.keep = keep;
  g.logit = logit;
  g.err = err;
  const WaitTest wt = wait_test();
  g.wait_limit = wt.mode == kWaitTestGate ? wt.limit : kGateWaitLimit;
  g.skip_first_mma = wt.mode == kWaitTestGate ? 1 : 0;
  launch_k(gate_forward_kernel<true>, grid, kTile * kFwdGroups, FLay::TOTAL, s, g);
}

void launch_gate_train(const float* P, const float* X, const float* y, const float* wt, long long n,
                       float* grad, double* loss, unsigned* err, int grid, cudaStream_t s) {
  gate_attrs();
  GateTrainArgs g{P, X, y, wt, n, grad, loss, err};
  launch_k(gate_train_kernel, grid, kTrainThreads, TLay::TOTAL, s, g);
}

void launch_gate_zero(float* grad, double* loss, cudaStream_t s) {
  launch_k(gate_zero_kernel, (kGateNParam + 255) / 256, 256, 0, s, grad, loss);
}

void launch_gate_adam(float* P, const float* G, float* m, float* v, int t, float lr, float b1, float b2,
                      float eps, cudaStream_t s) {
  launch_k(gate_adam_kernel, (kGateNTrain + 255) / 256, 256, 0, s, P, G, m, v, t, lr, b1, b2, eps);
}

void launch_gate_features(const Model& md, const CompTable& ct, const PairTable& pt, const FrameDev* fs,
                          float* X, long long cap, int grid, cudaStream_t s) {
  launch_k(gate_features_kernel, grid, 256, 0, s, md, ct, pt, fs, X, cap);
}

void launch_gate_compact(const Model& md, const CompTable& ct, const PairTable& full, const uint8_t* keep,
                         const PairTable& gated, const FrameDev* fs, int grid, cudaStream_t s) {
  launch_k(gate_compact_kernel, grid, 256, 0, s, md, ct, full, keep, gated, fs);
}

void launch_gate_usage(const HypTable& par, const HypTable& out, const CompTable& A, const CompTable& B,
                       const long long* surv, int H_new, int h_up, int M, const PairTable& pt, const FrameDev* fs,
                       const float* logit, float thr, uint8_t* used, uint8_t* hflag, int capT, int grid,
                       cudaStream_t s) {
  const size_t smem = (size_t)capT * sizeof(int);
  if (smem > 48 * 1024) cudaFuncSetAttribute(gate_usage_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  launch_k(gate_usage_kernel, grid, 128, smem, s, par, out, A, B, surv, H_new, h_up, M, pt, fs, logit, thr, used,
           hflag, capT);
}

}  // namespace glmb
