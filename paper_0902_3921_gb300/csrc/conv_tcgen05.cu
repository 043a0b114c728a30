// conv_tcgen05.cu -- periodic 3x3 convolution of the learned surrogate as an
// implicit GEMM on the tcgen05 tensor cores.
//
// One tile is 128 consecutive pixels of one image row (the MMA's M = 128).  A
// CTA walks runs of rows down a 128-pixel column strip, and each input row is
// used once, when it arrives: it contributes to the output rows above, at and
// below it, so its MMAs have N = 3 Cout, the three weight rows ky = 2, 1, 0 side
// by side, and accumulate into three neighbouring accumulators of a ring of
// eight in tensor memory.  Per row and shift dx, Cin / 16 MMAs of K = 16 read
// the staged row (130 pixels wide, periodic halo of one) as the A operand
// shifted by dx pixels.  The MMAs of one shape read their operands from shared
// memory at 128 bytes a clock, 4 KiB of A each: one MMA with N = 96 instead of
// three with N = 32 reads A a third as often, 368 instead of 720 shared-memory
// wavefronts per tile of a 32 -> 32 layer, which had bound the layer (123 us at
// 2048^2: 80 us of operand reads beside 79 us of HBM traffic); now 104 us.
//
// Shared-memory operand layout (K-major, no swizzle): a "core matrix" is 8
// rows x 16 bytes stored as 128 contiguous bytes.  Staged rows are kept as
// one plane per 8-channel chunk, [chunk][slot][pixel][8 channels], so 8
// consecutive pixels of one chunk form a core matrix, consecutive 8-pixel
// groups are 128 bytes apart (the stride-dimension offset) and the two chunks
// of one K = 16 step are one plane apart (the leading-dimension offset).  The
// weights use the same form, [dx, chunk][ky block, output channel][8].
//
// Roles per CTA (persistent): a loader warp stages rows with bulk copies (one
// per chunk plane, three at the image's edges), an MMA warp issues the MMAs
// (one elected lane, warp-uniform operands) into FP32 accumulators in tensor
// memory, four epilogue warps read them back with tcgen05.ld; they meet only on
// mbarriers, and every wait is bounded.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <mutex>

#include "conv_tc.cuh"

namespace {

typedef __nv_bfloat16 bf16;
using hlbm::conv_act_index;
using hlbm::CONV_LINEAR_F32;
using hlbm::CONV_MASK;
using hlbm::CONV_PREDICT;
using hlbm::CONV_RELU;

constexpr int TM = 128;        // pixels per tile (MMA M)
constexpr int RW = TM + 2;     // staged pixels per row
constexpr int EG = 2;          // epilogue groups of four warps (32 accumulator lanes each), tiles g % EG
constexpr int WARP_MMA = 4 * EG, WARP_LOAD = WARP_MMA + 1, NTHREADS = 32 * (WARP_LOAD + 1);

__device__ int g_conv_tc_err = 0;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// shared-memory matrix descriptor: start address, leading- and stride-
// dimension byte offsets (all >> 4), descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t instr_desc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// The lane that issues (1) and the others (0), elected once per staged row.
__device__ __forceinline__ uint32_t elect_lane() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(e));
  return e;
}

// Issued by the whole warp in uniform control flow (so the operands can stay
// warp-uniform), by the lane whose `e` is set.
__device__ __forceinline__ void mma_bf16_ss(uint32_t e, uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 e, %5, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(e)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t e, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\tsetp.ne.b32 e, %1, 0;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(bar), "r"(e)
      : "memory");
}

__device__ __forceinline__ uint64_t globaltimer();

__device__ __forceinline__ bool mbar_test(uint32_t addr, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(addr), "r"(parity)
      : "memory");
  return done != 0;
}

// Waits for a phase; bounded: gives up after half a second of global time, or
// once another role has given up.  The clock and the flag are looked at only
// after a first test has failed.
__device__ __forceinline__ bool mbar_poll(uint32_t addr, uint32_t parity, const volatile int *abort_flag) {
  if (mbar_test(addr, parity)) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
#pragma unroll 1
    for (int k = 0; k < 64; ++k)
      if (mbar_test(addr, parity)) return true;
    if (*abort_flag || globaltimer() - t0 > 500000000ull) return false;
  }
}

// the same with the suspending test (the epilogue warps)
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity, const volatile int *abort_flag) {
  if (mbar_test(addr, parity)) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if ((abort_flag && *abort_flag) || globaltimer() - t0 > 500000000ull) return false;
  }
}

// mbar_wait for the end of a whole run of MMAs: bounded by 20 times as long
// (the issuer, whose every wait is bounded, ends or gives up well before)
__device__ __forceinline__ bool mbar_wait_long(uint32_t addr, uint32_t parity, const volatile int *abort_flag) {
  for (int k = 0; k < 20; ++k) {
    if (mbar_wait(addr, parity, abort_flag)) return true;
    if (*abort_flag) return false;
  }
  return false;
}

// 32 consecutive FP32 columns of this warp's 32 lanes (one pixel per thread)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[32]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
#pragma unroll
  for (int j = 16; j < 32; ++j) v[j] = 0.f;
}

__device__ __forceinline__ void tmem_zero16(uint32_t taddr) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
      "%1};" ::"r"(taddr),
      "r"(0)
      : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&h);
}

template <int CIN, int NM>
struct TcGeom {
  static constexpr int CH = CIN / 8;       // 8-channel chunks per pixel
  static constexpr int SLOTS = 8;          // staged input rows
  static constexpr int NACC = 8;           // accumulators (output rows) in tensor memory
  static constexpr int TMEM_COLS = NACC * NM;  // 256 or 128
  static constexpr int CTAS_TMEM = 512 / TMEM_COLS;
  // +32 bytes: the chunk planes start in different shared-memory bank groups
  static constexpr int PLANE_A = SLOTS * RW * 16 + 32;
  static constexpr int ABYTES = CH * PLANE_A;
  static constexpr int KCH = 3 * CH;       // weight chunk planes (dx, chunk)
  static constexpr int PLANE_B = 3 * NM * 16;  // ky = 2, 1, 0 of one plane
  static constexpr int BBYTES = KCH * PLANE_B;
  static constexpr int NBAR = 2 * NACC + 2 * SLOTS;
  static constexpr int USED = ABYTES + BBYTES + NM * 4 + 8 * NBAR + 16;
  // at least so much that no more CTAs share an SM than its tensor memory holds
  static constexpr int LEAST = 233472 / (CTAS_TMEM + 1) + 16;
  static constexpr int SMEM = USED > LEAST ? USED : LEAST;
  static constexpr uint32_t ROW_BYTES = CH * RW * 16;  // one staged row
  static_assert(PLANE_A % 16 == 0 && ABYTES % 16 == 0 && BBYTES % 16 == 0, "16-byte planes");
};

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_arrive(uint32_t addr) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}\n" ::"r"(addr)
               : "memory");
}

// Work item = a run of R tiles stacked in y (one 128-pixel column strip, rows
// y0 .. y0 + R - 1 of one image); CTAs take items round-robin and all roles
// walk the same sequence, numbering tiles g = 0, 1, ... (accumulator g % NACC)
// and staged rows q = 0, 1, ... per CTA (ring slot q % SLOTS; an item stages
// its rows y0 - 1 .. y0 + R).  The strips' x origins are multiples of 128 except
// the last one's, which ends at the image's edge and rewrites no pixel of the
// strip before it.
//
// Loader (last warp): requests each row's 130 staged pixels (periodic halo of one)
// by bulk copies once the slot's previous row has been released on sfree[slot];
// the copies complete loaded[slot].
// MMA issuer (one elected lane issues): per staged row j of an item
// (tiles j - 2, j - 1 and j use it) waits for the row and, for the new tile j,
// for its accumulator (aempty); the first MMA initialises the new tile's
// accumulator separately; commits sfree[slot] and, tile j - 2 being complete,
// full[its accumulator] (a commit arrives once all MMAs issued so far are
// complete).
// Epilogue (EG groups of four warps; group g % EG takes tile g, warp w of a group
// reads tensor-memory lanes 32 w .. 32 w + 31; with one group its latency bound
// the backward pass): wait full[g % NACC], load the accumulator, release it on aempty[g % NACC] (four
// arrivals), then bias/ReLU/mask, convert and store.
// Every barrier is refilled only by the side that waits on it, so a parity
// wait can never fall two phases behind; every wait is bounded.
template <int CIN, int NM, int COUTG, int EPI>
__global__ void __launch_bounds__(NTHREADS, 2)
    conv_tc_kernel(const bf16 *__restrict__ in, const bf16 *__restrict__ w, int ks,
                   const float *__restrict__ bias, const bf16 *__restrict__ mask, int N, int H,
                   int W, int R, bf16 *__restrict__ out_bf, float *out_f, const float *x0_,
                   const float *__restrict__ out_std) {
  using G = TcGeom<CIN, NM>;
  constexpr int S = G::SLOTS, NACC = G::NACC, CH = G::CH, COCH = COUTG / 8;
  static_assert(CIN % 16 == 0 && (NM == 16 || NM == 32) && COUTG <= NM && COUTG % 8 == 0, "shape");
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char *sB = smem + G::ABYTES;
  float *sbias = reinterpret_cast<float *>(sB + G::BBYTES);
  uint64_t *bars = reinterpret_cast<uint64_t *>(sbias + NM);  // full, aempty, loaded, sfree
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + G::NBAR);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles_x = (W + TM - 1) / TM, runs_y = (H + R - 1) / R;
  const long long nitems = (long long)N * runs_y * tiles_x;

  // weights -> [dx, chunk][ky = 2, 1, 0][co][8]; rows co >= COUTG are zero
  for (int k = tid; k < 3 * G::KCH * NM; k += NTHREADS) {
    const int co = k / (3 * G::KCH), kc = k - co * (3 * G::KCH);  // kc = (ky 3 + dx) CH + chunk
    const int ky = kc / G::KCH, pl = kc - ky * G::KCH;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (co < COUTG) v = __ldg(reinterpret_cast<const uint4 *>(w + (size_t)co * ks + kc * 8));
    *reinterpret_cast<uint4 *>(sB + pl * G::PLANE_B + ((2 - ky) * NM + co) * 16) = v;
  }
  if (tid < NM) sbias[tid] = (EPI != CONV_MASK && tid < COUTG) ? bias[tid] : 0.f;
  const uint32_t full0 = smem_u32(bars), aempty0 = full0 + 8 * NACC, loaded0 = aempty0 + 8 * NACC,
                 sfree0 = loaded0 + 8 * S;
  if (tid == 0) {
    for (int k = 0; k < NACC; ++k) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full0 + 8 * k), "r"(1) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(aempty0 + 8 * k), "r"(4) : "memory");
    }
    for (int k = 0; k < S; ++k) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(loaded0 + 8 * k), "r"(1) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sfree0 + 8 * k), "r"(1) : "memory");
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tslot)),
                 "r"(G::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const uint32_t abase = smem_u32(smem), bbase = smem_u32(sB);
  // The waits' loops end lane by lane, and the stores of a partial strip are some
  // lanes' only; tcgen05.ld and elect.sync need the whole warp.  So a role goes on
  // from a wait through a vote, which brings the lanes together and makes them give
  // up together.  The loader votes once its copies are issued: before them, the
  // vote's latency is the row's (training step 1515 -> 1545 us, 16 channels' forward
  // 170 -> 178).
  auto poll = [&](uint32_t bar, uint32_t parity) { return mbar_poll(bar, parity, abort_flag); };
  auto together = [](bool got) { return __all_sync(0xffffffffu, got) != 0; };

  if (warp == WARP_LOAD) {
    // ---------------- loader ----------------
    // lane c < CH copies chunk plane c of a row
    long long q = 0;
    bool ok = true;
    auto bulk = [&](uint32_t dst, const bf16 *src, uint32_t bytes, uint32_t bar) {
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
          "l"(src), "r"(bytes), "r"(bar)
          : "memory");
    };
    for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const int xt = (int)(item % tiles_x);
      const long long it = item / tiles_x;
      const int y0 = (int)(it % runs_y) * R;
      const long long row0 = (it / runs_y) * (long long)H;  // n H
      const int rows = min(R, H - y0);
      const int x0 = min(xt * TM, W - TM);
      const int first = x0 == 0 ? 1 : 0, last = x0 + TM == W ? RW - 2 : RW - 1;  // pixels of the main copy
      for (int r = 0; r < rows + 2; ++r, ++q) {
        const int slot = (int)(q % S);
        const bool got = q < S || poll(sfree0 + 8 * slot, (uint32_t)(q / S - 1) & 1u);
        int gy = y0 - 1 + r;
        gy = gy < 0 ? gy + H : (gy >= H ? gy - H : gy);
        const uint32_t bar = loaded0 + 8 * slot;
        if (lane == 0 && got)
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(G::ROW_BYTES)
                       : "memory");
        __syncwarp();
        if (lane < CH && got) {
          const bf16 *plane = in + conv_act_index(row0 + gy, lane, 0, W, CH);
          const uint32_t dst = abase + lane * G::PLANE_A + slot * RW * 16;
          bulk(dst + first * 16, plane + (long long)(x0 - 1 + first) * 8, (last - first + 1) * 16, bar);
          if (first) bulk(dst, plane + (long long)(W - 1) * 8, 16, bar);
          if (last == RW - 2) bulk(dst + (RW - 1) * 16, plane, 16, bar);
        }
        if (!(ok = together(got))) break;
      }
    }
    if (!ok) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicExch(&g_conv_tc_err, 1);
      }
      // no copy may land after the CTA has left (row q: lanes that did not give up
      // have issued theirs)
      for (long long k = max(q - S, 0ll); k <= q; ++k)
        mbar_wait(loaded0 + 8 * (uint32_t)(k % S), (uint32_t)(k / S) & 1u, nullptr);
    }
  } else if (warp == WARP_MMA) {
    // ---------------- MMA issuer (one elected lane issues) ----------------
    // descriptors of slot 0 / weight plane 0; start addresses advance in
    // 16-byte units and stay below 2^18 bytes, so they never carry out of
    // their 14-bit field
    const uint64_t a_desc0 = smem_desc(abase, G::PLANE_A, 128);
    const uint64_t b_desc0 = smem_desc(bbase, G::PLANE_B, 128);
    // The issue of a row is a serial chain in one warp, and at two rows in
    // flight per SM it bounds the kernel: descriptors are one addition each,
    // instruction descriptors immediates, and the ring's two wrapped positions
    // have paths of their own.
    constexpr uint32_t ID1 = instr_desc(TM, NM), ID2 = instr_desc(TM, 2 * NM), ID3 = instr_desc(TM, 3 * NM);
    constexpr int STEPS = 3 * CIN / 16;  // (dx, K step)
    uint32_t q = 0, gbase = 0;           // staged row; first tile of the item
    bool ok = true;
    for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const long long it = item / tiles_x;
      const int y0 = (int)(it % runs_y) * R;
      const int rows = min(R, H - y0);
      for (int j = 0; j < rows + 2; ++j, ++q) {
        const uint32_t slot = q % S;
        const bool fresh = j < rows;  // tile j starts here
        bool got = !(fresh && gbase + j >= NACC) || poll(aempty0 + 8 * ((gbase + j) % NACC), ((gbase + j) / NACC - 1) & 1u);
        got = got && poll(loaded0 + 8 * slot, (q / S) & 1u);
        ok = together(got);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t e = elect_lane();
        const uint64_t da0 = a_desc0 + (uint64_t)(slot * RW);
        auto da = [&](int step) {
          return da0 + (uint64_t)((2 * (step % (CIN / 16)) * G::PLANE_A) / 16 + step / (CIN / 16));
        };
        // B operand of tiles j - 2 + blk on: ky = 2, 1, 0 side by side
        auto db = [&](int step, int blk) { return b_desc0 + (uint64_t)((2 * step * G::PLANE_B) / 16 + blk * NM); };
        const uint32_t sl = (gbase + j - 2) % NACC;  // accumulator of tile j - 2
        const uint32_t tm = tmem + sl * NM;
        if (j >= 2 && fresh && sl < NACC - 2) {
          mma_bf16_ss(e, tm, da(0), db(0, 0), ID2, 1u);
          mma_bf16_ss(e, tm + 2 * NM, da(0), db(0, 2), ID1, 0u);
#pragma unroll
          for (int step = 1; step < STEPS; ++step) mma_bf16_ss(e, tm, da(step), db(step, 0), ID3, 1u);
        } else if (j >= 2 && fresh && sl == NACC - 2) {
#pragma unroll
          for (int step = 0; step < STEPS; ++step) {
            mma_bf16_ss(e, tm, da(step), db(step, 0), ID2, 1u);
            mma_bf16_ss(e, tmem, da(step), db(step, 2), ID1, step > 0);
          }
        } else if (j >= 2 && fresh) {
          mma_bf16_ss(e, tm, da(0), db(0, 0), ID1, 1u);
          mma_bf16_ss(e, tmem, da(0), db(0, 1), ID1, 1u);
          mma_bf16_ss(e, tmem + NM, da(0), db(0, 2), ID1, 0u);
#pragma unroll
          for (int step = 1; step < STEPS; ++step) {
            mma_bf16_ss(e, tm, da(step), db(step, 0), ID1, 1u);
            mma_bf16_ss(e, tmem, da(step), db(step, 1), ID2, 1u);
          }
        } else {
          // the first and last rows of an item: tile by tile
          const int lo = max(0, j - 2), hi = min(rows - 1, j);
          for (int t = lo; t <= hi; ++t) {
            const uint32_t acc = tmem + ((gbase + t) % NACC) * NM;
#pragma unroll
            for (int step = 0; step < STEPS; ++step)
              mma_bf16_ss(e, acc, da(step), db(step, 0) + (uint64_t)((t - (j - 2)) * NM), ID1, step > 0 || t != j);
          }
        }
        mma_commit(e, sfree0 + 8 * slot);
        if (j >= 2) mma_commit(e, full0 + 8 * sl);
      }
      gbase += rows;
    }
    if (!ok) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicExch(&g_conv_tc_err, 1);
      }
      if (q > 0) mbar_wait(sfree0 + 8 * ((q - 1) % S), ((q - 1) / S) & 1u, nullptr);
    }
  } else {
    // ---------------- epilogue ----------------
    int g = 0;
    bool ok = true;
    for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const int xt = (int)(item % tiles_x);
      const long long q = item / tiles_x;
      const int y0 = (int)(q % runs_y) * R;
      const long long row0 = (q / runs_y) * (long long)H;
      const int rows = min(R, H - y0);
      const int quarter = warp & 3;  // the accumulator lanes this warp may read
      const int x = min(xt * TM, W - TM) + quarter * 32 + lane;
      const bool mine = x >= xt * TM;
      for (int t = 0; t < rows; ++t, ++g) {
        if (g % EG != warp >> 2) continue;
        const uint32_t acc = (uint32_t)(g % NACC);
        if (!(ok = together(mbar_wait(full0 + 8 * acc, (uint32_t)(g / NACC) & 1u, abort_flag)))) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float v[32];
        const uint32_t taddr = tmem + acc * NM + ((uint32_t)(quarter * 32) << 16);
        if constexpr (NM == 32) tmem_ld32(taddr, v);
        else tmem_ld16(taddr, v);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(aempty0 + 8 * acc);
        if (!mine) continue;  // the lanes meet again at the next tile's vote
        const long long row = row0 + y0 + t;
        if constexpr (EPI == CONV_LINEAR_F32) {
          float4 *o = reinterpret_cast<float4 *>(out_f + (row * W + x) * COUTG);
#pragma unroll
          for (int c = 0; c < COUTG / 4; ++c)
            o[c] = make_float4(v[4 * c] + sbias[4 * c], v[4 * c + 1] + sbias[4 * c + 1],
                               v[4 * c + 2] + sbias[4 * c + 2], v[4 * c + 3] + sbias[4 * c + 3]);
        } else if constexpr (EPI == CONV_PREDICT) {
          const float4 b = *reinterpret_cast<const float4 *>(x0_ + (row * W + x) * 4);
          *reinterpret_cast<float4 *>(out_f + (row * W + x) * 4) =
              make_float4(b.x + (v[0] + sbias[0]) * __ldg(out_std), b.y + (v[1] + sbias[1]) * __ldg(out_std + 1),
                          b.z + (v[2] + sbias[2]) * __ldg(out_std + 2), b.w + (v[3] + sbias[3]) * __ldg(out_std + 3));
        } else {
#pragma unroll
          for (int c = 0; c < COCH; ++c) {
            const long long o = conv_act_index(row, c, x, W, COCH);
            float e[8];
            if constexpr (EPI == CONV_RELU) {
#pragma unroll
              for (int j = 0; j < 8; ++j) e[j] = fmaxf(v[8 * c + j] + sbias[8 * c + j], 0.f);
            } else {
              const uint4 mk = __ldg(reinterpret_cast<const uint4 *>(mask + o));
              const bf16 *mb = reinterpret_cast<const bf16 *>(&mk);
#pragma unroll
              for (int j = 0; j < 8; ++j) e[j] = __bfloat162float(mb[j]) > 0.f ? v[8 * c + j] : 0.f;
            }
            *reinterpret_cast<uint4 *>(out_bf + o) =
                make_uint4(pack_bf16(e[0], e[1]), pack_bf16(e[2], e[3]), pack_bf16(e[4], e[5]),
                           pack_bf16(e[6], e[7]));
          }
        }
      }
    }
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicExch(&g_conv_tc_err, 1);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(G::TMEM_COLS)
                 : "memory");
  }
}

// Rows of a run: the number of runs per strip that minimises waves of resident
// CTAs times the rows a run stages (R + 2, and about one row's latency).
int run_rows(int H, long long strips, long long ctas) {
  int R = H;
  long long best = -1;
  for (int runs = 1; runs <= H; ++runs) {
    const int r = (H + runs - 1) / runs;
    const long long waves = (strips * ((H + r - 1) / r) + ctas - 1) / ctas, cost = waves * (r + 3);
    if (best < 0 || cost < best) {
      best = cost;
      R = r;
    }
    if (strips * runs > 8 * ctas) break;
  }
  return R;
}

template <int CIN, int NM, int COUTG, int EPI>
cudaError_t launch(const void *in, const void *w, int ks, const float *bias, const void *mask,
                   int N, int H, int W, void *out_bf, float *out_f, cudaStream_t s, const float *x0 = nullptr,
                   const float *out_std = nullptr) {
  using G = TcGeom<CIN, NM>;
  auto *kern = conv_tc_kernel<CIN, NM, COUTG, EPI>;
  static int ctas_per_sm = -1;
  static int sms = 0;
  static std::once_flag once;
  static cudaError_t init_err = cudaSuccess;
  std::call_once(once, [&] {
    init_err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
    if (init_err == cudaSuccess)
      init_err = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                      (int)cudaSharedmemCarveoutMaxShared);
    int dev = 0;
    if (init_err == cudaSuccess) init_err = cudaGetDevice(&dev);
    if (init_err == cudaSuccess)
      init_err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // resident CTAs per SM from the shared memory (plus the driver's
    // reservation per CTA), the threads, and the 512 tensor-memory columns
    int smem_sm = 0, reserved = 0;
    if (init_err == cudaSuccess)
      init_err = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (init_err == cudaSuccess)
      init_err = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    cudaFuncAttributes fa{};
    if (init_err == cudaSuccess) init_err = cudaFuncGetAttributes(&fa, kern);
    const int warp_regs = (fa.numRegs * 32 + 255) / 256 * 256;  // allocated per warp
    const int by_regs = 65536 / std::max(1, warp_regs * (NTHREADS / 32));
    ctas_per_sm = std::min({smem_sm / (G::SMEM + reserved), 2048 / NTHREADS, G::CTAS_TMEM, by_regs});
    if (std::getenv("HLBM_CONV_VERBOSE")) {
      int api = -1;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&api, kern, NTHREADS, G::SMEM);
      std::fprintf(stderr, "hlbm conv_tc occupancy: %d CTAs/SM by resources, %d by the occupancy API\n",
                   ctas_per_sm, api);
    }
  });
  if (init_err != cudaSuccess) return init_err;
  if (ctas_per_sm < 1) return cudaErrorInvalidConfiguration;
  const long long ctas = (long long)ctas_per_sm * sms;
  const int tiles_x = (W + TM - 1) / TM;
  const long long strips = (long long)N * tiles_x;
  const int R = run_rows(H, strips, ctas);
  const long long nitems = strips * ((H + R - 1) / R);
  const long long grid = std::min(nitems, ctas);
  if (std::getenv("HLBM_CONV_VERBOSE"))
    std::fprintf(stderr,
                 "hlbm conv_tc cin=%d n=%d epi=%d %dx%dx%d: %d CTAs/SM x %d SMs, smem %d B, "
                 "runs of %d tiles, grid %lld\n",
                 CIN, NM, EPI, N, H, W, ctas_per_sm, sms, G::SMEM, R, grid);
  kern<<<(unsigned)grid, NTHREADS, G::SMEM, s>>>(
      static_cast<const bf16 *>(in), static_cast<const bf16 *>(w), ks, bias,
      static_cast<const bf16 *>(mask), N, H, W, R, static_cast<bf16 *>(out_bf), out_f, x0, out_std);
  return cudaGetLastError();
}

// ---- weight and bias gradients ------------------------------------------------------
// dW[co][ky, dx][ci] = sum over pixels of dz[y][x][co] in[y + ky - 1][x + dx - 1][ci], the
// reduction K of the MMAs running over the 128 pixels of a row.  Both operands
// are read MN-major: 8 channels of a pixel are 16 contiguous bytes, 8 pixels a
// 128-byte core matrix, so the row-chunk planes serve as they are staged.  M =
// 128 holds the three dx (three copies of the staged input row, each shifted by
// one pixel at the copy) of Cin channels and a plane of ones, whose row sums dz
// for the bias; N = 3 Cout holds the three dz rows that an input row meets, as
// in the forward kernel (ky = 2, 1, 0).  The rows of a CTA accumulate in turn
// into four accumulators, read and added once at the end (four short chains
// round less than one long one: the tensor cores truncate).  Per staged row 8
// MMAs (K = 16 pixels);
// the mma.sync kernel, which stages 8 x 16 tiles without overlap and takes 592
// MMAs per 128 pixels, stays for rows under 128 pixels and for small images.
// 8 x 512^2, 32 -> 32 channels: 265 -> 113 us a layer; distance from the FP32 SIMT sums
// 7.2e-6 (mma.sync) -> 3.6e-6.
template <int CINP, int DZS>
struct WgGeom {
  static constexpr int XCH = CINP / 8, DCH = DZS / 8;  // chunk planes of an input pixel, of a dz pixel
  static constexpr int SX = 4, SD = 8;                 // staged input and dz rows
  static constexpr int P = TM * 16 + 16;               // bytes of a plane; + 16: other banks
  static constexpr int XS = (3 * XCH + 1) * P, DS = DCH * P;  // bytes of a slot
  static constexpr int ABYTES = SX * XS, DBYTES = SD * DS;
  static constexpr int NBAR = 2 * SX + 2 * SD + 1;
  static constexpr int TMEM_COLS = 16 * DZS;  // 12 Cout used
  static constexpr int SMEM = ABYTES + DBYTES + 8 * NBAR + 16;
  static constexpr uint32_t XROW = 3 * XCH * TM * 16, DROW = DCH * TM * 16;  // bytes copied per row
  // the 16 plane strides that an A operand spans stay inside the allocation
  static_assert((SX - 1) * XS + 16 * P <= ABYTES + DBYTES, "operand reads in bounds");
};
constexpr int WG_THREADS = 192;   // epilogue warps 0-3, MMA warp 4, loader warp 5
constexpr int WG_SETS = 4;        // accumulators of three blocks of Cout FP32 columns
constexpr uint32_t MN_MAJOR = (1u << 15) | (1u << 16);  // both operands

template <int CINP, int COUTP, int DZS>
__global__ void __launch_bounds__(WG_THREADS, 1)
    wgrad_tc_kernel(const bf16 *__restrict__ x, const bf16 *__restrict__ dz, int N, int H, int W, int R,
                    float *__restrict__ partial) {
  using G = WgGeom<CINP, DZS>;
  constexpr int SX = G::SX, SD = G::SD, NB = DZS;
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + G::ABYTES + G::DBYTES);
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + G::NBAR);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tiles_x = (W + TM - 1) / TM, runs_y = (H + R - 1) / R;
  const long long nitems = (long long)N * runs_y * tiles_x;
  // the plane of ones behind each slot's input planes; everything else starts
  // as zeros (the operand reads planes past it, whose rows of D are not used)
  for (int k = tid; k < (G::ABYTES + G::DBYTES) / 16; k += WG_THREADS) {
    const int r = k * 16 % G::XS;
    const bool one = k * 16 < G::ABYTES && r >= 3 * G::XCH * G::P && r < 3 * G::XCH * G::P + TM * 16;
    const uint32_t v = one ? 0x3F803F80u : 0u;
    reinterpret_cast<uint4 *>(smem)[k] = make_uint4(v, v, v, v);
  }
  const uint32_t xload0 = smem_u32(bars), xfree0 = xload0 + 8 * SX, dload0 = xfree0 + 8 * SX, dfree0 = dload0 + 8 * SD,
                 done = dfree0 + 8 * SD;
  if (tid == 0) {
    for (int k = 0; k < G::NBAR; ++k)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(xload0 + 8 * k) : "memory");
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(G::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const uint32_t xbase = smem_u32(smem), dbase = xbase + G::ABYTES;
  if (warp < 4) {  // the accumulators start at zero
    for (int c = 0; c < WG_SETS * 3 * NB; c += 16) tmem_zero16(tmem + c + ((uint32_t)(warp * 32) << 16));
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  auto poll = [&](uint32_t bar, uint32_t parity) { return mbar_poll(bar, parity, abort_flag); };
  auto together = [](bool got) { return __all_sync(0xffffffffu, got) != 0; };  // as above
  auto give_up = [&]() {
    if (lane == 0) {
      *abort_flag = 1;
      atomicExch(&g_conv_tc_err, 1);
    }
  };

  if (warp == 5) {
    // ---------------- loader: lane (dx, chunk) copies one plane of an input row ----------------
    uint32_t q = 0, d = 0;  // staged input rows, staged dz rows
    bool ok = true;
    auto expect = [&](bool got, uint32_t bar, uint32_t bytes) {
      if (lane == 0 && got)
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
      __syncwarp();
    };
    auto bulk = [&](uint32_t dst, const bf16 *src, uint32_t bytes, uint32_t bar) {
      asm volatile(
          "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
          "l"(src), "r"(bytes), "r"(bar)
          : "memory");
    };
    for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const int x0 = min((int)(item % tiles_x) * TM, W - TM);
      const long long it = item / tiles_x;
      const int y0 = (int)(it % runs_y) * R;
      const long long row0 = (it / runs_y) * (long long)H;  // n H
      const int rows = min(R, H - y0);
      for (int j = 0; j < rows + 2; ++j) {
        bool got_d = true;
        if (j < rows) {
          const uint32_t slot = d % SD, bar = dload0 + 8 * slot;
          got_d = d < SD || poll(dfree0 + 8 * slot, (d / SD - 1) & 1u);
          expect(got_d, bar, G::DROW);
          if (lane < G::DCH && got_d)
            bulk(dbase + slot * G::DS + lane * G::P, dz + conv_act_index(row0 + y0 + j, lane, x0, W, G::DCH), TM * 16, bar);
          ++d;
        }
        const uint32_t slot = q % SX, bar = xload0 + 8 * slot;
        const bool got = q < SX || poll(xfree0 + 8 * slot, (q / SX - 1) & 1u);
        int gy = y0 - 1 + j;
        gy = gy < 0 ? gy + H : (gy >= H ? gy - H : gy);
        expect(got, bar, G::XROW);
        if (lane < 3 * G::XCH && got) {
          const int dx = lane / G::XCH, c = lane - dx * G::XCH;
          const bf16 *plane = x + conv_act_index(row0 + gy, c, 0, W, G::XCH);
          const uint32_t dst = xbase + slot * G::XS + lane * G::P;
          const int first = dx == 0 && x0 == 0 ? 1 : 0, last = dx == 2 && x0 + TM == W ? TM - 2 : TM - 1;
          bulk(dst + first * 16, plane + (long long)(x0 - 1 + dx + first) * 8, (last - first + 1) * 16, bar);
          if (first) bulk(dst, plane + (long long)(W - 1) * 8, 16, bar);
          if (last == TM - 2) bulk(dst + (TM - 1) * 16, plane, 16, bar);
        }
        if (!(ok = together(got && got_d))) break;
        ++q;
      }
    }
    if (!ok) {
      give_up();
      // no copy may land after the CTA has left (rows q and d - 1: lanes that did not
      // give up have issued theirs)
      for (uint32_t k = q > SX ? q - SX : 0; k <= q; ++k) mbar_wait(xload0 + 8 * (k % SX), (k / SX) & 1u, nullptr);
      for (uint32_t k = d > SD ? d - SD - 1 : 0; k < d; ++k) mbar_wait(dload0 + 8 * (k % SD), (k / SD) & 1u, nullptr);
    }
  } else if (warp == 4) {
    // ---------------- MMA issuer ----------------
    // MN-major: the stride-dimension offset steps 8 channels (a plane), the
    // leading-dimension offset 8 pixels (128 bytes)
    const uint64_t a0 = smem_desc(xbase, 128, G::P), b0 = smem_desc(dbase, 128, G::P);
    uint32_t q = 0, d0 = 0;  // staged input row; first dz row of the item
    bool ok = true;
    for (long long item = blockIdx.x; item < nitems && ok; item += gridDim.x) {
      const int y0 = (int)((item / tiles_x) % runs_y) * R;
      const int rows = min(R, H - y0);
      // the last strip of a row starts with pixels of the strip before it
      const int xt = (int)(item % tiles_x) * TM, step0 = (xt - min(xt, W - TM)) / 16;
      for (int j = 0; j < rows + 2; ++j, ++q) {
        const uint32_t slot = q % SX;
        const int lo = max(0, j - 2), hi = min(rows - 1, j);  // dz rows that meet this input row
        bool got = j >= rows || poll(dload0 + 8 * ((d0 + j) % SD), ((d0 + j) / SD) & 1u);
        got = got && poll(xload0 + 8 * slot, (q / SX) & 1u);
        ok = together(got);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t e = elect_lane();
        const uint64_t da = a0 + (uint64_t)(slot * (G::XS / 16));
        // dz rows t .. t + n - 1, split where their ring wraps; `step`: 16 pixels
        const uint32_t set = tmem + (q % WG_SETS) * (3 * NB);
        auto issue = [&](int t, int n, int step) {
          const uint32_t sl = (d0 + t) % SD;
          const int n0 = min(n, SD - (int)sl);
          const uint32_t col = set + (uint32_t)(t - (j - 2)) * NB;
          const uint64_t a = da + (uint64_t)(step * 16);
          mma_bf16_ss(e, col, a, b0 + (uint64_t)(sl * (G::DS / 16) + step * 16),
                      (instr_desc(TM, 0) | MN_MAJOR) + ((uint32_t)(n0 * NB >> 3) << 17), 1u);
          if (n > n0)
            mma_bf16_ss(e, col + n0 * NB, a, b0 + (uint64_t)(step * 16),
                        (instr_desc(TM, 0) | MN_MAJOR) + ((uint32_t)((n - n0) * NB >> 3) << 17), 1u);
        };
#pragma unroll
        for (int step = 0; step < TM / 16; ++step)
          if (step >= step0) issue(lo, hi - lo + 1, step);
        mma_commit(e, xfree0 + 8 * slot);
        if (j >= 2) mma_commit(e, dfree0 + 8 * ((d0 + j - 2) % SD));
      }
      d0 += rows;
    }
    if (ok) {
      mma_commit(elect_lane(), done);
    } else {
      give_up();
      if (q > 0) mbar_wait(xfree0 + 8 * ((q - 1) % SX), ((q - 1) / SX) & 1u, nullptr);
    }
  } else {
    // ---------------- read-out: warp w holds rows 32 w .. 32 w + 31 of D ----------------
    if (together(mbar_wait_long(done, 0, abort_flag))) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float *out = partial + (size_t)blockIdx.x * (COUTP * 9 * CINP + COUTP);
      const int m = warp * 32 + lane, dx = m / CINP, ci = m - dx * CINP;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        float v[32];
#pragma unroll
        for (int k = 0; k < WG_SETS; ++k) {
          float p[32];
          const uint32_t taddr = tmem + (k * 3 + b) * NB + ((uint32_t)(warp * 32) << 16);
          if constexpr (NB == 32) tmem_ld32(taddr, p);
          else tmem_ld16(taddr, p);
#pragma unroll
          for (int co = 0; co < NB; ++co) v[co] = k == 0 ? p[co] : v[co] + p[co];
        }
        if (dx < 3) {
#pragma unroll
          for (int co = 0; co < COUTP; ++co) out[(co * 9 + (2 - b) * 3 + dx) * CINP + ci] = v[co];
        } else if (m == 3 * CINP && b == 1) {  // the ones' row: each dz row once
#pragma unroll
          for (int co = 0; co < COUTP; ++co) out[COUTP * 9 * CINP + co] = v[co];
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    } else {
      give_up();
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(G::TMEM_COLS) : "memory");
  }
}

template <int CINP, int COUTP, int DZS>
cudaError_t wgrad_launch(const void *x, const void *dz, int N, int H, int W, float *partial, int most, int *parts,
                         cudaStream_t s) {
  using G = WgGeom<CINP, DZS>;
  auto *kern = wgrad_tc_kernel<CINP, COUTP, DZS>;
  static int sms = 0;
  static std::once_flag once;
  static cudaError_t init_err = cudaSuccess;
  std::call_once(once, [&] {
    init_err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
    int dev = 0;
    if (init_err == cudaSuccess) init_err = cudaGetDevice(&dev);
    if (init_err == cudaSuccess) init_err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  });
  if (init_err != cudaSuccess) return init_err;
  const long long ctas = std::min(sms, most), strips = (long long)N * ((W + TM - 1) / TM);
  const int R = run_rows(H, strips, ctas);
  const long long nitems = strips * ((H + R - 1) / R);
  *parts = (int)std::min(nitems, ctas);
  kern<<<(unsigned)*parts, WG_THREADS, G::SMEM, s>>>(static_cast<const bf16 *>(x), static_cast<const bf16 *>(dz), N, H,
                                                     W, R, partial);
  return cudaGetLastError();
}

}  // namespace

namespace hlbm {

cudaError_t conv_tc_wgrad(int cinp, int coutp, int dzs, const void *x, const void *dz, int N, int H, int W,
                          float *partial, int most, int *parts, cudaStream_t s) {
  if (N < 1 || H < 1 || W < TM || W % 16) return cudaErrorInvalidValue;
#define CASE(CI, CO, DS) \
  if (cinp == CI && coutp == CO && dzs == DS) return wgrad_launch<CI, CO, DS>(x, dz, N, H, W, partial, most, parts, s);
  CASE(16, 32, 32) CASE(32, 32, 32) CASE(32, 8, 16) CASE(16, 16, 16) CASE(16, 8, 16)
#undef CASE
  return cudaErrorInvalidValue;
}

bool conv_tc_supported(int cinp, int coutp, int W) {
  if (W < TM || W % 16) return false;
  return (cinp == 16 || cinp == 32) && (coutp == 8 || coutp == 16 || coutp == 32);
}

cudaError_t conv_tc(int cinp, int coutp, int epi, const void *in, const void *w, int ks,
                    const float *bias, const void *mask, int N, int H, int W, void *out_bf,
                    float *out_f, cudaStream_t s) {
  if (N < 1 || H < 1 || W < TM || W % 16 || ks < 9 * cinp || ks % 8) return cudaErrorInvalidValue;
#define CASE(CI, NMM, CO, E)                                                   \
  if (cinp == CI && coutp == CO && epi == E)                                   \
    return launch<CI, NMM, CO, E>(in, w, ks, bias, mask, N, H, W, out_bf, out_f, s);
  CASE(16, 32, 32, CONV_RELU) CASE(32, 32, 32, CONV_RELU) CASE(16, 16, 16, CONV_RELU)
  CASE(32, 16, 8, CONV_LINEAR_F32) CASE(16, 16, 8, CONV_LINEAR_F32)
  CASE(32, 32, 32, CONV_MASK) CASE(16, 32, 32, CONV_MASK) CASE(16, 16, 16, CONV_MASK)
#undef CASE
  return cudaErrorInvalidValue;
}

cudaError_t conv_tc_predict(int cinp, const void *in, const void *w, int ks, const float *bias, const float *x0,
                            const float *out_std, int N, int H, int W, float *x1, cudaStream_t s) {
  if (N < 1 || H < 1 || !conv_tc_supported(cinp, 8, W) || ks < 9 * cinp || ks % 8) return cudaErrorInvalidValue;
  return cinp == 32 ? launch<32, 16, 8, CONV_PREDICT>(in, w, ks, bias, nullptr, N, H, W, nullptr, x1, s, x0, out_std)
                    : launch<16, 16, 8, CONV_PREDICT>(in, w, ks, bias, nullptr, N, H, W, nullptr, x1, s, x0, out_std);
}

int conv_tc_error(bool reset) {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_conv_tc_err, sizeof v) != cudaSuccess) return -1;
  if (reset && v) {
    const int zero = 0;
    cudaMemcpyToSymbol(g_conv_tc_err, &zero, sizeof zero);
  }
  return v;
}

}  // namespace hlbm
