// RowSel on the tensor cores with the database streamed through tensor memory
// (the streaming kernel: tile variant 12, and the multi-job form for small and
// medium batches).
//
// What is computed: the per-point modular GEMM of Sec. 2.3 / Sec. 5.1 of the
// GPIR paper, out[p][m][n] = sum_k ct[p][m][k] * db[p][k][n] mod q, with
// p = (limb, slot), m = (client, polynomial), k = DB row, n = DB column.
//
// Why another kernel. With few clients the database is the traffic, and the
// tensor-memory kernel (rowsel_tmem.cu) reads it as 6 bytes of fp16 digits a
// residue, passes the ciphertexts through a ring in global memory (one writer
// CTA, other readers, counters between them) and writes single 4-byte slots of
// output, eight partial writes to a 32-byte sector. Here the operands change
// places: the database is the tensor-memory operand, kept at 4 bytes a residue
// (four 7-bit fields) and widened to fp16 on the way in, and one CTA owns all 8
// slots of a sector for 16 ciphertext rows x 32 columns, so that nothing passes
// between CTAs: the ciphertext box (8 slots wide, as a sector is) is converted
// by the CTA that uses it, and the 8 results of an output sector leave
// together.
//
// Exactness.
//   - A database residue v < 2^28 is sum_u f_u 2^(7u) with fields f_u in
//     [0, 127]. The fp16 operand is the byte itself as a bit pattern: the
//     subnormal f_u 2^-24, exact.
//   - A ciphertext residue x < 2^28 has fields e_0, e_1 (10 bits) and e_2 (8
//     bits); d_v = e_v - o_v with o = (512, 512, 128) lies in [-512, 511], and
//     x = sum_v d_v 2^(10v) + C, C = 512 + 512 2^10 + 128 2^20. The term of C
//     is the same for every row of a column: C sum_k db[k][n] mod q, made at
//     upload.
//   - |f d| <= 127 * 512, so the sums of 256 rows stay below 2^24 and every
//     partial sum is an integer multiple of 2^-24 that fp32 holds exactly. The
//     12 sums D_uv of a group are weighted by 2^(7u + 10v) mod q in 64-bit
//     integers (below 2^55.6 together) and reduced; groups add mod q.
//
// Work. A unit is (group of 8 slots, block of 32 columns, block of 16 rows),
// numbered so that units sharing a database tile or a ciphertext box are
// neighbours; CTA i runs units i, i + gridDim, ... Every role walks the same
// list, so nothing is claimed and no end is signalled. Per step (64 k) of a
// unit:
//   - warp 0 copies the 8 slots' database tiles (8 KB each, contiguous in the
//     packed layout) into a ring of shared-memory slots;
//   - warp 1 loads the raw boxes, 4 clients each; boxes past the batch are left
//     out (their rows' products are never stored);
//   - 8 ingest warps split the residues into fp16 digits and write the 8
//     slots' operand tiles (48 rows v*16 + m, 64 k, 128-byte swizzle);
//   - 8 converter warps (two sets of 4, alternating tiles) turn a tile's bytes
//     into fp16 in a tensor-memory buffer: thread = lane (column, digit), one
//     byte permute per pair;
//   - two warps (even and odd slots), each with one elected lane, issue M = 128,
//     N = 48, K = 16 MMAs into the slot's own accumulator (8 x 48 columns). A
//     tile is 96 cycles of tensor work, but its waits, MMA issue and commits
//     take the issuing warp several hundred beside 26 busy warps; it stays
//     converged, since a lone thread of a diverged warp takes still longer;
//   - 8 epilogue warps drain the slots' accumulators in turn, each handed back
//     at once, so the next group's first MMAs follow slot by slot.
// Costs per step (262,144 products): 64 KB of database and up to 32 KB of
// ciphertexts from L2 or DRAM (about 3,300 cycles at the copy rate with 8
// clients), about 2,300 cycles of shared-memory traffic (copies in, converter and
// ingest reads, operand tiles written and read by the MMAs) and as much
// instruction issue. Measured 5,200 cycles: every role is busy 40 to 65% of the
// time, and the chains between them (convert, issue, commit, drain) set the pace
// (256x64, 2 limbs: 8 clients 237 -> 154 us against the tensor-memory kernel, 67%
// of the copy rate; 3 clients 213 -> 132 us against the CUDA cores; 3 clients on
// 1024x128 1494 -> 898 us). Tried: four MMA warps (156 us), waits that suspend the
// warp (157 us), reads through generic pointers (179 us).
#include <cuda.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <shared_mutex>
#include <vector>

#include "common.cuh"
#include "tcgen05.cuh"

namespace gpir {
namespace {

constexpr int S_KCHUNK = 64;                       // k per step
constexpr int S_COLS = 32;                         // DB columns per tile (x 4 digits = 128 lanes)
constexpr int S_ROWS = 16;                         // ciphertext rows per unit (x 3 digits = MMA N)
constexpr int S_SLOTS = 8;                         // slots per unit
constexpr int S_N = 3 * S_ROWS;                    // 48
constexpr int S_KGROUP = 4;                        // steps per exact group: 256 rows
constexpr int S_TILE = S_COLS * S_KCHUNK * 4;      // 8 KB database tile
constexpr int S_BT = S_N * S_KCHUNK * 2;           // 6 KB ciphertext operand tile of one slot
constexpr int S_BSTEP = S_SLOTS * S_BT;            // 48 KB: one step's operand tiles
constexpr int S_BOX_CLIENTS = 4;
constexpr int S_BOX = S_BOX_CLIENTS * S_KCHUNK * 2 * S_SLOTS * 4;   // 16 KB raw box
constexpr int S_RING = 10;                         // database tiles in shared memory (even: two converter sets)
constexpr int S_ABUF = 4;                          // tensor-memory A buffers (32 columns each)
constexpr int S_OUT = S_SLOTS * S_ROWS * S_COLS * 4;   // 16 KB
constexpr uint32_t S_A_COL0 = S_SLOTS * S_N;       // 384
constexpr uint32_t S_TMEM_COLS = 512;
static_assert(S_A_COL0 + 32 * S_ABUF <= S_TMEM_COLS, "accumulators and A buffers fit tensor memory");
static_assert(S_RING % 2 == 0, "a ring slot's uses alternate within one converter set");
constexpr size_t S_SMEM = 1024 + 2 * (size_t)S_BSTEP + (size_t)S_RING * S_TILE + 2 * (size_t)S_BOX + S_OUT + 1024;
static_assert(S_SMEM <= 232448, "streaming kernel shared memory exceeds 227 KB");
constexpr uint32_t kOffC = 512u + (512u << 10) + (128u << 20);

// Warp roles (896 threads). Tensor-memory lane quarter of a warp = warp % 4.
constexpr int SW_PROD = 0, SW_BOX = 1, SW_MMA0 = 2;
constexpr int SW_CONV0 = 4, SW_EPI0 = 12, SW_ING0 = 20;
constexpr int SN_MMA = 2, SN_CONV = 8, SN_EPI = 8, SN_ING = 8;
static_assert(S_ABUF % SN_MMA == 0, "an A buffer belongs to one MMA warp");
constexpr int S_THREADS = 32 * (SW_ING0 + SN_ING);

struct StLimb {
  uint32_t q, one_s;     // prime, floor(2^32 / q)
  uint32_t r32, r32_s;   // 2^32 mod q and floor(r32 2^32 / q)
  uint64_t off56;        // multiple of q, >= 2^56
  int32_t w[4][3];       // 2^(7u + 10v) mod q
};

constexpr int S_MAX_JOBS = 8;
struct StJob {
  CUtensorMap ct_map;              // box (8 slots, 1, 2, 64 k, 4 clients)
  uint32_t M, batch, d1, cblk, rblk, kch;
  uint32_t unit0;                  // first unit of the job
  const uint8_t *tiles;            // [group][cblk][kch][spg] x 8 KB
  const uint32_t *corr;            // [slot][32 cblk]
  uint32_t *out;
};

struct StParams {
  StJob job[S_MAX_JOBS];
  uint32_t L, N, njobs, gpl, spg;  // groups per limb, slots per group
  uint32_t n_units;
  unsigned int *err;
  StLimb limb[GPIR_MAX_LIMBS];
};

// kind::f16, D = f32, A = B = f16, K-major, M = 128, N = 48.
constexpr uint32_t kIdescS = (1u << 4) | ((uint32_t)(S_N >> 3) << 17) | ((128u >> 4) << 24);

__device__ __forceinline__ void mma_stream(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(kIdescS), "r"(accumulate)
      : "memory");
}

// 32 consecutive tensor-memory columns of this warp's lane quarter <- r[0..31].
__device__ __forceinline__ void st_tmem32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
      "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
      "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
      "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

// Three loads of 8 columns each (the three ciphertext digits of 8 rows).
__device__ __forceinline__ void ld_tmem8x3(uint32_t t0, uint32_t t1, uint32_t t2, uint32_t (&r)[24]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%24];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%25];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%26];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23])
      : "r"(t0), "r"(t1), "r"(t2)
      : "memory");
}

__device__ __forceinline__ uint32_t hadd2_bits(uint32_t x, uint32_t c) {
  const __half2 h = __hadd2(*reinterpret_cast<const __half2 *>(&x), *reinterpret_cast<const __half2 *>(&c));
  return *reinterpret_cast<const uint32_t *>(&h);
}

// Digit pairs (fp16 x 2) of two ciphertext residues: fields under 0x6400
// (1024 + field exactly), then field - offset by one addition. lo / hi pick
// the low / high halves of the two words in k order.
__device__ __forceinline__ void ct_digit_pairs(uint32_t a, uint32_t b, uint32_t lo, uint32_t hi, uint32_t &d0,
                                               uint32_t &d1, uint32_t &d2) {
  const uint32_t f0 = (__byte_perm(a, b, lo) & 0x03FF03FFu) | 0x64006400u;
  const uint32_t f1 = (__byte_perm(a >> 10, b >> 10, lo) & 0x03FF03FFu) | 0x64006400u;
  const uint32_t f2 = ((__byte_perm(a, b, hi) >> 4) & 0x00FF00FFu) | 0x64006400u;
  d0 = hadd2_bits(f0, 0xE600E600u);   // - (1024 + 512)
  d1 = hadd2_bits(f1, 0xE600E600u);
  d2 = hadd2_bits(f2, 0xE480E480u);   // - (1024 + 128)
}

// Byte u of the result = bits [7u, 7u + 7) of v < 2^28, by two spreads done as
// adds: bits 14.. up by 2, then bits 7..13 of each 16-bit half up by 1.
__device__ __forceinline__ uint32_t db_fields(uint32_t v) {
  const uint32_t a = v + 3u * (v & 0xFFFFC000u);
  return a + (a & 0x7F807F80u);
}

// Any 64-bit x to [0, 4q): hi 2^32 + lo by two products with precomputed
// quotients (Shoup), of 2^32 and of 1, and one product by q.
__device__ __forceinline__ uint32_t red64_4q(uint64_t x, const StLimb &m) {
  const uint32_t hi = (uint32_t)(x >> 32), lo = (uint32_t)x;
  return hi * m.r32 + lo - (__umulhi(hi, m.r32_s) + __umulhi(lo, m.one_s)) * m.q;
}
__device__ __forceinline__ uint32_t min_sub(uint32_t x, uint32_t c) { return min(x, x - c); }

// ---- database packing (once per upload) -------------------------------------

struct PackStreamParams {
  uint32_t d0, d1, L, N, gpl, spg, cblk, kch;
  const uint32_t *db;
  uint8_t *tiles;
};

// One block per (group, column block, step), thread = (column n, k octet j).
// Row n of a tile (256 bytes): 16-byte chunk 2j + h holds, for k octet j, the
// bytes of digits 2h and 2h + 1 of its 8 residues, stored at position
// (2j + h) ^ (n % 8). The padding is digit 0.
__global__ void __launch_bounds__(256) stream_pack_kernel(const PackStreamParams p) {
  const uint32_t kc = blockIdx.x % p.kch, cb = (blockIdx.x / p.kch) % p.cblk, g = blockIdx.x / (p.kch * p.cblk);
  const uint32_t l = g / p.gpl, t0 = (g % p.gpl) * 8;
  const uint32_t n = threadIdx.x >> 3, j = threadIdx.x & 7, col = cb * S_COLS + n;
  uint32_t z[8][8];   // [k][slot]
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    const uint32_t k = kc * S_KCHUNK + j * 8 + kk;
    const bool in = col < p.d1 && k < p.d0;
    const uint32_t *src = p.db + (((uint64_t)k * p.d1 + col) * p.L + l) * p.N + t0;
    if (p.N >= 8) {
      const uint4 a = in ? *reinterpret_cast<const uint4 *>(src) : make_uint4(0, 0, 0, 0);
      const uint4 b = in ? *reinterpret_cast<const uint4 *>(src + 4) : make_uint4(0, 0, 0, 0);
      z[kk][0] = a.x, z[kk][1] = a.y, z[kk][2] = a.z, z[kk][3] = a.w;
      z[kk][4] = b.x, z[kk][5] = b.y, z[kk][6] = b.z, z[kk][7] = b.w;
    } else {
#pragma unroll
      for (uint32_t s = 0; s < 8; ++s) z[kk][s] = in && s < p.spg ? src[s] : 0u;
    }
  }
  uint8_t *tile = p.tiles + (uint64_t)blockIdx.x * p.spg * S_TILE + n * 256;
#pragma unroll
  for (uint32_t s = 0; s < 8; ++s) {
    if (s >= p.spg) break;
    uint32_t f[8], w[2][4];   // [k half][digit]: 4 bytes of one digit
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) f[kk] = db_fields(z[kk][s]);
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const uint32_t t0_ = __byte_perm(f[4 * hh], f[4 * hh + 1], 0x5140), t1 = __byte_perm(f[4 * hh], f[4 * hh + 1], 0x7362);
      const uint32_t t2 = __byte_perm(f[4 * hh + 2], f[4 * hh + 3], 0x5140), t3 = __byte_perm(f[4 * hh + 2], f[4 * hh + 3], 0x7362);
      w[hh][0] = __byte_perm(t0_, t2, 0x5410);
      w[hh][1] = __byte_perm(t0_, t2, 0x7632);
      w[hh][2] = __byte_perm(t1, t3, 0x5410);
      w[hh][3] = __byte_perm(t1, t3, 0x7632);
    }
    uint4 *row = reinterpret_cast<uint4 *>(tile + (uint64_t)s * S_TILE);
    row[(2 * j) ^ (n & 7)] = make_uint4(w[0][0], w[1][0], w[0][1], w[1][1]);
    row[(2 * j + 1) ^ (n & 7)] = make_uint4(w[0][2], w[1][2], w[0][3], w[1][3]);
  }
}

// corr[slot][n] = C sum_k db[k][n][slot] mod q.
__global__ void stream_corr_kernel(const PackStreamParams p, LimbTable limbs, uint32_t *corr) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t slots = p.L * p.N;
  if (i >= (uint64_t)slots * p.d1) return;
  const uint32_t slot = (uint32_t)(i % slots), n = (uint32_t)(i / slots), l = slot / p.N;
  uint64_t sum = 0;
  const uint32_t *src = p.db + (uint64_t)n * slots + slot;
#pragma unroll 8
  for (uint32_t k = 0; k < p.d0; ++k) sum += src[(uint64_t)k * p.d1 * slots];
  const uint32_t q = limbs.m[l].q;
  const uint64_t mu = limbs.m[l].mu;
  corr[(uint64_t)slot * (p.cblk * S_COLS) + n] = reduce64((uint64_t)reduce64(sum, q, mu) * reduce64(kOffC, q, mu), q, mu);
}

// ---- the persistent kernel -------------------------------------------------

struct StUnit {
  uint32_t j;              // job
  uint32_t g, cb, rb, kch;
  uint32_t l, t0;          // limb, first slot
};

__device__ __forceinline__ StUnit stream_unit(const StParams &p, uint32_t u) {
  StUnit x;
  x.j = 0;
  while (x.j + 1 < p.njobs && u >= p.job[x.j + 1].unit0) ++x.j;
  const StJob &jb = p.job[x.j];
  const uint32_t ul = u - jb.unit0, per = jb.cblk * jb.rblk;
  x.g = ul / per;
  const uint32_t w = ul - x.g * per;
  x.cb = w / jb.rblk;
  x.rb = w - x.cb * jb.rblk;
  x.kch = jb.kch;
  x.l = x.g / p.gpl;
  x.t0 = (x.g - x.l * p.gpl) * 8;
  return x;
}

__global__ void __launch_bounds__(S_THREADS, 1) tc_stream_kernel(const __grid_constant__ StParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);   // an offset: a shared-memory pointer to the compiler
  uint8_t *btiles = smem;                                     // [2][8 slots] x 6 KB
  uint8_t *ring = btiles + 2 * S_BSTEP;                       // [S_RING] x 8 KB
  uint8_t *boxes = ring + S_RING * S_TILE;                    // [2] x 16 KB
  uint32_t *stage = reinterpret_cast<uint32_t *>(boxes + 2 * S_BOX);   // [slot][row][column, swizzled]
  uint64_t *rfull = reinterpret_cast<uint64_t *>(boxes + 2 * S_BOX + S_OUT);   // [S_RING] tile landed
  uint64_t *rempty = rfull + S_RING;                          // [S_RING] tile read by its converters
  uint64_t *box_full = rempty + S_RING;                       // [2]
  uint64_t *box_empty = box_full + 2;                         // [2]
  uint64_t *bfull = box_empty + 2;                            // [2] operand tiles of a step written
  uint64_t *bempty = bfull + 2;                               // [2] ... read by its MMAs
  uint64_t *afull = bempty + 2;                               // [S_ABUF] converted
  uint64_t *aempty = afull + S_ABUF;                          // [S_ABUF] read by its MMAs
  uint64_t *acc_full = aempty + S_ABUF;                       // [8] group sums of the slot done
  uint64_t *acc_empty = acc_full + S_SLOTS;                   // [8] drained
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + S_SLOTS);
  volatile uint32_t *abort_flag = tmem_slot + 1;
  volatile uint32_t *epi_failed = tmem_slot + 2;             // an epilogue warp's wait has expired
  static_assert(8 * (2 * S_RING + 8 + 2 * S_ABUF + 2 * S_SLOTS + 2) <= 1024, "barrier area exceeds its reservation");

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < S_RING; ++i) {
      mbar_init(&rfull[i], 1);
      mbar_init(&rempty[i], 4);       // the 4 warps of the converter set that reads it
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&box_full[i], 1);
      mbar_init(&box_empty[i], SN_ING);
      mbar_init(&bfull[i], SN_ING);
      mbar_init(&bempty[i], SN_MMA);
    }
    for (int i = 0; i < S_ABUF; ++i) {
      mbar_init(&afull[i], 4);
      mbar_init(&aempty[i], 1);
    }
    for (int i = 0; i < S_SLOTS; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], SN_EPI);
    }
    *abort_flag = 0;
    *epi_failed = 0;
    fence_mbar_init();
  }
  if (warp == SW_MMA0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(S_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t spg = p.spg;

  auto wait = [&](uint64_t *bar, uint32_t parity, unsigned int code) -> bool {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (uint32_t n = 1;; ++n) {
      if (mbar_try_wait(bar, parity)) return true;
      if ((n & 63u) == 0) {
        if (*abort_flag) return false;
        if (globaltimer_ns() - t0 > kWaitLimitNs) {
          atomicCAS(p.err, 0u, code);
          *abort_flag = 1;
          return false;
        }
      }
    }
  };

  if (warp == SW_PROD) {
    // ---------------- database tiles ----------------
    if (lane == 0) {
      uint32_t r = 0, ph = 0, issued = 0, issued_ph = 0;
      bool ok = true;
      for (uint32_t u = blockIdx.x; u < p.n_units && ok; u += gridDim.x) {
        const StUnit x = stream_unit(p, u);
        const StJob &jb = p.job[x.j];
        const uint8_t *src = jb.tiles + ((uint64_t)x.g * jb.cblk + x.cb) * x.kch * spg * (uint64_t)S_TILE;
        for (uint32_t i = 0; i < x.kch * spg; ++i) {
          if (!(ok = wait(&rempty[r], ph ^ 1u, kErrTmaWait))) break;
          mbar_arrive_expect_tx(&rfull[r], S_TILE);
          bulk_g2s(ring + r * S_TILE, src + (uint64_t)i * S_TILE, S_TILE, &rfull[r]);
          issued |= 1u << r;
          issued_ph = (issued_ph & ~(1u << r)) | (ph << r);
          if (++r == S_RING) {
            r = 0;
            ph ^= 1u;
          }
        }
      }
      if (!ok)   // let the copies in flight land before the CTA leaves
        for (int i = 0; i < S_RING; ++i)
          if ((issued >> i) & 1u) mbar_wait_bounded(&rfull[i], (issued_ph >> i) & 1u, nullptr, 0);
    }
  } else if (warp == SW_BOX) {
    // ---------------- raw ciphertext boxes ----------------
    if (lane == 0) {
      uint32_t gb = 0;
      bool ok = true;
      for (uint32_t u = blockIdx.x; u < p.n_units && ok; u += gridDim.x) {
        const StUnit x = stream_unit(p, u);
        const StJob &jb = p.job[x.j];
        const uint32_t c0 = x.rb * (S_ROWS / 2);
        const uint32_t parts = jb.batch - c0 > S_BOX_CLIENTS ? 2 : 1;
        for (uint32_t kc = 0; kc < x.kch && ok; ++kc)
          for (uint32_t part = 0; part < parts; ++part, ++gb) {
            const uint32_t b = gb & 1u;
            if (!(ok = wait(&box_empty[b], ((gb >> 1) & 1u) ^ 1u, kErrTmaWait))) break;
            mbar_arrive_expect_tx(&box_full[b], S_BOX);
            tma_load_5d(boxes + b * S_BOX, &jb.ct_map, &box_full[b], (int)x.t0, (int)x.l, 0, (int)(kc * S_KCHUNK),
                        (int)(c0 + part * S_BOX_CLIENTS));
          }
      }
      if (!ok)   // the last two boxes may still be in flight
        for (uint32_t i = 0; i < 2 && i < gb; ++i) {
          const uint32_t k = gb - 1 - i;
          mbar_wait_bounded(&box_full[k & 1u], (k >> 1) & 1u, nullptr, 0);
        }
    }
  } else if (warp >= SW_ING0) {
    // ---------------- ingest: raw box -> operand tiles ----------------
    // Thread = (client cl, polynomial r, k octet j, slot pair sp) of a box: 8
    // residues of 2 slots. The slot pair turns with j / 2 and the k order with
    // j % 2, so that the 16 lanes of each half-warp read all 32 banks (8-byte
    // reads), and the 8 lanes of each 16-byte store have 8 different j, which
    // the swizzle sends to different banks.
    const int iw = warp - SW_ING0;
    const uint32_t j = lane & 7, rp = (lane >> 3) & 1, cl = (iw >> 2) * 2 + (lane >> 4);
    const uint32_t sp = ((iw & 3) + (j >> 1)) & 3u, j0 = j & 1u;
    const uint32_t sel_lo = j0 ? 0x1054u : 0x5410u, sel_hi = j0 ? 0x3276u : 0x7632u;
    const uint32_t src0 = ((cl * S_KCHUNK + 8 * j) * 2 + rp) * 8 + 2 * sp;
    uint32_t gb = 0, t = 0;
    bool ok = true;
    for (uint32_t u = blockIdx.x; u < p.n_units && ok; u += gridDim.x) {
      const StUnit x = stream_unit(p, u);
      const uint32_t parts = p.job[x.j].batch - x.rb * (S_ROWS / 2) > S_BOX_CLIENTS ? 2 : 1;
      for (uint32_t kc = 0; kc < x.kch && ok; ++kc, ++t) {
        const uint32_t bb = t & 1u;
        if (!(ok = __all_sync(0xffffffffu, wait(&bempty[bb], ((t >> 1) & 1u) ^ 1u, kErrMmaWait)))) break;
        for (uint32_t part = 0; part < parts; ++part, ++gb) {
          const uint32_t b = gb & 1u;
          if (!(ok = __all_sync(0xffffffffu, wait(&box_full[b], (gb >> 1) & 1u, kErrTmaWait)))) break;
          const uint32_t *be = reinterpret_cast<const uint32_t *>(boxes + b * S_BOX) + src0 + j0 * 16;
          const uint32_t *bo = be - 2 * j0 * 16;
          uint2 z[8];   // position kk holds k offset kk ^ j0
#pragma unroll
          for (int kk = 0; kk < 8; ++kk) z[kk] = *reinterpret_cast<const uint2 *>((kk & 1 ? bo : be) + kk * 16);
          const uint32_t row = part * 8 + cl * 2 + rp;
          uint8_t *dst = btiles + bb * S_BSTEP + 2 * sp * S_BT + row * 128 + ((j ^ (row & 7u)) << 4);
#pragma unroll
          for (int s = 0; s < 2; ++s) {
            uint32_t d[3][4];
#pragma unroll
            for (int m = 0; m < 4; ++m)
              ct_digit_pairs(s ? z[2 * m].y : z[2 * m].x, s ? z[2 * m + 1].y : z[2 * m + 1].x, sel_lo, sel_hi, d[0][m],
                             d[1][m], d[2][m]);
#pragma unroll
            for (int v = 0; v < 3; ++v)
              *reinterpret_cast<uint4 *>(dst + s * S_BT + v * S_ROWS * 128) =
                  make_uint4(d[v][0], d[v][1], d[v][2], d[v][3]);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&box_empty[b]);
        }
        if (!ok) break;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the MMAs read these tiles
        __syncwarp();
        if (lane == 0) mbar_arrive(&bfull[bb]);
      }
    }
  } else if (warp >= SW_CONV0 && warp < SW_CONV0 + SN_CONV) {
    // ---------------- converters: database tile -> fp16 in tensor memory ----------------
    // Thread = tensor-memory lane: column m = quarter * 8 + m_lo of the tile,
    // digit u. Set cs converts tiles cs, cs + 2, ...
    const uint32_t qw = (uint32_t)(warp & 3), cs = (uint32_t)(warp - SW_CONV0) >> 2;
    const int u4 = lane >> 3, m_lo = lane & 7, m = (int)qw * 8 + m_lo;
    const uint32_t lane_base = tmem_base + ((qw * 32u) << 16) + S_A_COL0;
    uint32_t total = 0;   // tiles of this CTA
    for (uint32_t u = blockIdx.x; u < p.n_units; u += gridDim.x) total += stream_unit(p, u).kch * spg;
    for (uint32_t i = cs; i < total; i += 2) {
      const uint32_t r = i % S_RING, ab = i % S_ABUF;
      if (!__all_sync(0xffffffffu, wait(&rfull[r], (i / S_RING) & 1u, kErrTmaWait))) break;
      const uint2 *row = reinterpret_cast<const uint2 *>(ring + r * S_TILE) + m * 32;
      uint32_t wv[32];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint2 z = row[(((2 * j + (u4 >> 1)) ^ (m & 7)) << 1) | (u4 & 1)];
        wv[4 * j] = __byte_perm(z.x, 0, 0x4140);   // bytes 0, 1 as two 16-bit subnormals
        wv[4 * j + 1] = __byte_perm(z.x, 0, 0x4342);
        wv[4 * j + 2] = __byte_perm(z.y, 0, 0x4140);
        wv[4 * j + 3] = __byte_perm(z.y, 0, 0x4342);
      }
      if (!__all_sync(0xffffffffu, wait(&aempty[ab], ((i / S_ABUF) & 1u) ^ 1u, kErrMmaWait))) break;
      tc_fence_after();
      st_tmem32(lane_base + ab * 32, wv);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      // The ring slot is handed back only here, where the store has consumed
      // every word read from it: arriving right after the reads were issued
      // let the next copy overwrite words still to be read (seen as a few
      // wrong columns in a million).
      if (lane == 0) {
        mbar_arrive(&rempty[r]);
        mbar_arrive(&afull[ab]);
      }
    }
  } else if (warp >= SW_MMA0 && warp < SW_MMA0 + SN_MMA) {
    // ---------------- MMA issuers (converged warps, one elected lane each) ----------------
    // Warp w takes slots w, w + 2, ... so that the warps share nothing but the
    // step's operand tiles: slot s uses A buffer s % 4 (a step is 8 tiles, or 4
    // when N = 4), so A buffers and accumulators have one issuing warp each.
    uint32_t leader;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(leader));
    const uint32_t w = (uint32_t)(warp - SW_MMA0);
    uint32_t t = 0, grp = 0;   // steps, groups so far
    uint32_t tiles = 0;        // tiles up to the last one this warp issued
    bool ok = true;
    for (uint32_t u = blockIdx.x; u < p.n_units && ok; u += gridDim.x) {
      const uint32_t kch = stream_unit(p, u).kch;
      for (uint32_t kc = 0; kc < kch && ok; ++kc, ++t) {
        const bool first = kc % S_KGROUP == 0, last = kc % S_KGROUP == S_KGROUP - 1 || kc + 1 == kch;
        if (!(ok = __all_sync(0xffffffffu, wait(&bfull[t & 1u], (t >> 1) & 1u, kErrTmaWait)))) break;
        const uint32_t sb = smem_u32(btiles + (t & 1u) * S_BSTEP);
#pragma unroll
        for (uint32_t k = 0; k < S_SLOTS / SN_MMA; ++k) {
          const uint32_t s = SN_MMA * k + w, i = t * spg + s, ab = s % S_ABUF;   // i: tile of this CTA
          if (s >= spg) break;
          if (first && !(ok = __all_sync(0xffffffffu, wait(&acc_empty[s], (grp & 1u) ^ 1u, kErrMmaWait)))) break;
          if (!(ok = __all_sync(0xffffffffu, wait(&afull[ab], (i / S_ABUF) & 1u, kErrTmaWait)))) break;
          tc_fence_after();
          if (leader) {
#pragma unroll
            for (int k16 = 0; k16 < S_KCHUNK / 16; ++k16)
              mma_stream(tmem_base + s * S_N, tmem_base + S_A_COL0 + ab * 32 + k16 * 8,
                         sw128_desc(sb + s * S_BT + k16 * 32), (!first || k16 > 0) ? 1u : 0u);
            mma_commit(&aempty[ab]);
            if (last) mma_commit(&acc_full[s]);
            if (s + SN_MMA >= spg) mma_commit(&bempty[t & 1u]);
          }
          __syncwarp();
          tiles = i + 1;
        }
        if (last) ++grp;
      }
    }
    // every MMA issued is done, and its commits have arrived, before the CTA leaves
    if (lane == 0) {
      for (uint32_t i = tiles, b = 0; b < S_ABUF / SN_MMA && i > 0; ++b, i = i > SN_MMA ? i - SN_MMA : 0)
        mbar_wait_bounded(&aempty[(i - 1) % S_ABUF], ((i - 1) / S_ABUF) & 1u, nullptr, 0);
      for (uint32_t b = 0; ok && b < 2 && b < t; ++b)
        mbar_wait_bounded(&bempty[(t - 1 - b) & 1u], ((t - 1 - b) >> 1) & 1u, nullptr, 0);
    }
    __syncwarp();
  } else if (warp >= SW_EPI0 && warp < SW_EPI0 + SN_EPI) {
    // ---------------- epilogue ----------------
    // Thread = lane (column m, digit u) and 8 of the 16 rows. After the
    // reduce-scatter over the four digits it holds rows 8 hf + u and + 4.
    const uint32_t qw = (uint32_t)(warp & 3), hf = (uint32_t)(warp - SW_EPI0) >> 2;
    const uint32_t u4 = lane >> 3, m = qw * 8 + (lane & 7);
    const int et = (int)threadIdx.x - 32 * SW_EPI0;
    const bool b0 = u4 & 1u, b1 = u4 >> 1;
    uint32_t *cell = stage + (8 * hf + u4) * S_COLS + (m ^ (u4 * 8));   // row 8 hf + u; + 4 rows: the same swizzle
    uint32_t grp = 0;
    bool ok = true;
    for (uint32_t u = blockIdx.x; u < p.n_units && ok; u += gridDim.x) {
      const StUnit x = stream_unit(p, u);
      const StJob &jb = p.job[x.j];
      const StLimb &lm = p.limb[x.l];
      const int32_t w0 = lm.w[u4][0], w1 = lm.w[u4][1], w2 = lm.w[u4][2];
      const uint32_t cpad = jb.cblk * S_COLS;
      const uint32_t *corr = jb.corr + ((uint64_t)x.l * p.N + x.t0) * cpad + x.cb * S_COLS + m;
      const uint32_t groups = (x.kch + S_KGROUP - 1) / S_KGROUP;
      for (uint32_t gi = 0; gi < groups && ok; ++gi, ++grp) {
#pragma unroll 1
        for (uint32_t s = 0; s < spg; ++s) {
          const uint32_t c = gi == 0 ? __ldg(corr + s * cpad) : 0u;
          if (!(ok = __all_sync(0xffffffffu, wait(&acc_full[s], grp & 1u, kErrMmaWait)))) break;
          tc_fence_after();
          uint32_t d[24];
          const uint32_t ta = tmem_base + ((qw * 32u) << 16) + s * S_N + hf * 8u;
          ld_tmem8x3(ta, ta + S_ROWS, ta + 2 * S_ROWS, d);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[s]);
          int64_t P[8];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            P[i] = (int64_t)__float2int_rn(__uint_as_float(d[i]) * 16777216.f) * w0 +
                   (int64_t)__float2int_rn(__uint_as_float(d[8 + i]) * 16777216.f) * w1 +
                   (int64_t)__float2int_rn(__uint_as_float(d[16 + i]) * 16777216.f) * w2;
          int64_t K1[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            K1[i] = (b0 ? P[2 * i + 1] : P[2 * i]) + __shfl_xor_sync(0xffffffffu, b0 ? P[2 * i] : P[2 * i + 1], 8);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int64_t sum = (b1 ? K1[2 * i + 1] : K1[2 * i]) +
                                __shfl_xor_sync(0xffffffffu, b1 ? K1[2 * i] : K1[2 * i + 1], 16);
            uint32_t v = red64_4q((uint64_t)(sum + (int64_t)lm.off56), lm);
            v = min_sub(min_sub(v, 2 * lm.q), lm.q);
            uint32_t *to = cell + s * (S_ROWS * S_COLS) + i * 4 * S_COLS;   // read and written by this thread only
            *to = min_sub(v + (gi == 0 ? c : *to), lm.q);
          }
        }
      }
      // the unit's 8 slots of every (row, column) leave together. After an
      // expired wait some of the 8 warps may still see their accumulator
      // arrive and others not: they agree here, by a word written before the
      // barrier only, so that none is left waiting at the next one for a warp
      // that has gone.
      if (!ok) *epi_failed = 1;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * SN_EPI) : "memory");
      if (*epi_failed) break;
      uint32_t v[2][8];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint32_t row = (uint32_t)et / S_COLS + 8 * i, col = (uint32_t)et % S_COLS;
#pragma unroll
        for (int s = 0; s < 8; ++s) v[i][s] = stage[s * (S_ROWS * S_COLS) + row * S_COLS + (col ^ ((row & 3u) * 8))];
      }
      asm volatile("bar.sync 1, %0;" ::"n"(32 * SN_EPI) : "memory");
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const uint32_t row = x.rb * S_ROWS + (uint32_t)et / S_COLS + 8 * i, col = x.cb * S_COLS + (uint32_t)et % S_COLS;
        if (row >= jb.M || col >= jb.d1) continue;
        uint32_t *o = jb.out + ((((uint64_t)(row >> 1) * jb.d1 + col) * 2 + (row & 1u)) * p.L + x.l) * p.N + x.t0;
        if (spg == 8) {
          reinterpret_cast<uint4 *>(o)[0] = make_uint4(v[i][0], v[i][1], v[i][2], v[i][3]);
          reinterpret_cast<uint4 *>(o)[1] = make_uint4(v[i][4], v[i][5], v[i][6], v[i][7]);
        } else {
#pragma unroll
          for (int s = 0; s < 8; ++s)
            if (s < (int)spg) o[s] = v[i][s];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == SW_MMA0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(S_TMEM_COLS) : "memory");
}

StLimb make_st_limb(uint32_t q) {
  StLimb t;
  t.q = q;
  t.one_s = (uint32_t)((1ull << 32) / q);
  t.r32 = (uint32_t)((1ull << 32) % q);
  t.r32_s = (uint32_t)(((uint64_t)t.r32 << 32) / q);
  t.off56 = (((1ull << 56) + q - 1) / q) * (uint64_t)q;
  for (int u = 0; u < 4; ++u)
    for (int v = 0; v < 3; ++v) t.w[u][v] = (int32_t)((1ull << (7 * u + 10 * v)) % q);
  return t;
}

std::mutex g_st_mu;
bool g_st_attr_done[64];

// The databases that hold tiles. A launch holds the lock shared until it is
// enqueued; tiles are added, freed and given back with it held alone.
std::shared_mutex g_tiles_mu;
std::vector<gpir_db *> g_tiles;

void free_tiles(gpir_db *db) {
  uint8_t *fields = db->db_fields;
  __atomic_store_n(&db->db_fields, (uint8_t *)nullptr, __ATOMIC_RELAXED);
  if (fields) cudaFree(fields);
  if (db->db_corr) cudaFree(db->db_corr);
  db->db_corr = nullptr;
  db->db_fields_bytes = db->db_corr_bytes = 0;
}

PackStreamParams stream_shape(const gpir_db *db) {
  PackStreamParams pp;
  memset(&pp, 0, sizeof(pp));
  pp.d0 = db->d0;
  pp.d1 = db->d1;
  pp.L = db->params.num_limbs;
  pp.N = db->params.n;
  pp.gpl = (pp.N + 7) / 8;
  pp.spg = pp.N < 8 ? pp.N : 8u;
  pp.cblk = (pp.d1 + S_COLS - 1) / S_COLS;
  pp.kch = (pp.d0 + S_KCHUNK - 1) / S_KCHUNK;
  pp.db = db->db_pmajor;
  return pp;
}

}  // namespace

bool rowsel_stream_has_tiles(const gpir_db *db) {
  return __atomic_load_n(&db->db_fields, __ATOMIC_RELAXED) != nullptr;
}

size_t rowsel_stream_bytes(const gpir_db *db) {
  std::shared_lock<std::shared_mutex> lk(g_tiles_mu);
  return db->db_fields_bytes + db->db_corr_bytes;
}

void rowsel_stream_release(gpir_db *db) {
  std::unique_lock<std::shared_mutex> lk(g_tiles_mu);
  g_tiles.erase(std::remove(g_tiles.begin(), g_tiles.end(), db), g_tiles.end());
  free_tiles(db);
}

// The tiles only make small batches faster, so no other allocation of the
// library fails for them: when the device is full, those that no captured
// launch refers to are freed (cudaFree synchronizes across all executing
// streams, so the launches that read them are done), and their databases are
// served by the other kernels from then on.
bool rowsel_stream_give_back() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::unique_lock<std::shared_mutex> lk(g_tiles_mu);
  const auto held = [&](const gpir_db *db) {
    return db->device != dev || __atomic_load_n(&db->tiles_captured, __ATOMIC_RELAXED) != 0;
  };
  const auto keep = std::partition(g_tiles.begin(), g_tiles.end(), held);
  if (keep == g_tiles.end()) return false;
  for (auto it = keep; it != g_tiles.end(); ++it) free_tiles(*it);
  g_tiles.erase(keep, g_tiles.end());
  return true;
}

// The database tiles and column corrections of the streaming kernel. A database
// that leaves no room for them is served by the other kernels: they are taken
// only where an eighth of the device's memory stays free, for the caller's
// buffers (128 clients' ciphertexts and outputs of a 4 GiB database are 10 GB of
// a GB300's 35).
int rowsel_stream_prepare(gpir_db *db, cudaStream_t stream) {
  PackStreamParams pp = stream_shape(db);
  const uint64_t blocks = (uint64_t)pp.gpl * pp.L * pp.cblk * pp.kch;
  const size_t bytes = (size_t)blocks * pp.spg * S_TILE;
  const uint64_t slots = (uint64_t)pp.L * pp.N;
  const size_t corr_bytes = (size_t)slots * pp.cblk * S_COLS * 4;
  if (blocks > 0x7fffffffull || (slots * pp.d1 + 255) / 256 > 0x7fffffffull) return GPIR_OK;
  size_t free_bytes = 0, total_bytes = 0;
  cudaError_t e = cudaMemGetInfo(&free_bytes, &total_bytes);
  if (e != cudaSuccess) return set_cuda_error(e);
  if (free_bytes < bytes + corr_bytes + total_bytes / 8) return GPIR_OK;
  e = dev_malloc(reinterpret_cast<void **>(&db->db_fields), bytes, true);
  if (e != cudaSuccess) db->db_fields = nullptr;
  if (e == cudaSuccess) {
    e = dev_malloc(reinterpret_cast<void **>(&db->db_corr), corr_bytes, true);
    if (e != cudaSuccess) {
      db->db_corr = nullptr;
      cudaFree(db->db_fields);
      db->db_fields = nullptr;
    }
  }
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return GPIR_OK;
  }
  if (e != cudaSuccess) return set_cuda_error(e);
  db->db_fields_bytes = bytes;
  db->db_corr_bytes = corr_bytes;
  pp.tiles = db->db_fields;
  stream_pack_kernel<<<(unsigned)blocks, 256, 0, stream>>>(pp);
  e = cudaMemsetAsync(db->db_corr, 0, corr_bytes, stream);
  if (e != cudaSuccess) return set_cuda_error(e);
  stream_corr_kernel<<<(unsigned)((slots * pp.d1 + 255) / 256), 256, 0, stream>>>(pp, db->params.limbs, db->db_corr);
  e = cudaGetLastError();
  if (e != cudaSuccess) return set_cuda_error(e);
  e = cudaStreamSynchronize(stream);
  if (e != cudaSuccess) return set_cuda_error(e);
  std::unique_lock<std::shared_mutex> lk(g_tiles_mu);
  try {
    g_tiles.push_back(db);
  } catch (...) {   // no exception crosses the C ABI
    free_tiles(db);
  }
  return GPIR_OK;
}

// Untuned batches take the streaming kernel when they are one block of 16 rows
// (8 clients) and its units fill the SMs. Measured at N = 4096, 2 limbs (us,
// tensor-memory / streaming): 4 and 8 clients 219 / 136 and 237 / 154 (256x64),
// 606 / 363 and 636 / 405 (500x90), 1180 / 894 and 1251 / 1004 (1024x128); at two blocks
// of rows the database is converted twice and the gain is gone: 16 clients
// 284 / 277 (256x64), 1375 / 1965 (1024x128).
bool rowsel_stream_preferred(const gpir_db *db, uint32_t batch) {
  if (batch > S_ROWS / 2 || !rowsel_stream_has_tiles(db)) return false;
  const PackStreamParams sh = stream_shape(db);
  return (uint64_t)sh.gpl * sh.L * sh.cblk >= (uint64_t)sm_count();
}

// Untuned batches of 2 to 7 clients: the streaming kernel or the CUDA cores.
// Both run one CTA per 8 slots x 32 columns of such a batch and take whole waves.
// A streaming wave (one unit per SM) costs a fixed part, a part per step of 64
// rows and a part per exact group of 256, all padded; a wave of the CUDA cores
// (four CTAs per SM) costs its rows, twice as much from 5 clients on, which take
// a tile of twice the height. In quarters of what a row costs the CUDA cores,
// the streaming parts are 20, 30 and 60 at up to 4 clients and 20, 14 and 23 above:
// fitted to 8,100 points (16 to 1025 rows, 1 to 300 columns, N = 128 to 8192, 1 to 4
// limbs, 160 to 8192 units), where the choice is at most 7% behind the faster
// kernel. us, CUDA cores / streaming: 5 clients 12.6 / 28.7 (16x48, N = 2048, 1
// limb), 7 clients 39 / 92 (16x1, N = 4096, 4 limbs) and 387 / 222 (257x64, N =
// 4096, 2 limbs); 3 clients 56 / 63 (257x33, N = 2048, 1 limb), but 56 / 33
// (257x192, N = 256, 1 limb) and 217 / 200 (257x64, N = 4096, 2 limbs). Up to 192
// rows batches of 2 to 4 clients stay on the CUDA cores.
bool rowsel_stream_beats_cc(const gpir_db *db, uint32_t batch) {
  if (batch < 2 || (batch < 5 && db->d0 <= 192) || !rowsel_stream_preferred(db, batch)) return false;
  const PackStreamParams sh = stream_shape(db);
  const uint64_t units = (uint64_t)sh.gpl * sh.L * sh.cblk, sms = (uint64_t)sm_count();
  const uint64_t waves = (units + sms - 1) / sms, cc_waves = (units + 4 * sms - 1) / (4 * sms);
  const uint64_t groups = (sh.kch + S_KGROUP - 1) / S_KGROUP;
  const uint64_t cost = batch < 5 ? 20 + 30 * (uint64_t)sh.kch + 60 * groups : 20 + 14 * (uint64_t)sh.kch + 23 * groups;
  return waves * cost <= 4 * cc_waves * db->d0;
}

// RowSel problems of one parameter set through the streaming kernel, at most
// S_MAX_JOBS per launch. It needs no workspace.
int rowsel_stream_launch(const gpir_job_t *jobs, uint32_t njobs, cudaStream_t stream) {
  std::shared_lock<std::shared_mutex> lk_tiles(g_tiles_mu);
  for (uint32_t k = 0; k < njobs; ++k)
    if (!jobs[k].db->db_fields || !jobs[k].db->db_corr) return GPIR_ENOTSUP;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(stream, &cs);
  if (e != cudaSuccess || cs != cudaStreamCaptureStatusNone)   // its replays will read these tiles
    for (uint32_t k = 0; k < njobs; ++k) __atomic_store_n(&jobs[k].db->tiles_captured, 1u, __ATOMIC_RELAXED);
  int dev = 0;
  e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return set_cuda_error(e);
  if (dev < 0 || dev >= 64) return GPIR_EINVAL;
  {
    std::lock_guard<std::mutex> lk(g_st_mu);
    if (!g_st_attr_done[dev]) {
      e = cudaFuncSetAttribute(tc_stream_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S_SMEM);
      if (e != cudaSuccess) return set_cuda_error(e);
      g_st_attr_done[dev] = true;
    }
  }
  const gpir_params &prm = jobs[0].db->params;
  const uint32_t L = prm.num_limbs, N = prm.n;
  for (uint32_t k0 = 0; k0 < njobs; k0 += S_MAX_JOBS) {
    StParams sp;
    memset(&sp, 0, sizeof(sp));
    sp.L = L;
    sp.N = N;
    sp.njobs = std::min<uint32_t>(S_MAX_JOBS, njobs - k0);
    sp.gpl = (N + 7) / 8;
    sp.spg = N < 8 ? N : 8u;
    sp.err = device_error_word();
    uint64_t units = 0;
    for (uint32_t k = 0; k < sp.njobs; ++k) {
      const gpir_job_t &job = jobs[k0 + k];
      const PackStreamParams sh = stream_shape(job.db);
      StJob &jb = sp.job[k];
      jb.batch = job.batch;
      jb.M = 2 * job.batch;
      jb.d1 = job.db->d1;
      jb.cblk = sh.cblk;
      jb.rblk = (jb.M + S_ROWS - 1) / S_ROWS;
      jb.kch = sh.kch;
      jb.tiles = job.db->db_fields;
      jb.corr = job.db->db_corr;
      jb.out = job.out;
      if (units > UINT32_MAX) return GPIR_ETOOBIG;
      jb.unit0 = (uint32_t)units;
      units += (uint64_t)sp.gpl * L * jb.cblk * jb.rblk;
      const uint64_t dims[5] = {N, L, 2, job.db->d0, job.batch};
      const uint64_t str[4] = {(uint64_t)N * 4, (uint64_t)L * N * 4, (uint64_t)2 * L * N * 4,
                               (uint64_t)job.db->d0 * 2 * L * N * 4};
      const uint32_t box[5] = {S_SLOTS, 1, 2, S_KCHUNK, S_BOX_CLIENTS};
      const int rc = encode_tiled_u32(&jb.ct_map, job.ct, 5, dims, str, box);
      if (rc != GPIR_OK) return rc;
    }
    if (units > UINT32_MAX - 1024) return GPIR_ETOOBIG;   // a role's next unit index is below 2^32
    sp.n_units = (uint32_t)units;
    for (uint32_t l = 0; l < L; ++l) sp.limb[l] = make_st_limb(prm.primes[l]);
    const unsigned grid = (unsigned)std::min<uint64_t>(units, (uint64_t)sm_count());
    const int tr = trace_begin("tc_stream", stream);
    tc_stream_kernel<<<grid, S_THREADS, S_SMEM, stream>>>(sp);
    trace_end(tr, stream);
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(e);
  }
  return GPIR_OK;
}

}  // namespace gpir
