// ColTor: the column tournament that follows RowSel (GPIR paper Sec. 2.2,
// "ColTor"), with the external product of Sec. 2.5.1.
//
// For every client, log2(D1) stages halve the client's D1 ciphertexts: stage s
// pairs the stage inputs (2k, 2k+1) and keeps
//     ct_{2k} + RGSW_s [x] (ct_{2k+1} - ct_{2k}).
// The external product of an RGSW ciphertext (2 ell rows of two polynomials)
// with a ciphertext (c_0, c_1), everything in the NTT domain:
//   1. inverse NTT of c_0 and c_1, limb by limb;
//   2. Dcp: every coefficient is rebuilt from its limbs (CRT) as x in [0, Q),
//      centred to (-Q/2, Q/2], and split into balanced base-2^22 digits
//      x = sum_{i<ell} d_i 2^(22 i), d_i in [-2^21, 2^21) (the last digit takes
//      the rest);
//   3. forward NTT of the 2 ell digit polynomials (digits reduced mod q_l);
//   4. out_r = sum_{p, i} NTT(d_{p,i}) (.) rgsw[p ell + i][r], r in {0, 1}.
//
// GPU mapping: stage-level kernels (Sec. 4.1.2): each tree node is done on
// chip, so the 2 ell digit polynomials never leave the SMs; one launch per
// stage. A node is one thread-block cluster of 2L CTAs, CTA (p, l) on input
// polynomial p and limb l: one inverse NTT, the Dcp (the CRT takes the other
// limb's residues, pushed through distributed shared memory), the forward NTTs
// of its ell digits together (see ntt.cuh), and the products with its ell RGSW
// rows. The two CTAs of a limb then swap partial sums: CTA (p, l) finishes
// output polynomial p. Nothing is computed twice, and thread b owns slots /
// coefficients b + (N/8) e throughout. 64 registers, 66 KB of shared memory at
// N = 4096, two CTAs per SM, so that one's loads overlap the other's
// transforms. The multiply-accumulate keeps 64-bit sums of at most 3 terms
// below 16q * q < 2^60 (the forward transform's lazy range times a key
// residue) for one slot at a time. No pipe is full (issue slots 47% busy, ALU
// 38%, FMA 20%): between the CTA-wide barriers of a transform's rounds the warps
// wait for each other, for key rows and for the multiply pipe. 32 clients x 64
// ciphertexts 0.612 -> 0.474 ms against one CTA per limb doing both
// polynomials digit by digit (two cluster shapes, chosen by node count); 3
// clients x 16 at N = 2048, L = 1: 57 -> 33 us, and 24.6 us with overlapping stages.

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <map>
#include <mutex>

#include "common.cuh"
#include "internal.h"
#include "ntt.cuh"

namespace gpir {
namespace {

struct ColTorParams {
  ntt::Ring ring;
  const uint32_t *in;                             // [B][d_in][2][L][N]
  const uint32_t *rgsw;                           // [B][stages][2 ell][2][L][N]
  uint32_t *out;                                  // [B][d_in / 2][2][L][N]
  uint32_t d_in, nodes_per_client, stage, stages;
};

// EARLY: the grid may start while the stage before it finishes, so it waits for
// that stage and reads its results with ordinary loads instead of read-only ones.
template <int L, int LOGN, bool EARLY>
__global__ void __launch_bounds__(ntt::threads<LOGN>(), ntt::ctas_per_sm<LOGN>())
    coltor_stage_kernel(const __grid_constant__ ColTorParams p) {
  using namespace ntt;
  constexpr uint32_t N = 1u << LOGN, S = N >> 3, PN = padn(N);
  constexpr int D = digits<L>();
  extern __shared__ __align__(16) uint32_t sm[];
  const Ring &R = p.ring;
  const uint32_t rank = cluster_rank();
  const uint32_t h = rank % L, pp = rank / L;      // this CTA's limb, and its input and output polynomial
  const uint32_t b = threadIdx.x;
  const bool act = b < S;
  const Limb &T = R.limb[h];
  const uint32_t q = T.q, ell = R.ell;
  uint32_t *work = sm;                             // [D][PN]: transforms; the last one also receives residues
  uint32_t *part = sm + D * PN + b;                // [N]: the other polynomial's partial sums

  const uint32_t node = blockIdx.x / (2 * L);
  const uint32_t c = node / p.nodes_per_client, k = node % p.nodes_per_client;
  constexpr size_t ctw = (size_t)2 * L * N;
  const uint32_t *lo = p.in + ((size_t)c * p.d_in + 2 * k) * ctw + (size_t)(pp * L + h) * N + b;
  const uint32_t *hi = lo + ctw;
  const uint32_t *row = p.rgsw + (((size_t)c * p.stages + p.stage) * 2 + pp) * ell * ctw + (size_t)h * N + b;
  const auto ld_in = [](const uint32_t *x) { return EARLY ? *x : __ldg(x); };
  cluster_arrive_relaxed();   // this CTA runs: its peers may push into it after the wait

  // 1. hi - lo on the owned slots of (pp, h), then its inverse NTT
  uint32_t a[1][8];
  uint2 w[7];
  if constexpr (EARLY) wait_for_previous_stage();
  else let_next_stage_start();
  if (act) {
    inv_first_twiddles<LOGN>(w, T, b);
#pragma unroll
    for (int e = 0; e < 8; ++e) a[0][e] = ld_in(hi + e * S) - ld_in(lo + e * S) + q;
  }
  inverse<LOGN>(a, work, w, T, b, act);
  cluster_wait();

  // 2. the other limb's residues of the owned coefficients, and the digits.
  // They arrive where this thread's first forward round will write, so no
  // other thread can overwrite them before they are read.
  uint32_t *inbox = work + (D - 1) * PN + pad(b);
  if constexpr (L > 1) {
    if (act) {
      const uint32_t to = peer_addr(inbox, rank ^ 1u);
#pragma unroll
      for (uint32_t kk = 0; kk < 8; ++kk) st_peer(to + 4 * pad(kk * S), a[0][kk]);
    }
    cluster_arrive();
    cluster_wait();
  }
  uint32_t d[D][8];
  if (act) {
#pragma unroll
    for (uint32_t kk = 0; kk < 8; ++kk) {
      const uint32_t own = a[0][kk], other = L > 1 ? inbox[pad(kk * S)] : 0u;
      uint32_t x[D];
      dcp_digits<L>(R, T, h == 0 ? own : other, h == 0 ? other : own, x);
#pragma unroll
      for (int i = 0; i < D; ++i) d[i][kk] = x[i];
    }
  }

  // 3. forward NTT of the digits, products with RGSW rows pp ell + i
  {
    uint32_t *bufs[D];
#pragma unroll
    for (int i = 0; i < D; ++i) bufs[i] = work + i * PN;
    forward<LOGN, D>(d, bufs, T, b, act);
  }
  const auto sum = [&](uint32_t r, uint32_t e) {
    uint64_t acc = 0;
#pragma unroll
    for (uint32_t i = 0; i < D; ++i)   // absent digits are zero: row 0 stands in for theirs
      acc += (uint64_t)d[i][e] * __ldg(row + (size_t)(((i < ell ? i : 0u) * 2 + r) * L) * N + e * S);
    return acc;
  };

  // 4. out_pp = lo_pp + both polynomials' sums for it, limb h
  if (act) {
    const uint32_t to = peer_addr(part, h + L * (pp ^ 1u));
#pragma unroll
    for (uint32_t e = 0; e < 8; ++e) st_peer(to + 4 * e * S, red64(sum(pp ^ 1u, e), T));
  }
  cluster_arrive();
  uint64_t own[8];
  if (act) {
#pragma unroll
    for (uint32_t e = 0; e < 8; ++e) own[e] = sum(pp, e) + ld_in(lo + e * S);
  }
  cluster_wait();
  if (act) {
    uint32_t *out = p.out + ((size_t)c * p.nodes_per_client + k) * ctw + (size_t)(pp * L + h) * N + b;
#pragma unroll
    for (uint32_t e = 0; e < 8; ++e) out[e * S] = csub4(red64(own[e] + part[e * S], T), q);
  }
}

template <int L, int LOGN>
constexpr size_t coltor_smem() {
  constexpr uint32_t N = 1u << LOGN, PN = ntt::padn(N);
  return (size_t)(ntt::digits<L>() * PN + N) * 4;
}

std::mutex g_ct_mu;
std::map<std::pair<int, cudaStream_t>, std::pair<uint32_t *, size_t>> g_ct_ws;

int get_workspace(int dev, cudaStream_t s, size_t words, uint32_t **out) {
  auto &w = g_ct_ws[std::make_pair(dev, s)];
  if (w.second < words) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone) return GPIR_EINVAL;
    if (w.first) {
      cudaStreamSynchronize(s);
      cudaFree(w.first);
      w.first = nullptr;
      w.second = 0;
    }
    cudaError_t e = dev_malloc(reinterpret_cast<void **>(&w.first), words * 4);
    if (e != cudaSuccess) {
      w.first = nullptr;
      return set_cuda_error(e);
    }
    w.second = words;
  }
  *out = w.first;
  return GPIR_OK;
}

bool g_attr_done[64][ntt::MAX_LIMBS][ntt::MAX_LOGN + 1] = {};

// One stage: one cluster of 2L CTAs per node (polynomial x limb). A stage that
// the chip holds at once is bound by its launch and its chain of barriers and
// starts while the one before it finishes (3 clients x 16 at N = 2048, L = 1:
// 32.8 -> 24.6 us for the four stages); in larger ones the read-only loads are
// worth more (all stages early: 32 clients x 64 at N = 4096, 472 -> 484 us).
template <int L, int LOGN>
int launch_stage(const ColTorParams &p, unsigned nodes, int dev, cudaStream_t s) {
  if (dev < 0 || dev >= 64) return GPIR_EINVAL;
  const size_t smem = coltor_smem<L, LOGN>();
  if (!g_attr_done[dev][L - 1][LOGN]) {
    cudaError_t e = cudaFuncSetAttribute(coltor_stage_kernel<L, LOGN, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(coltor_stage_kernel<L, LOGN, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)smem);
    if (e != cudaSuccess) return set_cuda_error(e);
    g_attr_done[dev][L - 1][LOGN] = true;
  }
  // stage 0 follows work that is not this call's
  const bool early = p.stage > 0 && (uint64_t)nodes * 2 * L <= (uint64_t)ntt::ctas_per_sm<LOGN>() * sm_count();
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(nodes * 2 * L);
  cfg.blockDim = dim3(ntt::threads<LOGN>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2 * L;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = early ? 2 : 1;
  const cudaError_t e = early ? cudaLaunchKernelEx(&cfg, coltor_stage_kernel<L, LOGN, true>, p)
                              : cudaLaunchKernelEx(&cfg, coltor_stage_kernel<L, LOGN, false>, p);
  return e == cudaSuccess ? GPIR_OK : set_cuda_error(e);
}

template <int L>
int launch_stage_n(const ColTorParams &p, unsigned nodes, int dev, cudaStream_t s) {
  switch (p.ring.logn) {
    case 4: return launch_stage<L, 4>(p, nodes, dev, s);
    case 5: return launch_stage<L, 5>(p, nodes, dev, s);
    case 6: return launch_stage<L, 6>(p, nodes, dev, s);
    case 7: return launch_stage<L, 7>(p, nodes, dev, s);
    case 8: return launch_stage<L, 8>(p, nodes, dev, s);
    case 9: return launch_stage<L, 9>(p, nodes, dev, s);
    case 10: return launch_stage<L, 10>(p, nodes, dev, s);
    case 11: return launch_stage<L, 11>(p, nodes, dev, s);
    case 12: return launch_stage<L, 12>(p, nodes, dev, s);
    default: return GPIR_ENOTSUP;
  }
}

}  // namespace
}  // namespace gpir

extern "C" int gpir_coltor_gadget_digits(const gpir_params_t *params) {
  if (!params) return GPIR_EINVAL;
  unsigned __int128 Q = 1;
  for (uint32_t l = 0; l < params->num_limbs; ++l) Q *= params->primes[l];
  uint32_t bits = 0;
  for (unsigned __int128 v = Q - 1; v; v >>= 1) ++bits;
  return (int)((bits + gpir::ntt::LOG_BASE - 1) / gpir::ntt::LOG_BASE);
}

extern "C" int gpir_coltor(const gpir_params_t *params, uint32_t batch, uint32_t d1, const uint32_t *ct_dev,
                           const uint32_t *rgsw_dev, uint32_t *out_dev, void *stream) {
  using namespace gpir;
  // every argument is checked here, on the host, before any CUDA call
  if (!params || !ct_dev || !rgsw_dev || !out_dev || batch == 0 || d1 < 2 || (d1 & (d1 - 1)) != 0)
    return GPIR_EINVAL;
  if (params->num_limbs < 1 || params->num_limbs > ntt::MAX_LIMBS || params->n < ntt::MIN_N || params->n > ntt::MAX_N)
    return GPIR_ENOTSUP;
  {
    const size_t ctw = (size_t)2 * params->num_limbs * params->n * 4;
    const uintptr_t i0 = (uintptr_t)ct_dev, i1 = i0 + (size_t)batch * d1 * ctw;
    const uintptr_t o0 = (uintptr_t)out_dev, o1 = o0 + batch * ctw;
    if (i0 < o1 && o0 < i1) return GPIR_EINVAL;   // the last stage reads ct_dev's results while writing out_dev
  }
  ntt::Ring ring;
  int rc = ring_tables(params, &ring);
  if (rc != GPIR_OK) return rc;
  const uint32_t L = ring.L, N = ring.N;
  cudaStream_t s = (cudaStream_t)stream;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return set_cuda_error(e);
  std::lock_guard<std::mutex> lk(g_ct_mu);
  uint32_t stages = 0;
  while ((1u << stages) < d1) ++stages;
  const size_t ct_words = (size_t)2 * L * N;
  // ping-pong buffers for the intermediate stages: d1/2 and d1/4 ciphertexts per client
  uint32_t *ws = nullptr;
  const size_t half = (size_t)batch * (d1 / 2) * ct_words;
  if (stages > 1) {
    rc = get_workspace(dev, s, half + half / 2, &ws);
    if (rc != GPIR_OK) return rc;
  }
  ColTorParams p;
  memset(&p, 0, sizeof(p));
  p.ring = ring;
  p.rgsw = rgsw_dev;
  p.stages = stages;
  const uint32_t *in = ct_dev;
  uint32_t d_in = d1;
  for (uint32_t st = 0; st < stages; ++st) {
    uint32_t *dst = (st + 1 == stages) ? out_dev : (st % 2 == 0 ? ws : ws + half);
    p.in = in;
    p.out = dst;
    p.d_in = d_in;
    p.stage = st;
    p.nodes_per_client = d_in / 2;
    const unsigned nodes = batch * (d_in / 2);
    const int tr = trace_begin("coltor_stage", s);
    rc = L == 1 ? launch_stage_n<1>(p, nodes, dev, s) : launch_stage_n<2>(p, nodes, dev, s);
    trace_end(tr, s);
    if (rc != GPIR_OK) return rc;
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(e);
    in = dst;
    d_in /= 2;
  }
  return GPIR_OK;
}
