// ExpandQuery: the query-expansion tree before RowSel (GPIR paper Sec. 2.2,
// "ExpandQuery"), with the homomorphic substitution Subs of Sec. 2.5.1.
//
// For every client, J stages turn its query ciphertext into 2^J ciphertexts
// (the first n_out are kept). Node k of stage j takes ciphertext c = list[k]
// and writes
//     list[k]       = c + t
//     list[k + 2^j] = X^(-2^j) (c - t),     t = Subs(c, N/2^j + 1, evk_j).
// Subs(ct = (a, b), k): the automorphism tau_k (X -> X^k) of both polynomials,
// then key switching with Dcp on tau_k(a) only:
//     t = ( sum_i NTT(d_i) (.) evk[i][0],  tau_k(b) + sum_i NTT(d_i) (.) evk[i][1] ),
// d_i the balanced base-2^22 digits of the centred CRT value of tau_k(a)'s
// coefficients (inverse NTT first, forward NTT of each digit polynomial after).
//
// In the NTT domain tau_k is a permutation of the slots: slot s of tau_k(A)
// is A[s'] with 2s'+1 = (2s+1) k mod 2N, so the kernel gathers tau_k(a) and
// tau_k(b) while it loads them. The slot values of X^(-2^j) are
// psi^-((2s+1) 2^j mod 2N), read from a table.
//
// GPU mapping: stage-level kernels (Sec. 4.1.2), one launch per stage, the
// cluster shape chosen per stage (Sec. 4.4):
//   - expand_stage_kernel: one thread-block cluster of L CTAs per tree node,
//     CTA l on limb l; the CRT of the Dcp takes the other limb's residues,
//     pushed through distributed shared memory. The limb's two polynomials are
//     brought into shared memory whole: tau(a) and tau(b) are gathers of odd
//     slot stride, which shared memory serves without bank conflicts (from
//     global memory each gather of a warp touched 32 lines), and the same copy
//     serves c's own slots at the end. All digit polynomials go through the
//     forward transform together (see ntt.cuh), and the multiply-accumulate
//     starts when they are done, so its 64-bit sums live for one slot at a
//     time: 64 registers, 82 KB of shared memory at N = 4096, two CTAs per SM;
//     2420 warp instructions a warp and node (3440 when each digit had its own
//     transform and reduced after every round): 32 clients, 274 outputs: 2.90 ->
//     1.96 ms. No pipe is full (issue slots 51% busy, ALU 37%, FMA 21%): between
//     the CTA-wide barriers of a transform's rounds the warps wait for each
//     other, for key rows and for the multiply pipe;
//   - expand_split_kernel: for stages with few nodes, L digits CTAs per node
//     (limb x digit), each repeating the inverse NTT and doing one digit.
// The tree runs in place in the output array: stage j reads list[k], k < 2^j,
// and writes list[k] and list[k + 2^j]; each CTA that writes reads only its
// limb of list[k], and has all of it in shared memory before it writes. (In
// the split kernel the cluster barriers order every CTA's read of tau(a)
// before the writes.) Only
// the outputs with index < n_out are computed at any stage (an intermediate
// list[k] feeds final outputs k, k + 2^(j+1), ..., so k < n_out is exactly the
// condition for it to be needed).

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <mutex>

#include "common.cuh"
#include "internal.h"
#include "ntt.cuh"
#include "tcgen05.cuh"

namespace gpir {
namespace {

struct ExpandParams {
  ntt::Ring ring;
  const uint32_t *query;                          // [B][2][L][N] (read by stage 0)
  const uint32_t *evk;                            // [B][J][ell][2][L][N]
  uint32_t *out;                                  // [B][n_out][2][L][N]
  uint32_t batch, n_out, J, stage, nodes;         // nodes = min(2^stage, n_out) per client
  uint32_t ksub;                                  // N / 2^stage + 1
  uint32_t bulk;                                  // inputs are 16-byte aligned: bulk copies
  unsigned int *err;
};

// One node: its client and index, inputs and outputs.
struct ExpandNode {
  const uint32_t *in, *evk;
  uint32_t *out0, *out1;
  bool has1;
};

template <int L, int LOGN>
__device__ __forceinline__ ExpandNode expand_node(const ExpandParams &p, uint32_t node) {
  constexpr uint32_t ctw = 2 * L << LOGN;
  const uint32_t c = node / p.nodes, k = node % p.nodes, k1 = k + (1u << p.stage);
  uint32_t *list = p.out + (size_t)c * p.n_out * ctw;
  ExpandNode n;
  n.in = p.stage == 0 ? p.query + (size_t)c * ctw : list + (size_t)k * ctw;
  n.out0 = list + (size_t)k * ctw;
  n.out1 = list + (size_t)k1 * ctw;
  n.has1 = k1 < p.n_out;
  n.evk = p.evk + ((size_t)c * p.J + p.stage) * p.ring.ell * ctw;
  return n;
}

// Limb h of the node's polynomials a and b into shared memory (a at `stage`,
// b at `stage` + N), visible to the whole CTA on return.
template <int L, int LOGN>
__device__ __forceinline__ void expand_load(const ExpandParams &p, const ExpandNode &n, uint32_t h, uint32_t *stage,
                                            uint64_t *bar) {
  constexpr uint32_t N = 1u << LOGN;
  if (p.bulk) {
    if (threadIdx.x == 0) {
      mbar_init(bar, 1);
      fence_mbar_init();
      mbar_arrive_expect_tx(bar, 8 * N);
      bulk_g2s(stage, n.in + (size_t)h * N, 4 * N, bar);
      bulk_g2s(stage + N, n.in + (size_t)(L + h) * N, 4 * N, bar);
    }
    __syncthreads();
    // on expiry the copies may still be in flight: one more bounded wait
    if (!mbar_wait_bounded(bar, 0, p.err, kErrTmaWait)) mbar_wait_bounded(bar, 0, nullptr, 0);
  } else {
    for (uint32_t s = threadIdx.x; s < N; s += blockDim.x) {
      stage[s] = n.in[(size_t)h * N + s];
      stage[N + s] = n.in[(size_t)(L + h) * N + s];
    }
    __syncthreads();
  }
}

// Slot of A that holds slot b of tau(A) (2 src + 1 = (2b + 1) ksub mod 2N), and
// the step of src from slot b + (N/8) e to the next e.
template <int LOGN>
__device__ __forceinline__ void tau_slots(uint32_t ksub, uint32_t b, uint32_t &src, uint32_t &step) {
  constexpr uint32_t N = 1u << LOGN;
  src = (b * ksub + (ksub >> 1)) & (N - 1);
  step = ((N >> 3) * ksub) & (N - 1);
}

// The node's outputs on limb h from t = (a', b') without tau(b): out0 = c + t
// and out1 = X^(-2^j) (c - t) on the owned slots. sum(r, e) returns
// (64-bit) component r of t at slot b + (N/8) e. With s = c + t in [0, 4q),
// c - t is 2c - s.
template <int L, int LOGN, class OwnA, class Sum>
__device__ __forceinline__ void expand_outputs(const ExpandParams &p, const ExpandNode &n, uint32_t h, uint32_t b,
                                               const uint32_t *pb, const OwnA &own_a, const Sum &sum) {
  using namespace ntt;
  constexpr uint32_t N = 1u << LOGN, S = N >> 3, MASK2N = 2 * N - 1;
  const Limb &T = p.ring.limb[h];
  const uint32_t q = T.q;
  uint32_t src, step;
  tau_slots<LOGN>(p.ksub, b, src, step);
  const uint32_t e0 = ((2 * b + 1) << p.stage) & MASK2N;
  uint2 m = __ldg(T.mono + e0);
  const bool early = p.stage < 3;
#pragma unroll
  for (uint32_t e = 0; e < 8; ++e) {
    const uint32_t s = b + e * S;
    // the exponent (2s + 1) 2^j mod 2N does not depend on e from stage 3 on
    if (e > 0 && early) m = __ldg(T.mono + ((e0 + (2 * S * e << p.stage)) & MASK2N));
    const uint32_t tb = pb[src];
    src = (src + step) & (N - 1);
#pragma unroll
    for (uint32_t r = 0; r < 2; ++r) {
      const uint32_t c = r == 0 ? own_a(e) : pb[s];
      const uint32_t x = red64(sum(r, e) + (r == 0 ? c : c + tb), T);
      n.out0[(size_t)(r * L + h) * N + s] = csub4(x, q);
      if (n.has1) n.out1[(size_t)(r * L + h) * N + s] = shoup(2 * c + 4 * q - x, m, q);
    }
  }
}

// Persistent: cluster i runs nodes i, i + clusters, ... Polynomial a of the next
// node and b of the current one are copied while the current node computes, so
// only the first node waits for its load.
template <int L, int LOGN>
__global__ void __launch_bounds__(ntt::threads<LOGN>(), ntt::ctas_per_sm<LOGN>())
    expand_stage_kernel(const __grid_constant__ ExpandParams p) {
  using namespace ntt;
  constexpr uint32_t N = 1u << LOGN, S = N >> 3, PN = padn(N);
  constexpr int D = digits<L>();
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ uint64_t bar[2];                      // a landed, b landed
  const uint32_t h = L > 1 ? ntt::cluster_rank() : 0u;  // this CTA's limb
  const uint32_t b = threadIdx.x;
  const bool act = b < S;
  const Limb &T = p.ring.limb[h];
  uint32_t *pa = sm, *pb = sm + N;                 // [N] each: a, b on limb h
  uint32_t *work = sm + 2 * N;                     // [D][PN]: transforms; the last one also receives residues
  const uint32_t total = p.nodes * p.batch, stride = gridDim.x / L;
  if constexpr (L > 1) cluster_arrive_relaxed();   // this CTA runs: its peer may push into it after the wait
  if (b == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
  }
  wait_for_previous_stage();
  if (b == 0 && p.bulk) {
    mbar_arrive_expect_tx(&bar[0], 4 * N);
    bulk_g2s(pa, expand_node<L, LOGN>(p, blockIdx.x / L).in + (size_t)h * N, 4 * N, &bar[0]);
  }
  __syncthreads();
  uint32_t ph = 0;
  for (uint32_t i = blockIdx.x / L; i < total; i += stride, ph ^= 1) {
    const ExpandNode node = expand_node<L, LOGN>(p, i);
    uint2 w[7];
    if (act) inv_first_twiddles<LOGN>(w, T, b);
    if (p.bulk) {
      // on expiry the copy may still be in flight: one more bounded wait
      if (!mbar_wait_bounded(&bar[0], ph, p.err, kErrTmaWait)) mbar_wait_bounded(&bar[0], ph, nullptr, 0);
    } else {
      __syncthreads();   // the previous node's b has been read
      for (uint32_t s = b; s < N; s += blockDim.x) {
        pa[s] = node.in[(size_t)h * N + s];
        pb[s] = node.in[(size_t)(L + h) * N + s];
      }
      __syncthreads();
    }

    // 1. tau(a) on the owned slots, then its inverse NTT
    uint32_t a[1][8];
    if (act) {
      uint32_t src, step;
      tau_slots<LOGN>(p.ksub, b, src, step);
#pragma unroll
      for (uint32_t e = 0; e < 8; ++e) {
        a[0][e] = pa[src];
        src = (src + step) & (N - 1);
      }
    }
    // (no barrier since the previous node's transform: it read what this thread writes first)
    inverse<LOGN>(a, work, w, T, b, act);
    if (b == 0 && p.bulk) {
      // every thread has read a, and the previous node's b, before the barriers of the transform
      mbar_arrive_expect_tx(&bar[1], 4 * N);
      bulk_g2s(pb, node.in + (size_t)(L + h) * N, 4 * N, &bar[1]);
      if (i + stride < total) {
        mbar_arrive_expect_tx(&bar[0], 4 * N);
        bulk_g2s(pa, expand_node<L, LOGN>(p, i + stride).in + (size_t)h * N, 4 * N, &bar[0]);
      }
    }

    // 2. the other limb's residues of the owned coefficients, and the digits.
    // They arrive where this thread's first forward round will write, so no
    // other thread can overwrite them before they are read.
    uint32_t *inbox = work + (D - 1) * PN + pad(b);
    if constexpr (L > 1) {
      cluster_wait();
      if (act) {
        const uint32_t to = peer_addr(inbox, h ^ 1u);
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) st_peer(to + 4 * pad(k * S), a[0][k]);
      }
      cluster_arrive();
      cluster_wait();
    }
    uint32_t d[D][8];
    if (act) {
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) {
        const uint32_t own = a[0][k], other = L > 1 ? inbox[pad(k * S)] : 0u;
        uint32_t x[D];
        dcp_digits<L>(p.ring, T, h == 0 ? own : other, h == 0 ? other : own, x);
#pragma unroll
        for (int j = 0; j < D; ++j) d[j][k] = x[j];
      }
    }

    // 3. forward NTT of the digits, multiply-accumulate with the key rows, outputs
    const uint32_t *row = node.evk + (size_t)h * N + b;
    const uint32_t ell = p.ring.ell;
    {
      uint32_t *bufs[D];
#pragma unroll
      for (int j = 0; j < D; ++j) bufs[j] = work + j * PN;
      forward<LOGN, D>(d, bufs, T, b, act);
    }
    if (p.bulk && !mbar_wait_bounded(&bar[1], ph, p.err, kErrTmaWait)) mbar_wait_bounded(&bar[1], ph, nullptr, 0);
    if (act) {
      expand_outputs<L, LOGN>(
          p, node, h, b, pb, [&](uint32_t e) { return node.in[(size_t)h * N + b + e * S]; },
          [&](uint32_t r, uint32_t e) {
            uint64_t acc = 0;
#pragma unroll
            for (uint32_t j = 0; j < D; ++j)   // absent digits are zero: row 0 stands in for theirs
              acc += (uint64_t)d[j][e] * __ldg(row + (size_t)(((j < ell ? j : 0u) * 2 + r) * L) * N + e * S);
            return acc;
          });
    }
    if constexpr (L > 1)
      if (i + stride < total) cluster_arrive_relaxed();   // done with this node's buffers
  }
}

template <int L, int LOGN>
constexpr size_t expand_smem() {
  constexpr uint32_t N = 1u << LOGN, PN = ntt::padn(N);
  return (size_t)(2 * N + ntt::digits<L>() * PN) * 4;
}

// The same node for the stages with few nodes (the early ones): one cluster of
// L D CTAs (D = digits<L>()), CTA (l, g) on limb l and digit g. Every CTA takes
// the inverse NTT of tau(a) (repeated across g: free while the GPU is not
// full), then one digit's forward NTT and multiply-accumulate; the digit-0 CTA
// of each limb receives the other digits' partial sums and writes the node's
// outputs.
template <int L, int LOGN>
__global__ void __launch_bounds__(ntt::threads<LOGN>(), 1)
    expand_split_kernel(const __grid_constant__ ExpandParams p) {
  using namespace ntt;
  constexpr uint32_t N = 1u << LOGN, S = N >> 3, PN = padn(N);
  constexpr int D = digits<L>();
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ uint64_t bar;
  const uint32_t rank = ntt::cluster_rank();
  const uint32_t h = rank % L, g = rank / L;       // this CTA's limb and digit
  const uint32_t b = threadIdx.x;
  const bool act = b < S;
  const Limb &T = p.ring.limb[h];
  const uint32_t ell = p.ring.ell;
  uint32_t *stage = sm;                            // [2][N]: a, b on limb h
  uint32_t *work = sm + 2 * N;                     // [PN]: transforms
  uint32_t *inbox = work + PN + pad(b);            // [PN]: the other limb's residues
  uint32_t *sums = work + 2 * PN;                  // [D - 1][2 N]: the other digits' partial sums (digit-0 CTAs)
  const ExpandNode node = expand_node<L, LOGN>(p, blockIdx.x / (L * D));
  cluster_arrive_relaxed();
  // the key values this thread multiplies with, early: they come from DRAM
  uint32_t key[2][8];
  if (act) {
    const uint32_t *row = node.evk + (size_t)((g < ell ? g : 0u) * 2 * L + h) * N + b;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int e = 0; e < 8; ++e) key[r][e] = __ldg(row + (size_t)r * L * N + e * S);
  }
  uint2 w[7];
  if (act) inv_first_twiddles<LOGN>(w, T, b);
  wait_for_previous_stage();
  expand_load<L, LOGN>(p, node, h, stage, &bar);

  // 1. tau(a) on the owned slots of limb h, then its inverse NTT
  uint32_t a[1][8];
  if (act) {
    uint32_t src, step;
    tau_slots<LOGN>(p.ksub, b, src, step);
#pragma unroll
    for (uint32_t e = 0; e < 8; ++e) {
      a[0][e] = stage[src];
      src = (src + step) & (N - 1);
    }
  }
  inverse<LOGN>(a, work, w, T, b, act);
  cluster_wait();   // every CTA of the cluster runs
  if constexpr (L > 1) {
    if (act) {
      const uint32_t to = peer_addr(inbox, (h ^ 1u) + L * g);
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k) st_peer(to + 4 * pad(k * S), a[0][k]);
    }
    cluster_arrive();
    cluster_wait();
  }

  // 2. digit g of the owned coefficients, forward NTT, product with key row g
  uint32_t d[1][8];
  if (act) {
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) {
      const uint32_t own = a[0][k], other = L > 1 ? inbox[pad(k * S)] : 0u;
      uint32_t x[D];
      dcp_digits<L>(p.ring, T, h == 0 ? own : other, h == 0 ? other : own, x);
      d[0][k] = x[0];
#pragma unroll
      for (uint32_t i = 1; i < D; ++i) d[0][k] = g == i ? x[i] : d[0][k];
    }
  }
  {
    uint32_t *const bufs[1] = {work};
    forward<LOGN, 1>(d, bufs, T, b, act);
  }
  if (g > 0 && act) {
    const uint32_t to = peer_addr(sums + (g - 1) * 2 * N + b, h);
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int e = 0; e < 8; ++e) st_peer(to + 4 * (r * N + e * S), red64((uint64_t)d[0][e] * key[r][e], T));
  }
  cluster_arrive();   // the partial sums have arrived after this pair
  cluster_wait();

  // 3. digit-0 CTAs: the node's outputs on limb h
  if (g > 0 || !act) return;
  expand_outputs<L, LOGN>(
      p, node, h, b, stage + N, [&](uint32_t e) { return stage[b + e * S]; },
      [&](uint32_t r, uint32_t e) {
        uint64_t acc = (uint64_t)d[0][e] * key[r][e];
#pragma unroll
        for (uint32_t i = 1; i < D; ++i) acc += sums[(i - 1) * 2 * N + r * N + e * S + b];
        return acc;
      });
}

template <int L, int LOGN>
constexpr size_t expand_split_smem() {
  constexpr uint32_t N = 1u << LOGN, PN = ntt::padn(N);
  return (size_t)(2 * N + 2 * PN + (ntt::digits<L>() - 1) * 2 * N) * 4;
}

bool g_ex_attr_done[64][2][ntt::MAX_LIMBS][ntt::MAX_LOGN + 1] = {};
std::mutex g_ex_mu;

// One stage. split: one cluster of L digits<L>() CTAs per node (limb x digit), else one
// cluster of L CTAs per node (limb).
template <int L, int LOGN>
int launch_stage(const ExpandParams &p, unsigned nodes, bool split, int dev, cudaStream_t s) {
  if (dev < 0 || dev >= 64) return GPIR_EINVAL;
  const size_t smem = split ? expand_split_smem<L, LOGN>() : expand_smem<L, LOGN>();
  void (*kern)(ExpandParams) = split ? expand_split_kernel<L, LOGN> : expand_stage_kernel<L, LOGN>;
  {
    std::lock_guard<std::mutex> lk(g_ex_mu);
    if (!g_ex_attr_done[dev][split][L - 1][LOGN]) {
      const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return set_cuda_error(e);
      g_ex_attr_done[dev][split][L - 1][LOGN] = true;
    }
  }
  const unsigned cl = split ? L * ntt::digits<L>() : L;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  // the limb form is persistent: as many clusters as the SMs hold
  const unsigned resident = (unsigned)(sm_count() * ntt::ctas_per_sm<LOGN>() / L);
  cfg.gridDim = dim3((split || nodes < resident ? nodes : resident) * cl);
  cfg.blockDim = dim3(ntt::threads<LOGN>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.stage > 0 ? 2 : 1;   // stage 0 follows work that is not this call's
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p);
  return e == cudaSuccess ? GPIR_OK : set_cuda_error(e);
}

template <int L>
int launch_stage_n(const ExpandParams &p, unsigned nodes, bool split, int dev, cudaStream_t s) {
  switch (p.ring.logn) {
    case 4: return launch_stage<L, 4>(p, nodes, split, dev, s);
    case 5: return launch_stage<L, 5>(p, nodes, split, dev, s);
    case 6: return launch_stage<L, 6>(p, nodes, split, dev, s);
    case 7: return launch_stage<L, 7>(p, nodes, split, dev, s);
    case 8: return launch_stage<L, 8>(p, nodes, split, dev, s);
    case 9: return launch_stage<L, 9>(p, nodes, split, dev, s);
    case 10: return launch_stage<L, 10>(p, nodes, split, dev, s);
    case 11: return launch_stage<L, 11>(p, nodes, split, dev, s);
    case 12: return launch_stage<L, 12>(p, nodes, split, dev, s);
    default: return GPIR_ENOTSUP;
  }
}

}  // namespace
}  // namespace gpir

extern "C" int gpir_expand_query(const gpir_params_t *params, uint32_t batch, uint32_t stages, uint32_t n_out,
                                 const uint32_t *query_dev, const uint32_t *evk_dev, uint32_t *out_dev,
                                 void *stream) {
  using namespace gpir;
  // every argument is checked here, on the host, before any CUDA call
  if (!params || !query_dev || !out_dev || batch == 0 || n_out == 0) return GPIR_EINVAL;
  if (stages > 0 && !evk_dev) return GPIR_EINVAL;
  if (params->num_limbs < 1 || params->num_limbs > ntt::MAX_LIMBS || params->n < ntt::MIN_N || params->n > ntt::MAX_N)
    return GPIR_ENOTSUP;
  uint32_t logn = 0;
  while ((1u << logn) < params->n) ++logn;
  // tau_k with k = N / 2^j + 1 is an automorphism (k odd) only for j < log2 N
  if (stages > logn || n_out > (1u << stages)) return GPIR_EINVAL;
  {
    const size_t ctw = (size_t)2 * params->num_limbs * params->n * 4;
    const uintptr_t q0 = (uintptr_t)query_dev, q1 = q0 + batch * ctw;
    const uintptr_t o0 = (uintptr_t)out_dev, o1 = o0 + (size_t)batch * n_out * ctw;
    if (q0 < o1 && o0 < q1) return GPIR_EINVAL;   // the tree runs in place in out_dev
  }
  ntt::Ring ring;
  int rc = ring_tables(params, &ring);
  if (rc != GPIR_OK) return rc;
  const uint32_t L = ring.L, N = ring.N;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t ct_words = (size_t)2 * L * N;
  if (stages == 0) {
    const cudaError_t e =
        cudaMemcpyAsync(out_dev, query_dev, (size_t)batch * ct_words * 4, cudaMemcpyDeviceToDevice, s);
    return e == cudaSuccess ? GPIR_OK : set_cuda_error(e);
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return set_cuda_error(e);
  ExpandParams p;
  memset(&p, 0, sizeof(p));
  p.ring = ring;
  p.query = query_dev;
  p.evk = evk_dev;
  p.out = out_dev;
  p.batch = batch;
  p.n_out = n_out;
  p.J = stages;
  p.bulk = (((uintptr_t)query_dev | (uintptr_t)out_dev) & 15u) == 0;
  p.err = device_error_word();
  for (uint32_t st = 0; st < stages; ++st) {
    p.stage = st;
    p.nodes = (1u << st) < n_out ? (1u << st) : n_out;
    p.ksub = (N >> st) + 1;
    const unsigned nodes = batch * p.nodes;
    // stage-aware choice (Sec. 4.4): the limb x digit split (which repeats the
    // inverse NTT per digit) when its clusters run at once, one CTA per SM, the
    // limb split otherwise. A cluster's CTAs share a GPC, so not every SM can be
    // used: 7/8 of them is below what fits. One stage at N = 4096, us, split /
    // limb: 12.7 / 14.6 up to 16 nodes, 14.1 / 14.7 at 22 and 23, but 20.9 / 14.6
    // at 24 and 25 (L = 2, 6 CTAs); 12.2 / 12.6 at 16 and equal at 30 to 38 (L = 1).
    const unsigned split_ctas = L * (L == 1 ? ntt::digits<1>() : ntt::digits<2>());
    const bool split = (uint64_t)nodes * split_ctas * 8 <= (uint64_t)sm_count() * 7;
    const int tr = trace_begin(split ? "expand_stage_split" : "expand_stage", s);
    rc = L == 1 ? launch_stage_n<1>(p, nodes, split, dev, s) : launch_stage_n<2>(p, nodes, split, dev, s);
    trace_end(tr, s);
    if (rc != GPIR_OK) return rc;
    e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(e);
  }
  return GPIR_OK;
}
