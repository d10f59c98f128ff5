// kvq_drift_metrics / kvq_drift_window: offline drift metrics on paired FP16
// and low-bit logits and the recovery-window rule (Sec. 4.1 "Adaptive
// recovery-window selection", Sec. 4.2 "Offline supervision and
// calibration").
//
// Per step (row) t, with p = softmax(z):
//   C(alpha)  the shortest prefix of the FP16 order (z_fp descending, lower
//             index first among equal values) whose mass reaches alpha; M_t
//             its size;
//   S         TopK(z_q, K), same order on z_q;
//   c_t       sum of p_fp over C and S;
//   d_loc     || p_fp / p_fp(U) - p_q / p_q(U) ||_2 over U = C union S;
//   y_t       d_loc > eps and c_t >= rho_c;
//   cov_t(k)  sum of p_fp over C and TopK(z_q, k), k = 1 .. k_max.
// K_b is the smallest k whose coverage averaged over the rows reaches rho_K.
//
// Two kernels.  The streaming kernel (below) takes every row with one CTA; a
// row that its guesses do not settle (thousands of nearly equal logits around
// a boundary, alpha = 1) it leaves to the general kernel, launched behind it,
// which takes any row with one cluster of 8 CTAs.  256 rows of 128256 on a
// GB300: 1050 us with the general kernel alone, 160 with both.  Launches of a
// few long rows go to the general kernel alone (launch_drift).
//
// The general kernel.  Each CTA stages an eighth of both logit rows in shared
// memory once (the only HBM read) and the CTAs combine their partial results
// through distributed shared memory:
//   1. maxima;
//   2. the FP16 boundary: a 2048-bin histogram of the depth (m - z) * 64
//      (count and mass per bin, the depth order is the FP16 order) and, in
//      the same pass, the normaliser S_fp = sum e^{z - m}, find the bin
//      where the prefix mass reaches alpha S_fp; that bin's elements are
//      sorted in one CTA and scanned for the exact element.  A bin with more
//      than 2048 elements is narrowed by histograms of its key range first;
//      a range of equal keys takes the lowest indices (counted per CTA in
//      index order);
//   3. the same selection by count on z_q gives the k_max-th element, then
//      the k_max best elements are gathered and sorted (the TopK order);
//   4. one pass over U: its masses and the sums of e_fp^2, e_fp e_q, e_q^2
//      (multiples of 2^-60), from which d_loc follows.
// A mass term e = expf(z - m) (fp32, in (0, 1]) is taken as an integer
// multiple of 2^-40 (round to nearest) and every mass sum is an exact 64-bit
// integer sum, the product sums likewise (Prod): the same numbers decide every
// comparison, in any order, no per-element fp64 arithmetic is needed, and a row
// has the same results in either kernel, in every run and beside any rows.

#include <float.h>

#include <atomic>

#include "common.cuh"

namespace kvq {
namespace {

constexpr int kT = 512;              // threads per CTA
constexpr int kW = kT / 32;
constexpr int kCl = 8;               // CTAs per row (one cluster)
constexpr int kSlice = 20480;        // logits per CTA and array: vocab <= 8 * kSlice
constexpr int kBins = 2048;          // histogram bins
constexpr int kCap = 2048;           // largest boundary set sorted in one CTA
constexpr int kMaxKcov = 256;        // longest coverage curve
constexpr float kDepthScale = 64.0f; // bins per unit of depth m - z
constexpr int kSlots = 32;           // exchange slots (one per cluster exchange)
constexpr int kXw = 4;               // words per exchange
typedef unsigned long long u64;

struct Sm {
  float zf[kSlice];
  float zq[kSlice];
  uint32_t hc[kBins];               // bin counts
  uint32_t hm[3][kBins];            // bin masses: 14-bit chunks of the fixed-point terms
  u64 buf[kCap];                    // rank 0: boundary set / TopK set
  u64 xd[kSlots][kXw];              // per-CTA partials read by the peers
  uint32_t xu[kSlots][2];
  uint32_t res_u[8];                // rank 0: results of a selection
  u64 res_q[4];                     // the boundary bin's owner: its result
  uint32_t nbuf;                    // rank 0: fill count of buf
  u64 rq[kW];
  // merged histogram of this CTA's eighth of the bins, and exchange scratch
  uint32_t rc[kBins / kCl];
  u64 rm[kBins / kCl];
  u64 xin[kCl][kXw];                // values loaded from the eight CTAs
  u64 xin3[kCl][3 * kXw];           // the same for the three slots of a row's sums
  u64 wsel[kMaxKcov];               // coverage terms of the TopK list
  uint32_t ru[kW];
  float rf[kW];
};

// ---- cluster primitives (distributed shared memory) ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ float ld_peer_f32(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ u64 ld_peer_u64(uint32_t a) {
  u64 v;
  asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t ld_peer_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_peer_u64(uint32_t a, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
__device__ __forceinline__ void st_peer_u32(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atom_add_peer(uint32_t a, uint32_t v) {
  uint32_t old;
  asm volatile("atom.shared::cluster.add.u32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(v) : "memory");
  return old;
}

// Order-preserving key of a float (larger float, larger key; -0 as +0) and
// back.  Every key of a non-NaN float is > 0.
__device__ __forceinline__ uint32_t fkey(float x) {
  uint32_t u = __float_as_uint(x);
  if ((u << 1) == 0u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fval(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}
// A mass term e in [0, 1] as a multiple of 2^-40, rounded to nearest: e 2^20
// splits exactly into its integer part and a fraction whose 2^20 multiple
// fits a u32.
__device__ __forceinline__ u64 fix40(float e) {
  const float a = e * 1048576.0f;
  const uint32_t hi = (uint32_t)a;
  const uint32_t lo = __float2uint_rn((a - (float)hi) * 1048576.0f);
  return ((u64)hi << 20) + lo;
}
constexpr double kFix = 1099511627776.0;  // 2^40

// A sum of products of terms in [0, 1] as whole multiples of 2^-60, so that
// neither the order nor the split of the additions can change it (at most
// 2047 products a thread).  A product is p + r exactly; adding 8 rounds p to a
// multiple of 2^-20, adding 1.5 2^-17 rounds what is left of p, and r, to
// multiples of 2^-40, and 1.5 2^-37 the last rest to one of 2^-60.  The
// largest term of either row is 1 and belongs to U, so the sums of squares are
// at least 1.
struct Prod {
  uint32_t hi = 0u, mid = 0u, low = 0u;  // in units of 2^-20, 2^-40 and 2^-60
  __device__ __forceinline__ void add(float a, float b) {
    constexpr float kMid = 1.5f / 131072.0f, kLow = 1.5f / 137438953472.0f;
    constexpr uint32_t kMidBits = 0x37400000u, kLowBits = 0x2d400000u;
    const float p = __fmul_rn(a, b), r = __fmaf_rn(a, b, -p);
    const float h = __fadd_rn(p, 8.0f);
    const float p1 = __fsub_rn(p, __fsub_rn(h, 8.0f));
    const float m = __fadd_rn(p1, kMid), n = __fadd_rn(r, kMid);
    const float p2 = __fsub_rn(p1, __fsub_rn(m, kMid)), r2 = __fsub_rn(r, __fsub_rn(n, kMid));
    hi += __float_as_uint(h) - 0x41000000u;
    mid += (__float_as_uint(m) - kMidBits) + (__float_as_uint(n) - kMidBits);
    low += __float_as_uint(__fadd_rn(__fadd_rn(p2, r2), kLow)) - kLowBits;
  }
  __device__ __forceinline__ u64 coarse() const {  // multiples of 2^-40
    return ((u64)hi << 20) + (u64)(long long)(int)mid;
  }
  __device__ __forceinline__ u64 fine() const { return (u64)(long long)(int)low; }
};
__device__ __forceinline__ double prod_value(u64 coarse, u64 fine) {
  return ((double)(long long)coarse + (double)(long long)fine / 1048576.0) / kFix;
}
// The words of a row's sums over U, all whole numbers: count, masses A, B and C
// (see write_row), then coarse and fine parts of the sums of e_fp^2, e_fp e_q
// and e_q^2.
constexpr int kSumWords = 10;
__device__ __forceinline__ void warp_sums(u64 (&w)[kSumWords], u64* out) {  // by lane 0
#pragma unroll
  for (int o = 16; o; o >>= 1)
#pragma unroll
    for (int k = 0; k < kSumWords; ++k) w[k] += __shfl_xor_sync(0xffffffffu, w[k], o);
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int k = 0; k < kSumWords; ++k) out[k] = w[k];
  }
}

// (key, index) packed so that a larger word ranks first: key descending,
// index ascending.
__device__ __forceinline__ unsigned long long pack(uint32_t k, uint32_t i) {
  return ((unsigned long long)k << 32) | (0xffffffffu - i);
}
__device__ __forceinline__ uint32_t pk_key(unsigned long long w) { return (uint32_t)(w >> 32); }
__device__ __forceinline__ uint32_t pk_idx(unsigned long long w) {
  return 0xffffffffu - (uint32_t)w;
}

// Programmatic dependent launch (no-ops without the launch attribute).
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- block reductions (all threads get the result) ----
__device__ u64 block_sum_q(u64 v, Sm& s) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s.rq[threadIdx.x >> 5] = v;
  __syncthreads();
  u64 r = 0ull;
  for (int w = 0; w < kW; ++w) r += s.rq[w];
  return r;
}
__device__ float block_max_f(float v, Sm& s) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s.rf[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = -INFINITY;
  for (int w = 0; w < kW; ++w) r = fmaxf(r, s.rf[w]);
  return r;
}
__device__ uint32_t block_sum_u(uint32_t v, Sm& s) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s.ru[threadIdx.x >> 5] = v;
  __syncthreads();
  uint32_t r = 0u;
  for (int w = 0; w < kW; ++w) r += s.ru[w];
  return r;
}
__device__ uint32_t block_min_u(uint32_t v, Sm& s) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s.ru[threadIdx.x >> 5] = v;
  __syncthreads();
  uint32_t r = 0xffffffffu;
  for (int w = 0; w < kW; ++w) r = min(r, s.ru[w]);
  return r;
}
__device__ uint32_t block_max_u(uint32_t v, Sm& s) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s.ru[threadIdx.x >> 5] = v;
  __syncthreads();
  uint32_t r = 0u;
  for (int w = 0; w < kW; ++w) r = max(r, s.ru[w]);
  return r;
}

// Cluster-wide reductions of two values per CTA: each CTA publishes its
// partials in slot `slot`, and after the barrier every CTA combines all eight
// in rank order (identical results everywhere).
// Publish up to four words in slot `slot`; after the barrier threads load the
// eight CTAs' words in parallel into s.xin[rank][word].
__device__ void cluster_gather(Sm& s, int slot, u64 a, u64 b, u64 c = 0ull, u64 d = 0ull) {
  if (threadIdx.x == 0) {
    s.xd[slot][0] = a;
    s.xd[slot][1] = b;
    s.xd[slot][2] = c;
    s.xd[slot][3] = d;
  }
  cluster_sync();
  if (threadIdx.x < kXw * kCl)
    s.xin[threadIdx.x / kXw][threadIdx.x % kXw] =
        ld_peer_u64(peer_addr(&s.xd[slot][threadIdx.x % kXw], threadIdx.x / kXw));
  __syncthreads();
}
__device__ __forceinline__ void cluster_gather2(Sm& s, int slot, u64 a, u64 b) {
  cluster_gather(s, slot, a, b);
}
// op 0: (sum, sum); op 1: (min, max); op 2: (max, max) on float bits >= 0
__device__ void cluster_red2_u(Sm& s, int slot, uint32_t& a, uint32_t& b, int op) {
  cluster_gather2(s, slot, (u64)a, (u64)b);
  uint32_t ra = op == 1 ? 0xffffffffu : 0u, rb = 0u;
  for (int r = 0; r < kCl; ++r) {
    const uint32_t x = (uint32_t)s.xin[r][0];
    const uint32_t y = (uint32_t)s.xin[r][1];
    if (op == 0) {
      ra += x;
      rb += y;
    } else if (op == 1) {
      ra = min(ra, x);
      rb = max(rb, y);
    } else {
      ra = max(ra, x);
      rb = max(rb, y);
    }
  }
  __syncthreads();
  a = ra;
  b = rb;
}

// Bitonic sort of buf[0, n) descending (n <= kCap), padding with 0.  A step
// of distance j <= 16 stays inside the 32 consecutive elements that one warp
// handles, so only the longer steps need the block's barrier.
template <int kN>
__device__ void sort_desc(u64* buf, int n) {
  int P = 2;
  while (P < n) P <<= 1;
  __syncthreads();
  for (int i = n + threadIdx.x; i < P; i += kN) buf[i] = 0ull;
  __syncthreads();
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P; i += kN) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = buf[i], b = buf[ixj];
          const bool desc = (i & k) == 0;
          if (desc ? (a < b) : (a > b)) {
            buf[i] = b;
            buf[ixj] = a;
          }
        }
      }
      const int next = j > 1 ? j >> 1 : k;  // the next step's distance
      if (j > 16 || next > 16) __syncthreads();
      else __syncwarp();
    }
  __syncthreads();
}

struct Ctx {
  int n;          // logits in this CTA's slice
  uint32_t i0;    // global index of its first logit
  uint32_t rank;  // cluster rank
};

// Result of a selection: the element (key, index) at which the prefix of
// the order (key descending, index ascending) first reaches the target, and
// the prefix length.  all = the target is never reached (everything).
struct Pick {
  uint32_t key, idx, len;
  bool all;
};

// The bin where the prefix weight (count, or mass in fixed point) in bin
// order (bin 0 ranks first) reaches `target`, over the histograms of all
// eight CTAs.  CTA r merges bins [256 r, 256 r + 256) of the eight
// histograms and publishes their total; the CTA whose range holds the target
// finds the bin and publishes it.  If the total stays below the target: with
// `clamp` the last non-empty bin is taken, else false is returned (in every
// CTA alike).
// With `norm` set, each CTA's *norm holds its part of S_fp on entry and the
// target is ceil(alpha S_fp) over the cluster: *norm and target return it.
__device__ bool boundary_bin(Sm& s, const Ctx& cx, bool weighted, u64& target, int& slot, int& bin,
                             uint32_t& cnt_above, u64& w_above, uint32_t& cnt_bin,
                             bool clamp = false, u64* norm = nullptr, double alpha = 0.0) {
  constexpr int kR = kBins / kCl;  // bins per CTA range
  cluster_sync();                  // every CTA's histogram is complete
  const int t = threadIdx.x;
  __shared__ uint32_t part_c[kT];
  __shared__ u64 part_m[kT];
  {
    // thread t merges bin (t % kR) of its range from four of the CTAs
    const int b = (int)cx.rank * kR + (t % kR);
    const uint32_t r0 = (uint32_t)(t / kR) * (kCl / (kT / kR));
    uint32_t c = 0u, m0 = 0u, m1 = 0u, m2 = 0u;
#pragma unroll
    for (uint32_t r = 0; r < kCl / (kT / kR); ++r) {
      c += ld_peer_u32(peer_addr(&s.hc[b], r0 + r));
      if (weighted) {
        m0 += ld_peer_u32(peer_addr(&s.hm[0][b], r0 + r));
        m1 += ld_peer_u32(peer_addr(&s.hm[1][b], r0 + r));
        m2 += ld_peer_u32(peer_addr(&s.hm[2][b], r0 + r));
      }
    }
    part_c[t] = c;
    part_m[t] = weighted ? (u64)m0 + ((u64)m1 << 14) + ((u64)m2 << 28) : (u64)c;
  }
  __syncthreads();
  // exclusive prefix over this range's bins (warp scans, then warp totals)
  __shared__ uint32_t wtot_c[kR / 32];
  __shared__ u64 wtot_m[kR / 32];
  uint32_t c = 0u, ic = 0u;
  u64 m = 0ull, im = 0ull;
  if (t < kR) {
    c = part_c[t] + part_c[t + kR];
    m = part_m[t] + part_m[t + kR];
    s.rc[t] = c;
    s.rm[t] = m;
    ic = c;
    im = m;
    const int l = t & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t tc = __shfl_up_sync(0xffffffffu, ic, o);
      const u64 tm = __shfl_up_sync(0xffffffffu, im, o);
      if (l >= o) {
        ic += tc;
        im += tm;
      }
    }
    if (l == 31) {
      wtot_c[t >> 5] = ic;
      wtot_m[t >> 5] = im;
    }
  }
  __syncthreads();
  uint32_t tot_c = 0u;
  u64 tot_m = 0ull;
  for (int w = 0; w < kR / 32; ++w) {
    tot_c += wtot_c[w];
    tot_m += wtot_m[w];
  }
  uint32_t ex_c = ic - c;
  u64 ex_m = im - m;
  if (t < kR)
    for (int w = 0; w < (t >> 5); ++w) {
      ex_c += wtot_c[w];
      ex_m += wtot_m[w];
    }
  // range totals of all eight CTAs (and their S_fp parts), in rank order
  cluster_gather(s, slot++, (u64)tot_c, tot_m, norm ? *norm : 0ull);
  if (norm) {
    u64 sf = 0ull;
    for (int r = 0; r < kCl; ++r) sf += s.xin[r][2];
    *norm = sf;
    // prefix mass >= alpha S  <=>  prefix >= ceil(alpha S) in fixed point
    target = (u64)ceil(alpha * (double)sf);
  }
  u64 pre_m[kCl + 1];
  uint32_t pre_c[kCl + 1];
  pre_m[0] = 0ull;
  pre_c[0] = 0u;
  int owner = -1, last = -1;
  for (int r = 0; r < kCl; ++r) {
    pre_c[r + 1] = pre_c[r] + (uint32_t)s.xin[r][0];
    pre_m[r + 1] = pre_m[r] + s.xin[r][1];
    if (owner < 0 && pre_m[r] < target && target <= pre_m[r + 1] && s.xin[r][0] > 0ull) owner = r;
    if (s.xin[r][0] > 0ull) last = r;
  }
  __syncthreads();
  bool use_last = false;
  if (owner < 0) {
    if (!clamp || last < 0) {
      cluster_sync();  // peers finished reading this CTA's histogram (all return alike)
      return false;
    }
    owner = last;
    use_last = true;
  }
  if ((int)cx.rank == owner && t < kR) {
    const u64 wa = pre_m[owner] + ex_m;
    bool hit;
    if (use_last) {
      // the last non-empty bin of the range: no later bin has a count
      hit = c > 0u && ex_c + c == tot_c;
    } else {
      hit = c > 0u && wa < target && target <= wa + m;
    }
    if (hit) {
      s.res_q[0] = (u64)(owner * kR + t);
      s.res_q[1] = (u64)(pre_c[owner] + ex_c);
      s.res_q[2] = wa;
      s.res_q[3] = (u64)c;
    }
  }
  cluster_sync();
  if (t < 4) s.xin[t][0] = ld_peer_u64(peer_addr(&s.res_q[t], (uint32_t)owner));
  __syncthreads();
  bin = (int)s.xin[0][0];
  cnt_above = (uint32_t)s.xin[1][0];
  w_above = s.xin[2][0];
  cnt_bin = (uint32_t)s.xin[3][0];
  cluster_sync();  // every CTA read the owner's result; histograms may be rewritten
  return true;
}

// The n-th set element (1-based) in index order among this CTA's elements
// whose key equals `key` (array a), as a global index; the caller knows it is
// here.
__device__ uint32_t nth_tie(Sm& s, const Ctx& cx, const float* a, uint32_t key, uint32_t nth) {
  __shared__ uint32_t base_s, ans_s;
  if (threadIdx.x == 0) {
    base_s = 0u;
    ans_s = 0xffffffffu;
  }
  __syncthreads();
  for (int t0 = 0; t0 < cx.n; t0 += kT) {
    const int i = t0 + threadIdx.x;
    const bool hit = i < cx.n && fkey(a[i]) == key;
    const uint32_t bal = __ballot_sync(0xffffffffu, hit);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) s.ru[w] = __popc(bal);
    __syncthreads();
    uint32_t before = base_s;
    for (int v = 0; v < w; ++v) before += s.ru[v];
    const uint32_t rank_in = before + __popc(bal & ((1u << l) - 1u)) + 1u;
    if (hit && rank_in == nth) ans_s = cx.i0 + (uint32_t)i;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t tot = 0u;
      for (int v = 0; v < kW; ++v) tot += s.ru[v];
      base_s += tot;
    }
    __syncthreads();
  }
  return ans_s;
}

// The elements i of this CTA's slice with hit(i), as packed (key(i), index)
// words, appended to rank 0's buf: compacted in this CTA's histogram area
// (free once a selection's bin is known), then one remote reservation on
// rank 0's fill count and parallel remote stores.  Rank 0's nbuf must be
// zero, and visible through a cluster barrier, before the call.
template <typename Hit, typename Key>
__device__ void gather_to_rank0(Sm& s, const Ctx& cx, const Hit& hit, const Key& key) {
  __shared__ uint32_t lcount, lbase;
  u64* loc = reinterpret_cast<u64*>(&s.hm[0][0]);  // 3 * kBins u32 >= kCap u64
  if (threadIdx.x == 0) lcount = 0u;
  __syncthreads();
  const int l = threadIdx.x & 31;
  for (int t0 = 0; t0 < cx.n; t0 += kT) {
    const int i = t0 + threadIdx.x;
    const bool h = i < cx.n && hit(i);
    const uint32_t bal = __ballot_sync(0xffffffffu, h);
    if (bal == 0u) continue;
    uint32_t base = 0u;
    if (l == 0) base = atomicAdd(&lcount, (uint32_t)__popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (h) {
      const uint32_t pos = base + __popc(bal & ((1u << l) - 1u));
      if (pos < (uint32_t)kCap) loc[pos] = pack(key(i), cx.i0 + (uint32_t)i);
    }
  }
  __syncthreads();
  const uint32_t n = min(lcount, (uint32_t)kCap);
  if (threadIdx.x == 0) lbase = n ? atom_add_peer(peer_addr(&s.nbuf, 0), n) : 0u;
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < n; j += kT) {
    const uint32_t pos = lbase + j;
    if (pos < (uint32_t)kCap) st_peer_u64(peer_addr(&s.buf[pos], 0), loc[j]);
  }
}

__device__ void clear_hist(Sm& s) {
  for (int i = threadIdx.x; i < kBins; i += kT) {
    s.hc[i] = 0u;
    s.hm[0][i] = 0u;
    s.hm[1][i] = 0u;
    s.hm[2][i] = 0u;
  }
  __syncthreads();
}
// Count one element in bin b and (weighted) its mass term in three 14-bit
// chunks: each chunk's sum over a CTA stays below 2^28.
__device__ __forceinline__ u64 add_hist(Sm& s, int b, bool weighted, float z, float m) {
  atomicAdd(&s.hc[b], 1u);
  if (!weighted) return 0ull;
  const u64 q = fix40(expf(z - m));
  atomicAdd(&s.hm[0][b], (uint32_t)(q & 0x3fffu));
  atomicAdd(&s.hm[1][b], (uint32_t)((q >> 14) & 0x3fffu));
  atomicAdd(&s.hm[2][b], (uint32_t)(q >> 28));
  return q;
}

// Selection over array a (maximum m): the first element of the order at
// which the prefix weight reaches target.  `slot` counts exchange slots.
__device__ Pick select(Sm& s, const Ctx& cx, const float* a, float m, bool weighted,
                       u64 target, int& slot, u64* norm = nullptr, double alpha = 0.0) {
  Pick pk;
  pk.all = false;
  // ---- round 0: depth bins ----
  clear_hist(s);
  u64 part = 0ull;
  for (int i = threadIdx.x; i < cx.n; i += kT) {
    const float z = a[i];
    const float t = (m - z) * kDepthScale;
    const int b = t < (float)(kBins - 1) ? (int)t : kBins - 1;
    part += add_hist(s, b, weighted, z, m);
  }
  if (norm) *norm = block_sum_q(part, s);
  int bin;
  uint32_t cnt_above, n_set;
  u64 w_above;
  if (!boundary_bin(s, cx, weighted, target, slot, bin, cnt_above, w_above, n_set, false, norm,
                    alpha)) {
    pk.all = true;
    pk.key = 0u;
    pk.idx = 0xffffffffu;
    pk.len = 0u;
    return pk;
  }
  // the set: elements of the bin, then (if too large) narrower key ranges
  bool by_bin = true;
  uint32_t klo = 0u, khi = 0u;
  auto in_set = [&](float z) -> bool {
    if (by_bin) {
      const float t = (m - z) * kDepthScale;
      const int b = t < (float)(kBins - 1) ? (int)t : kBins - 1;
      return b == bin;
    }
    const uint32_t k = fkey(z);
    return k >= klo && k <= khi;
  };
  for (int round = 0; n_set > (uint32_t)kCap; ++round) {
    // key range of the set
    uint32_t lo = 0xffffffffu, hi = 0u;
    for (int i = threadIdx.x; i < cx.n; i += kT)
      if (in_set(a[i])) {
        const uint32_t k = fkey(a[i]);
        lo = min(lo, k);
        hi = max(hi, k);
      }
    lo = block_min_u(lo, s);
    hi = block_max_u(hi, s);
    cluster_red2_u(s, slot++, lo, hi, 1);
    klo = lo;
    khi = hi;
    by_bin = false;
    if (klo == khi || round >= 3) break;  // equal keys: ties
    // sub-bins of the key range, largest key first
    const unsigned long long span = (unsigned long long)(khi - klo) + 1ull;
    clear_hist(s);
    for (int i = threadIdx.x; i < cx.n; i += kT) {
      const uint32_t k = fkey(a[i]);
      if (k < klo || k > khi) continue;
      const int sb = (int)(((unsigned long long)(khi - k) * kBins) / span);
      add_hist(s, sb, weighted, a[i], m);
    }
    int sbin;
    uint32_t ca, cb;
    u64 wa;
    // (rounding can leave the narrowed set below the target: its last
    // non-empty sub-bin is taken)
    u64 rel = target - w_above;
    boundary_bin(s, cx, weighted, rel, slot, sbin, ca, wa, cb, true);
    cnt_above += ca;
    w_above += wa;
    n_set = cb;
    // the new set is the sub-bin's key range: [klo', khi'] from its keys
    const uint32_t olo = klo, ohi = khi;
    uint32_t lo2 = 0xffffffffu, hi2 = 0u;
    for (int i = threadIdx.x; i < cx.n; i += kT) {
      const uint32_t k = fkey(a[i]);
      if (k < olo || k > ohi) continue;
      const int sb = (int)(((unsigned long long)(ohi - k) * kBins) / span);
      if (sb == sbin) {
        lo2 = min(lo2, k);
        hi2 = max(hi2, k);
      }
    }
    lo2 = block_min_u(lo2, s);
    hi2 = block_max_u(hi2, s);
    cluster_red2_u(s, slot++, lo2, hi2, 1);
    klo = lo2;
    khi = hi2;
  }

  if (n_set > (uint32_t)kCap) {
    // all keys equal (klo == khi): the lowest indices come first
    const u64 wt = weighted ? fix40(expf(fval(klo) - m)) : 1ull;
    const u64 rest = target > w_above ? target - w_above : 0ull;
    const u64 need_q = wt == 0ull ? (u64)n_set : (rest + wt - 1ull) / wt;
    const uint32_t need = need_q < 1ull ? 1u : (need_q > (u64)n_set ? n_set : (uint32_t)need_q);
    // ties per CTA, in rank (index) order
    uint32_t mine = 0u;
    for (int i = threadIdx.x; i < cx.n; i += kT) mine += fkey(a[i]) == klo;
    mine = block_sum_u(mine, s);
    cluster_gather2(s, slot++, (u64)mine, 0ull);
    uint32_t before = 0u;
    for (uint32_t r = 0; r < cx.rank; ++r) before += (uint32_t)s.xin[r][0];
    __syncthreads();
    if (cluster_rank() == 0 && threadIdx.x == 0) s.res_u[0] = 0xffffffffu;
    cluster_sync();
    if (need > before && need <= before + mine) {
      const uint32_t gi = nth_tie(s, cx, a, klo, need - before);
      if (threadIdx.x == 0) st_peer_u32(peer_addr(&s.res_u[0], 0), gi);
    }
    cluster_sync();
    if (threadIdx.x == 0) s.xin[0][0] = ld_peer_u32(peer_addr(&s.res_u[0], 0));
    __syncthreads();
    pk.key = klo;
    pk.idx = (uint32_t)s.xin[0][0];
    pk.len = cnt_above + need;
    cluster_sync();  // everyone has read rank 0's result
    return pk;
  }

  // ---- gather the set into rank 0, sort, scan ----
  if (cx.rank == 0 && threadIdx.x == 0) s.nbuf = 0u;
  cluster_sync();
  gather_to_rank0(s, cx, [&](int i) { return in_set(a[i]); }, [&](int i) { return fkey(a[i]); });
  cluster_sync();
  if (cx.rank == 0) {
    const int n = (int)min(s.nbuf, (uint32_t)kCap);
    sort_desc<kT>(s.buf, n);
    if (threadIdx.x < 32) {
      // first element whose prefix weight (above + own) reaches the target
      const int l = threadIdx.x;
      u64 run = w_above;
      int hit = -1;
      for (int j0 = 0; j0 < n && hit < 0; j0 += 32) {
        const int j = j0 + l;
        u64 w = 0ull;
        if (j < n) w = weighted ? fix40(expf(fval(pk_key(s.buf[j])) - m)) : 1ull;
        u64 inc = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const u64 t = __shfl_up_sync(0xffffffffu, inc, o);
          if (l >= o) inc += t;
        }
        const bool ok = j < n && run + inc >= target;
        const uint32_t bal = __ballot_sync(0xffffffffu, ok);
        if (bal) hit = j0 + __ffs(bal) - 1;
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (hit < 0) hit = n > 0 ? n - 1 : 0;  // rounding: the whole set
      if (l == 0) {
        s.res_u[0] = pk_key(s.buf[hit]);
        s.res_u[1] = pk_idx(s.buf[hit]);
        s.res_u[2] = cnt_above + (uint32_t)hit + 1u;
      }
    }
  }
  cluster_sync();
  if (threadIdx.x < 3) s.xin[threadIdx.x][0] = ld_peer_u32(peer_addr(&s.res_u[threadIdx.x], 0));
  __syncthreads();
  pk.key = (uint32_t)s.xin[0][0];
  pk.idx = (uint32_t)s.xin[1][0];
  pk.len = (uint32_t)s.xin[2][0];
  cluster_sync();  // everyone has read rank 0's result
  return pk;
}

__device__ __forceinline__ bool ranks_in(uint32_t k, uint32_t i, const Pick& p) {
  return p.all || k > p.key || (k == p.key && i <= p.idx);
}

// Row results from S_fp and the sums over U (kSumWords of them): masses A =
// e_fp(U), B = e_q(U), C = e_fp(C and S) and the product sums (one thread).
__device__ void write_row(int row, int32_t len, const u64* w, double sf, const kvq_drift_params& p,
                          int32_t* m_t, float* c_t, float* d_loc, uint8_t* y_t) {
  const double ia = kFix / (double)w[1], ib = kFix / (double)w[2];
  const double saa = prod_value(w[4], w[5]), sab = prod_value(w[6], w[7]),
               sbb = prod_value(w[8], w[9]);
  double dsum = saa * ia * ia - 2.0 * sab * ia * ib + sbb * ib * ib;
  if (dsum < 0.0) dsum = 0.0;  // rounding of an exact zero
  const double c = (double)w[3] / sf;
  const double d = sqrt(dsum);
  m_t[row] = len;
  c_t[row] = (float)c;
  d_loc[row] = (float)d;
  y_t[row] = (uint8_t)(d > (double)p.eps && c >= (double)p.rho_c);
}
// The coverage curve: prefix sums of the terms wsel over S_fp (one warp).
__device__ void write_curve(const u64* wsel, double sf, int row, int k_max, float* cov) {
  const int l = threadIdx.x & 31;
  const float inv = (float)(1.0 / sf);
  u64 run = 0ull;
  for (int j0 = 0; j0 < k_max; j0 += 32) {
    const int j = j0 + l;
    u64 inc = j < k_max ? wsel[j] : 0ull;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 t = __shfl_up_sync(0xffffffffu, inc, o);
      if (l >= o) inc += t;
    }
    if (j < k_max) cov[(long long)row * k_max + j] = (float)(run + inc) * inv;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
}

// One row of the general kernel (the CTAs of one cluster).
__device__ void drift_row(Sm& s, const float* __restrict__ z_fp, const float* __restrict__ z_q,
                          int row, int vocab, const kvq_drift_params& p,
                          int32_t* __restrict__ m_t, float* __restrict__ c_t,
                          float* __restrict__ d_loc, uint8_t* __restrict__ y_t,
                          float* __restrict__ cov) {
  Ctx cx;
  cx.rank = cluster_rank();
  const int sl = ((vocab + kCl - 1) / kCl + 3) & ~3;
  cx.i0 = (uint32_t)(cx.rank * sl);
  cx.n = max(0, min(vocab - (int)cx.i0, sl));
  const float* gf = z_fp + (long long)row * vocab + cx.i0;
  const float* gq = z_q + (long long)row * vocab + cx.i0;
  int slot = 0;

  // ---- stage the slices (one HBM read) and the maxima ----
  float mf = -INFINITY, mq = -INFINITY;
  const bool vec = ((reinterpret_cast<uintptr_t>(gf) | reinterpret_cast<uintptr_t>(gq)) & 15u) == 0;
  if (vec) {
    const int n4 = cx.n >> 2;
    for (int i = threadIdx.x; i < n4; i += kT) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(gf) + i);
      const float4 b = __ldg(reinterpret_cast<const float4*>(gq) + i);
      reinterpret_cast<float4*>(s.zf)[i] = a;
      reinterpret_cast<float4*>(s.zq)[i] = b;
      mf = fmaxf(mf, fmaxf(fmaxf(a.x, a.y), fmaxf(a.z, a.w)));
      mq = fmaxf(mq, fmaxf(fmaxf(b.x, b.y), fmaxf(b.z, b.w)));
    }
    for (int i = 4 * n4 + threadIdx.x; i < cx.n; i += kT) {
      s.zf[i] = gf[i];
      s.zq[i] = gq[i];
      mf = fmaxf(mf, s.zf[i]);
      mq = fmaxf(mq, s.zq[i]);
    }
  } else {
    for (int i = threadIdx.x; i < cx.n; i += kT) {
      s.zf[i] = gf[i];
      s.zq[i] = gq[i];
      mf = fmaxf(mf, s.zf[i]);
      mq = fmaxf(mq, s.zq[i]);
    }
  }
  mf = block_max_f(mf, s);
  mq = block_max_f(mq, s);
  {
    // maxima as order keys (max of keys = key of the max)
    uint32_t a = fkey(mf), b = fkey(mq);
    cluster_red2_u(s, slot++, a, b, 2);
    mf = fval(a);
    mq = fval(b);
  }

  // ---- C(alpha) (with S_fp) and TopK(z_q, k_max) boundaries ----
  u64 sf = 0ull;
  const Pick pf = select(s, cx, s.zf, mf, true, 0ull, slot, &sf, (double)p.alpha);
  const Pick pq = select(s, cx, s.zq, mq, false, (u64)p.k_max, slot);

  // ---- the k_max best of z_q, sorted, in rank 0 ----
  if (cx.rank == 0 && threadIdx.x == 0) s.nbuf = 0u;
  cluster_sync();
  gather_to_rank0(
      s, cx, [&](int i) { return ranks_in(fkey(s.zq[i]), cx.i0 + (uint32_t)i, pq); },
      [&](int i) { return fkey(s.zq[i]); });
  cluster_sync();
  if (cx.rank == 0) {
    sort_desc<kT>(s.buf, (int)min(s.nbuf, (uint32_t)kCap));
    if (threadIdx.x == 0) {
      const unsigned long long w = s.buf[p.window - 1];  // the K-th of TopK(z_q)
      s.res_u[4] = pk_key(w);
      s.res_u[5] = pk_idx(w);
    }
  }
  cluster_sync();
  if (threadIdx.x < 2) s.xin[threadIdx.x][0] = ld_peer_u32(peer_addr(&s.res_u[4 + threadIdx.x], 0));
  __syncthreads();
  Pick ps;
  ps.all = false;
  ps.key = (uint32_t)s.xin[0][0];
  ps.idx = (uint32_t)s.xin[1][0];
  ps.len = (uint32_t)p.window;
  __syncthreads();

  // ---- one pass over U = C union S ----
  // masses A = e_fp(U), B = e_q(U), c = e_fp(C and S) and the sums of e_fp^2,
  // e_fp e_q, e_q^2 (Prod) for
  //   d_loc^2 = Saa / A^2 - 2 Sab / (A B) + Sbb / B^2.
  // U is sparse: each warp queues its members (local index, bit 31 = in C
  // and S) in its own 64 entries of buf past the TopK list and works on them
  // 32 at a time, so the exponentials and products run on full warps.
  u64 A = 0ull, B = 0ull, Cs = 0ull;
  Prod saa, sab, sbb;
  {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t* uq = reinterpret_cast<uint32_t*>(&s.buf[kMaxKcov]) + warp * 64;
    auto member = [&](uint32_t e) {
      const int i = (int)(e & 0x7fffffffu);
      const float a = expf(s.zf[i] - mf), b = expf(s.zq[i] - mq);
      const u64 qa = fix40(a);
      A += qa;
      B += fix40(b);
      if (e >> 31) Cs += qa;
      saa.add(a, a);
      sab.add(a, b);
      sbb.add(b, b);
    };
    int qn = 0;
    for (int t0 = warp * 32; t0 < cx.n; t0 += kT) {
      const int i = t0 + lane;
      bool inc = false, ins = false;
      if (i < cx.n) {
        const uint32_t gi = cx.i0 + (uint32_t)i;
        inc = ranks_in(fkey(s.zf[i]), gi, pf);
        ins = ranks_in(fkey(s.zq[i]), gi, ps);
      }
      const bool mem = inc || ins;
      const uint32_t bal = __ballot_sync(0xffffffffu, mem);
      if (mem) uq[qn + __popc(bal & ((1u << lane) - 1u))] = (uint32_t)i | (inc && ins ? 0x80000000u : 0u);
      qn += __popc(bal);
      __syncwarp();
      if (qn >= 32) {
        member(uq[lane]);
        __syncwarp();
        if (lane < qn - 32) uq[lane] = uq[32 + lane];  // the rest (< 32) to the front
        qn -= 32;
        __syncwarp();
      }
    }
    if (lane < qn) member(uq[lane]);
  }
  // the sums of the warps, of the CTA and, after one exchange, of the cluster
  // (the count is the prefix length already)
  {
    u64 w[kSumWords] = {0ull,          A,          B,            Cs,         saa.coarse(),
                        saa.fine(), sab.coarse(), sab.fine(), sbb.coarse(), sbb.fine()};
    u64* wpart = reinterpret_cast<u64*>(s.wsel);  // [kW][kSumWords] (wsel is free until the outputs)
    warp_sums(w, wpart + (threadIdx.x >> 5) * kSumWords);
    __syncthreads();
    if (threadIdx.x < kSumWords) {
      u64 v = 0ull;
      for (int k = 0; k < kW; ++k) v += wpart[k * kSumWords + threadIdx.x];
      s.xd[slot + threadIdx.x / kXw][threadIdx.x % kXw] = v;
    }
    cluster_sync();
    if (threadIdx.x < kSumWords * kCl) {
      const uint32_t k = threadIdx.x % kSumWords, r = threadIdx.x / kSumWords;
      s.xin3[r][k] = ld_peer_u64(peer_addr(&s.xd[slot + k / kXw][k % kXw], r));
    }
    __syncthreads();
    if (threadIdx.x < kSumWords) {
      u64 v = 0ull;
      for (int r = 0; r < kCl; ++r) v += s.xin3[r][threadIdx.x];
      s.xin3[0][threadIdx.x] = v;
    }
    __syncthreads();
    slot += 3;
  }

  // ---- outputs (rank 0) ----
  if (cx.rank == 0) {
    if (threadIdx.x == 0)
      write_row(row, pf.all ? vocab : (int32_t)pf.len, s.xin3[0], (double)sf, p, m_t, c_t, d_loc,
                y_t);
    // coverage curve: prefix sums of p_fp over TopK(z_q, k) within C; the
    // FP16 logits of the list come from the CTAs that hold them
    const int sl = ((vocab + kCl - 1) / kCl + 3) & ~3;
    if (threadIdx.x < p.k_max) {
      const uint32_t gi = pk_idx(s.buf[threadIdx.x]);
      u64 w = 0ull;
      if (gi < (uint32_t)vocab) {
        const uint32_t owner = gi / (uint32_t)sl;
        const float zf = ld_peer_f32(peer_addr(&s.zf[gi - owner * (uint32_t)sl], owner));
        if (ranks_in(fkey(zf), gi, pf)) w = fix40(expf(zf - mf));
      }
      s.wsel[threadIdx.x] = w;
    }
    __syncthreads();
    if (threadIdx.x < 32) write_curve(s.wsel, (double)sf, row, p.k_max, cov);
  }
  cluster_sync();  // no CTA goes on while a peer may read its shared memory
}

// kAll: every row, one cluster each (no streaming kernel ran).
template <bool kAll>
__global__ void __cluster_dims__(kCl, 1, 1) __launch_bounds__(kT, 1)
    drift_general_kernel(const float* __restrict__ z_fp, const float* __restrict__ z_q, int rows,
                         int vocab, kvq_drift_params p, int32_t* __restrict__ m_t,
                         float* __restrict__ c_t, float* __restrict__ d_loc,
                         uint8_t* __restrict__ y_t, float* __restrict__ cov) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Sm& s = *reinterpret_cast<Sm*>(smem_raw);
  pdl_launch_dependents();
  pdl_wait();  // the streaming kernel's marks
  if constexpr (kAll) {
    drift_row(s, z_fp, z_q, blockIdx.y, vocab, p, m_t, c_t, d_loc, y_t, cov);
    return;
  }
  // Marks are read kT rows at a time (usually none is set).  Every CTA of the
  // cluster reads them before the barriers that come before rank 0 overwrites
  // one.
  for (int r0 = blockIdx.y; r0 < rows; r0 += kT * (int)gridDim.y) {
    const int mine = r0 + (int)threadIdx.x * (int)gridDim.y;
    const bool left = mine < rows && *reinterpret_cast<volatile int32_t*>(m_t + mine) < 0;
    if (!__syncthreads_or(left)) continue;
    const uint32_t bal = __ballot_sync(0xffffffffu, left);
    __shared__ uint32_t marks[kT / 32];
    if ((threadIdx.x & 31) == 0) marks[threadIdx.x >> 5] = bal;
    __syncthreads();
    for (int w = 0; w < kT / 32; ++w)
      for (uint32_t bits = marks[w]; bits; bits &= bits - 1u)
        drift_row(s, z_fp, z_q, r0 + (32 * w + __ffs(bits) - 1) * (int)gridDim.y, vocab, p, m_t,
                  c_t, d_loc, y_t, cov);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// The streaming kernel: one CTA per row, the logits read straight from global
// memory; 512 threads, two rows per SM, or 1024 threads for launches of at
// most one row per SM.
//
//   sample  eight runs of elements spread over the row: where the histogram's
//           grid begins, and below which logits neither boundary can lie.
//   pass A  both rows once (the HBM read): maxima, a guess of S_fp (relative
//           to the sample's maximum), a count per 1/64 unit of z_fp logit
//           (shared-memory histogram) and the positions of the z_q logits
//           above the sample's bound.
//   plan    a few bins around the place where the prefix mass should reach
//           alpha (each bin weighed by the exponential of its centre), and
//           the bin where the count of z_q reaches k_max.
//   pass B  z_fp again (from L2 as far as it holds it): S_fp; elements above
//           the bins (certainly in C) add to the masses and the d_loc sums;
//           the few hundred inside the bins are listed.  The noted z_q logits
//           down to its bin are listed too.
//   finish  the exact boundary element among the listed ones (the masses
//           above them must bracket the target, which is checked), the z_q
//           list sorted, the listed members of U added, the row written.
//
// The sample, the guess of S_fp and the histogram only steer: masses,
// comparisons and orders are the ones defined above, over the same exact
// integers as in the general kernel, so a bad guess is noticed.  A row that is
// not settled (more than kL nearly equal logits at a boundary, a boundary more
// than 20 units below the sample's maximum, a sample far from the row) is
// marked m_t = -1 and left to the general kernel, launched behind it.
//
// What bounds it: the HBM reads (both rows, and z_fp once more beyond what L2
// keeps), then the latency of the serial steps of a row; one CTA per row has
// block barriers only and keeps up to 304 rows in flight, where a cluster of
// 2, 4 or 8 CTAs per row spent 25 us per row on cluster barriers and
// distributed shared memory (190, 203 and 230 us for 256 rows of 128256).
// ---------------------------------------------------------------------------

constexpr int kL = 1024;             // listed elements of a row
constexpr int kUp = 12;              // units above the sample's maximum in the histogram
constexpr uint32_t kSpread = 300;    // elements listed on either side of the estimate
constexpr float kMagic = 8388608.0f; // 2^23: floats in [2^23, 2^24) are whole numbers
constexpr int kU = 2;                // 16-byte loads of the next step in flight per thread
constexpr int kRuns = 8;             // sample elements per thread
constexpr int kMemCap = 16;          // members a thread notes before its warp works on them
constexpr int kTopCap = 12;          // z_q candidates a thread notes

template <int kS>
struct Ss {
  static constexpr int kSw = kS / 32;
  union {
    uint32_t hf[kBins];           // pass A
    u64 lf[kL];                   // pass B: z_fp elements inside the bins
  };
  union {
    uint32_t hq[kBins];           // z_q counts
    uint16_t mem[kMemCap][kS];    // pass B: positions of members
    u64 mass[kL];                 // finish: masses of the listed elements' key ranges
  };
  u64 lq[kL];                     // pass B: z_q elements down to the k_max bin
  u64 top[kL];                    // the same, best first
  uint16_t cand[kTopCap][kS];     // pass A: positions of z_q candidates
  union {
    uint16_t flat[kSw][32 * kMemCap];  // a warp's members, side by side
    u64 set[kS];                  // finish: the elements around the boundary
  };
  u64 wsel[kMaxKcov];             // coverage terms
  u64 part[kSw][kSumWords];       // warps' sums
  u64 su[kSw], sv[kSw];
  float rf[4][kSw];
  uint32_t sc[2][kSw];
  uint32_t pick[12];
  uint32_t nf, nq;                // list lengths
};

// A row of n floats (4-byte aligned) as each thread streams it: vectors
// u = 0, 1, ... of thread t at 16-byte positions u kS + t past the first
// boundary, then one vector with the single elements before and after them
// (missing elements are -inf).
template <int kS>
struct Stream {
  const float* p;
  int head, nv, n, steps;  // steps: full vectors per thread (the last may be empty)
  __device__ Stream(const float* q, int m) : p(q), n(m) {
    head = min(m, (int)((16u - (reinterpret_cast<uintptr_t>(q) & 15u)) & 15u) >> 2);
    nv = (m - head) >> 2;
    steps = (nv + kS - 1) / kS;
  }
  // Index of element k of vector u of thread t.
  __device__ __forceinline__ int index(int t, int u, int k) const {
    return u < steps ? head + 4 * (u * kS + t) + k : (t < head ? t : 4 * nv + t);
  }
  __device__ __forceinline__ float4 load(int u) const {
    const int j = u * kS + (int)threadIdx.x;
    return j < nv ? __ldg(reinterpret_cast<const float4*>(p + head) + j)
                  : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  }
  // f(vector, u) for every vector of this thread; all threads call f equally
  // often.  The next kU loads are issued before the current ones are used.
  template <typename F>
  __device__ __forceinline__ void each(const F& f) const {
    float4 v[kU], w[kU];
#pragma unroll
    for (int k = 0; k < kU; ++k) v[k] = load(k);
    for (int u = 0; u < steps; u += kU) {
#pragma unroll
      for (int k = 0; k < kU; ++k) w[k] = load(u + kU + k);
#pragma unroll
      for (int k = 0; k < kU; ++k)
        if (u + k < steps) f(v[k], u + k);
#pragma unroll
      for (int k = 0; k < kU; ++k) v[k] = w[k];
    }
    const int ends = n - 4 * nv;
    if (ends > 0) {
      float4 e = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      if ((int)threadIdx.x < ends) e.x = p[index(threadIdx.x, steps, 0)];
      f(e, steps);
    }
  }
};
// positions (vector, lane, element) fit 16 bits
static_assert((kCl * kSlice / 4 / 512 + 2) * 128 <= 65536, "positions fit 16 bits");

__device__ __forceinline__ float max4(const float4& v) {
  return fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w));
}
// About e^(z - m), for the plan only.
__device__ __forceinline__ float exp_guess(float z, float m) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(fmaf(z, 1.44269504f, -1.44269504f * m)));
  return y;
}
// The integer a (even) whose bin a - 64 z is 0 for z = kUp units above x.
__device__ __forceinline__ int bin_origin(float x) {
  const float a = 2.0f * rintf((kDepthScale / 2.0f) * (x + (float)kUp));
  return fabsf(a) < 4194304.0f ? (int)a : 0;  // |a| < 2^22 (and not NaN), else the guess is void
}
// The bin of z on the grid of origin a, clamped at bin 0 (z >= bin_floor(a)),
// as a float 2^23 + bin; without the clamp it orders all z alike.
__device__ __forceinline__ float bin_place(float z, float a) {
  return fmaf(-kDepthScale, z, a + kMagic);
}
__device__ __forceinline__ uint32_t bin_of(float z, float a) {
  return __float_as_uint(fmaxf(bin_place(z, a), kMagic)) - 0x4b000000u;
}
__device__ __forceinline__ float bin_floor(float a) {
  return (a - (float)(kBins - 1)) * (1.0f / kDepthScale);
}

// A sum of terms e in [0, 1] as multiples of 2^-40 (fix40's value, at most
// 4095 terms): e + 8 rounds e to a multiple of 2^-20, the exact rest + 1.5
// 2^-17 to one of 2^-40.
struct Fixed {
  uint32_t hi = 0u, lo = 0u;
  __device__ __forceinline__ void add(float e) {
    const float h = e + 8.0f;
    hi += __float_as_uint(h) - 0x41000000u;
    lo += __float_as_uint((e - (h - 8.0f)) + 1.5f / 131072.0f) - 0x37400000u;
  }
  __device__ __forceinline__ u64 value() const {
    return ((u64)hi << 20) + (u64)(long long)(int)lo;
  }
};
// A thread's sums over members of U.
struct Sums {
  uint32_t cnt = 0u;
  Fixed A, B;
  u64 C = 0ull;
  Prod aa, ab, bb;
  __device__ __forceinline__ void add(float a, float b) {
    A.add(a);
    B.add(b);
    aa.add(a, a);
    ab.add(a, b);
    bb.add(b, b);
  }
};
__device__ __forceinline__ void warp_sums(const Sums& v, u64* out) {
  u64 w[kSumWords] = {v.cnt,       v.A.value(),   v.B.value(), v.C,           v.aa.coarse(),
                      v.aa.fine(), v.ab.coarse(), v.ab.fine(), v.bb.coarse(), v.bb.fine()};
  warp_sums(w, out);
}

// Exclusive prefix of x over the threads; *total the sum.  buf: one word per
// warp, not read by anyone when the call begins.
template <int kS, typename T>
__device__ __forceinline__ T scan(T x, T* buf, T* total) {
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5;
  T i = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, i, o);
    if (l >= o) i += y;
  }
  if (l == 31) buf[w] = i;
  __syncthreads();
  // (the warps' totals by shuffles: a loop over 32 of them in every thread is
  // longer than the scan)
  T y = l < kS / 32 ? buf[l] : (T)0;
#pragma unroll
  for (int o = 1; o < kS / 32; o <<= 1) {
    const T z = __shfl_up_sync(0xffffffffu, y, o);
    if (l >= o) y += z;
  }
  *total = __shfl_sync(0xffffffffu, y, kS / 32 - 1);
  const T before = __shfl_sync(0xffffffffu, y, w > 0 ? w - 1 : 0);
  return (w > 0 ? before : (T)0) + i - x;
}

// The bins [b1, b2] of z_fp to list, around the place where the prefix mass
// should reach `goal` (in units of e^top), into pick[3..4] (pick[7] = 1 if
// they hold at most kL elements), and the bin of z_q where the count reaches
// k_max into pick[8] (pick[9] = 1 if at most kL elements rank above or in it).
// `counted` is the mass of the counted elements: the goal is met from the end
// of the histogram, where many small terms per bin leave no error, and not
// from its start, where one token can hold a third of the mass and its bin's
// width is 0.8% of that (44 rows of 20772 tokens, alpha = 0.99: some rows went
// to the general kernel).
template <int kS>
__device__ void make_plan(Ss<kS>& s, float top, float a_f, float goal, float counted,
                          uint32_t k_max) {
  constexpr int kPer = kBins / kS;
  const int t = threadIdx.x;
  if (t < 12) s.pick[t] = t == 0 || t == 8 ? kBins : 0u;
  uint32_t c[kPer], cs = 0u, d[kPer], ds = 0u;
  float w[kPer], ws = 0.0f;
  const float b0 = fmaf(-kDepthScale, top, a_f);  // its place among the bins (maybe below 0)
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    c[k] = s.hf[kPer * t + k];
    d[k] = s.hq[kPer * t + k];
    // bin 0 may hold elements above it: weighed like the maximum
    const float b = kPer * t + k == 0 ? fminf(b0, 0.0f) : (float)(kPer * t + k);
    w[k] = (float)c[k] * exp2f((b0 - b) * (1.44269504f / kDepthScale));
    cs += c[k];
    ds += d[k];
    ws += w[k];
  }
  float all_w;
  uint32_t all_c, all_d;
  const float wb = scan<kS>(ws, s.rf[0], &all_w);
  uint32_t x = scan<kS>(cs, s.sc[0], &all_c), y = scan<kS>(ds, s.sc[1], &all_d);
  goal += all_w - counted;
  {
    uint32_t b = kBins;  // the first bin whose prefix mass reaches the goal
    float q = wb;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      q += w[k];
      if (b == (uint32_t)kBins && c[k] > 0u && q >= goal) b = (uint32_t)(kPer * t + k);
      if (y < k_max && y + d[k] >= k_max) {
        s.pick[8] = (uint32_t)(kPer * t + k);
        s.pick[9] = y + d[k] <= (uint32_t)kL ? 1u : 0u;
      }
      y += d[k];
    }
    if (b < (uint32_t)kBins) atomicMin(&s.pick[0], b);
  }
  __syncthreads();
  const uint32_t bc = s.pick[0];
  if (bc / kPer == (uint32_t)t) {  // counts before it and up to it
    uint32_t u = x, v = 0u;
#pragma unroll
    for (uint32_t k = 0; k < (uint32_t)kPer; ++k) {
      u += k < bc % kPer ? c[k] : 0u;
      v = k == bc % kPer ? c[k] : v;
    }
    s.pick[1] = u;
    s.pick[2] = u + v;
    s.pick[3] = bc;
    s.pick[4] = bc;
  }
  __syncthreads();
  if (bc < (uint32_t)kBins) {
    const uint32_t c0 = s.pick[1], c1 = s.pick[2];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t b = (uint32_t)(kPer * t + k);
      if (b < bc && x + c[k] + kSpread > c0) atomicMin(&s.pick[3], b);
      if (b > bc && x < c1 + kSpread) atomicMax(&s.pick[4], b);
      x += c[k];
    }
  }
  __syncthreads();
  {
    const uint32_t b1 = s.pick[3], b2 = s.pick[4];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {  // the elements in them
      const uint32_t b = (uint32_t)(kPer * t + k);
      if (b >= b1 && b <= b2 && c[k]) atomicAdd(&s.pick[5], c[k]);
    }
  }
  __syncthreads();
  if (t == 0) {
    const bool wide = s.pick[5] <= (uint32_t)kL;
    if (!wide) s.pick[3] = s.pick[4] = bc;
    s.pick[7] = bc < (uint32_t)kBins && (wide || s.pick[2] - s.pick[1] <= (uint32_t)kL) ? 1u : 0u;
  }
  __syncthreads();
}

// The first of the n listed z_fp elements, in order, whose prefix mass (on
// top of `above`) reaches `target`, into pick[0..1] (key, index), with
// pick[2] = 1.  The elements' key range is cut into kL parts, the part where
// the mass reaches the target is found by a scan, and the few elements in it
// are compared pairwise (pick[2] = 0 if they are more than kS, or the target
// lies elsewhere).
template <int kS>
__device__ void find_boundary(Ss<kS>& s, int n, u64 above, u64 target, float mf) {
  constexpr int kPer = kL / kS;
  const int t = threadIdx.x, l = t & 31, w = t >> 5;
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (int j = t; j < n; j += kS) {
    const uint32_t k = pk_key(s.lf[j]);
    lo = min(lo, k);
    hi = max(hi, k);
  }
#pragma unroll
  for (int k = 0; k < kPer; ++k) s.mass[k * kS + t] = 0ull;
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (t == 0) {
    s.pick[1] = s.pick[2] = s.pick[3] = 0u;
    s.pick[0] = 0xffffffffu;
    s.pick[4] = kL;
  }
  if (l == 0) {
    s.sc[0][w] = lo;
    s.sc[1][w] = hi;
  }
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, l < kS / 32 ? s.sc[0][l] : 0xffffffffu);
  hi = __reduce_max_sync(0xffffffffu, l < kS / 32 ? s.sc[1][l] : 0u);
  const int sh = n > 0 ? max(0, 22 - __clz(hi - lo)) : 0;  // (hi - lo) >> sh < 1024 = kL
  auto part_of = [&](u64 e) { return (hi - pk_key(e)) >> sh; };
  auto mass_of = [&](u64 e) { return fix40(expf(fval(pk_key(e)) - mf)); };
  for (int j = t; j < n; j += kS) atomicAdd(&s.mass[part_of(s.lf[j])], mass_of(s.lf[j]));
  __syncthreads();
  u64 m[kPer], sum = 0ull, all;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    m[k] = s.mass[kPer * t + k];
    sum += m[k];
  }
  u64 run = above + scan<kS>(sum, s.su, &all);
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (run < target && target <= run + m[k]) {
      s.pick[4] = (uint32_t)(kPer * t + k);
      s.sv[0] = run;
    }
    run += m[k];
  }
  __syncthreads();
  const uint32_t part = s.pick[4];
  if (part >= (uint32_t)kL) return;
  for (int j = t; j < n; j += kS) {
    const u64 e = s.lf[j];
    if (part_of(e) == part) {
      const uint32_t q = atomicAdd(&s.pick[3], 1u);
      if (q < (uint32_t)kS) s.set[q] = e;
    }
  }
  __syncthreads();
  const int k = (int)s.pick[3];
  if (k <= kS && t < k) {
    const u64 e = s.set[t], own = mass_of(e);
    u64 pre = s.sv[0];
    for (int j = 0; j < k; ++j)
      if (s.set[j] > e) pre += mass_of(s.set[j]);
    if (pre < target && target <= pre + own) {
      s.pick[0] = pk_key(e);
      s.pick[1] = pk_idx(e);
      s.pick[2] = 1u;
    }
  }
  __syncthreads();
}

template <int kS>
__global__ void __launch_bounds__(kS, 1024 / kS)
    drift_stream_kernel(const float* __restrict__ z_fp, const float* __restrict__ z_q, int vocab,
                        kvq_drift_params p, int32_t* __restrict__ m_t, float* __restrict__ c_t,
                        float* __restrict__ d_loc, uint8_t* __restrict__ y_t,
                        float* __restrict__ cov) {
  constexpr int kSw = kS / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Ss<kS>& s = *reinterpret_cast<Ss<kS>*>(smem_raw);
  const int row = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31, n = vocab;
  pdl_launch_dependents();
  const float* rf = z_fp + (long long)row * vocab;
  const float* rq = z_q + (long long)row * vocab;
  const Stream<kS> f(rf, n), q(rq, n);

  // ---- sample ----
  // The grid begins kUp units above the sample's maximum (elements above go
  // to bin 0, elements kBins / 64 units below are not counted).  z_fp below
  // cut_f is not counted: with the smallest of four quarter-sample means of
  // e^z as a low guess of the row's, all of it weighs less than half of the
  // mass outside C.  z_q below cut_q, the least of the warps' maxima of 256
  // elements (the upper 1.2% or 1.5% of the row in the middle), is not a
  // candidate when k_max is under 1/400 of the vocabulary.
  // Two kinds of row are seen here to be the general kernel's: with alpha = 1 a
  // token that still has mass below the grid, and logits so close together
  // that their bins hold far more than the lists do.
  float mf = -INFINITY, mq = -INFINITY, cut_f, cut_q;
  float least = INFINITY, least_mass = INFINITY;  // of all and of those with mass
  {
    float z[kRuns];
#pragma unroll
    for (int u = 0; u < kRuns; ++u) {
      const int i = n >= kRuns * kS ? u * (n / kRuns) + t : u * kS + t;
      z[u] = i < n ? __ldg(rf + i) : -INFINITY;
      mf = fmaxf(mf, z[u]);
      mq = fmaxf(mq, i < n ? __ldg(rq + i) : -INFINITY);
    }
    for (int i = t; i < kBins; i += kS) s.hf[i] = s.hq[i] = 0u;
    if (t == 0) s.nf = s.nq = 0u;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
      mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o));
    }
    // (a warp's terms are relative to its own maximum)
    float e = 0.0f;
#pragma unroll
    for (int u = 0; u < kRuns; ++u) {
      e += z[u] > -INFINITY ? exp2f((z[u] - mf) * 1.44269504f) : 0.0f;
      const int i = n >= kRuns * kS ? u * (n / kRuns) + t : u * kS + t;
      least = fminf(least, i < n ? z[u] : INFINITY);
      least_mass = fminf(least_mass, z[u] > mf - 27.0f ? z[u] : INFINITY);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      least = fminf(least, __shfl_xor_sync(0xffffffffu, least, o));
      least_mass = fminf(least_mass, __shfl_xor_sync(0xffffffffu, least_mass, o));
    }
    if (lane == 0) {
      s.rf[0][warp] = mf;
      s.rf[1][warp] = mq;
      s.rf[2][warp] = e;
      s.rf[3][warp] = least;
      s.su[warp] = __float_as_uint(least_mass);
    }
    __syncthreads();
    // second level: lane = warp
    const float mw = lane < kSw ? s.rf[0][lane] : -INFINITY;
    const float qw = lane < kSw ? s.rf[1][lane] : -INFINITY;
    cut_q = lane < kSw ? qw : INFINITY;
    mf = mw;
    mq = qw;
    least = lane < kSw ? s.rf[3][lane] : INFINITY;
    least_mass = lane < kSw ? __uint_as_float((uint32_t)s.su[lane]) : INFINITY;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      least = fminf(least, __shfl_xor_sync(0xffffffffu, least, o));
      least_mass = fminf(least_mass, __shfl_xor_sync(0xffffffffu, least_mass, o));
      mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
      mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o));
      cut_q = fminf(cut_q, __shfl_xor_sync(0xffffffffu, cut_q, o));
    }
    // four sums over every fourth warp (xor 4, 8, 16), then their least
    float low = mw > -INFINITY ? s.rf[2][lane] * exp2f((mw - mf) * 1.44269504f) : 0.0f;
#pragma unroll
    for (int o = 16; o > 2; o >>= 1) low += __shfl_xor_sync(0xffffffffu, low, o);
    low = fminf(low, __shfl_xor_sync(0xffffffffu, low, 1));
    low = fminf(low, __shfl_xor_sync(0xffffffffu, low, 2));
    cut_f = mf + logf(0.5f * (1.0f - p.alpha) * low * (4.0f / (kRuns * kS)));
    if (n < kRuns * kS) cut_f = -INFINITY;
    if (n < kRuns * kS || (long long)p.k_max * 400 > vocab) cut_q = -INFINITY;
    __syncthreads();
  }
  const float af = (float)bin_origin(mf), aq = (float)bin_origin(mq);
  const float m0 = mf > -INFINITY ? mf : 0.0f;  // reference of the guess
  if ((p.alpha >= 1.0f && least_mass < bin_floor(af)) ||
      (mf - least) * kDepthScale + 1.0f < (float)(n / (4 * kL))) {
    if (t == 0) m_t[row] = -1;
    return;
  }

  // ---- pass A (z_fp last: pass B reads it again) ----
  int n_cand = 0;  // z_q candidates of this thread
  if (cut_q > -INFINITY)
    q.each([&](const float4& v, int u) {
      const float m = max4(v);
      mq = fmaxf(mq, m);
      if (m >= cut_q) {
        const float z[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (z[k] >= cut_q) {
            if (n_cand < kTopCap) s.cand[n_cand][t] = (uint16_t)(4 * u + k);
            ++n_cand;
          }
      }
    });
  // candidates that fit are counted from the lists, else in a pass of its own
  const bool listed = __syncthreads_and(n_cand <= kTopCap) && cut_q > -INFINITY;
  if (listed) {
    float z[kTopCap];
#pragma unroll
    for (int c = 0; c < kTopCap; ++c) {
      const int e = c < n_cand ? s.cand[c][t] : 0;
      z[c] = c < n_cand ? __ldg(rq + q.index(t, e >> 2, e & 3)) : -INFINITY;
    }
#pragma unroll
    for (int c = 0; c < kTopCap; ++c)
      if (z[c] >= bin_floor(aq)) atomicAdd(&s.hq[bin_of(z[c], aq)], 1u);
  } else {
    const float low = bin_floor(aq);
    q.each([&](const float4& v, int) {
      mq = fmaxf(mq, max4(v));
      const float z[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (z[k] >= low) atomicAdd(&s.hq[bin_of(z[k], aq)], 1u);
    });
  }
  cut_f = fmaxf(cut_f, bin_floor(af));  // (NaN: the floor)
  float guess = 0.0f, counted = 0.0f;   // S_fp times e^(m - m0), about, and the counted part
  f.each([&](const float4& v, int) {
    const float m = max4(v);
    mf = fmaxf(mf, m);
    const float z[4] = {v.x, v.y, v.z, v.w};
    float e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) e[k] = exp_guess(z[k], m0);
    guess += (e[0] + e[1]) + (e[2] + e[3]);
    if (m >= cut_f) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (z[k] >= cut_f) {
          atomicAdd(&s.hf[bin_of(z[k], af)], 1u);
          counted += e[k];
        }
    }
  });
  {
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
      mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o));
      guess += __shfl_xor_sync(0xffffffffu, guess, o);
      counted += __shfl_xor_sync(0xffffffffu, counted, o);
    }
    if (lane == 0) {
      s.rf[0][warp] = guess;
      s.rf[3][warp] = counted;
      s.rf[1][warp] = mf;
      s.rf[2][warp] = mq;
    }
    __syncthreads();
    guess = lane < kSw ? s.rf[0][lane] : 0.0f;
    counted = lane < kSw ? s.rf[3][lane] : 0.0f;
    mf = lane < kSw ? s.rf[1][lane] : -INFINITY;
    mq = lane < kSw ? s.rf[2][lane] : -INFINITY;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      guess += __shfl_xor_sync(0xffffffffu, guess, o);
      counted += __shfl_xor_sync(0xffffffffu, counted, o);
      mf = fmaxf(mf, __shfl_xor_sync(0xffffffffu, mf, o));
      mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o));
    }
    __syncthreads();
  }

  // ---- the plan ----
  make_plan(s, m0, af, p.alpha * guess, counted, (uint32_t)p.k_max);
  const float y1 = kMagic + (float)s.pick[3], y2 = kMagic + (float)s.pick[4];
  const float y3 = kMagic + (float)s.pick[8];
  const bool planned = s.pick[7] != 0u && s.pick[9] != 0u;
  __syncthreads();  // (the histograms and pick are free)
  if (!planned) {
    if (t == 0) m_t[row] = -1;
    return;
  }

  // ---- pass B ----
  Sums sums;
  Fixed norm;
  {
    // z_q candidates down to its bin
    auto list_q = [&](float z, int i) {
      if (bin_place(z, aq) <= y3) {
        const uint32_t pos = atomicAdd(&s.nq, 1u);
        if (pos < (uint32_t)kL) s.lq[pos] = pack(fkey(z), (uint32_t)i);
      }
    };
    // (the noted ones are all of them if even cut_q itself lies below the bin)
    if (listed && bin_place(cut_q, aq) > y3) {
      float z[kTopCap];
#pragma unroll
      for (int c = 0; c < kTopCap; ++c) {
        const int e = c < n_cand ? s.cand[c][t] : 0;
        z[c] = c < n_cand ? __ldg(rq + q.index(t, e >> 2, e & 3)) : -INFINITY;
      }
#pragma unroll
      for (int c = 0; c < kTopCap; ++c)
        if (c < n_cand) list_q(z[c], q.index(t, s.cand[c][t] >> 2, s.cand[c][t] & 3));
    } else {
      q.each([&](const float4& v, int u) {
        if (bin_place(max4(v), aq) <= y3) {
          list_q(v.x, q.index(t, u, 0));
          list_q(v.y, q.index(t, u, 1));
          list_q(v.z, q.index(t, u, 2));
          list_q(v.w, q.index(t, u, 3));
        }
      });
    }
    int n_mem = 0;
    // The noted members of the warp, laid side by side so that every lane has
    // work: those above the bins into the sums, the others into the list.
    auto flush = [&]() {
      int at = n_mem;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += x;
      }
      const int total = __shfl_sync(0xffffffffu, at, 31);
      at -= n_mem;
      for (int c = 0; c < n_mem; ++c)
        s.flat[warp][at + c] = (uint16_t)((s.mem[c][t] << 5) | lane);  // (vector, element, lane)
      __syncwarp();
      for (int j0 = 0; j0 < total; j0 += 64) {
        int i[2];
        float z[2], w[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int j = j0 + 32 * k + lane;
          const int e = j < total ? s.flat[warp][j] : 0;
          i[k] = j < total ? f.index((t & ~31) | (e & 31), e >> 7, (e >> 5) & 3) : -1;
          z[k] = i[k] >= 0 ? __ldg(rf + i[k]) : -INFINITY;
          w[k] = i[k] >= 0 ? __ldg(rq + i[k]) : -INFINITY;
        }
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (i[k] < 0) continue;
          if (bin_place(z[k], af) >= y1) {
            const uint32_t pos = atomicAdd(&s.nf, 1u);
            if (pos < (uint32_t)kL) s.lf[pos] = pack(fkey(z[k]), (uint32_t)i[k]);
          } else {
            ++sums.cnt;
            sums.add(expf(z[k] - mf), expf(w[k] - mq));
          }
        }
      }
      __syncwarp();
      n_mem = 0;
    };
    f.each([&](const float4& v, int u) {
      const float z[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) norm.add(expf(z[k] - mf));
      if (bin_place(max4(v), af) <= y2) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (bin_place(z[k], af) <= y2) s.mem[n_mem++][t] = (uint16_t)(4 * u + k);
      }
      if (__any_sync(0xffffffffu, n_mem > kMemCap - 4)) flush();
    });
    flush();
  }
  {  // the mass above the listed elements, and S_fp
    u64 a = sums.A.value(), b = norm.value();
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) {
      s.su[warp] = a;
      s.sv[warp] = b;
    }
  }
  __syncthreads();

  // ---- finish ----
  u64 above = lane < kSw ? s.su[lane] : 0ull, sum_f = lane < kSw ? s.sv[lane] : 0ull;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    above += __shfl_xor_sync(0xffffffffu, above, o);
    sum_f += __shfl_xor_sync(0xffffffffu, sum_f, o);
  }
  const uint32_t nf = s.nf, nq = s.nq;
  const double sf = (double)sum_f;
  __syncthreads();
  bool ok = nf <= (uint32_t)kL && nq <= (uint32_t)kL && nq >= (uint32_t)p.k_max;
  if (ok) {
    // prefix mass >= alpha S  <=>  prefix >= ceil(alpha S) in fixed point
    find_boundary(s, (int)nf, above, (u64)ceil((double)p.alpha * sf), mf);
    ok = s.pick[2] != 0u;
  }
  if (!ok) {
    if (t == 0) m_t[row] = -1;
    return;
  }
  Pick pf;
  pf.all = false;
  pf.key = s.pick[0];
  pf.idx = s.pick[1];
  const u64* top = s.top;  // TopK(z_q, k_max) first
  if (nq <= (uint32_t)kS) {  // by rank
    if ((t & ~31) < (int)nq) {
      const u64 e = t < (int)nq ? s.lq[t] : 0ull;
      int r = 0;
#pragma unroll 8
      for (uint32_t k = 0; k < nq; ++k) r += s.lq[k] > e;
      if (t < (int)nq) s.top[r] = e;
    }
    __syncthreads();
  } else {
    sort_desc<kS>(s.lq, (int)nq);
    top = s.lq;
  }
  // the listed members of C; the first `window` of TopK(z_q, k_max) are S
  for (int j = t; j < (int)nf; j += kS) {
    const u64 w = s.lf[j];
    if (ranks_in(pk_key(w), pk_idx(w), pf)) {
      ++sums.cnt;
      sums.add(expf(fval(pk_key(w)) - mf), expf(__ldg(rq + pk_idx(w)) - mq));
    }
  }
  if (t < p.k_max) {
    const u64 w = top[t];
    const uint32_t gi = pk_idx(w);
    const float z = __ldg(rf + gi), a = expf(z - mf);
    const bool in_c = ranks_in(fkey(z), gi, pf);
    s.wsel[t] = in_c ? fix40(a) : 0ull;
    if (t < p.window) {
      if (in_c) sums.C = fix40(a);
      else sums.add(a, expf(fval(pk_key(w)) - mq));
    }
  }
  warp_sums(sums, s.part[warp]);
  __syncthreads();
  if (warp == 0) {
    u64 w[kSumWords];
#pragma unroll
    for (int k = 0; k < kSumWords; ++k) w[k] = lane < kSw ? s.part[lane][k] : 0ull;
    __syncwarp();
    warp_sums(w, s.part[0]);
    if (lane == 0)
      write_row(row, (int32_t)s.part[0][0], s.part[0], sf, p, m_t, c_t, d_loc, y_t);
  } else if (warp == 1) {
    write_curve(s.wsel, sf, row, p.k_max, cov);
  }
}

// K_b: column means of cov over the rows and the smallest k whose mean reaches
// rho_K (0 if none).  One CTA, or a cluster of 8 for more than kWinRows rows
// of every thread: a thread takes one column of every (CTAs kWinT / k_max)-th
// row, sixteen loads in flight, and adds its rows up in fp64; the partial sums
// are added in a fixed order (pairwise in a CTA, then CTAs).  K_b compares these
// means with rho_K, so they keep fp64's precision throughout (a pair of floats
// whose low word is not renormalised loses 6 to 9 bits of it over 512 to 2048
// rows).  What bounds it is fp64: two additions a cycle and SM, and conversions
// slower by far (24 rows of 64: 12.0 us with them, 4.9 with widen).
constexpr int kWinT = 1024;
constexpr int kWinLoads = 16;
constexpr int kWinRows = 8;  // 4 rows a thread: 7.1 us in one CTA and in eight; 16: 13.8 and 7.1
// A float as a double, by integer steps where it is a normal number.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x);
  if ((u & 0x7f800000u) - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)(((u >> 3) & 0x0fffffffu) + 0x38000000u | (u & 0x80000000u)),
                            (int)(u << 29));
  return (double)x;
}
__global__ void __launch_bounds__(kWinT)
    drift_window_kernel(const float* cov, int rows, int k_max, float rho_k,
                        float* __restrict__ mean_cov, int32_t* __restrict__ k_b) {
  __shared__ double part[kWinT];
  __shared__ double col[kMaxKcov];
  __shared__ int best[kMaxKcov / 32];
  const int t = threadIdx.x, rank = (int)blockIdx.x, ctas = (int)gridDim.x;  // one cluster
  pdl_wait();  // this kernel may start while cov is still being written: the loads
               // below are coherent ones (not __ldg, nor through a restrict pointer)
  const int per = kWinT / k_max;  // rows per sweep of a CTA
  const int step = per * ctas;
  if (t < per * k_max) {
    double sum = 0.0;
    const int k = t % k_max;
    for (long long r = rank * per + t / k_max; r < rows; r += kWinLoads * step) {
      float v[kWinLoads];
#pragma unroll
      for (int i = 0; i < kWinLoads; ++i)
        v[i] = r + i * step < rows ? __ldcg(cov + (r + i * step) * k_max + k) : 0.0f;
#pragma unroll
      for (int i = 0; i < kWinLoads; ++i)
        if (r + i * step < rows) sum += widen(v[i]);
    }
    part[t] = sum;
  }
  __syncthreads();
  for (int n = min(per, rows); n > 1;) {  // the threads of a column, pairwise
    const int h = (n + 1) / 2;
    if (t < (n - h) * k_max) part[t] += part[t + h * k_max];
    __syncthreads();
    n = h;
  }
  if (t < k_max) col[t] = part[t];
  cluster_sync();  // (one CTA: a block barrier)
  int mine = 0x7fffffff;
  if (rank == 0 && t < kMaxKcov) {
    if (t < k_max) {
      double total = 0.0;
      for (int r = 0; r < ctas; ++r)
        total += __longlong_as_double((long long)ld_peer_u64(peer_addr(&col[t], (uint32_t)r)));
      const double mean = total / rows;
      mean_cov[t] = (float)mean;
      if (mean >= (double)rho_k) mine = t + 1;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) mine = min(mine, __shfl_xor_sync(0xffffffffu, mine, o));
    if ((t & 31) == 0) best[t >> 5] = mine;
  }
  cluster_sync();  // the columns are read
  if (rank == 0 && t == 0) {
    int b = 0x7fffffff;
    for (int w = 0; w < kMaxKcov / 32; ++w) b = min(b, best[w]);
    *k_b = b == 0x7fffffff ? 0 : b;
  }
}

}  // namespace

int drift_max_vocab() { return kCl * kSlice; }
int drift_max_kcov() { return kMaxKcov; }
int drift_cap() { return kCap; }

namespace {
// SMs of the current device and the clusters of the general kernel that it runs
// at once (looked up once per device; 152 SMs do not hold 19 of them: a second
// wave of the rest took 1.6 times as long).
cudaError_t device_limits(int* sms, int* clusters) {
  static std::atomic<int> known[64];  // clusters << 16 | SMs
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int k = dev < 64 ? known[dev].load(std::memory_order_relaxed) : 0;
  if (k == 0) {
    e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(drift_general_kernel<false>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Sm));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kCl, *sms);
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = sizeof(Sm);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveClusters(clusters, drift_general_kernel<false>, &cfg);
    if (e != cudaSuccess) return e;
    k = (*clusters < 1 ? 1 : *clusters) << 16 | *sms;
    if (dev < 64) known[dev].store(k, std::memory_order_relaxed);
  }
  *sms = k & 0xffff;
  *clusters = k >> 16;
  return cudaSuccess;
}

template <int kS>
cudaError_t launch_stream(const float* z_fp, const float* z_q, int rows, int vocab,
                          const kvq_drift_params& p, int32_t* m_t, float* c_t, float* d_loc,
                          uint8_t* y_t, float* cov, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(
      drift_stream_kernel<kS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Ss<kS>));
  if (e != cudaSuccess) return e;
  drift_stream_kernel<kS><<<rows, kS, sizeof(Ss<kS>), st>>>(z_fp, z_q, vocab, p, m_t, c_t, d_loc,
                                                           y_t, cov);
  return cudaGetLastError();
}
}  // namespace

cudaError_t drift_plan(int rows, int vocab, float alpha, DriftPlan* plan) {
  int sms = 0, clusters = 0;
  const cudaError_t e = device_limits(&sms, &clusters);
  if (e != cudaSuccess) return e;
  // A few long rows: a cluster spreads each over eight SMs, and up to 15 run at
  // once.  The line lies where a CTA's stream of a row takes as long, which
  // falls with alpha (more of the row belongs to C): 7 rows, sigma 2.1 to 3.9,
  // alpha 0.9: 32768: 32 to 36 us streamed, 36 to 40 in clusters; 49152: 36 to 44
  // and 39 to 44; 98304: 51 to 63 and 47 to 54.  alpha 0.99: 24576: 30 to 38 and
  // 36 to 40; 32768: 34 to 44 and 37 to 42; 98304: 56 to 81 and 50 to 59.
  // With alpha = 1 every token with mass belongs to C, and a streamed row takes
  // as long as three waves of clusters where it is settled at all: 16 rows of
  // 128256, sigma 1 and 3: 196 and 116 us streamed, 112 in clusters.
  if ((rows * 10 <= sms && vocab > (alpha > 0.97f ? 28672 : 40960)) ||
      (alpha >= 1.0f && rows * 10 <= 3 * sms)) {
    plan->stream_threads = 0;
    plan->clusters = rows;
  } else {
    plan->stream_threads = rows <= sms ? 1024 : 512;  // one row per SM: all its threads on it
    plan->clusters = rows < clusters ? rows : clusters;
  }
  return cudaSuccess;
}

cudaError_t launch_drift(const DriftPlan& plan, const float* z_fp, const float* z_q, int rows,
                         int vocab, const kvq_drift_params& p, int32_t* m_t, float* c_t,
                         float* d_loc, uint8_t* y_t, float* cov, cudaStream_t st) {
  const auto general =
      plan.stream_threads ? drift_general_kernel<false> : drift_general_kernel<true>;
  cudaError_t e = cudaFuncSetAttribute(general, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(Sm));
  if (e != cudaSuccess) return e;
  if (plan.stream_threads) {
    e = plan.stream_threads == 1024
            ? launch_stream<1024>(z_fp, z_q, rows, vocab, p, m_t, c_t, d_loc, y_t, cov, st)
            : launch_stream<512>(z_fp, z_q, rows, vocab, p, m_t, c_t, d_loc, y_t, cov, st);
    if (e != cudaSuccess) return e;
  }
  // behind a streaming kernel: the rows it leaves, usually none, so the launch
  // overlaps its end
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = plan.stream_threads ? 1 : 0;
  cfg.gridDim = dim3(kCl, plan.clusters);
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = sizeof(Sm);
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, general, z_fp, z_q, rows, vocab, p, m_t, c_t, d_loc, y_t, cov);
}

cudaError_t launch_drift_window(const float* cov, int rows, int k_max, float rho_k,
                                float* mean_cov, int32_t* k_b, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  const int ctas = (long long)rows * k_max > kWinRows * kWinT ? kCl : 1;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = ctas > 1 ? 2 : 1;
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kWinT);
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, drift_window_kernel, cov, rows, k_max, rho_k, mean_cov, k_b);
}

}  // namespace kvq
