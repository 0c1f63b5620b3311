// select.cu -- keep-set selection (Algorithm DoMemRefresh: sigma = argsort of
// the surprise scores, largest first; keep sigma[1:J]).
//
// One cluster of 1, 2, 4 or 8 CTAs per sequence (cluster_size), each CTA over a
// contiguous segment of slots.  Slots rank by the 32-bit monotone key of their
// score, ties toward the later slot.  The J-th largest key T is found by an
// MSB radix select of 11 + 11 + 10 bits: each pass every CTA counts its
// segment's digits in shared memory, the cluster sums the histograms (each
// CTA a slice of the bins, then the slice totals, through distributed shared
// memory), and the pass ends early once the bucket holding the boundary has
// exactly as many keys as are still needed (then every key at or above the
// prefix is kept; 1-2 passes on continuous scores).  If all 32 bits leave a
// tie, the last of the tied slots are kept.  A final pass flags the kept slots
// and writes them in ascending order through block and cluster prefix sums.
//
// Latency bounds it: a pass is a few barriers and round trips.  The segment's
// keys stay in shared memory when they fit.  One CTA per sequence with 256-bin
// passes over the scores in global memory took 18.8 us for 16384 slots and
// 151 us for 131072 (launch after launch); a cluster of eight takes 11.5 and 23.
#include "select.cuh"

#include <atomic>

namespace cc {

namespace {

constexpr int kThreads = 1024;
constexpr int kBins = 2048;
constexpr int kMaxCached = 44 * 1024;        // keys of a segment kept in shared memory at most
constexpr uint32_t kKeyPosInf = 0xFF800000u;   // monotone key of +inf
constexpr uint32_t kKeyNegInf = 0x007FFFFFu;   // monotone key of -inf

// float -> uint32 whose unsigned order is the float order; NaN ranks as -inf.
// -0.0 and +0.0 compare equal as floats, so both take the key of +0.0 (a
// score -logit is -0.0 for a logit of exactly zero); their tie then goes to
// the later slot like any other.
CC_DEV uint32_t monotone_key(float f) {
  uint32_t u = __float_as_uint(f);
  if ((u & 0x7F800000u) == 0x7F800000u && (u & 0x007FFFFFu)) return kKeyNegInf;
  if ((u & 0x7FFFFFFFu) == 0u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The variable at p in CTA `rank` of the cluster of CS.
template <int CS>
CC_DEV uint32_t ld_rank(const uint32_t *p, int rank) {
  if constexpr (CS == 1) return *p;
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_addr(p, rank)) : "memory");
  return v;
}

template <int CS>
CC_DEV void sync_all() {
  if constexpr (CS == 1) __syncthreads();
  else cluster_sync();
}

// Exclusive block scan of x; *total = block sum.  ws: 33 ints of shared memory.
CC_DEV int block_excl_scan(int x, int *ws, int *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int w = ws[lane];
    int wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
      if (lane >= o) wi += y;
    }
    ws[lane] = wi - w;            // exclusive warp offsets
    if (lane == 31) ws[32] = wi;  // block total
  }
  __syncthreads();
  const int r = incl - x + ws[warp];
  *total = ws[32];
  __syncthreads();
  return r;
}

template <int CS>
__global__ void __launch_bounds__(kThreads, 1)
    select_kernel(const float *scores, const int32_t *seq_len, int cap, const int32_t *budget,
                  int n_sink, int32_t *keep_idx, int32_t *keep_count, unsigned *status,
                  int cached) {
  extern __shared__ uint32_t keys[];               // [cached ? segment : 0]
  __shared__ unsigned hist[2][kBins];              // this CTA's digits, two passes in turn
  // keys of this CTA's slice of the bins (over the cluster) in its bins >= i
  __shared__ unsigned at_least[2][kBins + 1];
  __shared__ int ws[33];
  __shared__ int s_digit, s_above, s_count;
  __shared__ unsigned n_kept, n_tied;              // of this CTA's segment
  const int rank = CS == 1 ? 0 : (int)cluster_ctarank();
  const int b = blockIdx.x / CS, tid = threadIdx.x, lane = tid & 31;
  pdl_trigger();
  pdl_wait();   // the scores come from the kernel before
  const int n = seq_len[b];
  if (n < 0 || n > cap) {   // the same in every CTA of the cluster
    if (tid == 0 && rank == 0) {
      set_status(status, CC_ERR_DEVICE_ARG);
      keep_count[b] = 0;
    }
    return;
  }
  const float *s = scores + (size_t)b * cap;
  int32_t *out = keep_idx + (size_t)b * cap;
  int J = budget[b];
  const int forced = min(n, 1 + max(n_sink, 0));
  if (J < forced) {
    if (tid == 0 && rank == 0) set_status(status, CC_ERR_BUDGET);
    J = forced;
  }
  if (J >= n) {  // everything fits: identity
    for (int j = rank * kThreads + tid; j < n; j += CS * kThreads) out[j] = j;
    if (tid == 0 && rank == 0) keep_count[b] = n;
    return;
  }
  // segment [j0, j1) of this CTA: a multiple of 4 slots
  const int seg = ((n + CS - 1) / CS + 3) & ~3;
  const int j0 = min(n, rank * seg), j1 = min(n, j0 + seg);
  auto key_of = [&](int j) -> uint32_t {
    return j < n_sink ? kKeyPosInf : monotone_key(s[j]);
  };
  auto key_at = [&](int j) -> uint32_t { return cached ? keys[j - j0] : key_of(j); };
  for (int i = tid; i < kBins; i += kThreads) hist[0][i] = 0;
  if (cached) {
#pragma unroll 4
    for (int j = j0 + tid; j < j1; j += kThreads) keys[j - j0] = key_of(j);
  }
  __syncthreads();

  // ---- radix select of T = the J-th largest key
  uint32_t prefix = 0;
  int k = J;
  bool settled = false;
  constexpr int per = kBins / CS;   // bins of a slice
#pragma unroll 1
  for (int pass = 0; pass < 3 && !settled; ++pass) {
    const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
    const int bits = pass == 2 ? 10 : 11;
    const uint32_t hi_mask = pass == 0 ? 0u : ~0u << (shift + bits);
    const uint32_t digit_mask = (1u << bits) - 1;
    unsigned *h = hist[pass & 1];
#pragma unroll 4
    for (int j = j0 + tid; j < j1; j += kThreads) {
      const uint32_t key = key_at(j);
      if ((key & hi_mask) == prefix) atomicAdd(&h[(key >> shift) & digit_mask], 1u);
    }
    for (int i = tid; i < kBins; i += kThreads) hist[(pass & 1) ^ 1][i] = 0;   // the next pass's
    sync_all<CS>();
    // this CTA's slice, bins descending over the threads: running counts
    constexpr int PT = per > kThreads ? per / kThreads : 1;   // bins of a thread
    unsigned c[PT], sum = 0;
#pragma unroll
    for (int e = 0; e < PT; ++e) {
      const int i = per - 1 - (tid * PT + e);
      c[e] = 0;
      if (i >= 0) {
#pragma unroll
        for (int r = 0; r < CS; ++r) c[e] += ld_rank<CS>(&h[rank * per + i], r);
      }
      sum += c[e];
    }
    int total;
    unsigned run = (unsigned)block_excl_scan((int)sum, ws, &total);
    unsigned *al = at_least[pass & 1];
#pragma unroll
    for (int e = 0; e < PT; ++e) {
      const int i = per - 1 - (tid * PT + e);
      run += c[e];
      if (i >= 0) al[i] = run;
    }
    if (tid == 0) al[per] = 0;
    sync_all<CS>();
    // the slice that holds the boundary (digits descend from the last slice):
    // every warp reads the slices' totals and finds it alike
    unsigned t = 0;
    if (lane < CS) t = ld_rank<CS>(&al[0], lane);
    unsigned above = 0;   // keys in the slices after this lane's
#pragma unroll
    for (int r = 1; r < CS; ++r) {
      const unsigned y = __shfl_sync(0xFFFFFFFFu, t, r);
      if (r > lane) above += y;
    }
    const unsigned holds =
        __ballot_sync(0xFFFFFFFFu, lane < CS && above < (unsigned)k && (unsigned)k <= above + t);
    const int owner = __ffs((int)holds) - 1;
    above = __shfl_sync(0xFFFFFFFFu, above, owner);
    const unsigned want = (unsigned)k - above;
#pragma unroll
    for (int e = 0; e < PT; ++e) {
      const int i = tid * PT + e;
      if (i >= per) break;
      const unsigned at = ld_rank<CS>(&al[i], owner), over = ld_rank<CS>(&al[i + 1], owner);
      if (over < want && want <= at) {
        s_digit = owner * per + i;
        s_above = (int)(above + over);
        s_count = (int)(at - over);
      }
    }
    __syncthreads();
    prefix |= (uint32_t)s_digit << shift;
    k -= s_above;
    settled = s_count == k;   // the whole bucket is kept
    __syncthreads();
  }
  // Kept: key > T, and of the keys equal to T the last k (all bits used, not
  // settled); settled: key >= prefix (lower bits zero).
  const uint32_t T = prefix;
  const bool ties = !settled;
  if (tid == 0) n_kept = n_tied = 0;
  __syncthreads();
  unsigned kept = 0, tied = 0;
#pragma unroll 4
  for (int j = j0 + tid; j < j1; j += kThreads) {
    const uint32_t key = key_at(j);
    kept += ties ? key > T : key >= T;
    tied += key == T;
  }
  kept = __reduce_add_sync(0xFFFFFFFFu, kept);
  tied = __reduce_add_sync(0xFFFFFFFFu, tied);
  if (lane == 0 && kept) atomicAdd(&n_kept, kept);
  if (lane == 0 && tied) atomicAdd(&n_tied, tied);
  sync_all<CS>();
  int base = 0, tie_base = 0, tie_total = 0;   // before this segment; over the sequence
#pragma unroll
  for (int r = 0; r < CS; ++r) {
    const int a = (int)ld_rank<CS>(&n_kept, r);
    const int t = (int)ld_rank<CS>(&n_tied, r);
    if (r < rank) {
      base += a;
      tie_base += t;
    }
    tie_total += t;
  }
  if (ties) {   // tied slots before the segment that are kept: those past the first total - k
    const int first = tie_total - k;
    base += max(0, tie_base - first);
  }

  // ---- flag and emit the kept slots in ascending order
  int carry = base, tie_carry = tie_base;
  for (int jb = j0; jb < j1; jb += kThreads * 4) {
    const int ja = jb + tid * 4;
    int f[4], t[4], cnt = 0, tcnt = 0, total;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int j = ja + e;
      const uint32_t key = j < j1 ? key_at(j) : 0u;
      f[e] = j < j1 && (ties ? key > T : key >= T);
      t[e] = ties && j < j1 && key == T;
      tcnt += t[e];
    }
    if (ties) {
      int idx = tie_carry + block_excl_scan(tcnt, ws, &total);
      tie_carry += total;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (t[e] && idx >= tie_total - k) f[e] = 1;
        idx += t[e];
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) cnt += f[e];
    int off = carry + block_excl_scan(cnt, ws, &total);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (f[e]) out[off++] = ja + e;
    carry += total;
  }
  if (tid == 0 && rank == CS - 1) {
    keep_count[b] = J;
    if (carry != J) set_status(status, CC_ERR_DEVICE_ARG);   // cannot happen
  }
  sync_all<CS>();   // no CTA reads this one's counts any more
}

// CTAs per sequence of a launch: one up to 8192 slots (launch after launch, one and
// eight CTAs: 9.2 / 10.8 us there, 14.3 / 11.5 at 16384), eight above while every
// sequence's cluster is resident; else the least estimated time over the sizes, the
// clusters in as many waves as they need.  Fitted to every size at batches of 1 to
// 256 and caps of 4096 to 131072: a lone CTA 5.5 us + 0.65 ns a slot, 1.24 ns past
// the slots whose keys it holds; a cluster 12 us + 0.8 ns a slot of a CTA.  Eight
// CTAs whatever the batch took 103 us for 128 sequences of 16384 slots, one CTA each
// 16 us.
int cluster_size(int batch, int cap, uint64_t resident) {   // (16 bits per size)
  if (cap <= 8192) return 1;
  if (batch <= (int)(resident >> 48)) return 8;
  int best = 1;
  double least = 1e300;
  for (int i = 0; i < 4; ++i) {
    const int cs = 1 << i;
    const double seg = (double)cap / cs;
    const double one = (i == 0 ? 5.5e3 : 12e3) +
                       seg * (seg > kMaxCached ? 1.24 : i == 0 ? 0.65 : 0.8);
    const double t = ceil((double)batch / (double)(resident >> (16 * i) & 0xFFFF)) * one;
    if (t < least) {
      least = t;
      best = cs;
    }
  }
  return best;
}

}  // namespace

cudaError_t launch_select(const float *scores, const int32_t *seq_len, int batch, int cap,
                          const int32_t *budget, int n_sink, int32_t *keep_idx,
                          int32_t *keep_count, unsigned *status, cudaStream_t st) {
  if (batch <= 0) return cudaSuccess;
  using Kernel = decltype(&select_kernel<1>);
  const Kernel kerns[4] = {select_kernel<1>, select_kernel<2>, select_kernel<4>, select_kernel<8>};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  static std::atomic<uint64_t> resident[64];   // clusters resident with full segments (0: unknown)
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  uint64_t fit = resident[dev].load();
  if (fit == 0) {
    for (int i = 0; i < 4; ++i) {
      cudaError_t e = cudaFuncSetAttribute(kerns[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kMaxCached * 4);
      if (e != cudaSuccess) return e;
      attr[0].val.clusterDim.x = 1u << i;
      cfg.gridDim = dim3(1u << i);
      cfg.dynamicSmemBytes = kMaxCached * 4;
      cfg.numAttrs = 1;
      int n = 0;
      e = cudaOccupancyMaxActiveClusters(&n, kerns[i], &cfg);
      if (e != cudaSuccess) return e;
      fit |= (uint64_t)(n < 1 ? 1 : n > 0xFFFF ? 0xFFFF : n) << (16 * i);
    }
    resident[dev].store(fit);
  }
  const int cs = cluster_size(batch, cap, fit);
  const int seg = ((cap + cs - 1) / cs + 3) & ~3;   // slots of a segment at most
  const int cached = seg <= kMaxCached ? 1 : 0;
  attr[0].val.clusterDim.x = (unsigned)cs;
  cfg.gridDim = dim3((unsigned)(batch * cs));
  cfg.dynamicSmemBytes = cached ? (size_t)seg * 4 : 0;
  cfg.numAttrs = 2;
  const Kernel kern = cs == 1 ? kerns[0] : cs == 2 ? kerns[1] : cs == 4 ? kerns[2] : kerns[3];
  return cudaLaunchKernelEx(&cfg, kern, scores, seq_len, cap, budget, n_sink, keep_idx,
                            keep_count, status, cached);
}

}  // namespace cc
