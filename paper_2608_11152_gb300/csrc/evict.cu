// Eviction down to capacity (K4c): after a commit's inserts, each instance whose index
// holds E = size - Cap_w > 0 entries too many loses its E smallest (meta, key): the
// least recently committed blocks, deepest first among equal ticks (Sec. 4.4 reading:
// LRU; the commit-tick order keeps every index prefix-closed).
//
// Admissions concentrate on few instances (every cold request of a round prefers the
// same cheapest instance), so E ranges from 0 to a large part of an instance; the work
// is spread over many CTAs per instance and the one serial step is kept small:
//   k4_evict_estimate  (1 CTA / instance)  histogram of the metas of up to 2048 buckets -> a meta
//                      bracket [lo, hi] that contains the E-th smallest w.h.p. (for sure where
//                      that is the whole table)
//   k4_evict_collect   (many CTAs / instance, streaming)  fullness bitmap; entries with
//                      meta < lo are certainly evicted (slot list D), entries with
//                      lo <= meta <= hi go to a short list U with their values and slots
//   k4_evict_select    (1 CTA / instance)  theta = the (E - |D|)-th smallest of U: the bin of
//                      a histogram that holds it, then by counting ranks; if the bracket
//                      missed, the CTA re-collects the whole instance and selects exactly anyway
//   k4_evict_delete    deletes D and the entries of U at or below theta; those that leave a hole
//                      in a full bucket are listed
//   k4_evict_shift     refills the holes of every run of full buckets that lost an entry
//                      with backward shifts (no tombstones), one thread per run
#include "common.cuh"
#include "kernels.h"
#include "tick_scale.h"

namespace misat {

namespace {
constexpr unsigned kFull = 0xffffffffu;
constexpr int kEstThreads = 512;
constexpr int kBins = kTickBins;
constexpr int kEstBuckets = 2048;  // sampled per instance, four by each thread
constexpr int kSelSmem = 1024;      // candidates kept in shared memory
constexpr int kRankMax = 64;        // candidates that are ranked by counting

__device__ __forceinline__ bool le128(uint64_t ma, uint64_t ka, uint64_t mb, uint64_t kb) {
  return ma < mb || (ma == mb && ka <= kb);
}

__device__ __forceinline__ uint64_t v_hi(const uint4& v) { return ((unsigned long long)v.y << 32) | v.x; }
__device__ __forceinline__ uint64_t v_lo(const uint4& v) { return ((unsigned long long)v.w << 32) | v.z; }

// Block-wide (T threads): bin t with cum(<t) < E <= cum(<=t), 1 <= E <= all; cum(<t) in
// *below.
template <int T>
__device__ int find_threshold_bin(const uint32_t* hist, uint32_t E, uint32_t* below) {
  constexpr int kPer = kBins / T;
  __shared__ uint32_t s_tmp[32];
  __shared__ int s_bin;
  __shared__ uint32_t s_below;
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  uint32_t h[kPer], local = 0;
#pragma unroll
  for (int i = 0; i < kPer; i += 4) {
    const uint4 v = reinterpret_cast<const uint4*>(hist + kPer * t)[i / 4];
    h[i] = v.x;
    h[i + 1] = v.y;
    h[i + 2] = v.z;
    h[i + 3] = v.w;
    local += v.x + v.y + v.z + v.w;
  }
  uint32_t incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s_tmp[wid] = incl;
  if (t == 0) s_bin = -1;
  __syncthreads();
  uint32_t c = incl - local + __reduce_add_sync(kFull, lane < wid ? s_tmp[lane] : 0u);
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    if (c < E && E <= c + h[i]) {
      s_bin = kPer * t + i;
      s_below = c;
    }
    c += h[i];
  }
  __syncthreads();
  *below = s_below;
  const int bin = s_bin;
  __syncthreads();
  return bin;
}

// 12 bits of the 128-bit value (hi:lo) starting at bit `shift`.
__device__ __forceinline__ uint32_t digit128(uint64_t hi, uint64_t lo, int shift) {
  if (shift >= 64) return (uint32_t)(hi >> (shift - 64)) & (kBins - 1);
  uint64_t v = lo >> shift;
  if (shift > 0 && shift + 12 > 64) v |= hi << (64 - shift);
  return (uint32_t)v & (kBins - 1);
}

}  // namespace

struct EstPart {
  unsigned long long mn, mx;   // smallest and largest sampled meta
  unsigned occ, arr, dep;      // samples, their largest arrival and depth
};
constexpr int kEstMetas = 4 * kEstBuckets / kEstThreads;  // per thread

// The thread's metas of nsb of the table's NB buckets (powers of two), evenly spaced: slot s of
// sampled bucket threadIdx.x + k kEstThreads is m[4k + s].
__device__ __forceinline__ void load_metas(const InstDesc& d, uint32_t NB, uint32_t nsb, unsigned long long* m) {
#pragma unroll
  for (int k = 0; k < kEstMetas / 4; ++k) {
    const uint32_t i = threadIdx.x + k * kEstThreads;
    ulonglong2 m01 = make_ulonglong2(0, 0), m23 = m01;
    if (i < nsb) {
      const ulonglong2* mp = reinterpret_cast<const ulonglong2*>(d.tab[i * (NB / nsb)].meta);
      m01 = __ldcg(mp);
      m23 = __ldcg(mp + 1);
    }
    m[4 * k] = m01.x;
    m[4 * k + 1] = m01.y;
    m[4 * k + 2] = m23.x;
    m[4 * k + 3] = m23.y;
  }
}

// Range of the block's metas (one block barrier).
__device__ __forceinline__ EstPart sample_range(const unsigned long long* m, EstPart* s_part) {
  unsigned long long mn = ~0ull, mx = 0;
  unsigned occ = 0, arr = 0, dep = 0;
#pragma unroll
  for (int k = 0; k < kEstMetas; ++k)
    if (m[k]) {
      ++occ;
      mn = m[k] < mn ? m[k] : mn;
      mx = m[k] > mx ? m[k] : mx;
      arr = max(arr, (unsigned)(m[k] >> 16) & 0xfffffu);
      dep = max(dep, 0xffffu - ((unsigned)m[k] & 0xffffu));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long a1 = __shfl_xor_sync(kFull, mn, o), a2 = __shfl_xor_sync(kFull, mx, o);
    mn = a1 < mn ? a1 : mn;
    mx = a2 > mx ? a2 : mx;
  }
  occ = __reduce_add_sync(kFull, occ);
  arr = __reduce_max_sync(kFull, arr);
  dep = __reduce_max_sync(kFull, dep);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = EstPart{mn, mx, occ, arr, dep};
  __syncthreads();
  EstPart all = s_part[0];
#pragma unroll
  for (int k = 1; k < kEstThreads / 32; ++k) {
    const EstPart p = s_part[k];
    all.mn = p.mn < all.mn ? p.mn : all.mn;
    all.mx = p.mx > all.mx ? p.mx : all.mx;
    all.occ += p.occ;
    all.arr = max(all.arr, p.arr);
    all.dep = max(all.dep, p.dep);
  }
  return all;
}

// Bound by latency: one round of loads and a few block barriers.  The samples stay in registers,
// and a bin is a shift (with 128-bit quotients of equal bins it took 16 us, on tables of any
// size); 2,048 buckets instead of 512 make the bracket, and U with it, half as wide.
__global__ void __launch_bounds__(kEstThreads) k4_evict_estimate(EvictArgs a) {
  constexpr int kPer = kEstBuckets / kEstThreads;
  __shared__ __align__(16) uint32_t hist[kBins];
  __shared__ EstPart s_part[kEstThreads / 32];
  chain_wait();
  const int w = a.only_w ? *a.only_w : blockIdx.x;
  if (block_error(a.err)) return;
  const long long size = a.size[w];
  const InstDesc d = a.desc[w];
  const long long E = size - d.cap;
  const int tid = threadIdx.x;
  if (tid == 0) {
    a.active[w] = E > 0 ? 1 : 0;
    a.n_d[w] = 0;
    a.n_cand[w] = 0;
    a.n_holes[w] = 0;
    if (E > 0) a.act[atomicAdd(a.n_act, 1u)] = w;  // the streaming passes visit only these
  }
  if (E <= 0) return;
  const uint32_t NB = 1u << d.log2nb;
  const uint32_t nsb = NB < (uint32_t)kEstBuckets ? NB : (uint32_t)kEstBuckets;  // powers of two
  unsigned long long m[4 * kPer];
  load_metas(d, NB, nsb, m);
  for (int i = tid; i < kBins; i += kEstThreads) hist[i] = 0;
  const EstPart all = sample_range(m, s_part);
  const unsigned n = all.occ;
  const TickScale ts{32 - __clz(all.arr), 32 - __clz(all.dep)};
  unsigned long long lo = 0, hi = ~0ull;
  if (n > 0) {
    // histogram of the samples from their minimum on, bins of 2^shift
    const unsigned long long smin = ts.pack(all.mn);
    const int shift = bin_shift(ts.pack(all.mx) - smin);
#pragma unroll
    for (int k = 0; k < 4 * kPer; ++k)
      if (m[k]) atomicAdd(&hist[(uint32_t)((ts.pack(m[k]) - smin) >> shift)], 1u);
    __syncthreads();
    // the E-th smallest sits near sample rank p = E n / size (exactly there in a whole table);
    // bracket it by ~3 standard deviations of the sample count plus a constant on both sides
    // (in 32 bits: 64-bit floating point is slow here, and a miss costs time only)
    const float p = (float)E * ((float)n / (float)size);
    const float margin = 3.0f * sqrtf(p + 1.0f) + 16.0f;
    const long long rl = nsb == NB ? E : (long long)(p - margin), rh = nsb == NB ? E : (long long)(p + margin) + 1;
    uint32_t below;
    const int bl = rl >= 1 && rl <= (long long)n ? find_threshold_bin<kEstThreads>(hist, (uint32_t)rl, &below) : -1;
    const int bh = rh < 1 || rh > (long long)n ? -1
                   : rh == rl                  ? bl
                                               : find_threshold_bin<kEstThreads>(hist, (uint32_t)rh, &below);
    // every sample of bin b packs to [smin + b 2^shift, smin + (b + 1) 2^shift - 1]
    if (bl >= 0) lo = ts.unpack(smin + ((unsigned long long)bl << shift));
    if (bh >= 0) hi = ts.unpack(smin + ((unsigned long long)(bh + 1) << shift)) - 1;
  }
  if (tid == 0) {
    a.thr_lo[w] = lo;
    a.thr_hi[w] = hi;
    a.scale[w] = make_int2(ts.ab, ts.db);
  }
}

// Streaming pass over the instance's metas: chunk `cidx` of `chunks` of instance w, a range
// of whole 32-bucket bitmap words.  A CTA takes 4 x blockDim buckets at a time: each thread
// loads the metas of four buckets (all loads in flight together), keeps only which slots
// are certainly evicted (meta < lo) or candidates (lo <= meta <= hi) as bit masks, writes
// the fullness bitmap words and clears the deleted-slot masks; the list entries are
// reserved with one CTA-wide scan per step, and only candidates re-read their meta and key.
__device__ __forceinline__ void collect_chunk(const EvictArgs& a, int w, uint32_t cidx, uint32_t chunks) {
  __shared__ unsigned s_wd[32], s_wu[32], s_bd, s_bu;
  const InstDesc d = a.desc[w];
  const uint32_t NB = 1u << d.log2nb;
  const unsigned long long lo = a.thr_lo[w], hi = a.thr_hi[w];
  uint32_t* bitmap = a.bitmaps[w];
  uint32_t* dmask = a.dmask[w];
  uint32_t* dsl = a.dslots[w];
  uint4* u = a.cand_a[w];
  uint32_t* usl = a.slots[w];
  const int lane = threadIdx.x & 31;
  const int wid = threadIdx.x >> 5;
  const uint32_t words = (NB + 31) >> 5;
  const uint32_t b_beg = (uint32_t)(((uint64_t)words * cidx / chunks) << 5);
  const uint32_t b_end = min(NB, (uint32_t)(((uint64_t)words * (cidx + 1) / chunks) << 5));
  for (uint32_t base = b_beg; base < b_end; base += 4 * blockDim.x) {
    ulonglong2 m01[4], m23[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t b = base + k * blockDim.x + threadIdx.x;
      if (b < b_end) {
        const ulonglong2* mp = reinterpret_cast<const ulonglong2*>(d.tab[b].meta);
        m01[k] = __ldcg(mp);
        m23[k] = __ldcg(mp + 1);
      } else {
        m01[k] = make_ulonglong2(0, 0);
        m23[k] = make_ulonglong2(0, 0);
      }
    }
    unsigned dm = 0, um = 0;  // bit 4k + s: slot s of this thread's k-th bucket
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t b = base + k * blockDim.x + threadIdx.x;
      const unsigned long long m[4] = {m01[k].x, m01[k].y, m23[k].x, m23[k].y};
      const bool full = m[0] && m[1] && m[2] && m[3];
      const unsigned bits = __ballot_sync(kFull, full);
      if (lane == 0 && b < b_end) bitmap[b >> 5] = bits;
      if ((lane & 7) == 0 && b < b_end) dmask[b >> 3] = 0;
#pragma unroll
      for (int sl = 0; sl < 4; ++sl) {
        if (!m[sl]) continue;
        if (m[sl] < lo) dm |= 1u << (4 * k + sl);
        else if (m[sl] <= hi) um |= 1u << (4 * k + sl);
      }
    }
    const int nd = __popc(dm), nu = __popc(um);
    // CTA-wide reservation in both lists: warp scans, then one atomic pair per CTA
    int id = nd, iu = nu;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int vd = __shfl_up_sync(kFull, id, o), vu = __shfl_up_sync(kFull, iu, o);
      if (lane >= o) {
        id += vd;
        iu += vu;
      }
    }
    if (lane == 31) {
      s_wd[wid] = id;
      s_wu[wid] = iu;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned td = 0, tu = 0;
      for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
        const unsigned xd = s_wd[k], xu = s_wu[k];
        s_wd[k] = td;
        s_wu[k] = tu;
        td += xd;
        tu += xu;
      }
      s_bd = td ? atomicAdd(&a.n_d[w], td) : 0;
      s_bu = tu ? atomicAdd(&a.n_cand[w], tu) : 0;
    }
    __syncthreads();
    unsigned bd = s_bd + s_wd[wid] + (unsigned)(id - nd);
    unsigned bu = s_bu + s_wu[wid] + (unsigned)(iu - nu);
    __syncthreads();  // the shared offsets are rewritten by the next step
    while (dm) {
      const int bit = __ffs(dm) - 1;
      dm &= dm - 1;
      const uint32_t b = base + (bit >> 2) * blockDim.x + threadIdx.x;
      dsl[bd++] = b * 4 + (bit & 3);
    }
    while (um) {
      const int bit = __ffs(um) - 1;
      um &= um - 1;
      const uint32_t b = base + (bit >> 2) * blockDim.x + threadIdx.x;
      const int sl = bit & 3;
      const unsigned long long x = __ldcg(&d.tab[b].meta[sl]);
      const unsigned long long key = __ldcg(&d.tab[b].key[sl]);
      u[bu] = make_uint4((uint32_t)x, (uint32_t)(x >> 32), (uint32_t)key, (uint32_t)(key >> 32));
      usl[bu] = b * 4 + sl;
      ++bu;
    }
  }
}

// Work items (active instance, chunk), taken by a grid of resident CTAs: instances within
// capacity cost nothing (their list entries are never made).
__global__ void __launch_bounds__(256) k4_evict_collect(EvictArgs a, uint32_t chunks) {
  chain_wait();
  if (block_error(a.err)) return;
  const uint32_t items = *(volatile const unsigned*)a.n_act * chunks;
  for (uint32_t it = blockIdx.x; it < items; it += gridDim.x) collect_chunk(a, a.act[it / chunks], it % chunks, chunks);
}

// T: 1,024 threads while there is an SM per instance; where there are more instances (their tables
// are small then) 256, so that eight or more of them share an SM.
template <int T>
__global__ void __launch_bounds__(T) k4_evict_select(EvictArgs a) {
  __shared__ __align__(16) uint32_t hist[kBins];
  __shared__ uint4 s_v[kSelSmem], s_r[kRankMax];
  __shared__ unsigned s_cnt;
  __shared__ unsigned long long s_or_hi, s_or_lo;
  chain_wait();
  const int w = a.only_w ? *a.only_w : blockIdx.x;
  if (block_error(a.err)) return;
  if (a.active[w] != 1) return;
  const InstDesc d = a.desc[w];
  const long long E = a.size[w] - d.cap;
  const int tid = threadIdx.x;
  const uint32_t NB = 1u << d.log2nb;
  uint4* c0 = a.cand_a[w];
  unsigned cnt = a.n_cand[w];
  const unsigned nd = a.n_d[w];
  long long Erem = E - (long long)nd;
  const bool bracketed = Erem > 0 && Erem <= (long long)cnt, open = a.thr_hi[w] == ~0ull;
  if (!bracketed) {
    // the bracket missed the E-th smallest: collect every entry of the instance here
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    uint32_t* usl = a.slots[w];
    for (uint32_t b = tid; b < NB; b += T) {
      for (int s = 0; s < 4; ++s) {
        const unsigned long long m = __ldcg(&d.tab[b].meta[s]);
        if (!m) continue;
        const unsigned long long key = __ldcg(&d.tab[b].key[s]);
        const unsigned pos = atomicAdd(&s_cnt, 1u);
        c0[pos] = make_uint4((uint32_t)m, (uint32_t)(m >> 32), (uint32_t)key, (uint32_t)(key >> 32));
        usl[pos] = b * 4 + s;
      }
    }
    __syncthreads();
    cnt = s_cnt;
    __syncthreads();  // the counter is cleared again below
    Erem = E;
    if (tid == 0) {
      a.n_cand[w] = cnt;
      a.n_d[w] = 0;
    }
  }
  // radix narrowing while there are many candidates, keeping the bin that holds the target, in
  // shared memory as soon as it fits (the collected list, with its slots, is kept for the delete
  // pass).  The first pass spreads the bracket over the bins in the samples' scale, which leaves a
  // few entries; the others, hardly ever needed, take the 12 bits below the highest bit in which
  // the entries differ.
  const int2 sc = a.scale[w];
  const TickScale ts{sc.x, sc.y};
  const unsigned long long plo = ts.pack(a.thr_lo[w]);
  const int tick_shift = bin_shift(ts.pack(a.thr_hi[w]) - plo);
  const uint4* cur = c0;
  for (int iter = 0; iter < 16 && cnt > (unsigned)kRankMax; ++iter) {
    const bool tick = iter == 0 && bracketed && !open;
    int shift = 0;
    if (tid == 0) {
      s_or_hi = 0;
      s_or_lo = 0;
      s_cnt = 0;
    }
    for (int i = tid; i < kBins; i += T) hist[i] = 0;
    __syncthreads();
    if (!tick) {
      const uint4 v0 = cur[0];
      unsigned long long oh = 0, ol = 0;
#pragma unroll 4
      for (unsigned i = tid; i < cnt; i += T) {
        const uint4 v = cur[i];
        oh |= v_hi(v) ^ v_hi(v0);
        ol |= v_lo(v) ^ v_lo(v0);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        oh |= __shfl_xor_sync(kFull, oh, o);
        ol |= __shfl_xor_sync(kFull, ol, o);
      }
      if ((tid & 31) == 0) {
        if (oh) atomicOr(&s_or_hi, oh);
        if (ol) atomicOr(&s_or_lo, ol);
      }
      __syncthreads();
      const unsigned long long dh = s_or_hi, dl = s_or_lo;
      if (dh == 0 && dl == 0) break;  // all equal (cannot happen for distinct keys)
      const int top = dh ? 64 + 63 - __clzll((long long)dh) : 63 - __clzll((long long)dl);
      shift = top >= 11 ? top - 11 : 0;
    }
    auto bin_of = [&](const uint4& v) {
      return tick ? (uint32_t)((ts.pack(v_hi(v)) - plo) >> tick_shift) : digit128(v_hi(v), v_lo(v), shift);
    };
#pragma unroll 4
    for (unsigned i = tid; i < cnt; i += T) {
      const uint4 v = cur[i];
      atomicAdd(&hist[bin_of(v)], 1u);
    }
    __syncthreads();
    uint32_t bl;
    const int bin = find_threshold_bin<T>(hist, (uint32_t)Erem, &bl);
    if (bin < 0) {  // the table holds fewer entries than its size says
      if (tid == 0) set_error(a.err, MISAT_ERR_INTERNAL);
      return;
    }
    Erem -= bl;
    const unsigned kept = hist[bin];
    uint4* nxt = kept <= (unsigned)kRankMax                 ? s_r
                 : kept <= (unsigned)kSelSmem && cur != s_v ? s_v
                                                            : (cur == a.cand_b[w] ? a.cand_c[w] : a.cand_b[w]);
#pragma unroll 4
    for (unsigned i0 = 0; i0 < cnt; i0 += T) {
      // keep the target bin: one shared add per warp, positions by ballot rank
      const unsigned i = i0 + tid;
      uint4 v = make_uint4(0, 0, 0, 0);
      bool keep = false;
      if (i < cnt) {
        v = cur[i];
        keep = bin_of(v) == (uint32_t)bin;
      }
      const unsigned bal = __ballot_sync(kFull, keep);
      unsigned base = 0;
      if ((tid & 31) == 0 && bal) base = atomicAdd(&s_cnt, (unsigned)__popc(bal));
      base = __shfl_sync(kFull, base, 0);
      if (keep) nxt[base + __popc(bal & lanemask_lt())] = v;
    }
    __syncthreads();
    cnt = kept;
    cur = nxt;
  }
  if (cnt > (unsigned)kRankMax || cnt < 1) {  // no instance holds two equal entries
    if (tid == 0) set_error(a.err, MISAT_ERR_TABLE_FULL);
    return;
  }
  if (cur != s_r)
    for (unsigned i = tid; i < cnt; i += T) s_r[i] = cur[i];
  __syncthreads();
  // the target has Erem - 1 entries below it
  if (tid < (int)cnt) {
    const uint64_t mh = v_hi(s_r[tid]), ml = v_lo(s_r[tid]);
    int rank = 0;
#pragma unroll 4
    for (unsigned j = 0; j < cnt; ++j) {
      const uint64_t oh = v_hi(s_r[j]), ol = v_lo(s_r[j]);
      rank += oh < mh || (oh == mh && ol < ml);
    }
    if (rank == (int)(Erem - 1)) {
      a.theta[2 * w] = mh;
      a.theta[2 * w + 1] = ml;
    }
  }
}

namespace {
// The apply passes take the entries of all instances over capacity as one index space, so
// that every thread gets about the same number whatever the instances' shares: entry g
// belongs to the k-th active instance with s_pre[k] <= g < s_pre[k + 1].  Built by each CTA in
// shared memory from the instances' list lengths; returns the total.
template <class F>
__device__ unsigned long long list_prefix(const EvictArgs& a, unsigned long long* s_pre, int nact, F&& len) {
  // the lengths are loaded in parallel, then warp 0 scans them 32 at a time
  for (int k = threadIdx.x; k < nact; k += blockDim.x) {
    s_pre[k + 1] = len(a.act[k]);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    unsigned long long carry = 0;
    for (int k0 = 0; k0 < nact; k0 += 32) {
      const int k = k0 + lane;
      const unsigned long long v = k < nact ? s_pre[k + 1] : 0;
      unsigned long long incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += t;
      }
      if (k < nact) s_pre[k + 1] = carry + incl;
      carry += __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) s_pre[0] = 0;
  }
  __syncthreads();
  return s_pre[nact];
}

// The k with s_pre[k] <= g < s_pre[k + 1] (binary search over nact entries).
__device__ __forceinline__ int list_owner(const unsigned long long* s_pre, int nact, unsigned long long g) {
  int lo = 0, hi = nact - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (s_pre[mid] <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

}  // namespace

// Delete D and the candidates at or below theta; record them in the deleted-slot masks, and those in
// full buckets in the list of holes to refill (a fifth of them).  A CTA takes pieces of 1,024
// entries of one instance's lists (D first), four a thread with their loads in flight together:
// what bounds it is the chain slot -> bitmap, slot -> key -> global index of scattered accesses.
// The counters get one atomic per piece (with one per warp the pass waited for them: 95 us for
// 1.5 million deletions).
constexpr int kDelPer = 4;
constexpr int kDelPiece = 256 * kDelPer;
__global__ void __launch_bounds__(256) k4_evict_delete(EvictArgs a) {
  __shared__ unsigned long long s_pre[kMaxW + 1];
  __shared__ unsigned s_cnt[2], s_base;
  chain_wait();
  if (block_error(a.err)) return;
  const int nact = (int)*(volatile const unsigned*)a.n_act;
  auto len = [&](int w) { return (unsigned long long)a.n_d[w] + a.n_cand[w]; };
  const unsigned long long total =
      list_prefix(a, s_pre, nact, [&](int w) { return (len(w) + kDelPiece - 1) / kDelPiece; });
  const int lane = threadIdx.x & 31;
  unsigned long long mine = 0;
  for (unsigned long long it = blockIdx.x; it < total; it += gridDim.x) {
    const int k = list_owner(s_pre, nact, it);
    const int w = a.act[k];
    const unsigned nd = a.n_d[w], n = nd + a.n_cand[w];
    const unsigned i0 = (unsigned)(it - s_pre[k]) * kDelPiece + threadIdx.x;
    const unsigned long long tm = a.theta[2 * w], tk = a.theta[2 * w + 1];
    const uint32_t* bitmap = a.bitmaps[w];
    Bucket* tab = a.desc[w].tab;
    uint32_t* dmask = a.dmask[w];
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    uint32_t sl[kDelPer];
    bool del[kDelPer], hole[kDelPer];
#pragma unroll
    for (int j = 0; j < kDelPer; ++j) {
      const unsigned i = i0 + 256 * j;
      del[j] = i < n;
      sl[j] = 0;
      if (del[j]) {
        sl[j] = i < nd ? a.dslots[w][i] : a.slots[w][i - nd];
        if (i >= nd) {
          const uint4 v = a.cand_a[w][i - nd];
          del[j] = le128(v_hi(v), v_lo(v), tm, tk);
        }
      }
    }
    // a hole in a bucket that was not full, the last of its run, needs no refill
#pragma unroll
    for (int j = 0; j < kDelPer; ++j) hole[j] = del[j] && ((bitmap[sl[j] >> 7] >> ((sl[j] >> 2) & 31)) & 1u);
    unsigned at[kDelPer];
#pragma unroll
    for (int j = 0; j < kDelPer; ++j) {
      const unsigned md = __ballot_sync(kFull, del[j]), mh = __ballot_sync(kFull, hole[j]);
      unsigned base = 0;
      if (lane == 0) {
        if (md) atomicAdd(&s_cnt[0], (unsigned)__popc(md));
        if (mh) base = atomicAdd(&s_cnt[1], (unsigned)__popc(mh));
      }
      at[j] = __shfl_sync(kFull, base, 0) + __popc(mh & lanemask_lt());
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      if (s_cnt[0]) atomic_add_i64(&a.size[w], -(long long)s_cnt[0]);
      mine += s_cnt[0];
      s_base = s_cnt[1] ? atomicAdd(&a.n_holes[w], s_cnt[1]) : 0;
    }
    if (a.gix.keys) {
      unsigned long long key[kDelPer];
#pragma unroll
      for (int j = 0; j < kDelPer; ++j) key[j] = del[j] ? tab[sl[j] >> 2].key[sl[j] & 3] : 0;
#pragma unroll
      for (int j = 0; j < kDelPer; ++j)
        if (del[j] && gix_clear(a.gix, key[j], w) < 0) set_error(a.err, MISAT_ERR_INTERNAL);
    }
#pragma unroll
    for (int j = 0; j < kDelPer; ++j)
      if (del[j]) {
        const uint32_t b = sl[j] >> 2, s = sl[j] & 3;
        tab[b].key[s] = kEmpty;
        tab[b].meta[s] = 0;
        atomicOr(&dmask[b >> 3], 1u << ((b & 7) * 4 + s));
      }
    __syncthreads();
    uint32_t* list = reinterpret_cast<uint32_t*>(a.cand_b[w]) + s_base;
#pragma unroll
    for (int j = 0; j < kDelPer; ++j)
      if (hole[j]) list[at[j]] = sl[j];
  }
  if (threadIdx.x == 0 && mine) atomicAdd(a.evicted, mine);
}

namespace {
// Refills the holes of the run of full buckets that deleted slot sl of a full bucket belongs to, if
// that is the run's first deleted slot (lowest bucket, then lowest slot).  full, dmask: the
// table's fullness bits and deleted slots (four bits a bucket) before any refill.
__device__ __forceinline__ void refill_run(const InstDesc d, const uint32_t* full, const uint32_t* dmask, uint32_t sl) {
  const uint32_t NB = 1u << d.log2nb, mask = NB - 1;
  // the bitmap and deleted-mask words last read (runs are short: mostly one word each)
  uint32_t fw_i = 0xffffffffu, fw = 0, dw_i = 0xffffffffu, dw = 0;
  auto is_full = [&](uint32_t b) {
    if ((b >> 5) != fw_i) {
      fw_i = b >> 5;
      fw = full[fw_i];
    }
    return (fw >> (b & 31)) & 1u;
  };
  auto dmask_at = [&](uint32_t b) {
    if ((b >> 3) != dw_i) {
      dw_i = b >> 3;
      dw = dmask[dw_i];
    }
    return (dw >> ((b & 7) * 4)) & 0xFu;
  };
  const uint32_t x = sl >> 2, sx = sl & 3;
  // my deletion must be the lowest deleted slot of bucket x (the masks are not modified
  // by this kernel, unlike the buckets)
  if ((uint32_t)(__ffs(dmask_at(x)) - 1) != sx) return;
  // run start: walk back over full buckets; no earlier bucket of the run may hold a deletion
  uint32_t s0 = x, len = 0;
  bool lead = true;
  while (is_full((s0 - 1) & mask) && len < NB) {
    s0 = (s0 - 1) & mask;
    ++len;
    if (dmask_at(s0)) {
      lead = false;
      break;
    }
  }
  if (!lead) return;
  // run end: the first bucket after x that was not full
  uint32_t e = x, rl = 0;
  while (is_full(e) && rl < NB) {
    e = (e + 1) & mask;
    ++rl;
  }
  const uint32_t runlen = ((e - s0) & mask);  // buckets s0 .. e-1 are full, e ends the run
  for (uint32_t ii = 0; ii < runlen; ++ii) {
    Bucket* X = d.tab + ((s0 + ii) & mask);
    unsigned long long xk[4];
    {
      const ulonglong2* p = reinterpret_cast<const ulonglong2*>(X->key);
      const ulonglong2 u0 = p[0], u1 = p[1];
      xk[0] = u0.x;
      xk[1] = u0.y;
      xk[2] = u1.x;
      xk[3] = u1.y;
    }
    bool stop = false;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (stop || xk[s] != kEmpty) continue;
      bool moved = false;
      for (uint32_t j = ii + 1; j <= runlen && !moved; ++j) {
        Bucket* Y = d.tab + ((s0 + j) & mask);
        const ulonglong2* p = reinterpret_cast<const ulonglong2*>(Y->key);
        const ulonglong2 u0 = p[0], u1 = p[1];
        const unsigned long long yk[4] = {u0.x, u0.y, u1.x, u1.y};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const unsigned long long k = yk[t];
          if (moved || k == kEmpty) continue;
          const uint32_t rel = (home_bucket(k, d.log2nb) - s0) & mask;
          if (rel <= ii) {
            X->key[s] = k;
            X->meta[s] = Y->meta[t];
            Y->key[t] = kEmpty;
            Y->meta[t] = 0;
            xk[s] = k;
            moved = true;
          }
        }
      }
      if (!moved) stop = true;  // no later entry of the run can move into this bucket
    }
  }
}
}  // namespace

// Refill the holes of every run of full buckets that lost an entry.  The thread of the
// run's first deleted slot (lowest bucket, then lowest slot) owns the run.  Bound by the latency of
// its owner's dependent reads, five to ten for most runs, and lanes of a warp that walk different
// runs take turns: only holes that may need a refill are listed (with all deletions and
// candidates, ten a thread, it took 148 us in a batch of 65,536 requests), and neighbours in
// the list go to different warps, so that a warp has more than one only when all have.
__global__ void __launch_bounds__(256) k4_evict_shift(EvictArgs a) {
  __shared__ unsigned long long s_pre[kMaxW + 1];
  chain_wait();
  if (block_error(a.err)) return;
  const int nact = (int)*(volatile const unsigned*)a.n_act;
  const unsigned long long total = list_prefix(a, s_pre, nact, [&](int w) { return (unsigned long long)a.n_holes[w]; });
  const unsigned warps = gridDim.x * (blockDim.x >> 5), warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  for (unsigned long long g = (unsigned long long)(threadIdx.x & 31) * warps + warp; g < total; g += 32ull * warps) {
    const int k = list_owner(s_pre, nact, g);
    const int w = a.act[k];
    const uint32_t sl = reinterpret_cast<const uint32_t*>(a.cand_b[w])[g - s_pre[k]];
    const InstDesc d = a.desc[w];  // (a copy: the refill writes memory that may be anything)
    refill_run(d, a.bitmaps[w], a.dmask[w], sl);
  }
}

// The whole eviction of an instance whose table the sample covers (up to kEstBuckets buckets), by one
// CTA: the metas stay in registers from the first histogram to the choice of what goes, which is then
// listed in shared memory and spread over the threads.  In place of five kernels (8 + 6 + 5 + 8 + 13
// us, each little more than its latency, for 4 instances of 1,024 buckets; 21 us this one).
__global__ void __launch_bounds__(kEstThreads) k4_evict_small(EvictArgs a) {
  constexpr int kPer = kEstBuckets / kEstThreads;
  __shared__ __align__(16) uint32_t hist[kBins];
  __shared__ EstPart s_part[kEstThreads / 32];
  __shared__ uint4 s_v[kRankMax];
  __shared__ uint32_t s_full[kEstBuckets / 32], s_dmask[kEstBuckets / 8];
  __shared__ uint16_t s_del[4 * kEstBuckets], s_hole[kEstBuckets];
  __shared__ unsigned s_cnt, s_ndel, s_nholes;
  __shared__ unsigned long long s_theta[2];
  chain_wait();
  if (block_error(a.err)) return;
  const int w = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const long long size = a.size[w];
  const InstDesc d = a.desc[w];
  const long long E = size - d.cap;
  if (E <= 0) return;
  const uint32_t NB = 1u << d.log2nb;
  unsigned long long m[4 * kPer];
  load_metas(d, NB, NB, m);
  for (int i = tid; i < kEstBuckets / 8; i += kEstThreads) s_dmask[i] = 0;
  if (tid == 0) s_cnt = s_ndel = s_nholes = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const unsigned bits = __ballot_sync(kFull, m[4 * k] && m[4 * k + 1] && m[4 * k + 2] && m[4 * k + 3]);
    if (lane == 0) s_full[(tid + k * kEstThreads) >> 5] = bits;
  }
  const EstPart all = sample_range(m, s_part);
  const TickScale ts{32 - __clz(all.arr), 32 - __clz(all.dep)};
  // the bin of the E-th smallest, then that bin's values over the bins, until it holds a few
  unsigned long long lo = ts.pack(all.mn);
  int shift = bin_shift(ts.pack(all.mx) - lo);
  uint32_t rest = (uint32_t)E, cnt = 0;
  while (true) {
    for (int i = tid; i < kBins; i += kEstThreads) hist[i] = 0;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4 * kPer; ++k) {
      const unsigned long long x = ts.pack(m[k]);
      if (m[k] && x >= lo && ((x - lo) >> shift) < (unsigned)kBins) atomicAdd(&hist[(uint32_t)((x - lo) >> shift)], 1u);
    }
    __syncthreads();
    uint32_t below;
    const int bin = find_threshold_bin<kEstThreads>(hist, rest, &below);
    if (bin < 0) {  // the table holds fewer entries than its size says
      if (tid == 0) set_error(a.err, MISAT_ERR_INTERNAL);
      return;
    }
    rest -= below;
    cnt = hist[bin];
    lo += (unsigned long long)bin << shift;
    if (cnt <= (unsigned)kRankMax || shift == 0) break;
    // (values behind the bin that fall into the next pass's bins come after the target)
    shift = max(0, shift - 12);
    __syncthreads();  // hist is cleared again
  }
  // its entries in order of (meta, key): the threshold has rest - 1 of them below it.  (Only
  // equal ticks, which a commit never writes, can be more than kRankMax; they are ranked from the
  // work list.)
  uint4* list = cnt <= (unsigned)kRankMax ? s_v : a.cand_a[w];
#pragma unroll
  for (int k = 0; k < 4 * kPer; ++k) {
    const unsigned long long x = ts.pack(m[k]);
    if (!m[k] || x < lo || (x - lo) >> shift) continue;  // (the bin may end beyond 64 bits)
    const unsigned long long key = d.tab[tid + (k / 4) * kEstThreads].key[k & 3];
    list[atomicAdd(&s_cnt, 1u)] = make_uint4((uint32_t)m[k], (uint32_t)(m[k] >> 32), (uint32_t)key, (uint32_t)(key >> 32));
  }
  __syncthreads();
  for (unsigned i = tid; i < cnt; i += kEstThreads) {
    const uint64_t mh = v_hi(list[i]), ml = v_lo(list[i]);
    uint32_t rank = 0;
    for (unsigned j = 0; j < cnt; ++j) {
      const uint64_t oh = v_hi(list[j]), ol = v_lo(list[j]);
      rank += oh < mh || (oh == mh && ol < ml);
    }
    if (rank == rest - 1) {
      s_theta[0] = mh;
      s_theta[1] = ml;
    }
  }
  __syncthreads();
  const unsigned long long tm = s_theta[0], tk = s_theta[1];
  // deletions: listed by the buckets' owners, then a thread each (an owner's would be a chain of up
  // to sixteen key reads and global-index lookups)
  unsigned del = 0;  // bit k: entry m[k]
#pragma unroll
  for (int k = 0; k < 4 * kPer; ++k) {
    if (!m[k] || m[k] > tm) continue;
    if (m[k] == tm && d.tab[tid + (k / 4) * kEstThreads].key[k & 3] > tk) continue;
    del |= 1u << k;
  }
  const unsigned mine = __popc(del);
  unsigned incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  unsigned at = 0;
  if (lane == 31) at = atomicAdd(&s_ndel, incl);
  at = __shfl_sync(kFull, at, 31) + incl - mine;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const uint32_t b = tid + k * kEstThreads;
    const unsigned four = (del >> (4 * k)) & 0xfu;
    if (!four) continue;
    atomicOr(&s_dmask[b >> 3], four << (4 * (b & 7)));
    if ((s_full[b >> 5] >> (b & 31)) & 1u) s_hole[atomicAdd(&s_nholes, 1u)] = (uint16_t)(4 * b + __ffs(four) - 1);
    for (unsigned left = four; left; left &= left - 1) s_del[at++] = (uint16_t)(4 * b + __ffs(left) - 1);
  }
  __syncthreads();
  const unsigned ndel = s_ndel, nholes = s_nholes;
  for (unsigned i = tid; i < ndel; i += kEstThreads) {
    const uint32_t sl = s_del[i];
    Bucket* B = d.tab + (sl >> 2);
    if (a.gix.keys && gix_clear(a.gix, B->key[sl & 3], w) < 0) set_error(a.err, MISAT_ERR_INTERNAL);
    B->key[sl & 3] = kEmpty;
    B->meta[sl & 3] = 0;
  }
  if (tid == 0) {
    a.size[w] = size - (long long)ndel;
    atomicAdd(a.evicted, (unsigned long long)ndel);
  }
  __syncthreads();
  // neighbours in the list go to different warps (lanes that walk different runs take turns)
  for (unsigned i = (tid >> 5) + (kEstThreads / 32) * lane; i < nholes; i += kEstThreads)
    refill_run(d, s_full, s_dmask, s_hole[i]);
}

namespace {
int stream_grid(const EvictArgs& a, int chunks_per_inst, int resident) {
  // streaming passes: resident CTAs over (active instance, chunk) items
  const int64_t items = (int64_t)(a.only_w ? 1 : a.W) * chunks_per_inst;
  return (int)(items < (int64_t)resident ? items : (int64_t)resident);
}
}  // namespace

void launch_evict_select(const EvictArgs& a, int chunks_per_inst, int num_sms, cudaStream_t st,
                         const cudaEvent_t* marks) {
  const int W = a.only_w ? 1 : a.W;
  launch_chained(k4_evict_estimate, W, kEstThreads, 0, st, a);
  if (marks) cudaEventRecord(marks[0], st);
  launch_chained(k4_evict_collect, stream_grid(a, chunks_per_inst, resident_grid<k4_evict_collect>(256, 0, num_sms)), 256,
                 0, st, a, (uint32_t)chunks_per_inst);
  if (marks) cudaEventRecord(marks[1], st);
  if (W <= num_sms) launch_chained(k4_evict_select<1024>, W, 1024, 0, st, a);
  else launch_chained(k4_evict_select<256>, W, 256, 0, st, a);
  if (marks) cudaEventRecord(marks[2], st);
}

bool evict_is_small(uint32_t max_log2nb) { return ((uint64_t)1 << max_log2nb) <= (uint64_t)kEstBuckets; }

void launch_evict_small(const EvictArgs& a, cudaStream_t st) {
  launch_chained(k4_evict_small, a.W, kEstThreads, 0, st, a);
}

void launch_evict_apply(const EvictArgs& a, int num_sms, cudaStream_t st, const cudaEvent_t* marks) {
  // one grid-stride pass over the list entries of every instance over capacity, one wave each
  launch_chained(k4_evict_delete, resident_grid<k4_evict_delete>(256, 0, num_sms), 256, 0, st, a);
  if (marks) cudaEventRecord(marks[0], st);
  launch_chained(k4_evict_shift, resident_grid<k4_evict_shift>(256, 0, num_sms), 256, 0, st, a);
  if (marks) cudaEventRecord(marks[1], st);
}

// Compaction of one instance table: delete entries with meta == 0 (marked) or
// (meta, key) <= theta, then restore the probing invariant inside each run of full
// buckets.  A run starts after a bucket that was not full before the pass and ends at
// the next such bucket; runs are disjoint, so each is owned by one thread.
__global__ void __launch_bounds__(256) k4_evict_compact(EvictArgs a) {
  const int w = a.only_w ? *a.only_w : blockIdx.y;
  if (block_error(a.err)) return;
  // active: 0 nothing to do (bitmap not built), 1 theta eviction, 2 marked entries only
  const int act = a.active[w];
  if (act == 0) return;
  const InstDesc d = a.desc[w];
  const uint32_t NB = 1u << d.log2nb;
  const uint32_t mask = NB - 1;
  const uint32_t* bitmap = a.bitmaps[w];
  const unsigned long long tm = a.theta[2 * w], tk = a.theta[2 * w + 1];
  const uint32_t nthreads = gridDim.x * blockDim.x;
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t per = (NB + nthreads - 1) / nthreads;
  const uint32_t lo = tid * per;
  const uint32_t hi = lo + per < NB ? lo + per : NB;
  long long deleted = 0;
  auto is_full = [&](uint32_t b) { return (bitmap[b >> 5] >> (b & 31)) & 1u; };
  for (uint32_t x0 = lo; x0 < hi; ++x0) {
    if (is_full((x0 - 1) & mask)) continue;  // not a run start
    // run [x0, e]: e = first bucket at or after x0 that was not full
    uint32_t e = x0, len = 0;
    while (is_full(e) && len < NB) {
      e = (e + 1) & mask;
      ++len;
    }
    // delete
    for (uint32_t i = 0; i <= len; ++i) {
      Bucket* B = d.tab + ((x0 + i) & mask);
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const unsigned long long k = B->key[s];
        if (k == kEmpty) continue;
        const unsigned long long m = B->meta[s];
        if (m == 0 || (act == 1 && le128(m, k, tm, tk))) {
          if (a.gix.keys && gix_clear(a.gix, k, w) < 0) set_error(a.err, MISAT_ERR_INTERNAL);
          B->key[s] = kEmpty;
          B->meta[s] = 0;
          ++deleted;
        }
      }
    }
    if (len == 0) continue;
    // backward shift: fill free slots of bucket x from the first later entry of the run
    // whose home lies in [x0, x]
    for (uint32_t i = 0; i < len; ++i) {
      Bucket* X = d.tab + ((x0 + i) & mask);
      for (int s = 0; s < 4; ++s) {
        if (X->key[s] != kEmpty) continue;
        bool moved = false;
        for (uint32_t j = i + 1; j <= len && !moved; ++j) {
          Bucket* Y = d.tab + ((x0 + j) & mask);
          for (int t = 0; t < 4; ++t) {
            const unsigned long long k = Y->key[t];
            if (k == kEmpty) continue;
            const uint32_t rel = (home_bucket(k, d.log2nb) - x0) & mask;
            if (rel <= i) {
              X->key[s] = k;
              X->meta[s] = Y->meta[t];
              Y->key[t] = kEmpty;
              Y->meta[t] = 0;
              moved = true;
              break;
            }
          }
        }
        if (!moved) break;  // no later entry can move into x
      }
    }
  }
  const long long tot = block_sum(deleted);
  if (threadIdx.x == 0 && tot) {
    atomic_add_i64(&a.size[w], -tot);
    atomicAdd(a.evicted, (unsigned long long)tot);
  }
}

void launch_compact_marked(const EvictArgs& a, cudaStream_t st) {
  k4_evict_compact<<<dim3(8, 1), 256, 0, st>>>(a);
}

}  // namespace misat
