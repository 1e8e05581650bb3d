// Selection of one batch: the leaders (first request of each session in the batch) are
// decided one at a time in arrival order, as the online router of Sec. 4 decides requests.
// Each sees the snapshot taken at batch start (caches, sessions, backlog d_w, throughput
// mu_w) and the sessions admitted before it, which are pending on their instances
// (P_w, Sec. 4.1-4.2).  A leader takes the cheapest instance of Eq. (1) where Admit holds
// (Eq. 6 with the class cap of Sec. 4.2; Sec. 4.4: placement among instances with
// headroom), or is held when no instance has headroom for it; a released continuation may
// prefer to wait for its cached instance (Eq. 7).
//
// This serial policy is a serial dictatorship with capacities, and its outcome is the unique
// stable matching of the leaders (who rank instances by cost, ties to the lower index) and
// the instances (which all rank leaders by arrival, under a class and a global quota).  It is
// therefore found by deferred acceptance (Gale & Shapley 1962) instead of one leader after
// the other: every undecided leader proposes to the cheapest instance that has not
// refused it, every instance keeps the earliest proposers its quotas admit, and the refused
// ones propose again until nobody is refused.  In terms of thresholds: te[b][w] is the
// arrival position of the proposer that takes instance w's last headroom for class b (infinite
// while some is left); a leader at position i may choose w exactly when i < te[b][w], and
// thresholds only fall, so a choice stays right until its threshold passes it.  After r
// rounds the r earliest events (an instance running out) are exact, so there are at most
// 4 W + 1 rounds, and a round takes in every event whose proposers are already settled: 15
// to 70 rounds a window for batches in which the serial chain has 100 to 500 events.
//
// Eq. (7) breaks the scheme in one way: a released continuation that proposes to w while
// its cached instance w_hit has headroom may have to wait instead once w_hit is full, which
// gives w's headroom back.  Everything before such a leader is unaffected, so when the
// rounds have settled, the first one found so is fixed as held, the thresholds at or behind it
// are lifted, and the leaders behind it propose again.  (A leader that waits and then sees
// the instance it would have waited against fill up is not an exception: waiting takes
// nothing, it simply proposes later.)
#include "common.cuh"
#include "kernels.h"

namespace misat {

namespace {
constexpr unsigned kFull = 0xffffffffu;
constexpr int kNever = 0x7fff;       // threshold of an instance with headroom left (positions are below 2^14)
constexpr int kRecInt4 = kSelectRecInt4;
constexpr int kTop = 8;              // cached instances kept per leader, cheapest first

// A choice that is not an instance.
constexpr int kNone = -1;            // no instance has headroom
constexpr int kWait = -2;            // Eq. (7): waiting for the cached instance is cheaper
constexpr int kFixed = -3;           // the same, decided for good
}  // namespace

// ---------------------------------------------------------------------------
// Per-leader records of the selection (64 bytes), compact per block of 256 requests:
//   [0] = {L, class | state << 8, protected / last instance, hbest}
//   [1] = {cached instances the leader may use, request, theta low, theta high}
//   [2], [3] = the kTop cheapest of those, (w << 16 | H), by (cost, w)
// theta is Eq. (7)'s bound: the released leader waits for a full w_hit when the chosen
// instance's d_w is above theta.  H rows are read 16 bytes at a time, and only of leaders with
// a cached prefix, Ahead pieces in flight (3,001 requests of 1,000 instances: one entry at a time
// 130 us, one piece 31, four 20; with 64 or 128 instances four are 1 us slower than one).
template <int Ahead>
__global__ void __launch_bounds__(256) k3_select_prep(SelectPrepArgs a) {
  __shared__ int s_wc[8];
  chain_wait();
  if (block_error(a.err)) return;
  const int leaders = (a.n + 255) / 256;
  if ((int)blockIdx.x >= leaders) {  // the caller's copy of H, beside the records
    const int64_t total = (int64_t)a.n * a.W, t = (int64_t)(blockIdx.x - leaders) * blockDim.x + threadIdx.x,
                  stride = (int64_t)(gridDim.x - leaders) * blockDim.x;
    int64_t done = 0;
    if ((reinterpret_cast<uintptr_t>(a.out_H) & 15) == 0) {
      const uint4* src = reinterpret_cast<const uint4*>(a.H);
      uint4* dst = reinterpret_cast<uint4*>(a.out_H);
#pragma unroll 4
      for (int64_t i = t; i < total >> 3; i += stride) dst[i] = __ldcg(src + i);
      done = total & ~(int64_t)7;
    }
    for (int64_t i = done + t; i < total; i += stride) a.out_H[i] = __ldcg(a.H + i);
    return;
  }
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool lead = r < a.n && a.rq.status[r] == kStUnresolved;
  const unsigned ml = __ballot_sync(kFull, lead);
  if (lane == 0) s_wc[wid] = __popc(ml);
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int k = 0; k < 8; ++k) t += s_wc[k];
    a.segcnt[blockIdx.x] = t;
  }
  if (!lead) return;
  int off = __popc(ml & lanemask_lt());
  for (int k = 0; k < wid; ++k) off += s_wc[k];
  const int64_t x = a.rq.L[r];
  const int b = a.rq.cls[r], sst = a.rq.sst[r], sinst = a.rq.sinst[r];
  const int pw = sst == (int)kSessProtected ? sinst : -1;
  const uint32_t hb = a.rq.hbest[r];
  int nh = 0;
  int64_t theta = INT64_MAX;
  int64_t cost[kTop];
  uint32_t ent[kTop];
#pragma unroll
  for (int i = 0; i < kTop; ++i) {
    cost[i] = INT64_MAX;
    ent[i] = 0;
  }
  if (hb >> 16) {
    if (sst == (int)kSessReleased) {
      const int hmax = (int)(hb >> 16), whit = 65535 - (int)(hb & 0xffffu);
      theta = a.hold_delay_q + a.backlog[whit] - 16 * (int64_t)hmax * a.tokcost[whit];
    }
    // the row's entries in 16-byte pieces (its first and last piece may hold neighbours)
    const uint16_t* row = a.H + (int64_t)r * a.W;
    const int lead_in = (int)((reinterpret_cast<uintptr_t>(row) & 15) >> 1);
    const uint4* p = reinterpret_cast<const uint4*>(row - lead_in);
    const int pieces = (lead_in + a.W + 7) >> 3;
    for (int q0 = 0; q0 < pieces; q0 += Ahead) {
      uint4 ahead[Ahead];
#pragma unroll
      for (int k = 0; k < Ahead; ++k) ahead[k] = q0 + k < pieces ? __ldcg(p + q0 + k) : make_uint4(0, 0, 0, 0);
#pragma unroll 1
      for (int k = 0; k < Ahead; ++k) {
        const uint4 v = ahead[0];
#pragma unroll
        for (int i = 0; i + 1 < Ahead; ++i) ahead[i] = ahead[i + 1];
        const int q = q0 + k;
        if ((v.x | v.y | v.z | v.w) == 0) continue;
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const uint32_t h = (u[e >> 1] >> (16 * (e & 1))) & 0xffffu;
          const int w = 8 * q + e - lead_in;
          if (!h || w < 0 || w >= a.W) continue;
          if (w != pw && (a.gh[w] <= 0 || a.ch[w * 3 + b] <= 0)) continue;
          ++nh;
          const int64_t c = a.backlog[w] + (x - 16 * (int64_t)h) * a.tokcost[w];
          if (c < cost[kTop - 1]) {  // instances come in index order: equal costs keep it
            cost[kTop - 1] = c;
            ent[kTop - 1] = ((uint32_t)w << 16) | h;
#pragma unroll
            for (int i = kTop - 1; i > 0; --i)
              if (cost[i] < cost[i - 1]) {
                const int64_t tcost = cost[i];
                cost[i] = cost[i - 1];
                cost[i - 1] = tcost;
                const uint32_t te = ent[i];
                ent[i] = ent[i - 1];
                ent[i - 1] = te;
              }
          }
        }
      }
    }
  }
  int4* rec = a.rec + (int64_t)kRecInt4 * (blockIdx.x * 256 + off);
  rec[0] = make_int4((int)x, b | (sst << 8), sinst, (int)hb);
  rec[1] = make_int4(nh, r, (int)(uint32_t)theta, (int)(theta >> 32));
  if (nh > 0) {
    rec[2] = make_int4((int)ent[0], (int)ent[1], (int)ent[2], (int)ent[3]);
    rec[3] = make_int4((int)ent[4], (int)ent[5], (int)ent[6], (int)ent[7]);
  }
}

void launch_select_prep(const SelectPrepArgs& a, int num_sms, cudaStream_t st) {
  if (a.n <= 0) return;
  int grid = (a.n + 255) / 256;
  if (a.out_H) {
    const int64_t copy = ((int64_t)a.n * a.W + 8191) / 8192;
    grid += (int)(copy < 8 * num_sms ? copy : 8 * num_sms);
  }
  launch_chained(a.W > 256 ? k3_select_prep<4> : k3_select_prep<1>, grid, 256, 0, st, a);
}

// ---------------------------------------------------------------------------
// The selection kernel: one thread-block cluster takes the leaders in windows of one leader
// per thread (up to 16 CTAs x 1024).  A leader's position in the window is its thread's rank
// in the cluster.  Every CTA keeps a copy of the thresholds and the proposals of its own
// leaders (one bit per instance and thread, and their number per class; a refused proposal's
// bit stays, it lies behind its threshold for good).  A round:
//   1. leaders without a standing proposal are packed into as few warps as hold them, choose
//      and set their bits;                                                  cluster barrier
//   2. the warp that owns instance w adds up w's proposals per class over the CTAs (distributed
//      shared memory).  Where a quota is reached by new ones, a scan over the CTAs' numbers and
//      one over the words of the CTA it ends in give the new threshold, which is written into
//      every CTA;                                                           cluster barrier
//   3. leaders whose proposal lies behind its threshold are refused.
// What bounds it: latency.  A round of 16 CTAs at 128 instances takes 9,000 to 10,000 cycles: 2,000 to
// 2,700 for the choices and about 2,000 for the thresholds of an ordinary CTA, and after each 2,000 to
// 4,000 until the slowest CTA has reached the barrier.  The SMs are mostly idle.
namespace {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t ld_cluster(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_u16(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(addr), "h"((unsigned short)v) : "memory");
}
// Barrier over all threads of the cluster (a plain block barrier for one CTA).
__device__ __forceinline__ void cluster_barrier(int cs) {
  if (cs == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// Bits of word q (positions 32q .. 32q + 31) at or before position t.
__device__ __forceinline__ unsigned upto_mask(int q, int t) {
  const int k = t - 32 * q;
  return k >= 31 ? ~0u : (k < 0 ? 0u : (2u << k) - 1u);
}

__device__ __forceinline__ int warp_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// Inclusive scans of two registers over the warp, side by side.
__device__ __forceinline__ void warp_scan_pair(unsigned* a, unsigned* b) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(kFull, *a, o), v = __shfl_up_sync(kFull, *b, o);
    if (lane >= o) {
      *a += u;
      *b += v;
    }
  }
}

struct SelSmem {
  longlong2* ln;   // [W] {d_w, 1/mu_w}
  unsigned* prop;  // [W][warps] proposals of this CTA's leaders, one bit per thread
  unsigned* n01;   // [W] their number: class 0 | class 1 << 16
  unsigned* n2;    // [W] class 2
  int16_t* te;     // [3][W] position of the proposer that takes the class's last headroom, kNever
  int16_t* tg;     // [W] position of the proposer that takes the last global headroom, kNever
  // of the instances this CTA owns (w mod CTAs = its rank), by w / CTAs:
  int4* hr;        // headroom left: classes 0..2, global
  unsigned* seen;  // proposals when its thresholds were last computed
  unsigned* cm;    // [3][words] the window's leaders of each class, one bit per position
  int* pre;        // [blocks] leaders before each block of 256 requests
  // per leader of the CTA's part of the window
  uint32_t* lx;    // prompt tokens | class << 20 | (Eq. 7 may apply) << 22
  uint32_t* lpos;  // price cell | (its order before this position has no headroom for the leader) << 16
  uint32_t* lcp;   // protected instance + 1 | cached instances passed over << 16
  int32_t* lrec;   // record
  int16_t* lch;    // choice: an instance, kNone, kWait or kFixed
  uint16_t* queue; // leaders that choose in this round
  // copies that spare the rounds their global loads (the barriers' acquire drops L1); NULL
  // when they do not fit, and the originals are read
  uint4* ord;      // [kPriceCells][stride] price orders
  uint32_t* list;  // [kTop][threads] the leaders' cached instances
  int4* eq7;       // [threads] Eq. (7): {w_hit, -, theta low, theta high}
};
constexpr size_t kSelSmemMax = 226 * 1024;

__host__ __device__ inline size_t sel_smem_layout(int W, int cs, int warps, int nblk, SelSmem* s, unsigned char* p) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) & ~(size_t)15;
    return at;
  };
  const size_t own = (size_t)((W + cs - 1) / cs) * 16;
  const size_t ln = take((size_t)W * 16), prop = take((size_t)W * warps * 4), n01 = take((size_t)W * 4),
               n2 = take((size_t)W * 4), te = take((size_t)W * 6), tg = take((size_t)W * 2), hr = take(own),
               seen = take(own / 4), cm = take((size_t)cs * warps * 12), pre = take((size_t)nblk * 4),
               lx = take((size_t)warps * 128), lpos = take((size_t)warps * 128), lcp = take((size_t)warps * 128),
               lrec = take((size_t)warps * 128), lch = take((size_t)warps * 64), queue = take((size_t)warps * 64);
  const size_t base = o;
  const size_t ord = take((size_t)kPriceCells * price_order_stride(W) * 2), list = take((size_t)kTop * warps * 128),
               eq7 = take((size_t)warps * 512);
  const bool copies = o <= kSelSmemMax;
  if (s) {
    s->ln = reinterpret_cast<longlong2*>(p + ln);
    s->prop = reinterpret_cast<unsigned*>(p + prop);
    s->n01 = reinterpret_cast<unsigned*>(p + n01);
    s->n2 = reinterpret_cast<unsigned*>(p + n2);
    s->te = reinterpret_cast<int16_t*>(p + te);
    s->tg = reinterpret_cast<int16_t*>(p + tg);
    s->hr = reinterpret_cast<int4*>(p + hr);
    s->seen = reinterpret_cast<unsigned*>(p + seen);
    s->cm = reinterpret_cast<unsigned*>(p + cm);
    s->pre = reinterpret_cast<int*>(p + pre);
    s->lx = reinterpret_cast<uint32_t*>(p + lx);
    s->lpos = reinterpret_cast<uint32_t*>(p + lpos);
    s->lcp = reinterpret_cast<uint32_t*>(p + lcp);
    s->lrec = reinterpret_cast<int32_t*>(p + lrec);
    s->lch = reinterpret_cast<int16_t*>(p + lch);
    s->queue = reinterpret_cast<uint16_t*>(p + queue);
    s->ord = copies ? reinterpret_cast<uint4*>(p + ord) : nullptr;
    s->list = copies ? reinterpret_cast<uint32_t*>(p + list) : nullptr;
    s->eq7 = copies ? reinterpret_cast<int4*>(p + eq7) : nullptr;
  }
  return copies ? o : base;
}

// The choice of the CTA's leader t at window position pos given the thresholds: an instance,
// kNone or kWait.
__device__ __forceinline__ int sel_choose(const SelSmem& s, const SelectArgs& a, int64_t tc_min, int T, int t, int pos) {
  const int W = a.W;
  const uint32_t lx = s.lx[t], lcell = s.lpos[t], lcp = s.lcp[t];
  const int64_t x = lx & 0xfffffu;
  const int16_t* te = s.te + ((lx >> 20) & 3) * W;
  const int pw = (int)(lcp & 0xffffu) - 1;
  const int cell = (int)(lcell & 0xffffu);
  int p0 = (int)(lcell >> 16), cp = (int)(lcp >> 16);
  int64_t best_c = INT64_MAX;
  int best_w = kNone;
  auto consider = [&](int w, int64_t c) {
    if (c < best_c || (c == best_c && w < best_w)) {
      best_c = c;
      best_w = w;
    }
  };
  // cached instances, cheapest first (an empty entry ends the list, cp is kTop + 1 from then on);
  // beyond the kept ones the whole row
  if (cp <= kTop) {
    const int cp0 = cp;
    while (cp < kTop) {
      const uint32_t e = s.list ? s.list[cp * T + t] : reinterpret_cast<const uint32_t*>(a.rec + s.lrec[t] + 2)[cp];
      if (e == 0) {
        cp = kTop + 1;
        break;
      }
      const int w = (int)(e >> 16);
      if (te[w] > pos || w == pw) {
        const longlong2 q = s.ln[w];
        consider(w, q.x + (x - 16 * (int64_t)(e & 0xffffu)) * q.y);
        break;
      }
      ++cp;
    }
    if (cp == kTop && a.rec[s.lrec[t] + 1].x <= kTop) cp = kTop + 1;
    if (cp != cp0) s.lcp[t] = (lcp & 0xffffu) | ((uint32_t)cp << 16);
    if (cp == kTop) {
      const uint16_t* row = a.H + (int64_t)a.rec[s.lrec[t] + 1].y * W;
      const int lead_in = (int)((reinterpret_cast<uintptr_t>(row) & 15) >> 1);
      const uint4* p = reinterpret_cast<const uint4*>(row - lead_in);
      const int pieces = (lead_in + W + 7) >> 3;
      for (int q = 0; q < pieces; ++q) {
        const uint4 v = __ldcg(p + q);
        if ((v.x | v.y | v.z | v.w) == 0) continue;
        for (int e = 0; e < 8; ++e) {
          const uint32_t u = e < 2 ? v.x : (e < 4 ? v.y : (e < 6 ? v.z : v.w));
          const uint32_t h = (u >> (16 * (e & 1))) & 0xffffu;
          const int w = 8 * q + e - lead_in;
          if (!h || w < 0 || w >= W || !(te[w] > pos || w == pw)) continue;
          const longlong2 y = s.ln[w];
          consider(w, y.x + (x - 16 * (int64_t)h) * y.y);
        }
      }
    }
  }
  // the protected instance is eligible without headroom (its cached cost was considered above)
  if (pw >= 0) {
    const longlong2 y = s.ln[pw];
    consider(pw, y.x + x * y.y);
  }
  // without a cached prefix: the price order of the cell, eight entries at a time (one load,
  // then eight independent threshold reads): first the piece with headroom, then its entries
  const int Wp = price_order_stride(W);
  const uint4* ord = (s.ord ? s.ord : reinterpret_cast<const uint4*>(a.orders)) + cell * (Wp >> 3);
  uint4 v = make_uint4(0, 0, 0, 0);
  auto open_of = [&](int k) -> unsigned {
    v = ord[k >> 3];
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
    unsigned av = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (te[(u[e >> 1] >> (16 * (e & 1))) & kPriceMask] > pos) av |= 1u << e;
    // (the row's padding names instance 0)
    return k + 8 > W ? av & ((1u << (W - k)) - 1u) : av;
  };
  const int p_in = p0;
  unsigned av = 0;
  while (p0 < Wp && !(av = open_of(p0))) p0 += 8;
  if (p0 != p_in) s.lpos[t] = (uint32_t)cell | ((uint32_t)p0 << 16);
  const int64_t xg = price_cell_start(cell), dx = x - xg;
  const int64_t slack = dx * tc_min;
  int k = p0;
  while (k < Wp) {
    if (!av) {
      k += 8;
      if (k < Wp) av = open_of(k);
      continue;
    }
    const int e = __ffs(av) - 1;
    av &= av - 1;
    const uint32_t pair = e < 4 ? (e < 2 ? v.x : v.y) : (e < 6 ? v.z : v.w);
    const uint32_t ent = pair >> (16 * (e & 1));
    const int w = (int)(ent & kPriceMask);
    const longlong2 y = s.ln[w];
    const int64_t cg = y.x + xg * y.y;
    const int64_t bound = cg + slack;  // of this and every later entry
    if (bound > best_c) break;
    consider(w, cg + dx * y.y);
    // Entries behind this one that cost as little as the bound have the same cost at x_g, and so a
    // larger index: at an equal bound they can win only while this one's is below the best's (the
    // best may be a cached instance with any index).  A fast entry is cheaper than all behind it over
    // the whole cell.
    const bool last = (bound == best_c && w >= best_w) || (ent & kPriceFast);
    if (last) break;
  }
  if (best_w >= 0 && ((lx >> 22) & 1u)) {
    int4 q;
    if (s.eq7) {
      q = s.eq7[t];
    } else {
      q = a.rec[s.lrec[t] + 1];
      q.x = 65535 - (a.rec[s.lrec[t]].w & 0xffff);
    }
    const int64_t theta = ((int64_t)q.w << 32) | (uint32_t)q.z;
    if (te[q.x] <= pos && s.ln[best_w].x > theta) return kWait;
  }
  return best_w;
}

// The two halves of finding the position of the (rank + 1)-th proposal in a set whose number per
// CTA lane c holds in n (c < cs): the CTA and the rank in it, ...
__device__ __forceinline__ int find_cta(int n, int* rank) {
  const int incl = warp_scan(n);
  const int src = __ffs(__ballot_sync(kFull, incl > *rank)) - 1;
  *rank -= __shfl_sync(kFull, incl - n, src);
  return src;
}
// ... and the position from that CTA's words of the set, word i in lane i.
__device__ __forceinline__ int find_pos(unsigned x, int rank, int first_word) {
  const int lane = threadIdx.x & 31;
  const int n = __popc(x);
  const int incl = warp_scan(n);
  const int i = __ffs(__ballot_sync(kFull, incl > rank)) - 1;
  const int k = rank - __shfl_sync(kFull, incl - n, i);
  const unsigned y = __shfl_sync(kFull, x, i);
  const unsigned bit = __ballot_sync(kFull, ((y >> lane) & 1u) && __popc(y & lanemask_lt()) == k);
  return 32 * (first_word + i) + __ffs(bit) - 1;
}

}  // namespace

__global__ void __launch_bounds__(1024, 1) k4_select(SelectArgs a, int cs) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_ws[32];
  __shared__ int s_total;
  __shared__ int s_queued;          // leaders in the queue
  __shared__ int s_changed[2];      // some threshold moved in this round (written by any CTA)
  __shared__ int s_fix[16];         // per CTA: first leader of the window to fix as held
  __shared__ int s_fixmin;
  __shared__ int s_tgmax;
  __shared__ unsigned long long s_tcmin;
  chain_wait();
  if (block_error(a.err)) return;
  const int W = a.W;
  const int T = blockDim.x, NW = T >> 5;
  const int words = cs * NW;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int cta = cs == 1 ? 0 : (int)blockIdx.x;
  const int pos = cta * T + tid;    // position of this thread's leader in the window
  const int nblk = (a.n + 255) >> 8;
  SelSmem s;
  sel_smem_layout(W, cs, NW, nblk, &s, smem);
  const uint32_t sm_te = smem_addr(s.te), sm_tg = smem_addr(s.tg), sm_cm = smem_addr(s.cm),
                 sm_prop = smem_addr(s.prop), sm_n01 = smem_addr(s.n01), sm_n2 = smem_addr(s.n2),
                 sm_changed = smem_addr(s_changed), sm_fix = smem_addr(s_fix);

  // ---- state at batch start
  if (tid == 0) {
    s_changed[0] = s_changed[1] = 0;
    s_queued = 0;
    s_tcmin = ~0ull;
  }
  __syncthreads();
  for (int w = tid; w < W; w += T) {
    const longlong2 t = make_longlong2(a.backlog[w], a.tokcost[w]);
    s.ln[w] = t;
    atomicMin(&s_tcmin, (unsigned long long)t.y);
    const int g = a.gh[w], c0 = a.ch[w * 3], c1 = a.ch[w * 3 + 1], c2 = a.ch[w * 3 + 2];
    s.tg[w] = g > 0 ? kNever : -1;
    s.te[w] = g > 0 && c0 > 0 ? kNever : -1;
    s.te[W + w] = g > 0 && c1 > 0 ? kNever : -1;
    s.te[2 * W + w] = g > 0 && c2 > 0 ? kNever : -1;
    s.n01[w] = 0;
    s.n2[w] = 0;
    if (w % cs == cta) {
      s.hr[w / cs] = make_int4(c0, c1, c2, g);
      s.seen[w / cs] = 0;
    }
  }
  for (int i = tid; i < W * NW; i += T) s.prop[i] = 0;
  if (s.ord) {
    const uint4* src = reinterpret_cast<const uint4*>(a.orders);
    const int pieces = kPriceCells * (price_order_stride(W) >> 3);
#pragma unroll 4
    for (int i = tid; i < pieces; i += T) s.ord[i] = __ldcg(src + i);
  }
  // leaders before each block of 256 requests (exclusive scan of the prep kernel's counts)
  {
    const int per = (nblk + T - 1) / T;
    int t = 0;
    for (int u = 0; u < per; ++u) {
      const int j = tid * per + u;
      if (j < nblk) t += a.segcnt[j];
    }
    const int incl = warp_scan(t);
    if (lane == 31) s_ws[wid] = incl;
    __syncthreads();
    if (wid == 0) {
      const int v = lane < NW ? s_ws[lane] : 0;
      const int sc = warp_scan(v);
      s_ws[lane] = sc - v;
      if (lane == 31) s_total = sc;
    }
    __syncthreads();
    int off = s_ws[wid] + incl - t;
    for (int u = 0; u < per; ++u) {
      const int j = tid * per + u;
      if (j < nblk) {
        s.pre[j] = off;
        off += a.segcnt[j];
      }
    }
    __syncthreads();
  }
  const int nl = s_total;
  const int64_t tc_min = (int64_t)s_tcmin;
  // record of the g-th leader: its block is the last one whose offset is <= g
  auto leader_rec = [&](int g) -> int {
    int lo = 0, hi = nblk - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s.pre[mid] <= g) lo = mid;
      else hi = mid - 1;
    }
    return kRecInt4 * (lo * 256 + (g - s.pre[lo]));
  };
  auto decide = [&](int r, int choice, int pw, bool global_left) {
    if (choice >= 0) {
      a.rq.status[r] = kStResolved;
      a.rq.inst[r] = choice;
      a.rq.reason[r] = choice == pw ? MISAT_ADMIT_CONT : MISAT_ADMIT_NEW;
    } else {
      a.rq.status[r] = kStHeld;
      a.rq.inst[r] = -1;
      a.rq.last_reason[r] = choice == kWait || choice == kFixed
                                ? MISAT_HOLD_PREFER_CACHE
                                : (global_left ? MISAT_HOLD_CLASS_CAP : MISAT_HOLD_GLOBAL_CAP);
    }
  };
  // the other CTAs' shared memory is written from here on
  cluster_barrier(cs);

  int par = 0;  // parity of the round's changed flag
#pragma unroll 1
  for (int base = 0; base < nl; base += cs * T) {
    // no headroom left for any class: the leaders that remain are decided on their own (a
    // protected session continues on its instance, anyone else is held)
    {
      bool any = false, anyg = false;
      for (int w = tid; w < W; w += T) {
        any |= s.te[w] >= 0 || s.te[W + w] >= 0 || s.te[2 * W + w] >= 0;
        anyg |= s.tg[w] >= 0;
      }
      any = __syncthreads_or(any);
      if (!any) {
        anyg = __syncthreads_or(anyg);
        for (int g = base + pos; g < nl; g += cs * T) {
          const int4* rec = a.rec + leader_rec(g);
          const int4 q0 = rec[0];
          const int pw = ((q0.y >> 8) & 0xff) == (int)kSessProtected ? q0.z : -1;
          decide(rec[1].y, pw >= 0 ? pw : kNone, pw, anyg);
        }
        break;
      }
    }
    const bool valid = base + pos < nl;
    int b = 3;
    bool eq7 = false;
    if (valid) {
      const int at = leader_rec(base + pos);
      const int4 q0 = a.rec[at], q1 = a.rec[at + 1];
      b = q0.y & 0xff;
      eq7 = q1.w != (int)(INT64_MAX >> 32);
      s.lx[tid] = (uint32_t)q0.x | ((uint32_t)b << 20) | ((uint32_t)eq7 << 22);
      s.lpos[tid] = (uint32_t)price_cell((uint32_t)q0.x);
      s.lcp[tid] = (uint32_t)((((q0.y >> 8) & 0xff) == (int)kSessProtected ? q0.z : -1) + 1) |
                   ((q1.x > 0 ? 0u : kTop + 1u) << 16);
      s.lrec[tid] = at;
      if (eq7 && s.eq7) s.eq7[tid] = make_int4(65535 - (q0.w & 0xffff), 0, q1.z, q1.w);
      if (q1.x > 0 && s.list) {
        const int4 q2 = a.rec[at + 2], q3 = a.rec[at + 3];
        const int e[kTop] = {q2.x, q2.y, q2.z, q2.w, q3.x, q3.y, q3.z, q3.w};
#pragma unroll
        for (int k = 0; k < kTop; ++k) s.list[k * T + tid] = (uint32_t)e[k];
      }
    }
    s.lch[tid] = kNone;
    {
      const unsigned m0 = __ballot_sync(kFull, b == 0), m1 = __ballot_sync(kFull, b == 1),
                     m2 = __ballot_sync(kFull, b == 2);
      for (int i = lane; i < 3 * cs; i += 32) {
        const int c = i / cs, rank = i - c * cs;
        st_cluster(map_rank(sm_cm + 4 * (c * words + cta * NW + wid), rank), c == 0 ? m0 : (c == 1 ? m1 : m2));
      }
    }
    const int pw = valid ? (int)(s.lcp[tid] & 0xffffu) - 1 : -1;
    bool need = valid;
    int guard = 0;
#pragma unroll 1
    while (true) {
      // ---- 1. proposals, the leaders that choose packed into as few warps as hold them
      {
        const unsigned m = __ballot_sync(kFull, need);
        int at = 0;
        if (lane == 0 && m) at = atomicAdd(&s_queued, __popc(m));
        at = __shfl_sync(kFull, at, 0);
        if (need) s.queue[at + __popc(m & lanemask_lt())] = (uint16_t)tid;
      }
      __syncthreads();
      if (tid < s_queued) {
        const int t = s.queue[tid];
        const int c = sel_choose(s, a, tc_min, T, t, cta * T + t);
        s.lch[t] = (int16_t)c;
        if (c >= 0 && c != (int)(s.lcp[t] & 0xffffu) - 1) {
          atomicOr(&s.prop[c * NW + (t >> 5)], 1u << (t & 31));
          const int cb = (int)((s.lx[t] >> 20) & 3);
          atomicAdd(cb == 2 ? &s.n2[c] : &s.n01[c], cb == 1 ? 1u << 16 : 1u);
        }
      }
      cluster_barrier(cs);
      // ---- 2. thresholds of the instances this warp owns
      if (tid == 0) {
        s_changed[par ^ 1] = 0;
        s_queued = 0;
      }
      bool moved = false;
      for (int o = wid; o * cs + cta < W; o += NW) {
        const int w = o * cs + cta;
        const int4 h4 = s.hr[o];
        const unsigned seen = s.seen[o];
        if (h4.w <= 0) continue;
        // lane c: CTA c's proposals per class; totals
        unsigned p01 = 0, p2 = 0;
        if (lane < cs) {
          p01 = ld_cluster(map_rank(sm_n01 + 4 * w, lane));
          p2 = ld_cluster(map_rank(sm_n2 + 4 * w, lane));
        }
        const unsigned t01 = __reduce_add_sync(kFull, p01), t2 = __reduce_add_sync(kFull, p2);
        const int n[3] = {(int)(t01 & 0xffffu), (int)(t01 >> 16), (int)t2};
        const int h[3] = {h4.x, h4.y, h4.z};
        const unsigned all = (unsigned)(n[0] + n[1] + n[2]);
        // proposals are only added: the same number is the same set
        if (all == seen || !((h[0] > 0 && n[0] >= h[0]) || (h[1] > 0 && n[1] >= h[1]) ||
                             (h[2] > 0 && n[2] >= h[2]) || (int)all >= h4.w))
          continue;
        // per class: the position of its h-th proposal, through a scan over the CTAs and one over
        // the words of the CTA it is in; the three classes go through the same instructions
        // side by side (two share a register in the scans)
        unsigned i01 = p01, i2 = p2;
        warp_scan_pair(&i01, &i2);
        const int own[3] = {(int)(p01 & 0xffffu), (int)(p01 >> 16), (int)p2};
        const int inc[3] = {(int)(i01 & 0xffffu), (int)(i01 >> 16), (int)i2};
        int src[3], rank[3];
        unsigned x[3];
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) {
          const unsigned hit = __ballot_sync(kFull, inc[bb] >= h[bb]);
          src[bb] = hit ? __ffs(hit) - 1 : 0;
          rank[bb] = h[bb] - 1 - __shfl_sync(kFull, inc[bb] - own[bb], src[bb]);
        }
#pragma unroll
        for (int bb = 0; bb < 3; ++bb)
          x[bb] = lane < NW && h[bb] > 0 && n[bb] >= h[bb]
                      ? ld_cluster(map_rank(sm_prop + 4 * (w * NW + lane), src[bb])) & s.cm[bb * words + src[bb] * NW + lane]
                      : 0u;
        const int pc[3] = {__popc(x[0]), __popc(x[1]), __popc(x[2])};
        unsigned q01 = (unsigned)pc[0] | ((unsigned)pc[1] << 16), q2 = (unsigned)pc[2];
        warp_scan_pair(&q01, &q2);
        const int win[3] = {(int)(q01 & 0xffffu), (int)(q01 >> 16), (int)q2};
        int t[3], kept = 0;  // kept: lane c's proposals that pass the class quotas
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) {
          const unsigned hit = __ballot_sync(kFull, win[bb] > rank[bb]);
          const int i = hit ? __ffs(hit) - 1 : 0;
          const int k = rank[bb] - __shfl_sync(kFull, win[bb] - pc[bb], i);
          const unsigned y = __shfl_sync(kFull, x[bb], i);
          const unsigned bit = __ballot_sync(kFull, ((y >> lane) & 1u) && __popc(y & lanemask_lt()) == k);
          const bool full = n[bb] >= h[bb];
          t[bb] = h[bb] <= 0 ? -1 : (full ? 32 * (src[bb] * NW + i) + __ffs(bit) - 1 : kNever);
          kept += h[bb] <= 0 ? 0 : (!full || lane < src[bb] ? own[bb] : (lane == src[bb] ? rank[bb] + 1 : 0));
        }
        int tgw = kNever;
        // the proposals that pass the class quotas count against the global one
        if ((int)all >= h4.w && (int)__reduce_add_sync(kFull, (unsigned)kept) >= h4.w) {
          int r = h4.w - 1;
          const int c = find_cta(kept, &r);
          unsigned y = 0;
          if (lane < NW) {
            const int q = c * NW + lane;
            y = ld_cluster(map_rank(sm_prop + 4 * (w * NW + lane), c)) &
                ((s.cm[q] & upto_mask(q, t[0])) | (s.cm[words + q] & upto_mask(q, t[1])) |
                 (s.cm[2 * words + q] & upto_mask(q, t[2])));
          }
          tgw = find_pos(y, r, c * NW);
        }
        __syncwarp();
        if (lane == 0) s.seen[o] = all;
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) t[bb] = min(t[bb], tgw);
        if (t[0] != s.te[w] || t[1] != s.te[W + w] || t[2] != s.te[2 * W + w] || tgw != s.tg[w]) {
          moved = true;
          __syncwarp();
          for (int i = lane; i < 4 * cs; i += 32) {
            const int bb = i / cs, rank = i - bb * cs;
            st_cluster_u16(map_rank(bb < 3 ? sm_te + 2 * (bb * W + w) : sm_tg + 2 * w, rank),
                           bb == 0 ? t[0] : (bb == 1 ? t[1] : (bb == 2 ? t[2] : tgw)));
          }
        }
      }
      if (moved && lane < cs) st_cluster(map_rank(sm_changed + 4 * par, lane), 1u);
      cluster_barrier(cs);
      // ---- 3. refusals
      const bool changed = *(volatile int*)&s_changed[par] != 0;
      par ^= 1;
      if (changed) {
        if (++guard > 4 * W + 4) {  // at least one event becomes exact per round (uniform over the cluster)
          if (tid == 0) set_error(a.err, MISAT_ERR_INTERNAL);
          return;
        }
        const int c = s.lch[tid];
        need = valid && (c == kWait || (c >= 0 && c != pw && s.te[b * W + c] < pos));
        continue;
      }
      // settled: the first Eq. (7) leader whose cached instance filled up after it had
      // proposed elsewhere, where waiting is cheaper
      if (!__syncthreads_or(eq7) && cs == 1) break;
      {
        if (tid == 0) s_fixmin = kNever;
        __syncthreads();
        const int c = s.lch[tid];
        if (eq7 && c >= 0) {
          const int4 q0 = a.rec[s.lrec[tid]], q1 = a.rec[s.lrec[tid] + 1];
          const int whit = 65535 - (q0.w & 0xffff);
          const int64_t theta = ((int64_t)q1.w << 32) | (uint32_t)q1.z;
          if (c != whit && s.te[b * W + whit] <= pos && s.ln[c].x > theta) atomicMin(&s_fixmin, pos);
        }
        __syncthreads();
        if (tid < cs) st_cluster(map_rank(sm_fix + 4 * cta, tid), (uint32_t)s_fixmin);
        cluster_barrier(cs);
      }
      int fix = kNever;
      for (int i = 0; i < cs; ++i) fix = min(fix, *(volatile int*)&s_fix[i]);
      if (fix == kNever) break;
      // that leader waits; thresholds at or behind it are lifted (every CTA its own copy), its
      // proposal and those behind it withdrawn, and the leaders behind it start over
      for (int w = tid; w < W; w += T) {
        unsigned k01 = 0, k2 = 0;
        for (int i = 0; i < NW; ++i) {
          const int q = cta * NW + i;
          const unsigned x = s.prop[w * NW + i] & upto_mask(q, fix - 1);
          s.prop[w * NW + i] = x;
          k01 += __popc(x & s.cm[q]) + (__popc(x & s.cm[words + q]) << 16);
          k2 += __popc(x & s.cm[2 * words + q]);
        }
        s.n01[w] = k01;
        s.n2[w] = k2;
        if (w % cs == cta) s.seen[w / cs] = 0;
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (s.te[i * W + w] >= fix) s.te[i * W + w] = kNever;
        if (s.tg[w] >= fix) s.tg[w] = kNever;
      }
      if (pos == fix) s.lch[tid] = kFixed;
      need = valid && pos > fix;
      if (need) {
        s.lch[tid] = kNone;
        s.lpos[tid] &= 0xffffu;
        s.lcp[tid] = (s.lcp[tid] & 0xffffu) | ((a.rec[s.lrec[tid] + 1].x > 0 ? 0u : kTop + 1u) << 16);
      }
      guard = 0;
      cluster_barrier(cs);  // every CTA has read s_fix and lifted its copies
    }
    // ---- the window's decisions; behind position s_tgmax no instance has global headroom
    if (tid == 0) s_tgmax = -1;
    __syncthreads();
    for (int w = tid; w < W; w += T)
      if (s.tg[w] >= 0) atomicMax(&s_tgmax, (int)s.tg[w]);
    __syncthreads();
    if (valid) decide(a.rec[s.lrec[tid] + 1].y, s.lch[tid], pw, s_tgmax > pos);
    const bool more = base + cs * T < nl;
    // headroom left after the window (accepted proposals lie at or before their threshold)
    for (int o = wid; o * cs + cta < W; o += NW) {
      const int w = o * cs + cta;
      unsigned used01 = 0, used2 = 0;
      for (int q = lane; q < words; q += 32) {
        const unsigned v = ld_cluster(map_rank(sm_prop + 4 * (w * NW + q % NW), q / NW));
        used01 += __popc(v & s.cm[q] & upto_mask(q, s.te[w])) +
                  (__popc(v & s.cm[words + q] & upto_mask(q, s.te[W + w])) << 16);
        used2 += __popc(v & s.cm[2 * words + q] & upto_mask(q, s.te[2 * W + w]));
      }
      used01 = __reduce_add_sync(kFull, used01);
      used2 = __reduce_add_sync(kFull, used2);
      if (lane == 0) {
        int4 h = s.hr[o];
        h.x -= (int)(used01 & 0xffffu);
        h.y -= (int)(used01 >> 16);
        h.z -= (int)used2;
        const int all = (int)(used01 & 0xffffu) + (int)(used01 >> 16) + (int)used2;
        h.w -= all;
        s.hr[o] = h;
        // an instance that had global headroom ran out of it
        if (all && h.w <= 0) a.stats[25] = 1;
      }
    }
    cluster_barrier(cs);
    if (!more) break;
    for (int o = wid; o * cs + cta < W; o += NW) {
      const int w = o * cs + cta;
      const int4 h = s.hr[o];
      for (int i = lane; i < 4 * cs; i += 32) {
        const int bb = i / cs, rank = i - bb * cs;
        const bool left = h.w > 0 && (bb == 0 ? h.x : (bb == 1 ? h.y : (bb == 2 ? h.z : 1))) > 0;
        st_cluster_u16(map_rank(bb < 3 ? sm_te + 2 * (bb * W + w) : sm_tg + 2 * w, rank), left ? kNever : -1);
      }
      if (lane == 0) s.seen[o] = 0;
    }
    for (int i = tid; i < W * NW; i += T) s.prop[i] = 0;
    for (int w = tid; w < W; w += T) {
      s.n01[w] = 0;
      s.n2[w] = 0;
    }
    cluster_barrier(cs);
  }
  // no CTA leaves while another may still read its shared memory: the last access to another
  // CTA's is before the barrier that ends the last window (or before the loop)
}

namespace {

// CTAs and threads of the selection cluster for a batch of n requests and W instances.  One CTA, with
// block barriers, for small batches of few instances; else the whole cluster, whose warps share the
// instances' thresholds, with as few threads as hold the batch (a round's choices share an SM's
// issue slots), then windows of 16 x 1024.  A route in us by one CTA and by 16 of 256 threads:
// 4 instances 76/84 at 256 requests, 16 instances 121/133 at 512 and 133/123 at 1,000; 32
// instances 197/173 at 256; 64 332/269 at 1,000; 512 563/244 at 256; 1,000 981/465 at 512.
// (Windows of 16 x 512 suit batches without cached prefixes, 16,384 requests of 64 instances
// 391/355, but not the steady loop: 65,536 of 128 instances 992/1,099.)
void select_shape(int n, int W, int max_cs, int* cs, int* threads) {
  *cs = n <= 512 && W < 32 ? 1 : max_cs;
  *threads = 256;
  while (*threads < 1024 && *cs * *threads < n) *threads <<= 1;
}

}  // namespace

cudaError_t select_configure(int* max_cluster) {
  // sized for the largest instance count and batch, so that contexts of any size share the setting
  cudaError_t e = cudaFuncSetAttribute(k4_select, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSelSmemMax);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k4_select, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  // 16 CTAs per cluster where the device can hold one, else the portable 8
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 16;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(16);
  lc.blockDim = dim3(1024);
  lc.dynamicSmemBytes = kSelSmemMax;
  lc.attrs = &at;
  lc.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k4_select, &lc) != cudaSuccess) {
    cudaGetLastError();
    clusters = 0;
  }
  *max_cluster = clusters > 0 ? 16 : 8;
  return cudaSuccess;
}

void launch_select(const SelectArgs& a, int max_cluster, cudaStream_t st) {
  if (a.n <= 0) return;
  int cs, threads;
  select_shape(a.n, a.W, max_cluster, &cs, &threads);
  cudaLaunchAttribute at[2] = {};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3(cs);
  lc.blockDim = dim3(threads);
  lc.dynamicSmemBytes = sel_smem_layout(a.W, cs, threads / 32, (a.n + 255) / 256, nullptr, nullptr);
  lc.stream = st;
  lc.attrs = at;
  lc.numAttrs = 2;
  cudaLaunchKernelEx(&lc, k4_select, a, cs);
}

}  // namespace misat
