// K1: chained 16-token block hash (Sec. 4.4: the router's prefix index is keyed by
// block hashes of the engine's prefix cache).
//
// Key of block j of a prompt:  c_j = mix64(XOR_i (x_i + (i+1)G) M) over the block's
// eight 64-bit token pairs x_i (M odd: a bijection of each word), a_j = a_{j-1} G + c_j
// (a_{-1} = seed),
// k_j = mix64(a_j ^ (j+1)) (+2 if < 2).  The chain step is affine mod 2^64, so a
// warp evaluates 32 consecutive blocks as an inclusive scan of affine maps:
// in-chunk sums s_j = sum_{i<=j} c_i G^{j-i} (Hillis-Steele, multiplier G^d at
// distance d), then a_j = carry G^{j+1} + s_j.
//
// Layout.  A chunk of 32 blocks is 512 tokens = 2 KiB, copied to shared memory asynchronously as
// four coalesced 512-byte warp copies, two chunks ahead of the one being hashed; lane j then
// reads block j whole.  (With the block's words spread over four lanes, which read them from global
// memory coalesced, combining and moving the parts cost a seventh of the instructions.)  A block's four 16-byte pieces are stored rotated by its
// number, so that the lanes' reads meet no bank conflicts.  A prompt that does not start on a
// 16-byte boundary is realigned on the way to registers, with one more piece read: the misalignment
// (0..3 words) is the same for the whole prompt.  Keys are written coalesced.
//
// Who hashes what (a warp per prompt throughout left the longest prompt of a batch as a serial
// chain of 0.5 us a chunk, most lanes of a short prompt's only chunk idle, and one atomic on one
// address per prompt):
//   long prompts    a CTA each, its four warps a chunk each per step; the chain is an affine
//                   map per chunk, so a step's carries follow from four sums in shared memory
//   middle prompts  a warp each
//   short prompts   (below 32 blocks) a warp per group of neighbouring prompts, whose blocks are
//                   packed into full chunks and scanned in segments
// in this order, so that the longest chains start first.  Long is 8 chunks or more, and at least
// what the resident warps get each on average: below it a warp's chain is short beside
// the whole pass, and a warp wastes less on a ragged end than a CTA.
//
// What bounds it: instruction issue (about 340 a chunk, two thirds of them 64-bit multiplies and
// what is around them) in large batches, 0.7 of the copy rate at 65,536 requests of 2,500 tokens;
// the longest prompt, 256 chunks in 64 steps, where prompts reach 128K tokens; latency in small
// ones.  Measured, us before (a warp per prompt throughout) and now: 64 requests 11.9/7.8, 4,096
// of 2,500 tokens 34.6/21.5, 16,384 of 1,300 55/33, 9,216 with prompts up to 128K 251/98, 131,072 of
// 110 tokens 105/26, 65,536 of 2,500 147/153.
#include <mutex>

#include "common.cuh"
#include "kernels.h"

namespace misat {

namespace {

__host__ __device__ constexpr uint64_t gold_pow(int k) {
  uint64_t r = 1;
  for (int i = 0; i < k; ++i) r *= kGold;
  return r;
}

constexpr unsigned kFull = 0xffffffffu;
constexpr uint64_t kWordMul = 0x94d049bb133111ebull;  // the content hash's odd word multiplier

constexpr int kHashWarps = 4;
constexpr int kStages = 3;        // chunks of a warp in shared memory: one hashed, two on their way
constexpr int kHashTile = 1024;   // requests whose compact key positions one CTA works out
constexpr int kStageInt4 = 129;   // a chunk and the int4 behind it
constexpr int kHashCtas = 8;       // CTAs per SM: 64 registers a thread, 198 KB of shared memory
constexpr int kLongChunks = 8;     // chunks from which a prompt may be long

// Copy of 16 bytes to shared memory (of which the first `bytes` are read, the others zeros).
__device__ __forceinline__ void fetch_int4(int4* dst, const int4* src, int bytes) {
  asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(bytes)
               : "memory");
}

// Per-lane constants of the chunk loop.
struct LaneConst {
  int lane;
  int to;           // slot of the lane's 16 bytes within 512 copied ones
  int rot;          // rotation of the pieces of block `lane`
  uint64_t pw;      // G^(lane+1): multiplier of the incoming carry for block `lane`
};

__device__ __forceinline__ LaneConst lane_const() {
  LaneConst c;
  c.lane = threadIdx.x & 31;
  c.to = (c.lane & 28) | ((c.lane & 3) ^ (c.lane >> 3));
  c.rot = (c.lane >> 1) & 3;
  uint64_t pw = kGold;
  if (c.lane & 1) pw *= gold_pow(1);
  if (c.lane & 2) pw *= gold_pow(2);
  if (c.lane & 4) pw *= gold_pow(4);
  if (c.lane & 8) pw *= gold_pow(8);
  if (c.lane & 16) pw *= gold_pow(16);
  c.pw = pw;
  return c;
}

__device__ __forceinline__ uint64_t pair_product(int i, int lo, int hi) {
  // (x_i + (i + 1) G) M with the second product a constant
  return ((uint64_t)(uint32_t)lo | ((uint64_t)(uint32_t)hi << 32)) * kWordMul + (uint64_t)(i + 1) * kGold * kWordMul;
}
// XOR of the block's products: its tokens are words OFF .. OFF + 15 of v[0..4].
template <int OFF>
__device__ __forceinline__ uint64_t content_xor(const int4 v[5]) {
  uint64_t x = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (OFF == 0) x ^= pair_product(2 * i, v[i].x, v[i].y) ^ pair_product(2 * i + 1, v[i].z, v[i].w);
    if (OFF == 1) x ^= pair_product(2 * i, v[i].y, v[i].z) ^ pair_product(2 * i + 1, v[i].w, v[i + 1].x);
    if (OFF == 2) x ^= pair_product(2 * i, v[i].z, v[i].w) ^ pair_product(2 * i + 1, v[i + 1].x, v[i + 1].y);
    if (OFF == 3) x ^= pair_product(2 * i, v[i].w, v[i + 1].x) ^ pair_product(2 * i + 1, v[i + 1].y, v[i + 1].z);
  }
  return x;
}

// One step of the chain's scan: block `lane` takes in the sum of the `d` blocks that end `d` before it.
template <int D>
__device__ __forceinline__ uint64_t scan_step(uint64_t s, bool in) {
  const uint64_t t = __shfl_up_sync(kFull, s, D);
  return s + (in ? t : 0ull) * gold_pow(D);
}
// e: the blocks before the lane's that belong to its sum.
__device__ __forceinline__ uint64_t chain_scan(uint64_t s, int e) {
  s = scan_step<1>(s, e >= 1);
  s = scan_step<2>(s, e >= 2);
  s = scan_step<4>(s, e >= 4);
  s = scan_step<8>(s, e >= 8);
  return scan_step<16>(s, e >= 16);
}

// Starts the copy of chunk c of a prompt whose first token is in int4 q0, and of the int4 behind it
// (an empty group behind the prompt's end: the groups are counted).
__device__ __forceinline__ void fetch_chunk(int4* st, const int4* tok4, int64_t n_int4, int64_t q0, int c, int n_chunks,
                                            const LaneConst& lc) {
  if (c < n_chunks) {
    const int64_t b = q0 + 128ll * c;
    if (b + 128 < n_int4) {
      const int4* src = tok4 + b + lc.lane;
#pragma unroll
      for (int i = 0; i < 4; ++i) fetch_int4(st + 32 * i + lc.to, src + 32 * i, 16);
      if (lc.lane == 0) fetch_int4(st + 128, src + 128, 16);
    } else {  // zeros behind the tokens' end
#pragma unroll 1
      for (int i = 0; i < 5; ++i) {
        const int64_t at = b + 32 * i + lc.lane;
        if (i < 4 || lc.lane == 0)
          fetch_int4(st + 32 * i + (i < 4 ? lc.to : 0), tok4 + (at < n_int4 ? at : 0), at < n_int4 ? 16 : 0);
      }
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// The oldest chunk has arrived, for every lane of the warp.
__device__ __forceinline__ void chunk_arrived() {
  asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
  __syncwarp();
}

// In-chunk sums s_j of the chain (carry zero); `off`: word of the stage's first int4 that the chunk
// begins with.  Sums behind the prompt's last block are of no use, and nobody's.  Only the products
// depend on `off`: with the whole chunk loop specialised on it, a third of the warps of a 26 us
// pass waited for instructions.
__device__ __forceinline__ uint64_t chunk_sums(const int4* st, int off, const LaneConst& lc) {
  const int lane = lc.lane;
  int4 v[5];
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = st[4 * lane + (i ^ lc.rot)];
  v[4] = st[4 * (lane + 1) + (((lane + 1) >> 1) & 3)];
  uint64_t x;
  switch (off) {
    case 0: x = content_xor<0>(v); break;
    case 1: x = content_xor<1>(v); break;
    case 2: x = content_xor<2>(v); break;
    default: x = content_xor<3>(v); break;
  }
  return chain_scan(mix64(x), lane);
}

__device__ __forceinline__ uint64_t block_key(uint64_t av, int64_t j) {
  const uint64_t key = mix64(av ^ (uint64_t)(j + 1));
  return key + (key < 2 ? 2 : 0);
}

// Where the key of block 0 of request r goes.
__device__ __forceinline__ int64_t key_base(const HashArgs& a, int r, int64_t t0) {
  return a.off ? (int64_t)a.tile[r / kHashTile] + a.off[r] : t0 >> 4;
}

// The keys of request r, which has at least one full block, by one warp or (cta) by all warps of
// the CTA: in step t warp v hashes chunk kHashWarps t + v.  s_tot[t & 1][v] is that chunk's sum
// (its affine map is a -> a G^32 + sum; only the last chunk may be ragged, and nothing
// follows it), from which every warp works out its carry and the step's.
__device__ __forceinline__ void hash_prompt(const HashArgs& a, int r, bool cta, const LaneConst& lc,
                                            int4 (*ring)[kStageInt4], uint64_t (*s_tot)[kHashWarps]) {
  const int lane = lc.lane, wid = cta ? (int)(threadIdx.x >> 5) : 0, warps = cta ? kHashWarps : 1;
  const int64_t t0 = a.tok_off[r];
  const int32_t nb = (int32_t)((a.tok_off[r + 1] - t0) >> 4);
  const int64_t kb = key_base(a, r, t0);
  const int4* tok4 = reinterpret_cast<const int4*>(a.tokens);
  const int64_t n_int4 = (a.n_tokens + 3) >> 2, q0 = t0 >> 2, lim = a.keys_cap - kb;
  const int off = (int)(t0 & 3);
  uint64_t* out = a.keys + kb;
  uint64_t carry = a.seed;
  const int n_chunks = (nb + 31) >> 5;
  __syncwarp();  // the last prompt's chunks have been read
#pragma unroll 1
  for (int k = 0; k < kStages - 1; ++k) fetch_chunk(ring[k], tok4, n_int4, q0, warps * k + wid, n_chunks, lc);
  int now = 0, ahead = kStages - 1;
#pragma unroll 1
  for (int c0 = 0, par = 0; c0 < n_chunks; c0 += warps, par ^= 1) {
    const int c = c0 + wid;
    chunk_arrived();
    fetch_chunk(ring[ahead], tok4, n_int4, q0, c + warps * (kStages - 1), n_chunks, lc);
    const int cnt = min(32, nb - 32 * c);  // <= 0 behind the prompt's end
    const uint64_t s = cnt > 0 ? chunk_sums(ring[now], off, lc) : 0;
    uint64_t mine = carry;
    if (cta) {
      if (lane == 31) s_tot[par][wid] = s;
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kHashWarps; ++u) {
        if (u == wid) mine = carry;
        carry = carry * gold_pow(32) + s_tot[par][u];
      }
    } else {
      carry = carry * gold_pow(32) + __shfl_sync(kFull, s, 31);
    }
    const int64_t j = 32ll * c + lane;
    const uint64_t key = block_key(mine * lc.pw + s, j);
    if (lane < cnt && j < lim) out[j] = key;
    ahead = now;
    now = now + 1 == kStages ? 0 : now + 1;
  }
}

// The short prompts (1 .. kHashShort blocks) among requests [r0, r0 + a.group), one warp: lane i
// owns request r0 + i, the prompts' blocks in arrival order are numbered through, and chunk c takes
// numbers 32c .. 32c + 31, a lane each.
__device__ __forceinline__ void hash_group(const HashArgs& a, int r0, const LaneConst& lc) {
  const int lane = lc.lane;
  const int4* tok4 = reinterpret_cast<const int4*>(a.tokens);
  const int r = r0 + lane;
  const bool in = lane < a.group && r < a.n;
  const int64_t t0 = in ? a.tok_off[r] : 0;
  int nb = in ? (int)((a.tok_off[r + 1] - t0) >> 4) : 0;
  if (nb > kHashShort) nb = 0;  // on a list
  const int64_t kb = in ? key_base(a, r, t0) : 0;
  int incl = nb;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += u;
  }
  const int total = __shfl_sync(kFull, incl, 31);
  // token and key positions relative to the group's first request (below 32 x 2^20 tokens)
  const int64_t tb = __shfl_sync(kFull, t0, 0), kb0 = __shfl_sync(kFull, kb, 0);
  const int excl = incl - nb, trel = (int)(t0 - tb), krel = (int)(kb - kb0);
  uint64_t carry = a.seed;
  for (int x0 = 0; x0 < total; x0 += 32) {
    const int x = x0 + lane;
    // owner of block x: the first lane whose inclusive count is above x
    int o = 0;
#pragma unroll
    for (int h = 16; h > 0; h >>= 1)
      if (__shfl_sync(kFull, incl, o + h - 1) <= x) o += h;
    const int j = x - __shfl_sync(kFull, excl, o);
    const int w0 = __shfl_sync(kFull, trel, o) + 16 * j;
    const int kr = __shfl_sync(kFull, krel, o) + j;
    const bool live = x < total;
    int4 v[5];
    const int64_t t0b = tb + w0, at = t0b >> 2;
    const int off = (int)(t0b & 3);
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = live ? __ldg(tok4 + at + i) : make_int4(0, 0, 0, 0);
    v[4] = live && off ? __ldg(tok4 + at + 4) : make_int4(0, 0, 0, 0);
    if (off & 2) {
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        const int4 n = i < 4 ? v[i + 1] : v[i];
        v[i] = make_int4(v[i].z, v[i].w, n.x, n.y);
      }
    }
    if (off & 1) {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = make_int4(v[i].y, v[i].z, v[i].w, v[i + 1].x);
    }
    // segmented scan: block j of its prompt takes in the blocks before it in this chunk
    const int e = min(j, lane);
    const uint64_t s = chain_scan(live ? mix64(content_xor<0>(v)) : 0ull, e);
    // before the chunk's first block of this prompt: the last chunk's carry, or the seed
    const uint64_t pw = __shfl_sync(kFull, lc.pw, e & 31);
    const uint64_t av = (j > lane ? carry : a.seed) * pw + s;
    const uint64_t key = block_key(av, j);
    if (live && kb0 + kr < a.keys_cap) a.keys[kb0 + kr] = key;
    carry = __shfl_sync(kFull, av, 31);
  }
}

__device__ __forceinline__ void hash_batch(const HashArgs& a) {
  __shared__ int4 s_ring[kHashWarps][kStages][kStageInt4];
  __shared__ uint64_t s_tot[2][kHashWarps];
  __shared__ int s_item;
  const LaneConst lc = lane_const();
  const int wid = threadIdx.x >> 5;
  int4 (*ring)[kStageInt4] = s_ring[wid];
  const int n_long = (int)a.ctr[kHashNLong], n_mid = (int)a.ctr[kHashNMid];
  // The first items are the CTA's (the warp's) own number, the next ones come from a counter; where
  // CTAs come late from long prompts, the warps' first ones do too.
  const int own = wid * (int)gridDim.x + (int)blockIdx.x;
  const int first = n_long ? 0 : (int)(gridDim.x * kHashWarps);
  auto next = [&](int c) {
    int i = 0;
    if (lc.lane == 0) i = first + (int)atomicAdd(a.ctr + c, 1u);
    return __shfl_sync(kFull, i, 0);
  };
  bool cta = (int)blockIdx.x < n_long;
  int item = cta ? (int)blockIdx.x : (n_long ? (n_mid ? next(kHashWMid) : 0) : own);
#pragma unroll 1
  while (cta || item < n_mid) {
    hash_prompt(a, a.list[cta ? item : a.n - 1 - item], cta, lc, ring, s_tot);
    if (cta) {
      __syncthreads();
      if (threadIdx.x == 0) s_item = (int)(gridDim.x + atomicAdd(a.ctr + kHashWLong, 1u));
      __syncthreads();
      item = s_item;
      cta = item < n_long;
      if (cta) continue;
    }
    if (n_mid <= first) break;  // every warp had its own
    item = next(kHashWMid);
  }
  const int groups = (a.n + a.group - 1) / a.group;
  if (n_long + n_mid < a.n)
    for (int i = n_long ? next(kHashWGroup) : own; i < groups; i = groups <= first ? groups : next(kHashWGroup))
      hash_group(a, i * a.group, lc);
}

// Requests per group of short prompts: as many as leave every resident warp one.
int hash_group_size(int32_t n, int warps) {
  int g = 1;
  while (g < 32 && (int64_t)g * warps < n) g <<= 1;
  return g;
}

}  // namespace

int32_t hash_long_blocks(int64_t n_tokens, int num_sms) {
  const int64_t chunks = n_tokens / 512 / ((int64_t)num_sms * kHashCtas * kHashWarps);
  return (int32_t)(32 * (chunks < kLongChunks ? kLongChunks : (chunks > 2048 ? 2048 : chunks)));
}

__global__ void __launch_bounds__(32 * kHashWarps, kHashCtas) k1_block_hash(HashArgs a) {
  chain_wait();
  if (*a.err) return;
  hash_batch(a);
}

__global__ void __launch_bounds__(256) k1_lists(HashArgs a) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t nb = r < a.n ? (int32_t)((a.tok_off[r + 1] - a.tok_off[r]) >> 4) : 0;
  hash_list(a.ctr, a.list, a.n, r, nb, a.long_blocks);
}

void launch_hash_lists(const HashArgs& a, cudaStream_t st) {
  cudaMemsetAsync(a.ctr, 0, kHashCtrs * sizeof(unsigned), st);
  k1_lists<<<(a.n + 255) / 256, 256, 0, st>>>(a);
}

void launch_block_hash(HashArgs a, int num_sms, cudaStream_t st) {
  const int res = resident_grid<k1_block_hash>(32 * kHashWarps, 0, num_sms);
  a.group = hash_group_size(a.n, res * kHashWarps);
  launch_chained(k1_block_hash, a.n < res ? a.n : res, 32 * kHashWarps, 0, st, a);
}

// ---------------------------------------------------------------------------
// Allocation-free block hashing.
//
// Some callers of this library cannot allocate device memory: an inference engine
// that has already handed all free HBM to its KV-cache pool (a new cudaMalloc would
// fail, or fragment and shrink that pool), or a hook that runs inside another
// framework's allocator or memory-accounting scope, where new device allocations are
// not allowed.  misat_block_hash_noalloc serves them: it computes the same chained
// block keys as the routing path and allocates nothing.  Its only scratch -- key
// offsets, the list of longer prompts, counters and an error word -- lives in the
// file-scope array below, which every GPU that loads this library holds
// (about 512 KiB) until the process exits.

// scratch layout in 8-byte words: [0] error word | [1..3] counters of the hash | [8..39] blocks
// per tile of requests (32-bit) | [40 ..] key offsets within the tile, then the list of longer
// prompts (32-bit both: a batch has fewer than 2^32 blocks)
constexpr int kNoAllocMaxRequests = MISAT_NOALLOC_MAX_REQUESTS;
constexpr int kNoAllocHead = 40;
constexpr int kNoAllocWords = kNoAllocHead + kNoAllocMaxRequests;
static_assert(kNoAllocMaxRequests <= 64 * kHashTile, "tile sums");
static __device__ __align__(256) unsigned long long g_noalloc_scratch[kNoAllocWords];

namespace {

// A CTA per tile of kHashTile requests: validate the offsets, write the exclusive prefix of
// floor(L_r / 16) (compact key positions within the tile) and the tile's sum, list the longer
// prompts.  The hash adds up the sums of the tiles before a request's: one CTA that walked all
// tiles took 18.8 us at 20,001 requests, a memory round trip and a block scan per tile.
__global__ void __launch_bounds__(kHashTile) k1na_offsets(HashArgs a, unsigned long long* scratch) {
  __shared__ unsigned s_sum[kHashTile / 32];
  chain_wait();
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int r = blockIdx.x * kHashTile + t;
  int64_t o0 = 0, o1 = 0;
  if (r < a.n) {
    o0 = a.tok_off[r];
    o1 = a.tok_off[r + 1];
  }
  const bool ok = o0 >= 0 && o1 >= o0 && o1 <= a.n_tokens && o1 - o0 < (1 << 20) && (r != 0 || o0 == 0) &&
                  (r != a.n - 1 || o1 == a.n_tokens);
  if (!ok) scratch[0] = (unsigned long long)(long long)MISAT_ERR_INVALID_ARG;
  const int nb = ok ? (int)((o1 - o0) >> 4) : 0;
  unsigned incl = (unsigned)nb;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned u = __shfl_up_sync(kFull, incl, d);
    if (lane >= d) incl += u;
  }
  if (lane == 31) s_sum[wid] = incl;
  __syncthreads();
  const unsigned ws = lane < kHashTile / 32 ? s_sum[lane] : 0u;
  const unsigned before = __reduce_add_sync(kFull, lane < wid ? ws : 0u), all = __reduce_add_sync(kFull, ws);
  if (r < a.n) a.off[r] = before + incl - (unsigned)nb;
  if (t == 0) a.tile[blockIdx.x] = all;
  hash_list(a.ctr, a.list, a.n, r, nb, a.long_blocks);
}

// The block hash of k1_block_hash with compact output positions: block j of request r goes to
// keys[s_tile[tile of r] + off[r] + j].
__global__ void __launch_bounds__(32 * kHashWarps, kHashCtas) k1na_hash(HashArgs a, unsigned long long* scratch) {
  __shared__ uint32_t s_tile[65];  // blocks before each tile
  chain_wait();
  if (scratch[0]) return;
  const int tiles = (a.n + kHashTile - 1) / kHashTile, t = threadIdx.x;
  if (t <= 64) {
    uint32_t v = 0;
    for (int k = 0; k < t && k < tiles; ++k) v += a.tile[k];
    s_tile[t] = v;
  }
  __syncthreads();
  const int64_t total = s_tile[64];
  if (total > a.keys_cap) {
    if (blockIdx.x == 0 && t == 0) scratch[0] = (unsigned long long)(long long)MISAT_ERR_INVALID_ARG;
    return;
  }
  a.keys_cap = total;
  a.tile = s_tile;
  hash_batch(a);
}

std::mutex g_noalloc_mu;
unsigned long long* g_noalloc_ptr[256];  // device address of the scratch array, per device
int g_noalloc_sms[256], g_noalloc_ctas[256];  // SMs, resident CTAs of the hash

// Per device, once, with that device current: the device address of the scratch array.
int noalloc_setup(unsigned long long** scratch, int* sms, int* ctas) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return MISAT_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) {
      cudaGetLastError();
      return MISAT_ERR_CUDA;
    }
    int s = 0;
    if (cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return MISAT_ERR_CUDA;
    g_noalloc_sms[dev] = s;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k1na_hash, 32 * kHashWarps, 0) != cudaSuccess)
      return MISAT_ERR_CUDA;
    g_noalloc_ctas[dev] = s * (per_sm < 1 ? 1 : per_sm);
    g_noalloc_ptr[dev] = reinterpret_cast<unsigned long long*>(p);
  }
  *scratch = g_noalloc_ptr[dev];
  *sms = g_noalloc_sms[dev];
  *ctas = g_noalloc_ctas[dev];
  return MISAT_OK;
}

}  // namespace
}  // namespace misat

extern "C" int misat_block_hash_noalloc(const int64_t* tok_off, const int32_t* tokens, int32_t n, int64_t n_tokens,
                                        uint64_t seed, uint64_t* keys_out, int64_t keys_cap, void* cuda_stream) {
  using namespace misat;
  if (n < 0 || n_tokens < 0 || keys_cap < 0) return MISAT_ERR_INVALID_ARG;
  if (n > kNoAllocMaxRequests) return MISAT_ERR_BATCH_TOO_LARGE;
  if (n == 0) return MISAT_OK;
  if (!tok_off || (keys_cap > 0 && !keys_out)) return MISAT_ERR_INVALID_ARG;
  if (n_tokens > 0 && (!tokens || ((uintptr_t)tokens & 15) != 0)) return MISAT_ERR_INVALID_ARG;
  unsigned long long* scratch = nullptr;
  int sms = 1, res = 1;
  int rc = noalloc_setup(&scratch, &sms, &res);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  HashArgs a{};
  a.tok_off = tok_off;
  a.tokens = tokens;
  a.n_tokens = n_tokens;
  a.n = n;
  a.seed = seed;
  a.keys = keys_out;
  a.keys_cap = keys_cap;
  a.ctr = reinterpret_cast<unsigned*>(scratch + 1);
  a.tile = reinterpret_cast<uint32_t*>(scratch + 8);
  a.off = reinterpret_cast<uint32_t*>(scratch + kNoAllocHead);
  a.list = reinterpret_cast<int32_t*>(scratch + kNoAllocHead) + n;
  a.long_blocks = hash_long_blocks(n_tokens, sms);
  a.group = hash_group_size(n, res * kHashWarps);
  if (cudaMemsetAsync(scratch, 0, 8 * sizeof(*scratch), st) != cudaSuccess) return MISAT_ERR_CUDA;
  k1na_offsets<<<(n + kHashTile - 1) / kHashTile, kHashTile, 0, st>>>(a, scratch);
  launch_chained(k1na_hash, n < res ? n : res, 32 * kHashWarps, 0, st, a, scratch);
  if (cudaGetLastError() != cudaSuccess) return MISAT_ERR_CUDA;
  unsigned long long err = 0;
  if (cudaMemcpyAsync(&err, scratch, sizeof(err), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return MISAT_ERR_CUDA;
  return (int)(long long)err;
}
