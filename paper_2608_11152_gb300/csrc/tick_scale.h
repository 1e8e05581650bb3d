// Eviction ticks (metas, seq << 36 | arrival << 16 | 65535 - depth) in the bits that a sample of them
// uses, and the spread of a range over histogram bins.  Plain C++: a host test restates the
// eviction's arithmetic with it.
#pragma once

#ifdef __CUDACC__
#define MISAT_HD __host__ __device__ __forceinline__
#else
#define MISAT_HD inline
#endif

namespace misat {

// Metas without the bits that no sample uses (a commit's ticks fill a small part of the span between
// two sequence numbers): in this order the samples spread over the histogram's bins, while equal bins
// of the metas themselves held a whole commit each.  The order holds for every meta, sampled or
// not (m <= m' gives pack(m) <= pack(m')): a depth beyond the sampled ones counts as the deepest, and
// an arrival beyond them takes the last place of its sequence number, whatever its depth.
struct TickScale {
  int ab, db;      // bits of the samples' largest arrival and depth
  MISAT_HD unsigned long long pack(unsigned long long m) const {
    const unsigned long long low = (m & 0xffffu), base = 65536ull - (1ull << db);
    const unsigned long long arr = (m >> 16) & 0xfffffu, top = (1ull << ab) - 1;
    const unsigned long long in = arr <= top ? (arr << db) | (low > base ? low - base : 0ull) : (1ull << (ab + db)) - 1;
    return ((m >> 36) << (ab + db)) | in;
  }
  // the smallest meta that packs to x or more
  MISAT_HD unsigned long long unpack(unsigned long long x) const {
    const unsigned long long low = x & ((1ull << db) - 1), arr = (x >> db) & ((1ull << ab) - 1), seq = x >> (db + ab);
    if (seq >> 28) return ~0ull;
    return (seq << 36) | (arr << 16) | (low ? low + 65536ull - (1ull << db) : 0ull);
  }
};

constexpr int kTickBins = 4096;

// Shift that takes the values 0 .. range to bins 0 .. kTickBins - 1.
MISAT_HD int bin_shift(unsigned long long range) {
#ifdef __CUDA_ARCH__
  const int zeros = __clzll((long long)range);
#else
  const int zeros = range ? __builtin_clzll(range) : 64;
#endif
  return zeros < 52 ? 52 - zeros : 0;
}

}  // namespace misat
