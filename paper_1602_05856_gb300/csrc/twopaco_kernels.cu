// CUDA kernels of the junction-detection library (sm_103a).
//
// One run = pack, then per round (Algorithm 3, section "Multiple Rounds")
// the two passes of Algorithm 2 (Filter-Junctions-Two-Pass), each an
// instance of Algorithm 1 (Filter-Junctions): an insert loop and a probe
// loop, separated by a kernel boundary (the barrier of section
// "Parallelization Scheme"); then one emit of the junction positions.
//
// The first pass visits every position. An insert thread takes kInsertR
// consecutive positions and cuts their k-mers and reverse complements out of
// the packed words by shifts (rolling them from one to the next only across a
// string boundary); besides its filter OR it leaves an 8-byte
// descriptor per position, which the probe streams (4 rows of 32 positions
// per warp and step) instead of walking again. The second pass visits only
// the candidates the first pass left, from a compact list.
//
// Encoding: A,C,G,T = 0,1,2,3, 16 bases per 32-bit word, first base in the
// two most significant bits. A k-mer is the integer with its first base most
// significant, so integer order is lexicographic order (the normalized form
// of a k-mer is min(k-mer, reverse complement)), and complement is 3 - x.
#include "twopaco_internal.h"

#include <algorithm>
#include <atomic>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

// This file is compiled several times, so that its many instances build in
// parallel: on its own (the kernels that are no template of the k-mer width
// and the bits per item, and the library's entry points), and with
// TWOPACO_PART from the small files beside it, for the rounds, the class map
// and the partition pre-pass of one k-mer width and half of the bits per item:
//   1, 2  k <= 31, 1-4 and 5-8 bits      3, 4  k <= 63, 1-4 and 5-8 bits
//   5     k <= 127, the bits a run-time value

namespace twopaco {

// Optional per-kernel timing: CUDA events recorded on the launch stream
// right before and after every kernel (state shared by both halves).
struct ProfRecord {
  const char* name;
  cudaEvent_t start, stop;
};
extern std::atomic<unsigned long long> g_launches;
extern std::mutex g_prof_mu;
extern bool g_prof_on;
extern std::vector<ProfRecord> g_prof;
extern std::vector<cudaEvent_t> g_event_pool;
#ifndef TWOPACO_PART
std::atomic<unsigned long long> g_launches{0};
std::mutex g_prof_mu;
bool g_prof_on = false;
std::vector<ProfRecord> g_prof;
std::vector<cudaEvent_t> g_event_pool;
#endif

namespace {

cudaEvent_t take_event() {
  if (!g_event_pool.empty()) {
    cudaEvent_t e = g_event_pool.back();
    g_event_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

// Scope that brackets one kernel launch with events when profiling is on.
struct Timed {
  ProfRecord rec{nullptr, nullptr, nullptr};
  cudaStream_t s;
  unsigned flags = cudaEventRecordDefault;
  Timed(const char* name, cudaStream_t st) : s(st) {
    std::lock_guard<std::mutex> g(g_prof_mu);
    if (!g_prof_on) return;
    rec.name = name;
    rec.start = take_event();
    rec.stop = take_event();
    // inside a stream capture the events must become graph nodes of their own
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusActive)
      flags = cudaEventRecordExternal;
    cudaEventRecordWithFlags(rec.start, s, flags);
  }
  ~Timed() {
    if (!rec.name) return;
    cudaEventRecordWithFlags(rec.stop, s, flags);
    std::lock_guard<std::mutex> g(g_prof_mu);
    g_prof.push_back(rec);
  }
};

// Consecutive positions per thread (at most 16: one 32-bit word of successor
// bases) in the first-pass kernels and the partition pre-pass.
constexpr int kInsertR = 16;
// Inputs below kInsertSmall positions take fewer per thread, so that all SMs
// have warps to spare: 16 per thread left 0.2 M positions on 46 blocks. Whole builds at
// k = 25 and 63, 16 against 4 per thread: 0.2 M positions 71.5 to 66.2 and 85.8 to 78.1 us,
// 1 M 81.8 to 77.4 and 98.1 to 92.4, 2.1 M 92.2 to 90.2 and 125.1 to 125.2, 4 M 129.1 to 129.1
// and 225.2 to 232.4, 6 M 187.3 to 188.8 and 444 to 453.
constexpr int kInsertSmallR = 4;
constexpr uint64_t kInsertSmall = 1ull << 21;
constexpr int kProbeR = 8;
constexpr bool kProbePrefetch = true;  // the probe's descriptors loaded one step ahead
constexpr int kR = 8;  // partition pre-pass

using Ranges = std::vector<std::pair<uint64_t, uint64_t>>;

// ---------------------------------------------------------------------------
// k-mer words
// ---------------------------------------------------------------------------

struct Key {
  uint64_t hi, lo;  // value = hi * 2^64 + lo; hi == 0 for k <= 31
};

// k-mers of 64 to 127 bases: four words, w[0] the most significant.
struct Key4 {
  uint64_t w[4];
};

// The k-mer word of KW = 1 (k <= 31), 2 (k <= 63) or 4 (k <= 127).
template <int KW>
struct KeyOf {
  using T = Key;
};
template <>
struct KeyOf<4> {
  using T = Key4;
};
template <int KW>
using KeyT = typename KeyOf<KW>::T;

__device__ __forceinline__ bool key_less(const Key& a, const Key& b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}

__device__ __forceinline__ bool key_less(const Key4& a, const Key4& b) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (a.w[i] != b.w[i]) return a.w[i] < b.w[i];
  return false;
}

__device__ __forceinline__ bool key_eq(const Key4& a, const Key4& b) {
  return a.w[0] == b.w[0] && a.w[1] == b.w[1] && a.w[2] == b.w[2] && a.w[3] == b.w[3];
}

// a0:a1:a2:a3 (a0 most significant) shifted right by s bits, 0 <= s <= 128.
__device__ __forceinline__ Key4 shr256(uint64_t a0, uint64_t a1, uint64_t a2, uint64_t a3, int s) {
  if (s >= 64) {
    a3 = a2; a2 = a1; a1 = a0; a0 = 0; s -= 64;
  }
  if (s >= 64) {
    a3 = a2; a2 = a1; a1 = a0; a0 = 0; s -= 64;
  }
  if (s) {
    a3 = (a3 >> s) | (a2 << (64 - s));
    a2 = (a2 >> s) | (a1 << (64 - s));
    a1 = (a1 >> s) | (a0 << (64 - s));
    a0 >>= s;
  }
  return Key4{{a0, a1, a2, a3}};
}

// splitmix64 output finalizer (Steele, Lea & Flood, OOPSLA 2014).
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z ^= z >> 30;
  z *= 0xbf58476d1ce4e5b9ull;
  z ^= z >> 27;
  z *= 0x94d049bb133111ebull;
  z ^= z >> 31;
  return z;
}

// H of a k-mer: mix64(lo), mix64(lo ^ mix64(hi)), or for four words
// mix64(w3 ^ mix64(w2 ^ mix64(w1 ^ mix64(w0)))) -- the same value whenever the
// higher words are zero, as mix64(0) = 0.
template <int KW>
__device__ __forceinline__ uint64_t key_hash(const KeyT<KW>& v) {
  if constexpr (KW == 4) return mix64(v.w[3] ^ mix64(v.w[2] ^ mix64(v.w[1] ^ mix64(v.w[0]))));
  else return KW == 1 ? mix64(v.lo) : mix64(v.lo ^ mix64(v.hi));
}

// Second hash word: H times the 64-bit golden ratio; only its high bits are used.
__device__ __forceinline__ uint64_t second_hash(uint64_t H) { return H * 0x9e3779b97f4a7c15ull; }

// Start slot of a k-mer in the pass-2 table (bits above the partition bins).
__device__ __forceinline__ uint64_t slot_hash(uint64_t H) { return H >> 16; }

// Start slot of a k-mer in a pass-2 table of cap slots: bits 16-47 of H scaled
// to [0, cap) by a multiply-high (Lemire, "Fast random integer generation in an
// interval", 2019); larger tables take a remainder. Rounded down to a whole
// sector of N slots (cap is a multiple of N): a probe reads sector by sector.
template <int N>
__device__ __forceinline__ uint64_t slot_start(uint64_t H, uint64_t cap) {
  const uint64_t i = cap <= 0xFFFFFFFFull ? __umulhi((uint32_t)(H >> 16), (uint32_t)cap) : slot_hash(H) % cap;
  return i & ~(uint64_t)(N - 1);
}

// Reverse the order of the 32 two-bit groups of x.
__device__ __forceinline__ uint64_t rev_pairs(uint64_t x) {
  const uint64_t b = __brevll(x);
  return ((b >> 1) & 0x5555555555555555ull) | ((b & 0x5555555555555555ull) << 1);
}

__device__ __forceinline__ uint32_t base_at(const uint32_t* __restrict__ packed, uint64_t g) {
  return (__ldg(packed + (g >> 4)) >> (30u - 2u * (uint32_t)(g & 15))) & 3u;
}

// 16 bases starting at base g, first base in the two most significant bits.
__device__ __forceinline__ uint32_t bases16(const uint32_t* __restrict__ packed, uint64_t g) {
  const uint32_t* p = packed + (g >> 4);
  return __funnelshift_l(__ldg(p + 1), __ldg(p), 2u * (uint32_t)(g & 15));
}

// 32 bases starting at base g, first base in the two most significant bits
// (the word after the window is read too: the packed input ends in pad words).
__device__ __forceinline__ uint64_t bases32(const uint32_t* __restrict__ packed, uint64_t g) {
  const uint32_t* p = packed + (g >> 4);
  const uint32_t o2 = 2u * (uint32_t)(g & 15);
  const uint32_t w0 = __ldg(p), w1 = __ldg(p + 1), w2 = __ldg(p + 2);
  return ((uint64_t)__funnelshift_l(w1, w0, o2) << 32) | __funnelshift_l(w2, w1, o2);
}

// The k-mer starting at base g. KW = 1 for k <= 31 (one 64-bit word), 2 for
// 32 <= k <= 63, 4 for 64 <= k <= 127.
template <int KW>
__device__ __forceinline__ KeyT<KW> load_kmer(const uint32_t* __restrict__ packed, uint64_t g, int k) {
  if constexpr (KW == 4) {
    // 128 bases from g, then the first k of them
    return shr256(bases32(packed, g), bases32(packed, g + 32), bases32(packed, g + 64),
                  bases32(packed, g + 96), 256 - 2 * k);
  } else {
    const uint64_t a = bases32(packed, g);
    Key v;
    if (KW == 1) {
      v.hi = 0;
      v.lo = a >> (64 - 2 * k);
    } else {
      const uint64_t b = bases32(packed, g + 32);
      const int sh = 128 - 2 * k;  // 2 .. 64
      if (sh == 64) {
        v.hi = 0;
        v.lo = a;
      } else {
        v.hi = a >> sh;
        v.lo = (b >> sh) | (a << (64 - sh));
      }
    }
    return v;
  }
}

// Reverse complement of a k-mer.
template <int KW>
__device__ __forceinline__ KeyT<KW> revcomp(const KeyT<KW>& v, int k) {
  if constexpr (KW == 4) {
    return shr256(rev_pairs(~v.w[3]), rev_pairs(~v.w[2]), rev_pairs(~v.w[1]), rev_pairs(~v.w[0]),
                  256 - 2 * k);
  } else {
    Key r;
    if (KW == 1) {
      r.hi = 0;
      r.lo = rev_pairs(~v.lo) >> (64 - 2 * k);
    } else {
      const uint64_t nh = rev_pairs(~v.lo), nl = rev_pairs(~v.hi);
      const int sh = 128 - 2 * k;
      if (sh == 64) {
        r.hi = 0;
        r.lo = nh;
      } else {
        r.hi = nh >> sh;
        r.lo = (nl >> sh) | (nh << (64 - sh));
      }
    }
    return r;
  }
}

// Slide the k-mer one base to the right: f gains base b at its end, r (the
// reverse complement) gains 3 - b at its start.
template <int KW>
__device__ __forceinline__ void roll(KeyT<KW>& f, KeyT<KW>& r, uint32_t b, int k) {
  if constexpr (KW == 4) {
    f.w[0] = (f.w[0] << 2) | (f.w[1] >> 62);
    f.w[1] = (f.w[1] << 2) | (f.w[2] >> 62);
    f.w[2] = (f.w[2] << 2) | (f.w[3] >> 62);
    f.w[3] = (f.w[3] << 2) | b;
    const int hb = 2 * k - 128;  // bits above the two low words, 0 .. 126
    if (hb > 64) {
      f.w[0] &= (1ull << (hb - 64)) - 1ull;
    } else {
      f.w[0] = 0;
      if (hb < 64) f.w[1] &= (1ull << hb) - 1ull;
    }
    r.w[3] = (r.w[3] >> 2) | (r.w[2] << 62);
    r.w[2] = (r.w[2] >> 2) | (r.w[1] << 62);
    r.w[1] = (r.w[1] >> 2) | (r.w[0] << 62);
    r.w[0] >>= 2;
    const int top = 2 * k - 2;  // bit of the first base, from the least significant
    const uint64_t c = 3u - b;
    if (top >= 192) r.w[0] |= c << (top - 192);
    else if (top >= 128) r.w[1] |= c << (top - 128);
    else r.w[2] |= c << (top - 64);
  } else if (KW == 1) {
    f.lo = ((f.lo << 2) | b) & ((1ull << (2 * k)) - 1ull);
    r.lo = (r.lo >> 2) | ((uint64_t)(3u - b) << (2 * k - 2));
  } else {
    const int hb = 2 * k - 64;  // bits of the high word, 0 .. 62
    f.hi = ((f.hi << 2) | (f.lo >> 62)) & ((1ull << hb) - 1ull);
    f.lo = (f.lo << 2) | b;
    r.lo = (r.lo >> 2) | (r.hi << 62);
    r.hi >>= 2;
    if (hb >= 2) r.hi |= (uint64_t)(3u - b) << (hb - 2);
    else r.lo |= (uint64_t)(3u - b) << 62;
  }
}

// First base of a k-mer.
template <int KW>
__device__ __forceinline__ uint32_t first_base(const KeyT<KW>& f, int k) {
  if constexpr (KW == 4) {
    const int top = 2 * k - 2;
    const uint64_t x = top >= 192 ? f.w[0] >> (top - 192) : (top >= 128 ? f.w[1] >> (top - 128) : f.w[2] >> (top - 64));
    return (uint32_t)x & 3u;
  } else if (KW == 1) {
    return (uint32_t)(f.lo >> (2 * k - 2)) & 3u;
  } else {
    return (uint32_t)(k == 32 ? f.lo >> 62 : f.hi >> (2 * k - 66)) & 3u;
  }
}

// ---------------------------------------------------------------------------
// Positions and occurrences
// ---------------------------------------------------------------------------

struct Bounds {
  uint64_t start, end;
};

// [start, end) of the string that holds base g (largest t with offsets[t] <= g).
__device__ __forceinline__ Bounds seq_bounds(const RunView& v, uint64_t g) {
  uint32_t lo = 0, hi = v.n_seqs;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (__ldg(v.offsets + mid) <= g) lo = mid; else hi = mid;
  }
  return {__ldg(v.offsets + lo), __ldg(v.offsets + lo + 1)};
}

// The string bounds a k-mer at g must lie in. Without N splitting these are
// the input string's; with it, the N-free piece holding g, or the empty
// range [g, g) when base g is N (no k-mer starts there, and the next
// position looks its bounds up again).
__device__ __forceinline__ Bounds kmer_bounds(const RunView& v, uint64_t g) {
  if (!v.nmask) return seq_bounds(v, g);
  if ((__ldg(v.nmask + (g >> 5)) >> (g & 31)) & 1u) return {g, g};
  const uint64_t n = __ldcg(&v.hdr->n_runs);  // runs[n] = m
  uint64_t lo = 0, hi = n;                    // largest j < n with runs[j] <= g
  while (hi - lo > 1) {
    const uint64_t mid = (lo + hi) >> 1;
    if (__ldg(v.runs + mid) <= g) lo = mid; else hi = mid;
  }
  return {__ldg(v.runs + lo), __ldg(v.runs + lo + 1)};
}

// One k-mer occurrence, read in the orientation of its normalized form.
template <int KW>
struct OccT {
  KeyT<KW> key;    // normalized k-mer
  uint64_t H;      // key_hash(key)
  uint32_t j1, j2; // filter items this occurrence inserts (equal but for a palindrome)
  uint32_t tbits;  // pass-2 bits: in-bases 0-3, out-bases 4-7, sentinel 8
  bool sentinel;   // first or last k-mer of its string
  bool rc;         // the string reads the reverse complement of key here
};

// The (predecessor, successor) item of an occurrence, read in the k-mer's own
// orientation (jf) and on the other strand (jr = 4 (3 - succ) + (3 - pred)).
__device__ __forceinline__ uint32_t item_forward(uint32_t pred, uint32_t succ) { return 4u * pred + succ; }
__device__ __forceinline__ uint32_t item_reverse(uint32_t pred, uint32_t succ) { return 15u - 4u * succ - pred; }

// Pass-2 bits of an item (16: the sentinel item).
__device__ __forceinline__ uint32_t item_tbits(uint32_t j) {
  return j == 16u ? 1u << 8 : (1u << (j >> 2)) | (16u << (j & 3u));
}

// The filter items and pass-2 bits of one occurrence: its (predecessor,
// successor) pair read in the orientation of the normalized form (both
// orientations of a palindrome), or the sentinel item and bit.
__device__ __forceinline__ void occ_bits(uint32_t pred, uint32_t succ, bool use_f, bool use_r, bool sentinel,
                                         uint32_t* j1, uint32_t* j2, uint32_t* tbits) {
  const uint32_t jf = item_forward(pred, succ), jr = item_reverse(pred, succ);
  *j1 = sentinel ? 16u : (use_f ? jf : jr);
  *j2 = sentinel ? 16u : (use_r ? jr : jf);
  *tbits = item_tbits(*j1) | item_tbits(*j2);
}

template <int KW>
__device__ __forceinline__ void make_occ(const RunView& v, const KeyT<KW>& f, const KeyT<KW>& r,
                                         uint32_t pred, uint32_t succ, bool sentinel, OccT<KW>* oc) {
  const bool use_f = !v.both || !key_less(r, f);  // f is the normalized form
  const bool use_r = v.both && !key_less(f, r);   // r is (palindromes: both)
  oc->key = use_f ? f : r;
  oc->H = key_hash<KW>(oc->key);
  oc->sentinel = sentinel;
  oc->rc = !use_f;
  occ_bits(pred, succ, use_f, use_r, sentinel, &oc->j1, &oc->j2, &oc->tbits);
}

// The occurrence at global position g, read from scratch; false if no k-mer
// starts at g.
template <int KW>
__device__ __forceinline__ bool read_occurrence(const RunView& v, uint64_t g, OccT<KW>* oc) {
  const Bounds b = kmer_bounds(v, g);
  if (g + (uint64_t)v.k > b.end) return false;
  const KeyT<KW> f = load_kmer<KW>(v.packed, g, v.k);
  const bool has_pred = g > b.start, has_succ = g + (uint64_t)v.k < b.end;
  const uint32_t pred = has_pred ? base_at(v.packed, g - 1) : 0u;
  const uint32_t succ = has_succ ? base_at(v.packed, g + v.k) : 0u;
  const KeyT<KW> r = v.both ? revcomp<KW>(f, v.k) : f;
  make_occ<KW>(v, f, r, pred, succ, !has_pred || !has_succ, oc);
  return true;
}

// Distance from p0 to x, clamped to [-2^30, 2^30] (positions within one
// thread's chunk are compared in 32 bits).
__device__ __forceinline__ int32_t rel(uint64_t x, uint64_t p0) {
  constexpr int64_t kClamp = 1ll << 30;
  const int64_t d = (int64_t)(x - p0);
  return (int32_t)(d > kClamp ? kClamp : (d < -kClamp ? -kClamp : d));
}

// The occurrence of a listed candidate: its string bounds are not needed,
// because the list marks candidates at a string end (sentinel positions)
// and every other candidate has a predecessor and a successor. Those are read
// from one window with the k-mer, which starts at the predecessor: 2 KW + 1
// aligned words hold any 32 KW + 1 bases.
//
// word(i) gives word i of the window's packed words: the window starts at the
// base p (2 bits) of word 0 (the predecessor, or a sentinel's first base).
template <int KW, typename F>
__device__ __forceinline__ void read_window(const RunView& v, uint32_t p, bool sentinel, F&& word, OccT<KW>* oc) {
  static_assert(KW <= 2, "four-word k-mers are read apart");
  constexpr int W = 2 * KW;
  const int k = v.k;
  uint32_t w[W + 1], x[W + 1];
#pragma unroll
  for (int j = 0; j <= W; ++j) w[j] = word(j);
#pragma unroll
  for (int j = 0; j <= W; ++j) x[j] = __funnelshift_l(j < W ? w[j + 1] : 0u, w[j], 2u * p);
  uint32_t pred = 0, succ = 0;
  if (sentinel) {  // the window starts at the k-mer: move it to where the others have it
#pragma unroll
    for (int j = W; j >= 0; --j) x[j] = __funnelshift_r(x[j], j ? x[j - 1] : 0u, 2);
  } else {
    pred = x[0] >> 30;
    const int sw = (k + 1) >> 4;  // base k + 1 of the window
    uint32_t y = x[W];
#pragma unroll
    for (int j = 0; j < W; ++j)
      if (j == sw) y = x[j];
    succ = (y >> (30 - 2 * ((k + 1) & 15))) & 3u;
  }
  uint64_t top[KW];  // the 32 KW bases after the window's first
#pragma unroll
  for (int j = 0; j < KW; ++j)
    top[j] = ((uint64_t)__funnelshift_l(x[2 * j + 1], x[2 * j], 2) << 32) | __funnelshift_l(x[2 * j + 2], x[2 * j + 1], 2);
  Key f;
  if constexpr (KW == 1) {
    f.hi = 0;
    f.lo = top[0] >> (64 - 2 * k);
  } else {
    const int sh = 128 - 2 * k;  // 2 .. 64
    f.hi = sh == 64 ? 0ull : top[0] >> sh;
    f.lo = sh == 64 ? top[0] : (top[1] >> sh) | (top[0] << (64 - sh));
  }
  const Key r = v.both ? revcomp<KW>(f, k) : f;
  make_occ<KW>(v, f, r, pred, succ, sentinel, oc);
}

template <int KW>
__device__ __forceinline__ void read_listed(const RunView& v, uint64_t g, bool sentinel, OccT<KW>* oc) {
  if constexpr (KW == 4) {
    const int k = v.k;
    const Key4 f = load_kmer<4>(v.packed, g, k);
    const Key4 r = v.both ? revcomp<4>(f, k) : f;
    const uint32_t pred = sentinel ? 0u : base_at(v.packed, g - 1);
    const uint32_t succ = sentinel ? 0u : base_at(v.packed, g + k);
    make_occ<4>(v, f, r, pred, succ, sentinel, oc);
  } else {
    const uint64_t a = sentinel ? g : g - 1;
    const uint32_t* p = v.packed + (a >> 4);
    read_window<KW>(v, (uint32_t)a & 15u, sentinel, [&](int j) { return __ldg(p + j); }, oc);
  }
}

// A k-mer as 2 KW 32-bit words, w[0] the most significant.
template <int KW>
struct Words {
  uint32_t w[2 * KW];
};

template <int KW>
__device__ __forceinline__ Words<KW> to_words(const KeyT<KW>& x) {
  Words<KW> y;
  if constexpr (KW == 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      y.w[2 * i] = (uint32_t)(x.w[i] >> 32);
      y.w[2 * i + 1] = (uint32_t)x.w[i];
    }
  } else {
    if constexpr (KW == 2) {
      y.w[0] = (uint32_t)(x.hi >> 32);
      y.w[1] = (uint32_t)x.hi;
    }
    y.w[2 * KW - 2] = (uint32_t)(x.lo >> 32);
    y.w[2 * KW - 1] = (uint32_t)x.lo;
  }
  return y;
}

template <int KW>
__device__ __forceinline__ KeyT<KW> from_words(const Words<KW>& y) {
  KeyT<KW> x;
  if constexpr (KW == 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x.w[i] = ((uint64_t)y.w[2 * i] << 32) | y.w[2 * i + 1];
  } else {
    x.hi = KW == 2 ? ((uint64_t)y.w[0] << 32) | y.w[1] : 0ull;
    x.lo = ((uint64_t)y.w[2 * KW - 2] << 32) | y.w[2 * KW - 1];
  }
  return x;
}

// Visit the R consecutive positions p0 .. p0 + R - 1, all of them inside one
// string and none its first or last k-mer. Instead of rolling two k-mers from
// position to position (a serial chain of 64-bit shifts, masks and inserts of
// single bases), the forward k-mer and its reverse complement are each one
// word longer than the k-mer -- the R successor bases appended at their ends --
// and every position cuts its two k-mers out by funnel shifts of a
// compile-time distance: one per 32-bit word, and independent of each other.
// The integer instructions are what bounds every kernel that walks: 35 M
// positions at k = 25, insert 231 -> 202 us (k = 100: 505 -> 385); the class map
// of 6 G positions 33.3 -> 22.3 ms.
template <int KW, int R, typename F>
__device__ __forceinline__ void walk_inside(const RunView& v, uint64_t p0, F&& fn) {
  constexpr int W = 2 * KW;
  const int k = v.k;
  const KeyT<KW> f0 = load_kmer<KW>(v.packed, p0, k);
  const uint32_t next = bases16(v.packed, p0 + (uint64_t)k);
  const uint32_t before = bases16(v.packed, p0 - 1);  // predecessors of the positions
  const Words<KW> f = to_words<KW>(f0);
  const Words<KW> r = to_words<KW>(revcomp<KW>(f0, k));
  // mask of 2 k bits; only the upper half can hold bits beyond them (the whole of a k <= 31 word)
  uint32_t mask[W], rx[W + 1];
#pragma unroll
  for (int j = 0; j < W; ++j) {
    const int bits = 2 * k - 32 * (W - 1 - j);  // of word j
    mask[j] = bits >= 32 ? 0xFFFFFFFFu : (bits <= 0 ? 0u : (1u << bits) - 1u);
  }
  // the complements of the successor bases, the first lowest, above the 2 k bits of r
  const uint32_t t = (uint32_t)(rev_pairs(~(uint64_t)next) >> 32);
  rx[0] = 0;
#pragma unroll
  for (int j = 0; j < W; ++j) rx[j + 1] = r.w[j];
  const int at = (2 * k) >> 5, sh = (2 * k) & 31;  // rx[W - at] is the word that holds bit 2 k
#pragma unroll
  for (int j = 0; j <= W; ++j) {
    if (j == W - at) rx[j] |= t << sh;
    if (j == W - at - 1) rx[j] |= __funnelshift_l(t, 0u, sh);
  }
  const bool may_be_palindrome = !(k & 1);
#pragma unroll
  for (int i = 0; i < R; ++i) {
    Words<KW> fi, ri;
#pragma unroll
    for (int j = 0; j < W; ++j) {
      fi.w[j] = __funnelshift_l(j + 1 < W ? f.w[j + 1] : next, f.w[j], 2 * i);
      ri.w[j] = __funnelshift_r(rx[j + 1], rx[j], 2 * i);
      if (KW == 1 || j < W / 2) {
        fi.w[j] &= mask[j];
        ri.w[j] &= mask[j];
      }
    }
    const KeyT<KW> kf = from_words<KW>(fi), kr = from_words<KW>(ri);
    const bool use_r = v.both && key_less(kr, kf);
    OccT<KW> oc;
    oc.key = use_r ? kr : kf;
    oc.H = key_hash<KW>(oc.key);
    oc.sentinel = false;
    oc.rc = use_r;
    // the item from the bases before and after, or their complements after and before
    const uint32_t x = (use_r ? ~next : before) >> (30 - 2 * i), y = (use_r ? ~before : next) >> (30 - 2 * i);
    oc.j1 = oc.j2 = ((x & 3u) << 2) | (y & 3u);
    if (may_be_palindrome && v.both && !use_r && !key_less(kf, kr))
      oc.j2 = item_reverse((before >> (30 - 2 * i)) & 3u, (next >> (30 - 2 * i)) & 3u);
    oc.tbits = item_tbits(oc.j1) | item_tbits(oc.j2);
    fn(i, p0 + i, true, oc);
  }
}

// Visit the R consecutive positions p0 .. p0 + R - 1 (p0 < m), a string (or
// piece) boundary or the input's end among them: rolling the k-mer from each
// position to the next within a string and reading it from scratch after a
// string boundary. b: the bounds at p0.
template <int KW, int R, bool ROLLED, typename F>
__device__ __forceinline__ void walk_edges(const RunView& v, uint64_t p0, Bounds b, F&& fn) {
  static_assert(R >= 1 && R <= 16, "successor bases come from one 32-bit word");
  const int k = v.k;
  int32_t s_rel = rel(b.start, p0), e_rel = rel(b.end, p0);  // string bounds relative to p0
  const int32_t m_rel = rel(v.m, p0);
  // bases p0 + k .. p0 + k + R - 1: the successor of each position, which is
  // also the base that enters the k-mer when it slides to the next position
  const uint32_t next = bases16(v.packed, p0 + (uint64_t)k);
  KeyT<KW> f{}, r{};
  bool fresh = true;
  auto visit = [&](int i) {
    const uint64_t p = p0 + i;
    OccT<KW> oc;
    bool valid = false;
    if (i < m_rel) {
      if (i >= e_rel) {  // p starts a later string (or piece)
        b = kmer_bounds(v, p);
        s_rel = rel(b.start, p0);
        e_rel = rel(b.end, p0);
        fresh = true;
      }
      if (i + k <= e_rel) {
        valid = true;
        uint32_t pred;
        if (fresh) {
          f = load_kmer<KW>(v.packed, p, k);
          if (v.both) r = revcomp<KW>(f, k);
          pred = i > s_rel ? base_at(v.packed, p - 1) : 0u;
          fresh = false;
        } else {
          pred = first_base<KW>(f, k);  // the first base of the previous k-mer
          roll<KW>(f, r, i > 0 ? (next >> (32 - 2 * i)) & 3u : 0u, k);
        }
        const uint32_t succ = (next >> (30 - 2 * i)) & 3u;
        const bool sentinel = i == s_rel || i + k == e_rel;
        make_occ<KW>(v, f, v.both ? r : f, pred, succ, sentinel, &oc);
      } else {
        fresh = true;
      }
    }
    fn(i, p, valid, oc);
  };
  if constexpr (ROLLED) {
#pragma unroll 1
    for (int i = 0; i < R; ++i) visit(i);
  } else {
#pragma unroll
    for (int i = 0; i < R; ++i) visit(i);
  }
}


// Visit the R consecutive positions p0 .. p0 + R - 1 (p0 < m): fn(i, p, valid,
// occ) runs for every i, with i a compile-time constant once unrolled.
// ROLLED: the rare walks over a boundary stay a loop, with i a run-time value
// (an fn that does not index registers by it): unrolled beside the other walk
// they made the inserts of four-word k-mers miss the instruction cache.
template <int KW, int R, bool ROLLED = false, typename F>
__device__ __forceinline__ void walk(const RunView& v, uint64_t p0, F&& fn) {
  const Bounds b = kmer_bounds(v, p0);
  if (b.start < p0 && p0 + (uint64_t)(R - 1 + v.k) < b.end) walk_inside<KW, R>(v, p0, fn);
  else walk_edges<KW, R, ROLLED>(v, p0, b, fn);
}

__device__ __forceinline__ bool in_round(const RunView& v, uint64_t H, int round) {
  const uint32_t bin = (uint32_t)H & v.qmask;
  return bin >= __ldg(v.cuts + round) && bin < __ldg(v.cuts + round + 1);
}

// ---------------------------------------------------------------------------
// First-pass filter: b bits = b/256 blocks of four 64-bit words. A k-mer owns
// one 64-bit word: block from the top bits of H, word o from the top two bits
// of G. Each of its h bits u has a 5-bit base cut from G, in the low (u even)
// or high (u odd) half; item j sets bit (base_u + j) & 31 of that half. All 17
// items of a k-mer live in one word: an insert is one 64-bit atomic OR and a
// probe is one 8-byte load that answers all of its items at once.
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned long long* filter_word(const RunView& v, uint64_t H, uint64_t G) {
  // b <= 2^40 bits: the block index has at most 32 bits
  const uint32_t block = v.lg_blocks ? (uint32_t)(H >> (64 - v.lg_blocks)) : 0u;
  return v.filter + ((uint64_t)block * 4u + (uint32_t)(G >> 62));
}

__device__ __forceinline__ uint32_t bit_base(uint64_t G, int u) {
  const int sh = 57 - 5 * u;  // u is a compile-time constant once unrolled
  if (sh >= 32) return ((uint32_t)(G >> 32) >> (sh - 32)) & 31u;
  return (uint32_t)(G >> sh) & 31u;
}

// The bits of item 0 in each half of the word; item j is both halves
// rotated left by j (bit (base_u + j) mod 32).
struct ItemPattern {
  uint32_t lo, hi;
};

// HB > 0: that many bits per item, a compile-time constant; HB = 0: hb bits,
// a run-time value (the k > 63 kernels, to keep their instances few).
template <int HB>
__device__ __forceinline__ ItemPattern item_pattern(uint64_t G, int hb) {
  ItemPattern p{0u, 0u};
#pragma unroll
  for (int u = 0; u < (HB ? HB : 8); ++u) {
    if (!HB && u >= hb) break;
    const uint32_t b = 1u << bit_base(G, u);
    if (u & 1) p.hi |= b; else p.lo |= b;
  }
  return p;
}

__device__ __forceinline__ uint64_t item_bits(const ItemPattern& p, uint32_t j) {
  return ((uint64_t)__funnelshift_l(p.hi, p.hi, j) << 32) | __funnelshift_l(p.lo, p.lo, j);
}

template <int HB>
__device__ __forceinline__ uint64_t item_bits(uint64_t G, uint32_t j, int hb) {
  return item_bits(item_pattern<HB>(G, hb), j);
}

// Bit j of the result: item j is present (all of its bits are set).
template <int HB>
__device__ __forceinline__ uint32_t present_items(uint64_t G, uint64_t w, int hb) {
  const uint32_t lo = (uint32_t)w, hi = (uint32_t)(w >> 32);
  uint32_t pres = 0x1FFFFu;
#pragma unroll
  for (int u = 0; u < (HB ? HB : 8); ++u) {
    if (!HB && u >= hb) break;
    const uint32_t x = (u & 1) ? hi : lo;
    pres &= __funnelshift_r(x, x, bit_base(G, u));
  }
  return pres & 0x1FFFFu;
}

// Index of a k-mer's filter word (the word filter_word points to).
__device__ __forceinline__ uint64_t filter_index(const RunView& v, uint64_t H, uint64_t G) {
  const uint32_t block = v.lg_blocks ? (uint32_t)(H >> (64 - v.lg_blocks)) : 0u;
  return (uint64_t)block * 4u + (uint32_t)(G >> 62);
}

// ---------------------------------------------------------------------------
// Region-bucketed first-pass inserts. A filter far larger than L2 takes its
// random ORs at DRAM's random-access rate, about a tenth of the rate L2 takes
// them at. So for such a filter the insert loop turns every OR into an 8-byte
// record in the bucket of its filter region (32 MiB, which L2 holds), and the
// apply kernel then performs the ORs bucket by bucket, while the region stays
// in L2. A record: bits 0-21 the word within its region, 22-51 the bits 32-61
// of G (the bit bases of up to 6 bits per item), 52-56 and 57-61 the items (two
// for a palindrome's orientations). A full bucket takes the OR directly.
// ---------------------------------------------------------------------------

constexpr uint32_t kApplyPiece = 4096;  // records per apply work item
constexpr uint32_t kFillStride = 32;    // bucket counters 128 bytes apart (one L2 line each)

// A region's records go to one of its sub-buckets (chosen by the warp, so
// that every region has at least 256 counters between them): the bucket
// index is region * n_sub + sub, region-major, so that the apply's order
// still takes one region after the other.
__device__ __forceinline__ void stage_or(const RunView& v, uint64_t word, uint64_t G, uint32_t j1, uint32_t j2,
                                         uint64_t mask) {
  const uint32_t warp = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  const uint32_t b = (uint32_t)(word >> v.lg_region_words) * v.n_sub + (warp & (v.n_sub - 1u));
  const unsigned grp = __match_any_sync(__activemask(), b);
  const int lane = threadIdx.x & 31, leader = __ffs(grp) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(v.bucket_fill + (uint64_t)b * kFillStride, (uint32_t)__popc(grp));
  base = __shfl_sync(grp, base, leader);
  const uint64_t slot = (uint64_t)base + __popc(grp & ((1u << lane) - 1u));
  if (slot < v.bucket_cap) {
    const uint64_t local = word & ((1ull << v.lg_region_words) - 1ull);
    v.bucket_recs[(uint64_t)b * v.bucket_cap + slot] =
        local | (((G >> 32) & 0x3FFFFFFFull) << 22) | ((uint64_t)j1 << 52) | ((uint64_t)j2 << 57);
  } else {
    atomicOr(v.filter + word, (unsigned long long)mask);
  }
}

// The ORs of the staged records, in work items of kApplyPiece records taken in
// bucket order from a ticket (so that the blocks in flight work on one or two
// regions at a time). The counter after the last bucket's is the ticket.
template <int HB>
__global__ void __launch_bounds__(kBlock) filter_apply_kernel(RunView v) {
  __shared__ uint32_t first_s[kMaxBuckets + 1];  // first work item of every bucket
  __shared__ uint32_t item_s;
  const uint32_t R = v.n_regions * v.n_sub;  // buckets
  if (threadIdx.x == 0) {
    uint32_t acc = 0;
    for (uint32_t b = 0; b < R; ++b) {
      first_s[b] = acc;
      const uint64_t n = min((uint64_t)__ldcg(v.bucket_fill + (uint64_t)b * kFillStride), v.bucket_cap);
      acc += (uint32_t)((n + kApplyPiece - 1) / kApplyPiece);
    }
    first_s[R] = acc;
  }
  __syncthreads();
  const uint32_t total = first_s[R];
  for (;;) {
    if (threadIdx.x == 0) item_s = atomicAdd(v.bucket_fill + (uint64_t)R * kFillStride, 1u);
    __syncthreads();
    const uint32_t item = item_s;
    __syncthreads();
    if (item >= total) break;
    uint32_t lo = 0, hi = R;  // the bucket b with first_s[b] <= item < first_s[b + 1]
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (first_s[mid] <= item) lo = mid; else hi = mid;
    }
    const uint32_t b = lo;
    const uint64_t n = min((uint64_t)__ldcg(v.bucket_fill + (uint64_t)b * kFillStride), v.bucket_cap);
    const uint64_t i0 = (uint64_t)(item - first_s[b]) * kApplyPiece;
    const uint64_t i1 = min(i0 + kApplyPiece, n);
    const uint64_t* recs = v.bucket_recs + (uint64_t)b * v.bucket_cap;
    const uint64_t region = (uint64_t)(b / v.n_sub) << v.lg_region_words;
    for (uint64_t i = i0 + threadIdx.x; i < i1; i += kBlock) {
      const uint64_t r = __ldcs(recs + i);
      const uint64_t G = ((r >> 22) & 0x3FFFFFFFull) << 32;  // the bits bit_base reads for u < 6
      const ItemPattern pat = item_pattern<HB>(G, v.hashes);
      const uint32_t j1 = (uint32_t)(r >> 52) & 31u, j2 = (uint32_t)(r >> 57) & 31u;
      uint64_t m = item_bits(pat, j1);
      if (j2 != j1) m |= item_bits(pat, j2);
      atomicOr(v.filter + (region | (r & ((1ull << 22) - 1ull))), (unsigned long long)m);
    }
  }
}

// ---------------------------------------------------------------------------
// Pass-2 table: open addressing with linear probing, keyed by the normalized
// k-mer; the value is the 9-bit pass-2 mask. Empty keys are all ones, which
// no k-mer of k <= 63 can be.
// ---------------------------------------------------------------------------

struct alignas(16) Slot1 {
  unsigned long long key;
  unsigned int mask;
  unsigned int pad;
};

struct alignas(32) Slot2 {
  unsigned long long w0, w1;  // key.lo, key.hi (one 128-bit word, w0 low)
  unsigned int mask;
  unsigned int pad;
  unsigned long long pad2;
};

constexpr unsigned long long kEmpty = ~0ull;
constexpr int kMaskBits = 9;

__device__ __forceinline__ void cas128(unsigned long long* addr, uint64_t cmp_lo, uint64_t cmp_hi,
                                       uint64_t new_lo, uint64_t new_hi, uint64_t* old_lo,
                                       uint64_t* old_hi) {
  uint64_t ol, oh;
  asm volatile(
      "{\n\t.reg .b128 c, n, d;\n\t"
      "mov.b128 c, {%2, %3};\n\t"
      "mov.b128 n, {%4, %5};\n\t"
      "atom.global.cas.b128 d, [%6], c, n;\n\t"
      "mov.b128 {%0, %1}, d;\n\t}"
      : "=l"(ol), "=l"(oh)
      : "l"(cmp_lo), "l"(cmp_hi), "l"(new_lo), "l"(new_hi), "l"(addr)
      : "memory");
  *old_lo = ol;
  *old_hi = oh;
}

constexpr uint64_t kNoSlot = ~0ull;

// Slots of a 32-byte sector (four 8-byte slots, two 16-byte ones): a probe
// starts at a k-mer's sector and reads a whole sector at a time, so that a
// k-mer mostly costs one round trip. Slot by slot from any start, the longest
// of a warp's 32 chains -- six to eight slots at a load of 0.4 -- cost one each,
// and the rest of the warp its instructions. Tables hold whole sectors.
// That is for tables of up to about twice L2: larger ones (kSectorSlots) are probed slot
// by slot, from a k-mer's very slot, as the two loads of a sector are two misses in
// flight for one there. Pass-2 inserts, by sectors and by slots: one-word slots at 195 MB
// 502 and 545 us, 229 MB 634 and 680, 269 MB 800 and 734, 390 MB 1932 and 1359, 714 MB 4.60
// and 3.20 ms; 16-byte slots at 243 MB 428 and 437 us, 347 MB 1080 and 817, 1.4 GB 7.07 and
// 5.12 ms.
template <int TS>
struct SectorOf {
  static constexpr int kSlots = TS == 0 || TS == 3 ? 4 : (TS == 2 ? 1 : 2);
  unsigned long long key[kSlots];   // the slot's word (TS 0, 3), key (1) or low key word (2)
  unsigned long long more[kSlots];  // its mask (1) or high key word (2)
  unsigned int mask;                // TS 2: its mask

  __device__ __forceinline__ void load(const void* table, uint64_t first) {  // first: a multiple of kSlots
    const ulonglong2* p = reinterpret_cast<const ulonglong2*>(static_cast<const char*>(table) + first * (32 / kSlots));
    const ulonglong2 a = __ldcg(p), b = __ldcg(p + 1);
    if constexpr (TS == 0 || TS == 3) {
      key[0] = a.x; key[1] = a.y; key[2] = b.x; key[3] = b.y;
    } else if constexpr (TS == 2) {
      key[0] = a.x; more[0] = a.y;
      mask = (unsigned int)b.x;
    } else {
      key[0] = a.x; more[0] = a.y;
      key[1] = b.x; more[1] = b.y;
    }
  }
};

template <int TS>
constexpr uint64_t kSectorSlots = (256ull << 20) / (TS == 1 ? 16 : 8);

// A table of cap slots is probed by sectors (else slot by slot; kinds 0 and 1 only).
template <int TS>
__device__ __forceinline__ bool by_sectors(uint64_t cap) {
  return (TS != 0 && TS != 1) || cap <= kSectorSlots<TS>;
}

// Start slot of a k-mer in a pass-2 table of cap slots of kind TS.
template <int TS>
__device__ __forceinline__ uint64_t table_start(uint64_t H, uint64_t cap) {
  const uint64_t i = slot_start<1>(H, cap);
  return by_sectors<TS>(cap) ? i & ~(uint64_t)(SectorOf<TS>::kSlots - 1) : i;
}

// Insert into the one-word slots T[0 .. cap), probing from slot i (table_start; by
// sectors a multiple of 4): the key's slot, or kNoSlot if `tries` slots were tried
// (all of them: the table is full). Bits already present are not written again. A
// word is key << 9 | mask bits; never all ones for a key < 2^54.
__device__ __forceinline__ uint64_t word_insert(unsigned long long* T, uint64_t cap, uint64_t i, uint64_t key,
                                                uint32_t bits, uint64_t tries) {
  if (!by_sectors<0>(cap)) {
    for (uint64_t seen = 0; seen < tries; ++seen, i = i + 1 == cap ? 0 : i + 1) {
      unsigned long long cur = __ldcg(T + i);
      if (cur == kEmpty) {
        cur = atomicCAS(T + i, kEmpty, (key << kMaskBits) | bits);
        if (cur == kEmpty) return i;
      }
      if ((cur >> kMaskBits) != key) continue;
      if ((cur & bits) != bits) atomicOr(T + i, (unsigned long long)bits);
      return i;
    }
    return kNoSlot;
  }
  for (uint64_t seen = 0; seen < tries; seen += 4) {
    SectorOf<0> q;
    q.load(T, i);
    for (;;) {  // again only after another k-mer took the empty slot
      unsigned long long cur = 0;
      int at = 4;  // the first slot that is empty or the key's
#pragma unroll
      for (int k = 3; k >= 0; --k)
        if (q.key[k] == kEmpty || (q.key[k] >> kMaskBits) == key) {
          cur = q.key[k];
          at = k;
        }
      if (at == 4) break;
      unsigned long long* s = T + i + at;
      if (cur == kEmpty) {
        cur = atomicCAS(s, kEmpty, (key << kMaskBits) | bits);
        if (cur == kEmpty) return i + at;
      }
      if ((cur >> kMaskBits) == key) {
        if ((cur & bits) != bits) atomicOr(s, (unsigned long long)bits);
        return i + at;
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k == at) q.key[k] = cur;
    }
    i = i + 4 == cap ? 0 : i + 4;
  }
  return kNoSlot;
}

// Mask of key in the one-word slots T[0 .. cap), or -1 if absent.
__device__ __forceinline__ int word_find(const unsigned long long* T, uint64_t cap, uint64_t i, uint64_t key) {
  if (!by_sectors<0>(cap)) {
    for (uint64_t seen = 0; seen < cap; ++seen, i = i + 1 == cap ? 0 : i + 1) {
      const unsigned long long cur = __ldcg(T + i);
      if (cur == kEmpty) return -1;
      if ((cur >> kMaskBits) == key) return (int)(cur & ((1u << kMaskBits) - 1u));
    }
    return -1;
  }
  for (uint64_t seen = 0; seen < cap; seen += 4) {
    SectorOf<0> q;
    q.load(T, i);
    unsigned long long cur = 0;
    bool hit = false;
#pragma unroll
    for (int k = 3; k >= 0; --k)
      if (q.key[k] == kEmpty || (q.key[k] >> kMaskBits) == key) {
        cur = q.key[k];
        hit = true;
      }
    if (hit) return cur == kEmpty ? -1 : (int)(cur & ((1u << kMaskBits) - 1u));
    i = i + 4 == cap ? 0 : i + 4;
  }
  return -1;
}

// Insert (key, bits) into a table of cap TS-kind slots (table_slot_kind),
// probing from start (table_start); the key's slot, or kNoSlot if `tries` slots were tried (all of them: the table is full). Bits already present
// are not written again.
template <int TS>
__device__ __forceinline__ uint64_t table_insert(const RunView& v, uint64_t cap, const Key& key,
                                             uint64_t start, uint32_t bits, uint64_t tries) {
  if constexpr (TS == 0) {
    return word_insert(static_cast<unsigned long long*>(v.table), cap, start, key.lo, bits, tries);
  } else {
    constexpr uint64_t N = SectorOf<TS>::kSlots;
    uint64_t base = start;
    if constexpr (TS == 1) {
      if (!by_sectors<1>(cap)) {
        for (uint64_t seen = 0; seen < tries; ++seen, base = base + 1 == cap ? 0 : base + 1) {
          Slot1* s = static_cast<Slot1*>(v.table) + base;
          const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2*>(s));
          unsigned long long cur = w.x;
          uint32_t have = (uint32_t)w.y;
          if (cur == kEmpty) {
            cur = atomicCAS(&s->key, kEmpty, (unsigned long long)key.lo);
            if (cur == kEmpty) cur = key.lo;
            have = 0;
          }
          if (cur != key.lo) continue;
          if ((have & bits) != bits) atomicOr(&s->mask, bits);
          return base;
        }
        return kNoSlot;
      }
    }
    for (uint64_t seen = 0; seen < tries; seen += N) {
      SectorOf<TS> q;
      if constexpr (TS == 1) q.load(v.table, base);  // TS 2: the CAS itself is the first look
#pragma unroll
      for (uint64_t k = 0; k < N; ++k) {
        if constexpr (TS == 1) {
          Slot1* s = static_cast<Slot1*>(v.table) + base + k;
          unsigned long long cur = q.key[k];
          uint32_t have = (uint32_t)q.more[k];
          if (cur == kEmpty) {
            cur = atomicCAS(&s->key, kEmpty, (unsigned long long)key.lo);
            if (cur == kEmpty) cur = key.lo;
            have = 0;
          }
          if (cur != key.lo) continue;
          if ((have & bits) != bits) atomicOr(&s->mask, bits);
        } else {
          Slot2* s = static_cast<Slot2*>(v.table) + base;
          uint64_t ol, oh;
          cas128(&s->w0, kEmpty, kEmpty, key.lo, key.hi, &ol, &oh);
          if (!((ol == kEmpty && oh == kEmpty) || (ol == key.lo && oh == key.hi))) continue;
          if ((__ldcg(&s->mask) & bits) != bits) atomicOr(&s->mask, bits);
        }
        return base + k;
      }
      base = base + N == cap ? 0 : base + N;
    }
    return kNoSlot;
  }
}

// Mask of key, or -1 if absent.
template <int TS>
__device__ __forceinline__ int table_find(const RunView& v, uint64_t cap, const Key& key, uint64_t start) {
  if constexpr (TS == 0) {
    return word_find(static_cast<const unsigned long long*>(v.table), cap, start, key.lo);
  } else {
    constexpr uint64_t N = SectorOf<TS>::kSlots;
    uint64_t base = start;
    if constexpr (TS == 1) {
      if (!by_sectors<1>(cap)) {
        for (uint64_t seen = 0; seen < cap; ++seen, base = base + 1 == cap ? 0 : base + 1) {
          const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2*>(static_cast<const Slot1*>(v.table) + base));
          if (w.x == key.lo) return (int)(uint32_t)w.y;
          if (w.x == kEmpty) return -1;
        }
        return -1;
      }
    }
    for (uint64_t seen = 0; seen < cap; seen += N) {
      SectorOf<TS> q;
      q.load(v.table, base);
#pragma unroll
      for (uint64_t k = 0; k < N; ++k) {
        if constexpr (TS == 1) {
          if (q.key[k] == key.lo) return (int)(uint32_t)q.more[k];
          if (q.key[k] == kEmpty) return -1;
        } else {
          if (q.key[0] == key.lo && q.more[0] == key.hi) return (int)q.mask;
          if (q.key[0] == kEmpty && q.more[0] == kEmpty) return -1;
        }
      }
      base = base + N == cap ? 0 : base + N;
    }
    return -1;
  }
}

// Slots of k-mers of 64 to 127 bases (kind 3): instead of the key, a
// reference to one occurrence of it -- bits 0-47 its position + 1, bit 48
// whether the string reads the key's reverse complement there -- with the
// pass-2 mask (bits 49-57) and the top six bits of H as a tag (58-63). 0 is
// empty. Keys are compared by reading the referenced occurrence back from the
// packed input, so one 64-bit CAS claims a slot for a key of any length, its
// first bits included. (With the mask in a second word beside a 15-bit tag, a
// new k-mer took a CAS and an OR, and the table twice the memory: 672 us for
// 11.6 M candidates, 10 M of them new, in a 328 MB table.)
constexpr uint64_t kRefPos = (1ull << 48) - 1;
constexpr int kRefMask = 49, kRefTag = 58;

__device__ __forceinline__ bool ref_holds(const RunView& v, uint64_t ref, const Key4& key) {
  Key4 x = load_kmer<4>(v.packed, (ref & kRefPos) - 1, v.k);
  if ((ref >> 48) & 1u) x = revcomp<4>(x, v.k);
  return key_eq(x, key);
}

__device__ __forceinline__ uint64_t table_insert_ref(const RunView& v, uint64_t cap, const Key4& key,
                                                     uint64_t H, uint64_t start, uint32_t bits, uint64_t g,
                                                     bool rc) {
  const uint64_t tag = H >> kRefTag, add = (uint64_t)bits << kRefMask;
  const unsigned long long mine = (tag << kRefTag) | add | ((uint64_t)rc << 48) | (g + 1);
  uint64_t base = start;
  for (uint64_t seen = 0; seen < cap; seen += 4) {
    SectorOf<3> q;
    q.load(v.table, base);
#pragma unroll
    for (uint64_t k = 0; k < 4; ++k) {
      unsigned long long* s = static_cast<unsigned long long*>(v.table) + base + k;
      unsigned long long cur = q.key[k];
      if (cur == 0) {
        cur = atomicCAS(s, 0ull, mine);
        if (cur == 0) return base + k;
      }
      if ((cur >> kRefTag) != tag || !ref_holds(v, cur, key)) continue;
      if ((cur & add) != add) atomicOr(s, (unsigned long long)add);
      return base + k;
    }
    base = base + 4 == cap ? 0 : base + 4;
  }
  return kNoSlot;
}

__device__ __forceinline__ int ref_mask(unsigned long long slot) {
  return (int)(slot >> kRefMask) & ((1 << kMaskBits) - 1);
}

__device__ __forceinline__ int table_find_ref(const RunView& v, uint64_t cap, const Key4& key, uint64_t H) {
  const uint64_t tag = H >> kRefTag;
  uint64_t base = slot_start<4>(H, cap);
  for (uint64_t seen = 0; seen < cap; seen += 4) {
    SectorOf<3> q;
    q.load(v.table, base);
#pragma unroll
    for (uint64_t k = 0; k < 4; ++k) {
      if (q.key[k] == 0) return -1;
      if ((q.key[k] >> kRefTag) == tag && ref_holds(v, q.key[k], key)) return ref_mask(q.key[k]);
    }
    base = base + 4 == cap ? 0 : base + 4;
  }
  return -1;
}

// The table slot of an occurrence at g (inserted; after at most `tries` slots), or its
// mask (found).
template <int KW, int TS>
__device__ __forceinline__ uint64_t insert_occurrence(const RunView& v, uint64_t cap, const OccT<KW>& oc,
                                                      uint64_t g, uint64_t tries) {
  if constexpr (TS == 3) return table_insert_ref(v, cap, oc.key, oc.H, slot_start<4>(oc.H, cap), oc.tbits, g, oc.rc);
  else return table_insert<TS>(v, cap, oc.key, table_start<TS>(oc.H, cap), oc.tbits, tries);
}

template <int KW, int TS>
__device__ __forceinline__ uint64_t insert_occurrence(const RunView& v, uint64_t cap, const OccT<KW>& oc,
                                                      uint64_t g) {
  return insert_occurrence<KW, TS>(v, cap, oc, g, cap);
}

template <int KW, int TS>
__device__ __forceinline__ int find_occurrence(const RunView& v, uint64_t cap, const OccT<KW>& oc) {
  if constexpr (TS == 3) return table_find_ref(v, cap, oc.key, oc.H);
  else return table_find<TS>(v, cap, oc.key, table_start<TS>(oc.H, cap));
}

// Mask held by slot i (a slot that table_insert returned).
template <int TS>
__device__ __forceinline__ int table_mask(const RunView& v, uint64_t i) {
  if (TS == 0) return (int)(__ldcg(static_cast<const unsigned long long*>(v.table) + i) & ((1u << kMaskBits) - 1u));
  if (TS == 1) return (int)__ldcg(&(static_cast<const Slot1*>(v.table) + i)->mask);
  if (TS == 3) return ref_mask(__ldcg(static_cast<const unsigned long long*>(v.table) + i));
  return (int)__ldcg(&(static_cast<const Slot2*>(v.table) + i)->mask);
}

__device__ __forceinline__ bool is_junction_mask(int mk) {
  return ((mk >> 8) & 1) || __popc(mk & 15) > 1 || __popc((mk >> 4) & 15) > 1;
}

// ---------------------------------------------------------------------------
// Reductions
// ---------------------------------------------------------------------------

template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  return x;
}

// Exclusive scan of x over the block (blockDim.x == kBlock); *total gets the sum.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* total) {
  __shared__ uint32_t warp_tot[kBlock / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_tot[wid] = inc;
  __syncthreads();
  uint32_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kBlock / 32; ++w) {
    const uint32_t t = warp_tot[w];
    before += (w < wid) ? t : 0u;
    all += t;
  }
  __syncthreads();
  *total = all;
  return before + inc - x;
}

// Sum a counter over the block's threads into *dst (one atomic per block).
__device__ __forceinline__ void block_add(unsigned long long x, unsigned long long* dst) {
  __shared__ unsigned long long part[kBlock / 32];
  x = warp_sum(x);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < kBlock / 32; ++w) t += part[w];
    if (t) atomicAdd(dst, t);
  }
  __syncthreads();
}

// Linear counting (Whang, Vander-Zanden & Taylor 1990) of the distinct
// candidates, on the 2^-lc_sample_log2 of the k-mers that a few bits of their
// hash choose: sets the bit of a candidate whose k-mer hashes to h (table_setup
// counts the bits). Every k-mer counted (no sample) cost one random atomic per
// candidate; an atomic that returns whether the bit was new, to save the count,
// made the probe wait (181 -> 193 us).
__device__ __forceinline__ void lc_mark(const RunView& v, uint64_t h) {
  if ((uint32_t)(h >> 24) & ((1u << v.lc_sample_log2) - 1u)) return;
  const uint64_t x = h >> (64 - v.lc_log2);
  atomicOr(v.lc_bits + (x >> 5), 1u << (x & 31));
}

constexpr uint64_t kLcMul = 0xff51afd7ed558ccdull;

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

// Four ASCII bytes -> four 2-bit codes in the result's top byte (first byte in
// bits 31-30); *diff gets nonzero bytes exactly where a byte is not one of
// ACGTacgt. Bits 2-1 of a letter tell a, c, t, g = 0x61, 0x63, 0x74, 0x67 apart
// (0, 1, 2, 3); a byte permute turns them into the letter they stand for, which
// the byte must be, and one multiply gathers the four codes (no two of its
// partial products share a bit). The pack is bound by its instructions: with four byte
// compares and four shifts per word it ran at 54% issue and a third of the
// memory bandwidth.
__device__ __forceinline__ uint32_t pack4(uint32_t x, uint32_t* diff) {
  const uint32_t low = x | 0x20202020u;
  const uint32_t t = (low >> 1) & 0x03030303u;
  const uint32_t sel = __byte_perm(t | (t >> 4), 0u, 0x4420);  // the four t as nibbles
  *diff = low ^ __byte_perm(0x67746361u, 0u, sel);             // g t c a
  const uint32_t c = t ^ ((t >> 1) & 0x01010101u);             // a c t g = 0 1 2 3 -> 0 1 3 2
  return c * 0x40100401u;
}

// 0xFF in every byte that is an N (either case).
__device__ __forceinline__ uint32_t is_n_bytes(uint32_t x) { return __vcmpeq4(x | 0x20202020u, 0x6e6e6e6eu); }

// Bit j of the result: the top bit of byte j of e (for a __vcmpeq4 mask:
// byte j matched).
__device__ __forceinline__ uint32_t byte_bits(uint32_t e) {
  // the top bit of every byte to bits 0-3: the multiply moves bits 7, 15, 23
  // and 31 to bits 28-31, every other partial product lands elsewhere
  return ((e & 0x80808080u) * 0x00204081u) >> 28;
}

// Sixteen ASCII bytes at g (or fewer at the end of the input) -> one word;
// *bad_at gets the index of the first invalid byte. With N splitting (v.nmask)
// an N is valid and *nbits gets bit i for an N at g + i.
__device__ __forceinline__ uint32_t pack16(const RunView& v, uint64_t g, uint4 q, bool full,
                                           uint64_t* bad_at, uint32_t* nbits) {
  uint32_t out = 0, nb = 0;
  const bool split = v.nmask != nullptr;
  if (full) {
    const uint32_t part[4] = {q.x, q.y, q.z, q.w};
    uint32_t code[4], diff[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) code[c] = pack4(part[c], &diff[c]);
    out = __byte_perm(__byte_perm(code[3], code[2], 0x0073), __byte_perm(code[1], code[0], 0x0073), 0x5410);
    if (diff[0] | diff[1] | diff[2] | diff[3]) {  // a byte that is no base: rare
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t bad = diff[c];
        if (split) {
          const uint32_t is_n = is_n_bytes(part[c]);
          bad &= ~is_n;
          nb |= byte_bits(is_n) << (4 * c);
        }
        if (bad && *bad_at == ~0ull) *bad_at = g + 4 * c + (__ffs(bad) - 1) / 8;
      }
    }
  } else if (g < v.m) {
    for (int i = 0; i < 16 && g + i < v.m; ++i) {
      const uint32_t c = v.bases[g + i];
      uint32_t diff;
      const uint32_t code = pack4(c | 0x61616100u, &diff) >> 30;  // pad bytes are 'a'
      if (split && (is_n_bytes(c) & 0xFFu)) {
        diff = 0;
        nb |= 1u << i;
      }
      if ((diff & 0xFFu) && *bad_at == ~0ull) *bad_at = g + i;
      out |= code << (30 - 2 * i);
    }
  }
  *nbits = nb;
  return out;
}

// ASCII -> 2-bit words: 64 bytes (four 128-bit loads in flight) per thread,
// for the packed words [w_begin, w_end) (w_begin a multiple of 4; the input
// bytes of those words are read at v.bases + 16 * w, so that a chunk of the
// input staged elsewhere can be packed by passing v.bases offset back by the
// chunk's start). With `first`, block 0 also records where this run keeps its
// bitmaps (for inspection), and the grid clears the filter, the
// linear-counting bitmap, C_final and the emit's tile status for the first
// round.
__global__ void __launch_bounds__(kBlock) pack_kernel(RunView v, uint64_t w_begin, uint64_t w_end, int first) {
  if (first && blockIdx.x == 0 && threadIdx.x == 0) {
    DevHeader* h = v.hdr;
    h->ctemp = v.ctemp;
    h->cfinal = v.cfinal;
    h->bins = v.bins;
    h->cuts = v.cuts;
    h->bitmap_words = v.bitmap_words;
    h->q = (unsigned long long)v.qmask + 1ull;
    h->rounds = (unsigned long long)v.rounds;
    h->packed = v.packed;
    h->m = v.m;
    h->k = v.k;
    h->both = v.both;
    h->nmask = v.nmask;
    h->runs = v.runs;
    h->run_rank = v.run_rank;
    h->run_cap = v.run_cap;
    h->offsets = v.offsets;
    h->n_seqs = v.n_seqs;
    h->hashes = v.hashes;
    h->lg_blocks = v.lg_blocks;
    h->partial = v.partial;
    h->packed_words = v.packed_words;
  }
  const bool vec = (reinterpret_cast<uintptr_t>(v.bases) & 15) == 0;
  const uint64_t stride = (uint64_t)gridDim.x * kBlock * 4;
  uint64_t bad_at = ~0ull;
  for (uint64_t w0 = w_begin + ((uint64_t)blockIdx.x * kBlock + threadIdx.x) * 4; w0 < w_end; w0 += stride) {
    uint4 q[4];
    bool full[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint64_t g = (w0 + j) * 16;
      full[j] = vec && g + 16 <= v.m;
      if (full[j]) q[j] = __ldcs(reinterpret_cast<const uint4*>(v.bases + g));
    }
    uint32_t out[4], nb[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) out[j] = pack16(v, (w0 + j) * 16, q[j], full[j], &bad_at, &nb[j]);
    if (v.nmask) {  // two packed words per N-mask word (w0 is a multiple of 4)
      v.nmask[w0 / 2] = nb[0] | (nb[1] << 16);
      v.nmask[w0 / 2 + 1] = nb[2] | (nb[3] << 16);
    }
    if (w0 + 4 <= w_end) {
      *reinterpret_cast<uint4*>(v.packed + w0) = make_uint4(out[0], out[1], out[2], out[3]);
    } else {
      for (int j = 0; j < 4 && w0 + j < w_end; ++j) v.packed[w0 + j] = out[j];
    }
  }
  if (bad_at != ~0ull) atomicMax(&v.hdr->bad_inv, ~(unsigned long long)bad_at);
  if (!first) return;
  // clear what the first round and the emit need to start at zero
  const uint64_t tid = (uint64_t)blockIdx.x * kBlock + threadIdx.x, nthreads = (uint64_t)gridDim.x * kBlock;
  auto zero = [&](void* p, uint64_t bytes) {  // 16-byte multiples at 16-byte aligned addresses
    uint4* q = static_cast<uint4*>(p);
    for (uint64_t i = tid; i < bytes / 16; i += nthreads) q[i] = make_uint4(0u, 0u, 0u, 0u);
  };
  zero(v.filter, v.filter_words64 * 8);
  zero(v.lc_bits, (1ull << v.lc_log2) / 8);
  zero(v.cfinal, (v.bitmap_words + 3) / 4 * 16);
  zero(v.tile_prefix, (v.n_tiles + 1) / 2 * 16);
}

// Digest of the input (checkpoints record it and check it on resume): the
// packed words, the string offsets and the N mask, each term tagged with its
// kind and index.
__global__ void __launch_bounds__(kBlock) digest_kernel(DevHeader* hdr, const uint32_t* packed, uint64_t words,
                                                        const uint64_t* offsets, uint64_t n_off,
                                                        const uint32_t* nmask, uint64_t nmask_words) {
  const uint64_t stride = (uint64_t)gridDim.x * kBlock;
  const uint64_t tid = (uint64_t)blockIdx.x * kBlock + threadIdx.x;
  unsigned long long d = 0;
  for (uint64_t w = tid; w < words; w += stride) d += mix64((w << 32) ^ packed[w]);
  for (uint64_t t = tid; t < n_off; t += stride) d += mix64(mix64(t ^ 0x6f66667365747321ull) ^ offsets[t]);
  if (nmask)
    for (uint64_t w = tid; w < nmask_words; w += stride) d += mix64(mix64(w ^ 0x6e6d61736b212121ull) ^ nmask[w]);
  block_add(d, &hdr->input_digest);
}

// ---------------------------------------------------------------------------
// N splitting: the sorted boundaries of the N-free pieces and of the N runs.
// Bit g of the boundary bitmap is set iff g starts a string or base g is N
// and base g - 1 is not, or the other way round, inside one string. The set
// bits, in order, are runs[0 .. n_runs); runs[n_runs] = m.
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(kBlock) runs_mark_kernel(RunView v) {
  const uint64_t stride = (uint64_t)gridDim.x * kBlock;
  for (uint64_t w = (uint64_t)blockIdx.x * kBlock + threadIdx.x; w < v.bitmap_words; w += stride) {
    const uint32_t cur = v.nmask[w], prev = w ? v.nmask[w - 1] : 0u;
    uint32_t b = cur ^ ((cur << 1) | (prev >> 31));
    if (w == v.bitmap_words - 1 && (v.m & 31)) b &= (1u << (v.m & 31)) - 1u;
    v.bound_bits[w] = b;
  }
}

__global__ void __launch_bounds__(kBlock) runs_starts_kernel(RunView v) {
  const uint64_t stride = (uint64_t)gridDim.x * kBlock;
  for (uint64_t t = (uint64_t)blockIdx.x * kBlock + threadIdx.x; t < v.n_seqs; t += stride) {
    const uint64_t g = __ldg(v.offsets + t);
    if (g < v.m) atomicOr(v.bound_bits + (g >> 5), 1u << (g & 31));
  }
}

// Set bits of every chunk of kRunChunkWords boundary words.
__global__ void __launch_bounds__(kBlock) runs_count_kernel(RunView v) {
  __shared__ unsigned long long part[kBlock / 32];
  for (uint64_t c = blockIdx.x; c < v.n_chunks; c += gridDim.x) {
    unsigned long long n = 0;
    for (uint64_t w = c * kRunChunkWords + threadIdx.x; w < (c + 1) * kRunChunkWords && w < v.bitmap_words;
         w += kBlock)
      n += __popc(v.bound_bits[w]);
    n = warp_sum(n);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = n;
    __syncthreads();
    if (threadIdx.x == 0) {
      unsigned long long tot = 0;
      for (int i = 0; i < kBlock / 32; ++i) tot += part[i];
      v.chunk_counts[c] = tot;
    }
    __syncthreads();
  }
}

// Exclusive scan of the chunk counts (in place, one block); records the
// number of boundaries (at most run_cap, else the overflow flag) and closes
// the list with m.
__global__ void __launch_bounds__(1024) runs_scan_kernel(RunView v) {
  __shared__ unsigned long long wsum[32];
  __shared__ unsigned long long carry_s;
  if (threadIdx.x == 0) carry_s = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (uint64_t base = 0; base < v.n_chunks; base += 1024) {
    const uint64_t c = base + threadIdx.x;
    const unsigned long long x = c < v.n_chunks ? v.chunk_counts[c] : 0ull;
    unsigned long long inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    unsigned long long before = 0, all = 0;
    for (int w = 0; w < 32; ++w) {
      before += (w < wid) ? wsum[w] : 0ull;
      all += wsum[w];
    }
    const unsigned long long c0 = carry_s;
    if (c < v.n_chunks) v.chunk_counts[c] = c0 + before + inc - x;
    __syncthreads();
    if (threadIdx.x == 0) carry_s = c0 + all;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const unsigned long long total = carry_s;
    const unsigned long long n = total < v.run_cap ? total : v.run_cap;
    if (total > v.run_cap) v.hdr->overflow = 1;
    v.hdr->n_runs = n;
    v.runs[n] = v.m;
  }
}

// Positions of the set boundary bits, in order (chunk by chunk).
__global__ void __launch_bounds__(kBlock) runs_write_kernel(RunView v) {
  constexpr int kPer = (int)(kRunChunkWords / kBlock);  // consecutive words per thread
  for (uint64_t c = blockIdx.x; c < v.n_chunks; c += gridDim.x) {
    const uint64_t w0 = c * kRunChunkWords + (uint64_t)threadIdx.x * kPer;
    uint32_t words[kPer];
    uint32_t n = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      words[j] = (w0 + j < v.bitmap_words) ? v.bound_bits[w0 + j] : 0u;
      n += __popc(words[j]);
    }
    uint32_t tot;
    uint64_t at = v.chunk_counts[c] + block_exclusive_scan(n, &tot);
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      uint32_t bits = words[j];
      while (bits) {
        const uint32_t b = __ffs(bits) - 1;
        bits &= bits - 1;
        if (at < v.run_cap) v.runs[at] = (w0 + j) * 32 + b;
        ++at;
      }
    }
  }
}

// Probe descriptor of a position (64 bits): bit 63 active (probe it), bit 62
// sentinel position, bits 32-61 the bit bases of its k-mer (G >> 32, bases
// of u < 6), bits 0-31 its filter word index. 1 marks a position whose
// k-mer is in another round's class, 0 a position without a k-mer.
constexpr uint64_t kDescActive = 1ull << 63, kDescSentinel = 1ull << 62;

__device__ __forceinline__ uint64_t make_desc(const RunView& v, uint64_t H, uint64_t G, bool sentinel) {
  const uint64_t block = v.lg_blocks ? (H >> (64 - v.lg_blocks)) : 0ull;
  const uint64_t index = block * 4 + (G >> 62);  // < 2^32 for b <= 2^37
  return kDescActive | (sentinel ? kDescSentinel : 0ull) | (((G >> 32) & 0x3FFFFFFFull) << 32) | index;
}

// Algorithm 1, insert loop, first pass: every active position records its
// item(s) in its k-mer's filter word with one atomic OR. With DESC it also
// leaves the position's probe descriptor for the probe loop: the block's
// descriptors are staged in shared memory (16-byte pairs, columns swizzled by
// the owning thread so that neither side conflicts) and written out in
// order, whole sectors at a time.
// R consecutive positions per thread: kInsertR, or kInsertSmallR for small inputs.
template <int KW, bool ROUNDS, int HB, bool DESC, bool BKT = false, int R = kInsertR>
__global__ void __launch_bounds__(kBlock) pass1_insert_kernel(RunView v, int round) {
  constexpr int kTile = kBlock * R;  // positions per block per pass
  constexpr int kPairs = R / 2;      // 16-byte descriptor pairs per thread
  __shared__ ulonglong2 stage[DESC ? kTile / 2 : 1];
  const uint64_t stride = (uint64_t)gridDim.x * kTile;
  const int t = threadIdx.x;
  for (uint64_t base = v.p_begin + (uint64_t)blockIdx.x * kTile; base < v.p_end; base += stride) {
    const uint64_t p0 = base + (uint64_t)t * R;
    if (p0 < v.m) {
      uint64_t prev = 0;
      walk<KW, R, true>(v, p0, [&](int i, uint64_t, bool valid, const auto& oc) {
        uint64_t d = 0;
        if (valid) {
          if (ROUNDS && !in_round(v, oc.H, round)) {
            d = 1;
          } else {
            const uint64_t G = second_hash(oc.H);
            const ItemPattern pat = item_pattern<HB>(G, v.hashes);
            uint64_t m = item_bits(pat, oc.j1);
            if (oc.j2 != oc.j1) m |= item_bits(pat, oc.j2);  // a palindrome's two orientations
            if (BKT) stage_or(v, filter_index(v, oc.H, G), G, oc.j1, oc.j2, m);
            else atomicOr(filter_word(v, oc.H, G), (unsigned long long)m);
            if (DESC) d = make_desc(v, oc.H, G, oc.sentinel);
          }
        }
        if (DESC) {
          if (i & 1) stage[t * kPairs + ((i >> 1) ^ (t % kPairs))] = make_ulonglong2(prev, d);
          else prev = d;
        }
      });
    }
    if (DESC) {
      __syncthreads();
      // pair j covers positions base + 2j, base + 2j + 1; its owner is thread
      // j / kPairs (which wrote 0 for any of them past m). The region holds
      // m + 16 descriptors, so a pair that starts before m fits.
      for (int j = t; j < kTile / 2; j += kBlock) {
        const uint64_t p = base + 2 * (uint64_t)j;
        if (p >= v.m) break;
        const int owner = j / kPairs, c = j % kPairs;
        __stcs(reinterpret_cast<ulonglong2*>(v.desc + p), stage[owner * kPairs + (c ^ (owner % kPairs))]);
      }
      __syncthreads();
    }
  }
}

// Algorithm 1, probe loop, first pass: a position stays a candidate iff it is
// a sentinel position, its k-mer's sentinel item is present, or at least two
// of its 16 (predecessor, successor) items are present -- i.e. the filter
// does not show exactly one in-edge and one out-edge. Writes C_temp, appends
// every candidate's position to the warp's own segment of the pass-2 list,
// and sets the candidate's bit in a linear-counting bitmap that estimates how
// many distinct k-mers survive.
template <int KW, bool ROUNDS, int HB>
__global__ void __launch_bounds__(kBlock, 3) pass1_probe_kernel(RunView v, int round) {
  const int lane = threadIdx.x & 31;
  constexpr int kR = kProbeR;
  const uint64_t stride = (uint64_t)gridDim.x * kBlock * kR;
  constexpr int kLanesPerWord = 32 / kR;
  uint32_t kept = 0, valid_n = 0;  // per thread: below 2^32
  const uint32_t warp_id = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  uint64_t* seg = v.cands + (uint64_t)warp_id * v.seg_cap;  // wide records
  uint32_t* seg32 = reinterpret_cast<uint32_t*>(v.cands) + (uint64_t)warp_id * v.seg_cap;
  uint64_t seg_used = 0;
  for (uint64_t wbase = v.p_begin + ((uint64_t)blockIdx.x * kBlock + (threadIdx.x & ~31u)) * kR;
       wbase < v.p_end; wbase += stride) {
    const uint64_t p0 = wbase + (uint64_t)lane * kR;
    uint64_t word[kR], G[kR];
    uint32_t probe_bits = 0, sent_bits = 0, valid_bits = 0;
    if (p0 < v.m) {
      walk<KW, kR>(v, p0, [&](int i, uint64_t, bool valid, const auto& oc) {
        if (!valid) return;
        valid_bits |= 1u << i;
        if (ROUNDS && !in_round(v, oc.H, round)) return;
        G[i] = second_hash(oc.H);
        if (oc.sentinel) {
          sent_bits |= 1u << i;
        } else {
          word[i] = __ldcg(filter_word(v, oc.H, G[i]));
          probe_bits |= 1u << i;
        }
      });
    }
    uint32_t keep_bits = sent_bits;
#pragma unroll
    for (int i = 0; i < kR; ++i) {
      if ((probe_bits >> i) & 1u) {
        const uint32_t pres = present_items<HB>(G[i], word[i], v.hashes);
        if ((pres >> 16) || __popc(pres & 0xFFFFu) >= 2) keep_bits |= 1u << i;
      }
      if (((keep_bits >> i) & 1u) && !v.partial) lc_mark(v, G[i] * kLcMul);
    }
    // C_temp: kLanesPerWord lanes make up one 32-bit word
    uint32_t wv = keep_bits << (kR * (lane % kLanesPerWord));
#pragma unroll
    for (int o = 1; o < kLanesPerWord; o <<= 1) wv |= __shfl_xor_sync(0xffffffffu, wv, o);
    if (lane % kLanesPerWord == 0) {
      const uint64_t w = (wbase >> 5) + lane / kLanesPerWord;
      if (w < v.bitmap_words) {
        v.ctemp[w] = wv;
        if (v.partial) v.cfinal[w] |= wv;  // rounds own disjoint positions; one writer per word
      }
    }
    if (v.partial) {
      kept += __popc(keep_bits);
      valid_n += __popc(valid_bits);
      continue;
    }
    // candidate list: the warp appends to its own segment, in position order
    const uint32_t c = __popc(keep_bits);
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    uint64_t at = seg_used + (inc - c);
    uint32_t bits = keep_bits;
    while (bits) {
      const int i = __ffs(bits) - 1;
      bits &= bits - 1;
      if (at < v.seg_cap) {
        const uint64_t sent = (sent_bits >> i) & 1u;  // a string's first or last k-mer
        if (v.narrow) seg32[at] = (uint32_t)(p0 + (uint64_t)i) | ((uint32_t)sent << 31);
        else seg[at] = (p0 + (uint64_t)i) | (sent << 63);
      }
      ++at;
    }
    seg_used += __shfl_sync(0xffffffffu, inc, 31);
    kept += c;
    valid_n += __popc(valid_bits);
  }
  if (lane == 0) {
    v.seg_count[warp_id] = (uint32_t)(seg_used < v.seg_cap ? seg_used : v.seg_cap);
    if (seg_used > v.seg_cap) v.hdr->cand_overflow = 1;
  }
  block_add((unsigned long long)kept, &v.hdr->pass1_kept);
  block_add((unsigned long long)kept, v.partial ? &v.hdr->pass2_kept : &v.hdr->round_kept);
  if (round == v.count_round) block_add((unsigned long long)valid_n, &v.hdr->positions);
}

// The probe loop from descriptors (same decisions and outputs as
// pass1_probe_kernel). A warp takes kProbeR rows of 32 consecutive
// positions; lane l reads the descriptor of position row + l (one coalesced
// 256-byte load per row), loads the filter words of its active non-sentinel
// positions, then decides. A row's ballot is its C_temp word, and its kept
// positions go to the warp's list segment in order.
template <int HB>
__global__ void __launch_bounds__(kBlock) pass1_probe_desc_kernel(RunView v, int round) {
  static_assert(HB <= 6, "descriptors carry the bases of six bits");
  constexpr int kRows = 4;  // rows of 32 positions per warp and step (4 measured faster than 8 or 16)
  static_assert(kRows <= 32, "one C_temp word per lane");
  const int lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  const uint64_t stride = (uint64_t)gridDim.x * kBlock * kRows;
  uint32_t kept = 0, valid_n = 0;  // per thread: below 2^32
  const uint32_t warp_id = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  uint64_t* seg = v.cands + (uint64_t)warp_id * v.seg_cap;
  uint32_t* seg32 = reinterpret_cast<uint32_t*>(v.cands) + (uint64_t)warp_id * v.seg_cap;
  uint64_t seg_used = 0;
  // the descriptors of a step are loaded one step ahead (kProbePrefetch), so
  // that their stream overlaps the previous step's filter loads
  uint64_t dn[kRows];
  const uint64_t wfirst = v.p_begin + ((uint64_t)blockIdx.x * kBlock + (threadIdx.x & ~31u)) * kRows;
  if (kProbePrefetch) {
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
      const uint64_t p = wfirst + 32 * q + lane;
      dn[q] = p < v.m ? __ldcs(v.desc + p) : 0ull;
    }
  }
  for (uint64_t wbase = wfirst; wbase < v.p_end; wbase += stride) {
    uint64_t d[kRows], word[kRows];
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
      const uint64_t p = wbase + 32 * q + lane;
      if (kProbePrefetch) d[q] = dn[q];
      else d[q] = p < v.m ? __ldcs(v.desc + p) : 0ull;
    }
#pragma unroll
    for (int q = 0; q < kRows; ++q)
      if ((d[q] & (kDescActive | kDescSentinel)) == kDescActive) word[q] = __ldcg(v.filter + (uint32_t)d[q]);
    if (kProbePrefetch) {
#pragma unroll
      for (int q = 0; q < kRows; ++q) {
        const uint64_t p = wbase + stride + 32 * q + lane;
        dn[q] = p < v.m ? __ldcs(v.desc + p) : 0ull;
      }
    }
    uint32_t my_word = 0;
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
      bool keep = false;
      if (d[q] & kDescActive) {
        if (d[q] & kDescSentinel) {
          keep = true;
        } else {
          // descriptor bits 32-61 are G's, the only bits bit_base reads for u < 6
          const uint32_t pres = present_items<HB>(d[q], word[q], v.hashes);
          keep = (pres >> 16) || __popc(pres & 0xFFFFu) >= 2;
        }
      }
      valid_n += d[q] != 0;
      const uint32_t row = __ballot_sync(0xffffffffu, keep);
      if (lane == q) my_word = row;
      if (v.partial) {
        kept += keep;
        continue;
      }
      if (keep) {
        lc_mark(v, (d[q] & ~(kDescActive | kDescSentinel)) * kLcMul);
        const uint64_t at = seg_used + __popc(row & below);
        if (at < v.seg_cap) {
          const uint64_t p = wbase + 32 * q + lane;
          const uint64_t sent = (d[q] >> 62) & 1u;
          if (v.narrow) seg32[at] = (uint32_t)p | ((uint32_t)sent << 31);
          else seg[at] = p | (sent << 63);
        }
        ++kept;
      }
      seg_used += __popc(row);
    }
    if (lane < kRows) {
      const uint64_t w = (wbase >> 5) + lane;
      if (w < v.bitmap_words) {
        v.ctemp[w] = my_word;
        if (v.partial) v.cfinal[w] |= my_word;  // rounds own disjoint positions; one writer per word
      }
    }
  }
  if (lane == 0) {
    v.seg_count[warp_id] = (uint32_t)(seg_used < v.seg_cap ? seg_used : v.seg_cap);
    if (seg_used > v.seg_cap) v.hdr->cand_overflow = 1;
  }
  block_add((unsigned long long)kept, &v.hdr->pass1_kept);
  block_add((unsigned long long)kept, v.partial ? &v.hdr->pass2_kept : &v.hdr->round_kept);
  if (round == v.count_round) block_add((unsigned long long)valid_n, &v.hdr->positions);
}

// ---------------------------------------------------------------------------
// Class map (rounds > 1, at most kMaxMapRounds of them): Algorithm 3 marks,
// in round i, the positions whose k-mer is in class i. Instead of walking and
// hashing every position again in every round, one pass after the class cut
// records per position one byte -- bit 7: no k-mer starts here, bit 6: a
// sentinel position (the first or last k-mer of its string or N-free piece),
// bits 0-5: the class -- and each round's two first-pass loops then visit only
// the positions of their class, reading each k-mer from scratch. A warp takes
// a window of 512 consecutive positions, compacts the indices of the active
// ones in shared memory and shares them out evenly over its lanes.
// ---------------------------------------------------------------------------

constexpr uint32_t kCmNone = 0x80u, kCmSentinel = 0x40u, kCmClass = 0x3Fu;
constexpr int kCmWindow = 32 * 16;  // positions per warp window

// Class of a bin: the r with cuts[r] <= bin < cuts[r + 1] (cuts in shared memory).
__device__ __forceinline__ uint32_t class_of_bin(const uint32_t* cuts, int rounds, uint32_t bin) {
  int lo = 0, hi = rounds;  // cuts[lo] <= bin < cuts[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (cuts[mid] <= bin) lo = mid; else hi = mid;
  }
  return (uint32_t)lo;
}

// Filter region of a k-mer's word (region-ordered first pass).
__device__ __forceinline__ uint32_t ord_region(const RunView& v, uint64_t H, uint64_t G) {
  return (uint32_t)(filter_index(v, H, G) >> v.o_lg_region_words);
}

template <int KW>
__global__ void __launch_bounds__(kBlock) class_map_kernel(RunView v) {
  __shared__ uint32_t cuts_s[kMaxMapRounds + 1];
  for (int i = threadIdx.x; i <= v.rounds; i += kBlock) cuts_s[i] = v.cuts[i];
  __syncthreads();
  const uint64_t stride = (uint64_t)gridDim.x * kBlock * kInsertR;
  for (uint64_t p0 = ((uint64_t)blockIdx.x * kBlock + threadIdx.x) * kInsertR; p0 < v.m; p0 += stride) {
    uint32_t w[4] = {0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u};
    walk<KW, kInsertR>(v, p0, [&](int i, uint64_t, bool valid, const auto& oc) {
      if (!valid) return;
      const uint32_t c = class_of_bin(cuts_s, v.rounds, (uint32_t)oc.H & v.qmask) |
                         (oc.sentinel ? kCmSentinel : 0u);
      w[i >> 2] = (w[i >> 2] & ~(0xFFu << (8 * (i & 3)))) | (c << (8 * (i & 3)));
    });
    *reinterpret_cast<uint4*>(v.cmap + p0) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// The sorted tiles of a run with the region-ordered first pass, instead of a
// class map: every tile of kOrdTile positions lists the positions that have a
// k-mer, sorted by (class, filter region) -- 16 bits each, bits 0-13 the
// position within the tile, kOrdEntrySentinel for the first or last k-mer of a
// string -- with the first entry of every (class, region) pair and the end
// (o_toff). A round then reads exactly its members, in
// the order of the buckets their records go to: the scatter needs no
// compaction, no rank per member and no staging to write whole runs, and the
// gather reads the decisions of a run as consecutive bits. (With a class byte
// and a region byte per position instead, every round read 2 bytes of every
// position and compacted, ranked and staged its members: scatter and gather
// took 10.6 + 7.1 ps per position of a 6 Gbp build of four rounds.)
//
// A block sorts a tile in shared memory: the walk counts the pairs with
// atomics that return each position's rank, a scan gives every pair its place.
constexpr int kSortBlock = 512;
constexpr uint32_t kOrdEntryPos = 0x3FFFu, kOrdEntrySentinel = 0x4000u;
constexpr uint32_t kSortNone = 0xFFFFFFFFu;
// per position its pair, rank and sentinel flag, then the sorted list, then the counts
constexpr size_t kSortBytes = (size_t)kOrdTile * 6 + (size_t)kOrdMaxHist * 4;

template <int KW>
__global__ void __launch_bounds__(kSortBlock, 2) class_sort_kernel(RunView v) {
  extern __shared__ __align__(16) unsigned char sort_dyn_s[];
  uint32_t* ent = reinterpret_cast<uint32_t*>(sort_dyn_s);            // kOrdTile
  uint16_t* list = reinterpret_cast<uint16_t*>(ent + kOrdTile);       // kOrdTile
  uint32_t* hist = reinterpret_cast<uint32_t*>(list + kOrdTile);      // L * R
  __shared__ uint32_t cuts_s[kMaxMapRounds + 1];
  __shared__ uint32_t warp_s[kSortBlock / 32];
  constexpr int kUnits = (int)(kOrdTile / kInsertR);  // walks of 16 positions per tile
  const uint32_t R = v.o_regions, L = (uint32_t)v.rounds, nh = L * R;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (L > 1)
    for (uint32_t i = threadIdx.x; i <= L; i += kSortBlock) cuts_s[i] = v.cuts[i];
  // regions are runs of blocks (four words each): the top bits of H give them directly
  const bool by_block = v.o_lg_region_words >= 2;
  const int rshift = by_block ? 64 - v.lg_blocks + v.o_lg_region_words - 2 : 0;  // 64: one region
  for (uint64_t t = blockIdx.x; t < v.o_tiles; t += gridDim.x) {
    for (uint32_t i = threadIdx.x; i < nh; i += kSortBlock) hist[i] = 0;
    __syncthreads();
    for (int unit = threadIdx.x; unit < kUnits; unit += kSortBlock) {
      const uint64_t p0 = t * kOrdTile + (uint64_t)unit * kInsertR;
      if (p0 >= v.m) {
#pragma unroll
        for (int i = 0; i < kInsertR; ++i) ent[i * kUnits + unit] = kSortNone;
        continue;
      }
      walk<KW, kInsertR, true>(v, p0, [&](int i, uint64_t, bool valid, const auto& oc) {
        uint32_t e = kSortNone;
        if (valid) {
          const uint32_t cls = L > 1 ? class_of_bin(cuts_s, (int)L, (uint32_t)oc.H & v.qmask) : 0u;
          const uint32_t reg = by_block ? (rshift < 64 ? (uint32_t)(oc.H >> rshift) : 0u)
                                        : ord_region(v, oc.H, second_hash(oc.H));
          const uint32_t bin = cls * R + reg;
          e = (bin << 16) | atomicAdd(hist + bin, 1u) | (oc.sentinel ? kOrdEntrySentinel : 0u);
        }
        ent[i * kUnits + unit] = e;  // bin < 2^12, rank < 2^14
      });
    }
    __syncthreads();
    // exclusive scan of the counts (nh <= 4096: at most 8 per thread)
    uint32_t total;
    {
      const uint32_t per = (nh + kSortBlock - 1) / kSortBlock;
      const uint32_t i0 = min(nh, threadIdx.x * per), i1 = min(nh, i0 + per);
      uint32_t sum = 0;
      for (uint32_t i = i0; i < i1; ++i) sum += hist[i];
      uint32_t inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) warp_s[wid] = inc;
      __syncthreads();
      uint32_t before = 0;
      total = 0;
#pragma unroll
      for (int w = 0; w < kSortBlock / 32; ++w) {
        before += w < wid ? warp_s[w] : 0u;
        total += warp_s[w];
      }
      uint32_t at = before + inc - sum;
      uint16_t* toff = v.o_toff + t * (nh + 1);
      for (uint32_t i = i0; i < i1; ++i) {
        const uint32_t c = hist[i];
        hist[i] = at;
        toff[i] = (uint16_t)at;  // at most kOrdTile = 16384
        at += c;
      }
      if (threadIdx.x == 0) toff[nh] = (uint16_t)total;
    }
    __syncthreads();
    for (int e0 = threadIdx.x; e0 < (int)kOrdTile; e0 += kSortBlock) {
      const uint32_t e = ent[e0];
      if (e == kSortNone) continue;
      const uint32_t pos = (uint32_t)(e0 & (kUnits - 1)) * kInsertR + (uint32_t)(e0 / kUnits);
      list[hist[e >> 16] + (e & 0x3FFFu)] = (uint16_t)(pos | (e & kOrdEntrySentinel));
    }
    __syncthreads();
    uint4* out = reinterpret_cast<uint4*>(v.o_list + t * kOrdTile);
    const uint4* in = reinterpret_cast<const uint4*>(list);
    for (uint32_t i = threadIdx.x; i < (total + 7) / 8; i += kSortBlock) out[i] = in[i];
    __syncthreads();
  }
}

// The positions of this round's class in the warp's window [wbase, wbase + 512):
// their offsets (bits 0-8) with the sentinel flag (bit 9) go to idx[0 .. n), in
// position order; *valid gets the number of positions with a k-mer.
__device__ __forceinline__ uint32_t compact_window(const RunView& v, uint64_t wbase, int round, uint16_t* idx,
                                                   uint32_t* valid) {
  const int lane = threadIdx.x & 31;
  const uint64_t p0 = wbase + 16 * (uint64_t)lane;
  uint4 q = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
  if (p0 < v.m) q = __ldcs(reinterpret_cast<const uint4*>(v.cmap + p0));
  const uint32_t part[4] = {q.x, q.y, q.z, q.w};
  const uint32_t want = (uint32_t)round * 0x01010101u;
  uint32_t act = 0, sent = 0, val = 0;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    act |= byte_bits(__vcmpeq4(part[c] & 0xBFBFBFBFu, want)) << (4 * c);  // valid and in this class
    sent |= byte_bits(part[c] << 1) << (4 * c);  // bit 6: a sentinel
    val |= byte_bits(~part[c]) << (4 * c);       // bit 7 clear: a k-mer
  }
  const uint32_t n = __popc(act);
  uint32_t inc = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  uint32_t at = inc - n;
  while (act) {
    const uint32_t i = __ffs(act) - 1;
    act &= act - 1;
    idx[at++] = (uint16_t)((16 * lane + i) | (((sent >> i) & 1u) << 9));
  }
  *valid = __popc(val);
  __syncwarp();
  return __shfl_sync(0xffffffffu, inc, 31);
}

// The region-ordered kernels take the current round (its records fit).
__device__ __forceinline__ bool ordered_round(const RunView& v) {
  return v.o_regions && *reinterpret_cast<volatile const unsigned int*>(&v.hdr->ord_ok);
}

// Pass 2 of this (ordered) round runs on its records: no part of the table filled up.
__device__ __forceinline__ bool fused_pass2(const RunView& v) {
  return v.o_fused && !*reinterpret_cast<volatile const unsigned int*>(&v.hdr->part_full);
}

// Algorithm 1, insert loop, first pass, over this round's class only.
template <int KW, int HB, bool BKT = false>
__global__ void __launch_bounds__(kBlock) pass1_insert_cm_kernel(RunView v, int round) {
  __shared__ uint16_t idx_s[kBlock / 32][kCmWindow];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint16_t* idx = idx_s[wid];
  const uint64_t stride = (uint64_t)gridDim.x * kBlock * 16;
  for (uint64_t wbase = v.p_begin + ((uint64_t)blockIdx.x * kBlock + (threadIdx.x & ~31u)) * 16; wbase < v.p_end;
       wbase += stride) {
    uint32_t valid;
    const uint32_t n = compact_window(v, wbase, round, idx, &valid);
    for (uint32_t j = lane; j < n; j += 32) {
      const uint32_t e = idx[j];
      OccT<KW> oc;
      read_listed<KW>(v, wbase + (e & 511u), (e >> 9) & 1u, &oc);
      const uint64_t G = second_hash(oc.H);
      const ItemPattern pat = item_pattern<HB>(G, v.hashes);
      uint64_t m = item_bits(pat, oc.j1);
      if (oc.j2 != oc.j1) m |= item_bits(pat, oc.j2);  // a palindrome's two orientations
      if (BKT) stage_or(v, filter_index(v, oc.H, G), G, oc.j1, oc.j2, m);
      else atomicOr(filter_word(v, oc.H, G), (unsigned long long)m);
    }
    __syncwarp();
  }
}

// Algorithm 1, probe loop, first pass, over this round's class only: the same
// decisions and outputs as pass1_probe_kernel (C_temp words of the window, the
// candidate list segment of the warp, the linear-counting bits).
template <int KW, int HB>
__global__ void __launch_bounds__(kBlock) pass1_probe_cm_kernel(RunView v, int round) {
  __shared__ uint16_t idx_s[kBlock / 32][kCmWindow];
  __shared__ uint32_t keep_s[kBlock / 32][kCmWindow / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint16_t* idx = idx_s[wid];
  uint32_t* keep_w = keep_s[wid];
  const uint32_t below = (1u << lane) - 1u;
  uint32_t kept = 0, valid_n = 0;  // per thread: below 2^32
  const uint32_t warp_id = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  uint64_t* seg = v.cands + (uint64_t)warp_id * v.seg_cap;
  uint32_t* seg32 = reinterpret_cast<uint32_t*>(v.cands) + (uint64_t)warp_id * v.seg_cap;
  uint64_t seg_used = 0;
  if (lane < kCmWindow / 32) keep_w[lane] = 0;
  __syncwarp();
  const uint64_t stride = (uint64_t)gridDim.x * kBlock * 16;
  for (uint64_t wbase = v.p_begin + ((uint64_t)blockIdx.x * kBlock + (threadIdx.x & ~31u)) * 16; wbase < v.p_end;
       wbase += stride) {
    uint32_t valid;
    const uint32_t n = compact_window(v, wbase, round, idx, &valid);
    valid_n += valid;
    for (uint32_t j0 = 0; j0 < n; j0 += 32) {
      const uint32_t j = j0 + lane;
      bool keep = false;
      uint64_t G = 0, g = 0;
      uint32_t sentinel = 0;
      if (j < n) {
        const uint32_t e = idx[j];
        g = wbase + (e & 511u);
        sentinel = (e >> 9) & 1u;
        if (sentinel) {
          keep = true;
          OccT<KW> oc;
          read_listed<KW>(v, g, true, &oc);
          G = second_hash(oc.H);
        } else {
          OccT<KW> oc;
          read_listed<KW>(v, g, false, &oc);
          G = second_hash(oc.H);
          const uint64_t word = __ldcg(filter_word(v, oc.H, G));
          const uint32_t pres = present_items<HB>(G, word, v.hashes);
          keep = (pres >> 16) || __popc(pres & 0xFFFFu) >= 2;
        }
        if (keep) atomicOr(keep_w + ((e & 511u) >> 5), 1u << (e & 31u));
      }
      if (v.partial) {
        kept += keep;
        continue;
      }
      const uint32_t row = __ballot_sync(0xffffffffu, keep);
      if (keep) {
        lc_mark(v, G * kLcMul);
        const uint64_t at = seg_used + __popc(row & below);
        if (at < v.seg_cap) {
          if (v.narrow) seg32[at] = (uint32_t)g | (sentinel << 31);
          else seg[at] = g | ((uint64_t)sentinel << 63);
        }
        ++kept;
      }
      seg_used += __popc(row);
    }
    __syncwarp();
    if (lane < kCmWindow / 32) {
      const uint64_t w = (wbase >> 5) + lane;
      const uint32_t word = keep_w[lane];
      keep_w[lane] = 0;
      if (w < v.bitmap_words) {
        v.ctemp[w] = word;
        if (v.partial) v.cfinal[w] |= word;  // rounds own disjoint positions; one writer per word
      }
    }
    __syncwarp();
  }
  if (lane == 0) {
    v.seg_count[warp_id] = (uint32_t)(seg_used < v.seg_cap ? seg_used : v.seg_cap);
    if (seg_used > v.seg_cap) v.hdr->cand_overflow = 1;
  }
  block_add((unsigned long long)kept, &v.hdr->pass1_kept);
  block_add((unsigned long long)kept, v.partial ? &v.hdr->pass2_kept : &v.hdr->round_kept);
  if (round == v.count_round) block_add((unsigned long long)valid_n, &v.hdr->positions);
}

// ---------------------------------------------------------------------------
// Region-ordered first pass (class-map rounds). A filter far beyond L2 takes
// every random OR and every random probe at DRAM's random-access rate (about
// 64 bytes moved per 8-byte access). Here a round instead writes one 8-byte
// record per position of its class into the bucket of the position's filter
// region (at most 2^22 words: 32 MiB, which L2 holds), applies the ORs and
// then the probes bucket by bucket -- so that the random accesses of a region
// all hit L2 -- and gathers the probe's decisions back in position order.
//
// Buckets: the sorted tiles (class_sort_kernel) hold the count of every
// (class, region) pair per tile, so a round's buckets are laid out exactly
// (each a multiple of 32 slots). A tile's records for a bucket are consecutive
// in the bucket, in tile order and in the order of the tile's list: a scan over
// the tiles' counts gives every tile its room in every bucket (o_meta), and a
// member's slot is its bucket's start plus its tile's room plus its index
// within its run of the list.
//
// A record: bits 0-21 the word within its region, 22-51 the bits 32-61 of G
// (the bit bases of up to 6 bits per item), 52-56 and 57-61 the items (two
// for a palindrome's orientations), bit 62 the sentinel flag. With pass 2 on
// the records (k <= 31) a record holds the occurrence instead (fused_record).
// ---------------------------------------------------------------------------

constexpr uint32_t kOrdPiece = 4096;  // records per apply or probe work item (a multiple of 32)
constexpr unsigned long long kOrdSentinel = 1ull << 62;

// Fused records (k <= 31, o_fused): the round's pass 2 runs on the same
// records. The hash of a one-word k-mer is a bijection, and the bucket gives
// its top bits, so a record holds the k-mer as the low 64 - log2(R) bits of H
// (bits 6 up), with the item its occurrence inserts (bits 0-3), whether the
// k-mer is a palindrome (4: the other strand's item too) and whether it is a
// sentinel (5). The kernels that apply it hash nothing but G: with the k-mer
// and its bases in the record, each of them mixed it again, and the probe and
// the classify were bound by their integer instructions (73% issue).
constexpr uint32_t kFusedPalindrome = 16u, kFusedSentinel = 32u;
constexpr int kFusedBits = 6;

template <int KW>
__device__ __forceinline__ unsigned long long fused_record(const OccT<KW>& oc) {
  return (oc.H << kFusedBits) | (oc.sentinel ? kFusedSentinel : (oc.j1 | (oc.j2 != oc.j1 ? kFusedPalindrome : 0u)));
}

struct FusedOcc {
  uint64_t H, G;
  uint32_t j1, j2;
  bool sentinel;
};

// top: the bucket's bits of H, in place (fused_top).
__device__ __forceinline__ FusedOcc fused_occ(unsigned long long rec, uint64_t top, uint64_t low_mask) {
  FusedOcc o;
  o.H = top | ((rec >> kFusedBits) & low_mask);
  o.G = second_hash(o.H);
  const uint32_t f = (uint32_t)rec, j = f & 15u;
  o.sentinel = f & kFusedSentinel;
  o.j1 = o.sentinel ? 16u : j;
  o.j2 = (f & kFusedPalindrome) ? item_reverse(j >> 2, j & 3u) : o.j1;
  return o;
}

// Buckets are the top bits of H: R regions, a power of two of at least 64, each of
// whole filter blocks (four words or more).
__device__ __forceinline__ int fused_low_bits(const RunView& v) { return 64 - (31 - __clz(v.o_regions)); }

// The fused pass-2 table: bucket b owns the o_tcap one-word slots from b *
// o_tcap, so that its inserts and lookups stay in L2 beside the filter region.
// A slot: the k-mer as the low bits of H (bits 5 up), the item of its first
// occurrence (1-4), and whether it is a junction (0) -- a sentinel, or seen with
// two items, which differ in the in- or the out-base. Empty: all ones, which no
// slot is (58 bits of H at most). A k-mer starts at bits 16-47 of H scaled to
// o_tcap (Lemire's multiply-high) and probes linearly within the part. Slot by slot,
// unlike the direct table: the whole reserve is the table, at a load of a few
// percent, so that the first slot mostly decides (a sector at a time took the
// probe of 6 Gbp from 7.6 to 11.4 ps per position). A part counts as full when a
// k-mer finds no slot in kFusedChain steps (o_chain: in the whole of a smaller part): at
// a load of 0.9 the longest run of taken slots in a million is about 2600. A full part
// (its share of the k-mers varies, and a tight reserve has no room for that) is no error:
// the round's pass 2 then goes over the candidate list and one table of the whole reserve.
__device__ __forceinline__ bool fused_table_insert(const RunView& v, uint32_t b, const FusedOcc& o,
                                                   uint64_t low_mask) {
  const uint32_t cap = v.o_tcap;
  unsigned long long* T = static_cast<unsigned long long*>(v.table) + (uint64_t)b * cap;
  const bool junction = o.sentinel || o.j1 != o.j2;
  const unsigned long long mine = ((o.H & low_mask) << 5) | ((o.j1 & 15u) << 1) | (junction ? 1u : 0u);
  uint32_t i = __umulhi((uint32_t)(o.H >> 16), cap);
  for (uint32_t probe = 0; probe < v.o_chain; ++probe, i = i + 1 == cap ? 0u : i + 1) {
    unsigned long long cur = __ldcg(T + i);
    if (cur == kEmpty) {
      cur = atomicCAS(T + i, kEmpty, mine);
      if (cur == kEmpty) return true;
    }
    if ((cur ^ mine) >> 5) continue;
    if (!(cur & 1u) && cur != mine) atomicOr(T + i, 1ull);
    return true;
  }
  return false;
}

// 1 or 0: the k-mer of H is a junction or not; -1: absent.
__device__ __forceinline__ int fused_table_find(const RunView& v, uint32_t b, uint64_t H, uint64_t low_mask) {
  const uint32_t cap = v.o_tcap;
  const unsigned long long* T = static_cast<const unsigned long long*>(v.table) + (uint64_t)b * cap;
  const uint64_t key = H & low_mask;
  uint32_t i = __umulhi((uint32_t)(H >> 16), cap);
  for (uint32_t probe = 0; probe < kFusedChain; ++probe, i = i + 1 == cap ? 0u : i + 1) {
    const unsigned long long cur = __ldcg(T + i);
    if (cur == kEmpty) return -1;
    if ((cur >> 5) == key) return (int)(cur & 1u);
  }
  return -1;
}

// Exclusive scan of x over the block (blockDim.x == kBlock), 64-bit.
__device__ __forceinline__ unsigned long long block_exclusive_scan64(unsigned long long x, unsigned long long* total) {
  __shared__ unsigned long long warp_tot[kBlock / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_tot[wid] = inc;
  __syncthreads();
  unsigned long long before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kBlock / 32; ++w) {
    const unsigned long long t = warp_tot[w];
    before += (w < wid) ? t : 0ull;
    all += t;
  }
  __syncthreads();
  *total = all;
  return before + inc - x;
}

// The rooms of a round's tiles in its buckets, in tile order: o_meta[t * R + b]
// = the round's members of bucket b in the tiles before t. Three steps over
// chunks of kOrdScanTiles tiles: the chunks' sums, their prefix per bucket
// (with every bucket's total, o_btot), then every tile's room. The counts of
// kRoomAhead tiles are loaded before any of them is used: one after the other
// they were a chain of L2 round trips per thread.
constexpr int kRoomAhead = 8;
static_assert(kOrdScanTiles % kRoomAhead == 0, "whole groups of tiles");

// (Called by the whole block; fn runs for the threads of a bucket, b < R.)
template <typename F>
__device__ __forceinline__ void for_tile_counts(const RunView& v, int round, F&& fn) {
  const uint32_t R = v.o_regions, nh = (uint32_t)v.rounds * R, b = threadIdx.x;
  const uint64_t t0 = (uint64_t)blockIdx.x * kOrdScanTiles, t1 = min(t0 + kOrdScanTiles, v.o_tiles);
  const uint16_t* at = v.o_toff + (uint64_t)round * R + b;
  for (uint64_t t = t0; t < t1; t += kRoomAhead) {
    uint32_t c[kRoomAhead];
#pragma unroll
    for (int u = 0; u < kRoomAhead; ++u) {
      const uint16_t* q = at + (t + u) * (nh + 1);
      c[u] = (t + u < t1 && b <= R) ? __ldg(q) : 0u;
    }
#pragma unroll
    for (int u = 0; u < kRoomAhead; ++u) {  // a run ends where the next lane's starts
      uint32_t end = __shfl_down_sync(0xffffffffu, c[u], 1);
      if ((b & 31) == 31 && t + u < t1 && b < R) end = __ldg(at + (t + u) * (nh + 1) + 1);
      if (t + u < t1 && b < R) fn(t + u, end - c[u]);
    }
  }
}

__global__ void __launch_bounds__(kBlock) ord_room_sum_kernel(RunView v, int round) {
  uint32_t s = 0;
  for_tile_counts(v, round, [&](uint64_t, uint32_t c) { s += c; });
  if (threadIdx.x < v.o_regions) v.o_csum[(uint64_t)blockIdx.x * v.o_regions + threadIdx.x] = s;
}

__global__ void __launch_bounds__(kBlock) ord_room_prefix_kernel(RunView v, uint64_t chunks) {
  const uint32_t R = v.o_regions, b = blockIdx.x;
  __shared__ unsigned long long carry_s;
  if (threadIdx.x == 0) carry_s = 0;
  __syncthreads();
  for (uint64_t c0 = 0; c0 < chunks; c0 += kBlock) {
    const uint64_t c = c0 + threadIdx.x;
    const unsigned long long x = c < chunks ? v.o_csum[c * R + b] : 0ull;
    unsigned long long tot;
    const unsigned long long ex = block_exclusive_scan64(x, &tot);
    if (c < chunks) v.o_cpre[c * R + b] = carry_s + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry_s += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) v.o_btot[b] = carry_s;
}

__global__ void __launch_bounds__(kBlock) ord_room_scan_kernel(RunView v, int round) {
  const uint32_t R = v.o_regions;
  unsigned long long run = threadIdx.x < R ? v.o_cpre[(uint64_t)blockIdx.x * R + threadIdx.x] : 0ull;
  for_tile_counts(v, round, [&](uint64_t t, uint32_t c) {
    v.o_meta[t * R + threadIdx.x] = (uint32_t)run;  // within a bucket below 2^32 (the setup checks)
    run += c;
  });
}

// Before a round's scatter: the buckets' starts (each a multiple of 32), the
// work tickets cleared, and whether the round's records fit (else the direct
// kernels take the round). One block.
__global__ void __launch_bounds__(kBlock) ord_setup_kernel(RunView v, int round) {
  static_assert(kOrdMaxRegions <= kBlock, "one thread per bucket");
  const uint32_t R = v.o_regions, b = threadIdx.x;
  const unsigned long long n = b < R ? v.o_btot[b] : 0ull;
  unsigned long long total;
  const unsigned long long start = block_exclusive_scan64((n + 31) & ~31ull, &total);
  if (b < R) {
    v.o_fill[(uint64_t)b * kOrdFillStride] = (uint32_t)n;
    v.o_start[b] = start;
  }
  const int fits = __syncthreads_and(n < (1ull << 32));  // slots within a bucket are 32-bit
  if (threadIdx.x == 0) {
    v.o_start[R] = total;
    v.hdr->ord_ok = (fits && total <= v.o_rec_cap) ? 1u : 0u;
    v.hdr->ord_rounds += v.hdr->ord_ok;
    v.hdr->ord_ticket[0] = 0;
    v.hdr->ord_ticket[1] = 0;
    v.hdr->ord_ticket[2] = 0;
    v.hdr->ord_ticket[3] = 0;
    v.hdr->part_slots = 0;
    v.hdr->part_full = 0;
    v.hdr->cand_overflow = 0;  // the gather of the round before may have set it after its table_setup
  }
}

// A tile's members of a round, in the order of the tile's list (by bucket): the
// list from `list` on, `n` members; member i is in bucket bucket_s[i], at slot
// delta_s[bucket] + i of the round's records.
struct TileMembers {
  const uint16_t* list;
  uint32_t n;
};

// Load a tile's members (called by the whole block; ends with a barrier). The
// members' buckets are filled in by R / kBlock-th of the threads each, run by run.
__device__ __forceinline__ TileMembers ord_tile(const RunView& v, uint64_t t, int round, const uint64_t* start_s,
                                                unsigned long long* delta_s, uint32_t* run_s, uint8_t* bucket_s) {
  const uint32_t R = v.o_regions, b = threadIdx.x;
  const uint16_t* toff = v.o_toff + t * ((uint64_t)v.rounds * R + 1) + (uint64_t)round * R;
  const uint32_t first = toff[0];
  TileMembers tm;
  tm.list = v.o_list + t * kOrdTile + first;
  tm.n = toff[R] - first;
  if (b < R) {
    const uint32_t off = toff[b] - first, count = toff[b + 1] - toff[b];
    delta_s[b] = start_s[b] + __ldg(v.o_meta + t * R + b) - off;
    run_s[b] = off | (count << 16);  // both at most kOrdTile = 2^14
  }
  __syncthreads();
  // R is a power of two of at most kBlock: kBlock / R threads per run
  const uint32_t r = threadIdx.x & (R - 1u), x = run_s[r], end = (x & 0xFFFFu) + (x >> 16);
  for (uint32_t i = (x & 0xFFFFu) + threadIdx.x / R; i < end; i += kBlock / R) bucket_s[i] = (uint8_t)r;
  __syncthreads();
  return tm;
}

// Algorithm 1, insert loop, first pass, over this round's class: one record
// per member into the bucket of its filter region (tiles grid-strided). The
// members come in bucket order, so that consecutive threads write consecutive
// records of a run. A few members per thread are in flight at a time. Bound by
// the integer pipe (77% of its peak, L1 58%: 200 M members in 1.0 ms); reading the
// tile's packed words through shared memory changed nothing.
template <int KW, int HB, bool FUSED>
__global__ void __launch_bounds__(kBlock) tile_scatter_kernel(RunView v, int round) {
  __shared__ uint8_t bucket_s[kOrdTile];
  __shared__ unsigned long long delta_s[kOrdMaxRegions];
  __shared__ uint64_t start_s[kOrdMaxRegions];
  __shared__ uint32_t run_s[kOrdMaxRegions];
  if (!ordered_round(v)) return;
  for (uint32_t b = threadIdx.x; b < v.o_regions; b += kBlock) start_s[b] = v.o_start[b];
  const uint64_t local_mask = (1ull << v.o_lg_region_words) - 1ull;
  for (uint64_t t = blockIdx.x; t < v.o_tiles; t += gridDim.x) {
    const TileMembers tm = ord_tile(v, t, round, start_s, delta_s, run_s, bucket_s);
    constexpr int U = KW == 1 ? 4 : 2;
    for (uint32_t i0 = threadIdx.x; i0 < tm.n; i0 += U * kBlock) {
      uint32_t e[U];
#pragma unroll
      for (int u = 0; u < U; ++u) e[u] = i0 + u * kBlock < tm.n ? __ldcs(tm.list + i0 + u * kBlock) : 0u;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t i = i0 + u * kBlock;
        if (i >= tm.n) break;
        const bool sentinel = e[u] & kOrdEntrySentinel;
        OccT<KW> oc;
        read_listed<KW>(v, t * kOrdTile + (e[u] & kOrdEntryPos), sentinel, &oc);
        unsigned long long rec;
        if constexpr (FUSED) {
          rec = fused_record(oc);
        } else {
          const uint64_t G = second_hash(oc.H);
          const uint64_t word = filter_index(v, oc.H, G);
          rec = (word & local_mask) | (((G >> 32) & 0x3FFFFFFFull) << 22) | ((uint64_t)oc.j1 << 52) |
                ((uint64_t)oc.j2 << 57) | (sentinel ? kOrdSentinel : 0ull);
        }
        v.o_recs[delta_s[bucket_s[i]] + i] = rec;
      }
    }
    __syncthreads();  // the shared arrays serve the next tile
  }
}

// Work items of kOrdPiece records, taken in bucket order from a ticket, so
// that the blocks in flight work on one or two regions at a time. first_s[b]:
// the first item of bucket b (first_s[R]: the number of items).
__device__ __forceinline__ void ord_items(const RunView& v, uint32_t* first_s) {
  const uint32_t b = threadIdx.x;  // at most kBlock buckets
  const uint64_t n = b < v.o_regions ? __ldcg(v.o_fill + (uint64_t)b * kOrdFillStride) : 0ull;
  uint32_t total;
  const uint32_t first = block_exclusive_scan((uint32_t)((n + kOrdPiece - 1) / kOrdPiece), &total);
  if (b < v.o_regions) first_s[b] = first;
  if (b == 0) first_s[v.o_regions] = total;
  __syncthreads();
}

// Warm L2 with this work item's share of the next bucket's filter region, so
// that the region's first accesses do not wait on DRAM one random sector at
// a time (the items of a bucket together cover the whole next region).
__device__ __forceinline__ void ord_prefetch_next(const RunView& v, const uint32_t* first_s, uint32_t b,
                                                  uint32_t item) {
  if (b + 1 >= v.o_regions) return;
  const uint64_t rbytes = 8ull << v.o_lg_region_words;
  const uint64_t share = (rbytes / (first_s[b + 1] - first_s[b]) + 127) & ~127ull;
  const uint64_t off = (uint64_t)(item - first_s[b]) * share, end = min(off + share, rbytes);
  const char* next = reinterpret_cast<const char*>(v.filter + ((uint64_t)(b + 1) << v.o_lg_region_words));
  for (uint64_t o = off + 128 * (uint64_t)threadIdx.x; o < end; o += 128 * (uint64_t)kBlock)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(next + o));
}

__device__ __forceinline__ uint32_t ord_item_bucket(const uint32_t* first_s, uint32_t R, uint32_t item) {
  uint32_t lo = 0, hi = R;  // the bucket b with first_s[b] <= item < first_s[b + 1]
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (first_s[mid] <= item) lo = mid; else hi = mid;
  }
  return lo;
}

// The ORs of the round's records, bucket by bucket (four records in flight
// per thread).
template <int HB, bool FUSED>
__global__ void __launch_bounds__(kBlock) ord_or_kernel(RunView v) {
  __shared__ uint32_t first_s[kOrdMaxRegions + 1];
  __shared__ uint32_t item_s;
  if (!ordered_round(v)) return;
  ord_items(v, first_s);
  const uint32_t R = v.o_regions, total = first_s[R];
  for (;;) {
    if (threadIdx.x == 0) item_s = atomicAdd(&v.hdr->ord_ticket[0], 1u);
    __syncthreads();
    const uint32_t item = item_s;
    __syncthreads();
    if (item >= total) break;
    const uint32_t b = ord_item_bucket(first_s, R, item);
    ord_prefetch_next(v, first_s, b, item);
    const uint64_t n = __ldcg(v.o_fill + (uint64_t)b * kOrdFillStride);
    const uint64_t i0 = (uint64_t)(item - first_s[b]) * kOrdPiece, i1 = min(i0 + kOrdPiece, n);
    const uint64_t* recs = v.o_recs + __ldg(v.o_start + b);
    unsigned long long* region = v.filter + ((uint64_t)b << v.o_lg_region_words);
    const uint64_t low_mask = FUSED ? (1ull << fused_low_bits(v)) - 1ull : 0ull;
    const uint64_t top = FUSED ? (uint64_t)b << fused_low_bits(v) : 0ull;
    for (uint64_t i = i0 + threadIdx.x; i < i1; i += 4 * kBlock) {
      uint64_t r[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) r[u] = i + u * kBlock < i1 ? __ldcs(recs + i + u * kBlock) : ~0ull;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (r[u] == ~0ull) continue;
        if constexpr (FUSED) {
          const FusedOcc o = fused_occ(r[u], top, low_mask);
          const ItemPattern pat = item_pattern<HB>(o.G, v.hashes);
          uint64_t m = item_bits(pat, o.j1);
          if (o.j2 != o.j1) m |= item_bits(pat, o.j2);
          atomicOr(v.filter + filter_index(v, o.H, o.G), (unsigned long long)m);
        } else {
          const uint64_t G = ((r[u] >> 22) & 0x3FFFFFFFull) << 32;  // the bits bit_base reads for u < 6
          const ItemPattern pat = item_pattern<HB>(G, v.hashes);
          const uint32_t j1 = (uint32_t)(r[u] >> 52) & 31u, j2 = (uint32_t)(r[u] >> 57) & 31u;
          uint64_t m = item_bits(pat, j1);
          if (j2 != j1) m |= item_bits(pat, j2);
          atomicOr(region + (r[u] & 0x3FFFFFull), (unsigned long long)m);
        }
      }
    }
  }
}

// Algorithm 1, probe loop, first pass, over the round's records, bucket by
// bucket: a record's decision (its k-mer is a candidate: a sentinel, or its
// filter word holds a sentinel item or two distinct items) goes to its slot's
// bit; the linear-counting bit of every candidate is set from the k-mer's
// filter word index and bit bases. FUSED: instead, every candidate inserts
// its in/out bases into its region's part of the pass-2 table (Algorithm 1's
// insert loop, second pass) while the region is in L2, until a part fills up.
template <int HB, bool FUSED>
__global__ void __launch_bounds__(kBlock) ord_probe_kernel(RunView v) {
  __shared__ uint32_t first_s[kOrdMaxRegions + 1];
  __shared__ uint32_t item_s;
  __shared__ bool insert_s;
  if (!ordered_round(v)) return;
  ord_items(v, first_s);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t R = v.o_regions, total = first_s[R];
  uint32_t kept = 0;
  for (;;) {
    if (threadIdx.x == 0) item_s = atomicAdd(&v.hdr->ord_ticket[1], 1u);
    if (FUSED && threadIdx.x == 32) insert_s = fused_pass2(v);  // beside the ticket's round trip
    __syncthreads();
    const uint32_t item = item_s;
    const bool insert = FUSED && insert_s;
    __syncthreads();
    if (item >= total) break;
    const uint32_t b = ord_item_bucket(first_s, R, item);
    ord_prefetch_next(v, first_s, b, item);
    const uint64_t n = __ldcg(v.o_fill + (uint64_t)b * kOrdFillStride);
    const uint64_t i0 = (uint64_t)(item - first_s[b]) * kOrdPiece, i1 = min(i0 + kOrdPiece, n);
    const uint64_t start = __ldg(v.o_start + b);  // a multiple of 32, as is i0
    const uint64_t* recs = v.o_recs + start;
    const uint64_t region = (uint64_t)b << v.o_lg_region_words;
    // U chunks of 32 records per warp and step: their records, then their filter
    // words, all in flight at once
    constexpr int U = FUSED ? 2 : 4;
    const uint64_t low_mask = FUSED ? (1ull << fused_low_bits(v)) - 1ull : 0ull;
    const uint64_t top = FUSED ? (uint64_t)b << fused_low_bits(v) : 0ull;
    for (uint64_t w0 = i0 + 32 * wid; w0 < i1; w0 += U * kBlock) {
      unsigned long long rec[U], word[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t i = w0 + (uint64_t)u * kBlock + lane;
        rec[u] = i < i1 ? __ldcs(recs + i) : ~0ull;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        word[u] = 0;
        if (rec[u] == ~0ull) continue;
        if constexpr (FUSED) {
          const FusedOcc o = fused_occ(rec[u], top, low_mask);
          if (!o.sentinel) word[u] = __ldcg(v.filter + filter_index(v, o.H, o.G));
        } else {
          if (!(rec[u] & kOrdSentinel)) word[u] = __ldcg(v.filter + (region | (rec[u] & 0x3FFFFFull)));
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t c = w0 + (uint64_t)u * kBlock;
        if (c >= i1) break;  // the same for the whole warp
        bool keep = false;
        if (rec[u] != ~0ull) {
          if constexpr (FUSED) {  // the decision, and the candidate's edges into the region's table
            const FusedOcc o = fused_occ(rec[u], top, low_mask);
            const uint32_t pres = present_items<HB>(o.G, word[u], v.hashes);
            keep = o.sentinel || (pres >> 16) || __popc(pres & 0xFFFFu) >= 2;
            if (keep && insert && !fused_table_insert(v, b, o, low_mask)) v.hdr->part_full = 1;
          } else {
            const uint64_t G = ((rec[u] >> 22) & 0x3FFFFFFFull) << 32;
            const uint32_t pres = present_items<HB>(G, word[u], v.hashes);
            keep = (rec[u] & kOrdSentinel) || (pres >> 16) || __popc(pres & 0xFFFFu) >= 2;
            if (keep && !v.partial) {
              const uint64_t id = ((region | (rec[u] & 0x3FFFFFull)) << 30) | ((rec[u] >> 22) & 0x3FFFFFFFull);
              lc_mark(v, id * kLcMul);
            }
          }
        }
        const uint32_t row = __ballot_sync(0xffffffffu, keep);
        // word pairs, the candidates' bits then the junctions' (partial: no junctions)
        if (lane == 0) {
          v.o_dec[((start + c) >> 5) << (v.partial ? 0 : 1)] = row;
          kept += __popc(row);
        }
      }
    }
  }
  if (!v.partial) block_add((unsigned long long)kept, &v.hdr->round_kept);  // sizes the table and its work
}

// Algorithm 1, probe loop, second pass, on fused records, bucket by bucket:
// every candidate record (decision bit set) looks its k-mer up in the
// region's table; its bit in the junction word of o_dec says whether the
// k-mer is a junction.
__global__ void __launch_bounds__(kBlock, 8) ord_classify_kernel(RunView v) {
  __shared__ uint32_t first_s[kOrdMaxRegions + 1];
  __shared__ uint32_t item_s;
  if (!ordered_round(v) || !fused_pass2(v)) return;
  ord_items(v, first_s);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t R = v.o_regions, total = first_s[R];
  for (;;) {
    if (threadIdx.x == 0) item_s = atomicAdd(&v.hdr->ord_ticket[2], 1u);
    __syncthreads();
    const uint32_t item = item_s;
    __syncthreads();
    if (item >= total) break;
    const uint32_t b = ord_item_bucket(first_s, R, item);
    const uint64_t n = __ldcg(v.o_fill + (uint64_t)b * kOrdFillStride);
    const uint64_t i0 = (uint64_t)(item - first_s[b]) * kOrdPiece, i1 = min(i0 + kOrdPiece, n);
    const uint64_t start = __ldg(v.o_start + b);  // a multiple of 32, as is i0
    const uint64_t low_mask = (1ull << fused_low_bits(v)) - 1ull, top = (uint64_t)b << fused_low_bits(v);
    const uint64_t* recs = v.o_recs + start;
    // four chunks of 32 records per warp and step: their loads all in flight at once
    constexpr int U = 4;
    for (uint64_t w0 = i0 + 32 * wid; w0 < i1; w0 += U * kBlock) {
      uint32_t cand[U];
      unsigned long long rec[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t c = w0 + (uint64_t)u * kBlock;
        cand[u] = c < i1 ? __ldcg(v.o_dec + (((start + c) >> 5) << 1)) : 0u;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t i = w0 + (uint64_t)u * kBlock + lane;
        rec[u] = (i < i1 && ((cand[u] >> lane) & 1u)) ? __ldcs(recs + i) : ~0ull;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t c = w0 + (uint64_t)u * kBlock;
        bool junction = false;
        if (rec[u] != ~0ull) {
          const int j = fused_table_find(v, b, top | ((rec[u] >> kFusedBits) & low_mask), low_mask);
          if (j < 0) v.hdr->overflow = 1;
          junction = j != 0;
        }
        const uint32_t row = __ballot_sync(0xffffffffu, junction);
        if (lane == 0 && c < i1) v.o_dec[(((start + c) >> 5) << 1) + 1] = row;
      }
    }
  }
}

// Pass 2 bucket by bucket for k-mers that no record holds (32 <= k <= 63): the
// table has one part per filter region (table_setup), and the candidates of a
// bucket -- found by its records' decision bits, and their positions by the
// tiles' lists -- are inserted part by part, so that the table's random accesses
// hit L2. In position order, over a 6 GB table, they ran at DRAM's
// random-access rate: 15.0 + 5.3 of 31.7 ms for 62 genomes at k = 63.
// A work item is o_item_tiles tiles of one bucket, taken in bucket order from a
// ticket; a warp collects the candidates of its tiles' runs and inserts them 32
// at a time. The slot goes where the candidate's record was (the probe read it
// last), for the probe loop.
template <int KW, int TS>
__global__ void __launch_bounds__(kBlock) ord_insert2_kernel(RunView v, int round) {
  __shared__ uint32_t item_s;
  __shared__ uint32_t slot_s[kBlock / 32][64], ent_s[kBlock / 32][64];  // the warp's candidates: record, list entry
  const uint64_t part = __ldcg(&v.hdr->part_slots);
  if (!ordered_round(v) || !part) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t* slot_q = slot_s[wid];
  uint32_t* ent_q = ent_s[wid];
  const uint32_t below = (1u << lane) - 1u;
  const uint32_t R = v.o_regions, per = v.o_item_tiles;
  const uint32_t chunks = (uint32_t)((v.o_tiles + per - 1) / per), total = R * chunks;
  const uint64_t nh = (uint64_t)v.rounds * R;
  for (;;) {
    if (threadIdx.x == 0) item_s = atomicAdd(&v.hdr->ord_ticket[3], 1u);
    __syncthreads();
    const uint32_t item = item_s;
    __syncthreads();
    if (item >= total) break;
    const uint32_t b = item / chunks;
    const uint64_t t0 = (uint64_t)(item - b * chunks) * per, t1 = min(t0 + per, v.o_tiles);
    const uint64_t start = __ldg(v.o_start + b);
    RunView x = v;
    x.table = static_cast<char*>(v.table) + (uint64_t)b * part * (32 / SectorOf<TS>::kSlots);
    auto insert = [&](uint32_t n) {  // the first n candidates of the queue
      __syncwarp();
      if ((uint32_t)lane < n) {
        const uint32_t e = ent_q[lane];
        const uint64_t g = (t0 + (e >> 16)) * kOrdTile + (e & kOrdEntryPos);
        OccT<KW> oc;
        read_listed<KW>(v, g, e & kOrdEntrySentinel, &oc);
        const uint64_t at = insert_occurrence<KW, TS>(x, part, oc, g);
        if (at == kNoSlot) v.hdr->overflow = 1;
        v.o_recs[start + slot_q[lane]] = at;
      }
      __syncwarp();
    };
    uint32_t n = 0;
    // the runs of kGroup tiles at a time, one per lane
    constexpr int kGroup = 8;
    for (uint64_t tb = t0 + (uint64_t)kGroup * wid; tb < t1; tb += kGroup * (kBlock / 32)) {
      uint32_t off = 0, cnt = 0, room = 0;
      if (lane < kGroup && tb + lane < t1) {
        const uint16_t* q = v.o_toff + (tb + lane) * (nh + 1) + (uint64_t)round * R + b;
        off = q[0];
        cnt = q[1] - off;
        room = __ldg(v.o_meta + (tb + lane) * R + b);
      }
      const int tiles = (int)min((uint64_t)kGroup, t1 - tb);
      for (int i = 0; i < tiles; ++i) {
        const uint32_t c = __shfl_sync(0xffffffffu, cnt, i), r0 = __shfl_sync(0xffffffffu, room, i);
        const uint16_t* list = v.o_list + (tb + i) * kOrdTile + __shfl_sync(0xffffffffu, off, i);
        for (uint32_t j0 = 0; j0 < c; j0 += 32) {
          const uint32_t j = j0 + lane;
          const uint64_t s = start + r0 + j;
          const bool cand = j < c && ((__ldg(v.o_dec + ((s >> 5) << 1)) >> (s & 31)) & 1u);
          const uint32_t m = __ballot_sync(0xffffffffu, cand);
          if (cand) {
            const uint32_t at = n + __popc(m & below);
            slot_q[at] = r0 + j;
            ent_q[at] = (uint32_t)(tb + i - t0) << 16 | __ldcs(list + j);
          }
          n += __popc(m);
          if (n >= 32) {
            insert(32);
            n -= 32;
            if ((uint32_t)lane < n) {
              slot_q[lane] = slot_q[lane + 32];
              ent_q[lane] = ent_q[lane + 32];
            }
            __syncwarp();
          }
        }
      }
    }
    insert(n);
  }
}

// Its probe loop: a candidate's junction bit from the mask in the slot kept in
// place of its record (as ord_classify_kernel writes it).
template <int TS>
__global__ void __launch_bounds__(kBlock) ord_classify2_kernel(RunView v) {
  __shared__ uint32_t first_s[kOrdMaxRegions + 1];
  __shared__ uint32_t item_s;
  const uint64_t part = __ldcg(&v.hdr->part_slots);
  if (!ordered_round(v) || !part) return;
  ord_items(v, first_s);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t R = v.o_regions, total = first_s[R];
  for (;;) {
    if (threadIdx.x == 0) item_s = atomicAdd(&v.hdr->ord_ticket[2], 1u);
    __syncthreads();
    const uint32_t item = item_s;
    __syncthreads();
    if (item >= total) break;
    const uint32_t b = ord_item_bucket(first_s, R, item);
    const uint64_t n = __ldcg(v.o_fill + (uint64_t)b * kOrdFillStride);
    const uint64_t i0 = (uint64_t)(item - first_s[b]) * kOrdPiece, i1 = min(i0 + kOrdPiece, n);
    const uint64_t start = __ldg(v.o_start + b);  // a multiple of 32, as is i0
    RunView x = v;
    x.table = static_cast<char*>(v.table) + (uint64_t)b * part * (32 / SectorOf<TS>::kSlots);
    constexpr int U = 4;
    for (uint64_t w0 = i0 + 32 * wid; w0 < i1; w0 += U * kBlock) {
      uint64_t slot[U];
      bool cand[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t c = w0 + (uint64_t)u * kBlock;
        const uint32_t row = c < i1 ? __ldcg(v.o_dec + (((start + c) >> 5) << 1)) : 0u;
        cand[u] = (row >> lane) & 1u;
        slot[u] = cand[u] ? __ldcs(v.o_recs + start + c + lane) : kNoSlot;
      }
      int mk[U];
#pragma unroll
      for (int u = 0; u < U; ++u) mk[u] = slot[u] != kNoSlot ? table_mask<TS>(x, slot[u]) : -1;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t c = w0 + (uint64_t)u * kBlock;
        const uint32_t row = __ballot_sync(0xffffffffu, cand[u] && (mk[u] < 0 || is_junction_mask(mk[u])));
        if (lane == 0 && c < i1) v.o_dec[(((start + c) >> 5) << 1) + 1] = row;
      }
    }
  }
}

// What a tile's decisions leave behind, called by the whole block with the
// tile's candidate, junction and sentinel bits in shared memory: the tile's
// words of C_temp, its junctions (decided) or, partial, its candidates in
// C_final -- a tile has one block and rounds own disjoint positions, so no
// atomic -- or its candidates in the warp's segment of the pass-2 list, in
// position order. Clears the bits for the next tile.
constexpr uint32_t kOrdTileWords = (uint32_t)(kOrdTile / 32);

struct TileOut {
  unsigned long long kept, junctions;
  uint64_t seg_used;
};

__device__ __forceinline__ void ord_tile_out(const RunView& v, uint64_t t, bool decided, uint32_t* keep_s, uint32_t* jun_s,
                                             uint32_t* sent_s, TileOut* o) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t warp_id = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  constexpr uint32_t kPer = kOrdTileWords / (kBlock / 32);  // words per warp
  for (uint32_t w0 = wid * kPer; w0 < (wid + 1) * kPer; w0 += 32) {
    const uint64_t w = t * kOrdTileWords + w0 + lane;
    const uint32_t keep = keep_s[w0 + lane], jun = jun_s[w0 + lane], sent = sent_s[w0 + lane];
    keep_s[w0 + lane] = 0;
    jun_s[w0 + lane] = 0;
    sent_s[w0 + lane] = 0;
    if (w < v.bitmap_words) {
      v.ctemp[w] = keep;
      const uint32_t add = v.partial ? keep : jun;
      if (add) v.cfinal[w] |= add;
    }
    const uint32_t n = __popc(keep);
    o->kept += n;
    o->junctions += __popc(jun);
    if (v.partial || decided) continue;
    uint32_t inc = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += y;
    }
    uint64_t at = o->seg_used + inc - n;
    for (uint32_t x = keep; x; x &= x - 1, ++at) {
      const uint32_t i = __ffs(x) - 1;
      const uint64_t g = w * 32 + i;
      if (at < v.seg_cap) {
        const uint32_t sentinel = (sent >> i) & 1u;
        if (v.narrow) (reinterpret_cast<uint32_t*>(v.cands) + (uint64_t)warp_id * v.seg_cap)[at] = (uint32_t)g | (sentinel << 31);
        else (v.cands + (uint64_t)warp_id * v.seg_cap)[at] = g | ((uint64_t)sentinel << 63);
      }
    }
    o->seg_used += __shfl_sync(0xffffffffu, inc, 31);
  }
}

// The counts and the list segment's length after a block's last tile.
__device__ __forceinline__ void ord_counts_out(const RunView& v, bool decided, const TileOut& o) {
  const uint32_t warp_id = (blockIdx.x * kBlock + threadIdx.x) >> 5;
  if ((threadIdx.x & 31) == 0) {
    v.seg_count[warp_id] = (uint32_t)(o.seg_used < v.seg_cap ? o.seg_used : v.seg_cap);
    if (o.seg_used > v.seg_cap) v.hdr->cand_overflow = 1;
  }
  block_add(o.kept, &v.hdr->pass1_kept);
  if (v.partial) block_add(o.kept, &v.hdr->pass2_kept);
  if (decided) block_add(o.junctions, &v.hdr->pass2_kept);
}

// k-mer positions of a tile: the end of its list.
__device__ __forceinline__ uint32_t ord_tile_positions(const RunView& v, uint64_t t) {
  const uint64_t nh = (uint64_t)v.rounds * v.o_regions;
  return v.o_toff[t * (nh + 1) + nh];
}

// The probe loop's outputs in position order: every member of the round's
// class takes its decision from its record's slot -- the members of a run read
// consecutive bits -- and sets its bits of the tile in shared memory; then the
// tile's words, list entries and counts go out (ord_tile_out).
__global__ void __launch_bounds__(kBlock) tile_gather_kernel(RunView v, int round) {
  __shared__ uint8_t bucket_s[kOrdTile];
  __shared__ unsigned long long delta_s[kOrdMaxRegions];
  __shared__ uint64_t start_s[kOrdMaxRegions];
  __shared__ uint32_t run_s[kOrdMaxRegions];
  __shared__ uint32_t keep_s[kOrdTileWords], jun_s[kOrdTileWords], sent_s[kOrdTileWords];
  if (!ordered_round(v)) return;
  for (uint32_t b = threadIdx.x; b < v.o_regions; b += kBlock) start_s[b] = v.o_start[b];
  for (uint32_t i = threadIdx.x; i < kOrdTileWords; i += kBlock) keep_s[i] = jun_s[i] = sent_s[i] = 0;
  // the junctions are known: pass 2 ran on the records or bucket by bucket
  const bool decided = fused_pass2(v) || __ldcg(&v.hdr->part_slots) != 0;
  const bool listed = !decided && !v.partial;
  TileOut o{0, 0, 0};
  unsigned long long valid_n = 0;
  for (uint64_t t = blockIdx.x; t < v.o_tiles; t += gridDim.x) {
    const TileMembers tm = ord_tile(v, t, round, start_s, delta_s, run_s, bucket_s);
    if (threadIdx.x == 0) valid_n += ord_tile_positions(v, t);
    constexpr int U = 4;
    for (uint32_t i0 = threadIdx.x; i0 < tm.n; i0 += U * kBlock) {
      uint2 d[U];
      uint32_t e[U], bit[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t i = i0 + u * kBlock;
        d[u] = make_uint2(0u, 0u);
        if (i >= tm.n) continue;
        e[u] = __ldcs(tm.list + i);
        const uint64_t s = delta_s[bucket_s[i]] + i;
        bit[u] = (uint32_t)s & 31u;
        if (v.partial) d[u].x = __ldg(v.o_dec + (s >> 5));
        else d[u] = __ldg(reinterpret_cast<const uint2*>(v.o_dec) + (s >> 5));  // candidates, junctions
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (i0 + u * kBlock >= tm.n || !((d[u].x >> bit[u]) & 1u)) continue;  // a junction is a candidate
        const uint32_t pos = e[u] & kOrdEntryPos, m = 1u << (pos & 31u);
        atomicOr(keep_s + (pos >> 5), m);
        if (decided && ((d[u].y >> bit[u]) & 1u)) atomicOr(jun_s + (pos >> 5), m);
        if (listed && (e[u] & kOrdEntrySentinel)) atomicOr(sent_s + (pos >> 5), m);
      }
    }
    __syncthreads();
    ord_tile_out(v, t, decided, keep_s, jun_s, sent_s, &o);
    __syncthreads();  // the shared arrays serve the next tile
  }
  ord_counts_out(v, decided, o);
  if (round == v.count_round) block_add((unsigned long long)valid_n, &v.hdr->positions);
}

// The insert and the probe of a round whose records do not fit their room,
// directly on the filter, over the round's members of every tile's list.
template <int KW, int HB>
__global__ void __launch_bounds__(kBlock) list_insert_kernel(RunView v, int round) {
  if (ordered_round(v)) return;  // the region-ordered kernels took this round
  for (uint64_t t = blockIdx.x; t < v.o_tiles; t += gridDim.x) {
    const uint16_t* toff = v.o_toff + t * ((uint64_t)v.rounds * v.o_regions + 1) + (uint64_t)round * v.o_regions;
    const uint32_t a = toff[0], b = toff[v.o_regions];
    for (uint32_t i = a + threadIdx.x; i < b; i += kBlock) {
      const uint32_t e = v.o_list[t * kOrdTile + i];
      OccT<KW> oc;
      read_listed<KW>(v, t * kOrdTile + (e & kOrdEntryPos), e & kOrdEntrySentinel, &oc);
      const uint64_t G = second_hash(oc.H);
      const ItemPattern pat = item_pattern<HB>(G, v.hashes);
      uint64_t m = item_bits(pat, oc.j1);
      if (oc.j2 != oc.j1) m |= item_bits(pat, oc.j2);  // a palindrome's two orientations
      atomicOr(filter_word(v, oc.H, G), (unsigned long long)m);
    }
  }
}

template <int KW, int HB>
__global__ void __launch_bounds__(kBlock) list_probe_kernel(RunView v, int round) {
  __shared__ uint32_t keep_s[kOrdTileWords], jun_s[kOrdTileWords], sent_s[kOrdTileWords];
  if (ordered_round(v)) return;  // the region-ordered kernels took this round
  for (uint32_t i = threadIdx.x; i < kOrdTileWords; i += kBlock) keep_s[i] = jun_s[i] = sent_s[i] = 0;
  __syncthreads();
  TileOut o{0, 0, 0};
  unsigned long long valid_n = 0;
  for (uint64_t t = blockIdx.x; t < v.o_tiles; t += gridDim.x) {
    const uint16_t* toff = v.o_toff + t * ((uint64_t)v.rounds * v.o_regions + 1) + (uint64_t)round * v.o_regions;
    const uint32_t a = toff[0], b = toff[v.o_regions];
    if (threadIdx.x == 0) valid_n += ord_tile_positions(v, t);
    for (uint32_t i = a + threadIdx.x; i < b; i += kBlock) {
      const uint32_t e = v.o_list[t * kOrdTile + i], pos = e & kOrdEntryPos;
      const bool sentinel = e & kOrdEntrySentinel;
      OccT<KW> oc;
      read_listed<KW>(v, t * kOrdTile + pos, sentinel, &oc);
      const uint64_t G = second_hash(oc.H);
      bool keep = sentinel;
      if (!sentinel) {
        const uint32_t pres = present_items<HB>(G, __ldcg(filter_word(v, oc.H, G)), v.hashes);
        keep = (pres >> 16) || __popc(pres & 0xFFFFu) >= 2;
      }
      if (!keep) continue;
      atomicOr(keep_s + (pos >> 5), 1u << (pos & 31u));
      if (sentinel) atomicOr(sent_s + (pos >> 5), 1u << (pos & 31u));
      if (!v.partial) lc_mark(v, G * kLcMul);
    }
    __syncthreads();
    ord_tile_out(v, t, false, keep_s, jun_s, sent_s, &o);
    __syncthreads();
  }
  ord_counts_out(v, false, o);
  if (!v.partial) block_add(o.kept, &v.hdr->round_kept);
  if (round == v.count_round) block_add((unsigned long long)valid_n, &v.hdr->positions);
}

// Table slots per estimated distinct candidate: 2.5 for one-word slots
// (k <= 27), where probe chains cost more than memory, 2 for the wider slots,
// where a smaller table stays in L2 (measured at k = 25, 31 and 63).
constexpr double kTableLoadWord = 2.5, kTableLoad = 2.0;
// pass-2 list work: parts of about this many records, at most kMaxParts per segment
constexpr unsigned long long kPartRecords = 128, kMaxParts = 4096, kPartWarps = 8192;
// pass 2 bucket by bucket: tables of more than this (several times L2)
constexpr unsigned long long kPartTableBytes = 512ull << 20;

// Size the pass-2 table of this round: 2.5 or 2 times the number of distinct
// candidate k-mers, as the probe's linear counting estimates it (at least 1024
// slots, a multiple of 32, not rounded to a power of two), capped by the
// workspace. A saturated bitmap falls back to the number of candidate
// positions. The estimate only sets the table's size; an undersized table is
// detected and reported, never silently wrong. One block: the sampled bitmap is
// at most 1 MiB, and a grid that counts it and hands the sum to its last block
// took 10-13 us of every round.
template <int TS>
__global__ void __launch_bounds__(1024) table_setup_kernel(RunView v) {
  __shared__ unsigned int part[32];
  DevHeader* h = v.hdr;
  const bool parted = v.o_fused && ordered_round(v);  // the probe inserted into the table's parts
  if (parted && fused_pass2(v)) {  // that was the round's table: nothing to size or clear
    if (threadIdx.x == 0) {
      const unsigned long long used = (unsigned long long)v.o_tcap * v.o_regions;
      h->cand_overflow = 0;
      h->round_kept = 0;
      h->table_slots = 0;
      if (used > h->table_max) h->table_max = used;
    }
    return;
  }
  unsigned int c = 0;
  const uint32_t quads = 1u << (v.lc_log2 - 7);  // of four words; lc_log2 >= 16
#pragma unroll 8
  for (uint32_t i = threadIdx.x; i < quads; i += 1024) {
    const uint4 q = __ldcg(reinterpret_cast<const uint4*>(v.lc_bits) + i);
    c += __popc(q.x) + __popc(q.y) + __popc(q.z) + __popc(q.w);
  }
  c = warp_sum(c);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x != 0) return;
  unsigned long long set = 0;
  for (int w = 0; w < 32; ++w) set += part[w];
  const unsigned long long kept = h->round_kept;
  const unsigned int overflowed = h->cand_overflow;
  h->cand_overflow = 0;
  h->round_kept = 0;
  const double M = (double)(1ull << v.lc_log2);
  unsigned long long distinct = kept;
  if ((double)set < M - M / 1024.0) {  // at least 1/1024 of the bits still clear: about 7 per bit
    // a 2^-s sample of the k-mers was counted: scale it up, with eight standard
    // deviations of the sample's size to spare
    const int sl = v.lc_sample_log2;
    const double f = (double)(1u << sl);
    const double est = -M * log1p(-(double)set / M) * f;
    const unsigned long long e = (unsigned long long)(est * 1.1 + (sl ? 8.0 * sqrt(est * f) : 0.0)) + 64ull;
    if (e < distinct) distinct = e;
  }
  unsigned long long cap =
      (unsigned long long)((v.k <= 27 ? kTableLoadWord : kTableLoad) * (double)distinct);
  if (cap < 1024ull) cap = 1024ull;
  cap = (cap + 31) / 32 * 32;  // any capacity works (slot_start); whole 32-slot groups
  if (v.o_bucketed && ordered_round(v)) {
    // one part per region, of whole sectors: twice the region's share of the
    // estimate and 64 slots, which is more than eight standard deviations of the
    // share on top of it; a reserve without room for that keeps one table (and the
    // candidate list)
    const unsigned long long part = (cap / v.o_regions + 64 + 3) / 4 * 4;
    // worth it where the table is far beyond L2 and the candidates are not a small
    // share of the members, which all have to be looked at. Builds at k = 63, list against
    // parts: a table of 0.5-0.6 GB at shares of 10, 12 and 100% 9.7 to 10.6, 9.9 to 10.7 and
    // 1.59 to 1.26 ms; 100% at 212 and 304 MB 0.66 to 0.73 and 1.10 to 1.02; 14, 19, 27 and 32%
    // at 1.0, 1.8, 3.3 and 4.7 GB 11.0 to 11.3, 12.9 to 12.3, 16.0 to 13.9 and 18.5 to 15.3; 57%
    // at 6 GB 25.5 to 18.5. The two meet near 300 MB and 16%: both lines are on the
    // list's side of that.
    const bool pays = part * v.o_regions * (32 / SectorOf<TS>::kSlots) > kPartTableBytes && 4 * kept >= v.o_start[v.o_regions];
    if (pays && part * v.o_regions <= v.table_max_slots) {
      h->part_slots = part;
      cap = part * v.o_regions;
    }
  }
  // (no estimate in a round whose probe inserted; a part that filled up asks for all there is)
  if (parted || cap > v.table_max_slots) cap = v.table_max_slots;
  h->table_slots = cap;
  if (cap > h->table_max) h->table_max = cap;
  h->round_listed = overflowed ? 0u : 1u;
  // pass 2 cuts every list segment into parts of about kPartRecords records, or
  // down to one row where there are fewer such parts than warps
  unsigned long long parts = (kept / v.n_segments + kPartRecords) / kPartRecords;
  if (parts * v.n_segments < kPartWarps)
    parts = max(parts, min(kept / v.n_segments / 32 + 1, (unsigned long long)(kPartWarps / v.n_segments)));
  h->list_parts = (unsigned int)(parts < kMaxParts ? parts : kMaxParts);
}

template <int TS>
__global__ void __launch_bounds__(kBlock) table_clear_kernel(RunView v) {
  const uint64_t cap = *(volatile unsigned long long*)&v.hdr->table_slots;
  const uint64_t stride = (uint64_t)gridDim.x * kBlock;
  for (uint64_t i = (uint64_t)blockIdx.x * kBlock + threadIdx.x; i < cap; i += stride) {
    if (TS == 0) {
      static_cast<unsigned long long*>(v.table)[i] = kEmpty;
    } else if (TS == 1) {
      Slot1* s = static_cast<Slot1*>(v.table) + i;
      *reinterpret_cast<ulonglong2*>(s) = make_ulonglong2(kEmpty, 0ull);
    } else if (TS == 3) {
      static_cast<unsigned long long*>(v.table)[i] = 0ull;
    } else {
      Slot2* s = static_cast<Slot2*>(v.table) + i;
      reinterpret_cast<ulonglong2*>(s)[0] = make_ulonglong2(kEmpty, kEmpty);
      reinterpret_cast<ulonglong2*>(s)[1] = make_ulonglong2(0ull, 0ull);
    }
  }
}

// Candidate i of the list: its position, and whether it is a sentinel
// position (the record's top bit; 32-bit records when the input has fewer
// than 2^31 bases).
__device__ __forceinline__ uint64_t list_at(const RunView& v, uint64_t i, bool* sentinel, bool last_use) {
  if (v.narrow) {
    const uint32_t* p = reinterpret_cast<const uint32_t*>(v.cands) + i;
    const uint32_t r = last_use ? __ldcs(p) : __ldcg(p);
    *sentinel = r >> 31;
    return r & 0x7FFFFFFFu;
  }
  const uint64_t r = last_use ? __ldcs(v.cands + i) : __ldcg(v.cands + i);
  *sentinel = r >> 63;
  return r & ~(1ull << 63);
}

// Pass-2 work over the candidate list. Every list segment is cut into
// list_parts parts (interleaved 32-record rows), and the launched warps take
// the (segment, part) pairs in turn, so that the work spreads evenly over a
// grid that is resident all at once. fn(i) runs for list index i.
template <typename F>
__device__ __forceinline__ void for_listed(const RunView& v, F&& fn) {
  // 32-bit arithmetic: at most kMaxSegments segments of at most kMaxParts parts
  const uint32_t parts = *(volatile unsigned int*)&v.hdr->list_parts;
  const uint32_t pairs = v.n_segments * parts;
  const uint32_t warps = gridDim.x * (kBlock / 32);
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t w = (blockIdx.x * kBlock + threadIdx.x) >> 5; w < pairs; w += warps) {
    const uint32_t sgm = w / parts, part = w - sgm * parts;
    const uint32_t n = __ldcg(v.seg_count + sgm);
    const uint64_t first = (uint64_t)sgm * v.seg_cap;
    for (uint64_t r = part * 32; r < n; r += 32 * parts) {  // as often for every lane: the warp stays together
      if (r + lane < n) fn(first + r + lane);
      __syncwarp();
    }
  }
}

// for_listed that reads each record one ahead: fn(i, g, sentinel, slot)
// gets list index i with its position (and with SLOT its kept table slot)
// already loaded, while the lane's next record is in flight.
template <bool SLOT, typename F>
__device__ __forceinline__ void for_listed_ahead(const RunView& v, bool last_use, F&& fn) {
  const uint32_t parts = *(volatile unsigned int*)&v.hdr->list_parts;
  const uint32_t pairs = v.n_segments * parts;
  const uint32_t warps = gridDim.x * (kBlock / 32);
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t row = 32 * parts;
  for (uint32_t w = (blockIdx.x * kBlock + threadIdx.x) >> 5; w < pairs; w += warps) {
    const uint32_t sgm = w / parts, part = w - sgm * parts;
    const uint32_t n = __ldcg(v.seg_count + sgm);
    const uint64_t first = (uint64_t)sgm * v.seg_cap;
    uint32_t j = part * 32 + lane;
    bool sent = false;
    uint64_t g = j < n ? list_at(v, first + j, &sent, last_use) : 0;
    uint32_t slot = (SLOT && j < n) ? __ldcs(v.cand_slot + first + j) : 0u;
    while (j < n) {
      const uint32_t jn = j + row;
      bool sent_n = false;
      const uint64_t gn = jn < n ? list_at(v, first + jn, &sent_n, last_use) : 0;
      const uint32_t slot_n = (SLOT && jn < n) ? __ldcs(v.cand_slot + first + jn) : 0u;
      fn(first + j, g, sent, slot);
      j = jn;
      g = gn;
      sent = sent_n;
      slot = slot_n;
    }
  }
}

// Pass 2 of this round ran with the region-ordered kernels.
__device__ __forceinline__ bool pass2_done(const RunView& v) {
  return ordered_round(v) && (fused_pass2(v) || __ldcg(&v.hdr->part_slots) != 0);
}

// Pass 2 reads the list: every candidate of the round is in it (a region-ordered
// round writes its list after table_setup).
__device__ __forceinline__ bool list_complete(const RunView& v) {
  return *(volatile unsigned int*)&v.hdr->round_listed && !*(volatile unsigned int*)&v.hdr->cand_overflow;
}

// Slots tried by an insert into the one table that stands in for full parts: a
// cluster of 2^20 taken slots is to be expected from a load of 0.993 on. A reserve
// too small for the round reports so after this, not after a walk of the whole table
// for every k-mer that finds no room.
constexpr uint64_t kWholeTries = 1ull << 20;

__device__ __forceinline__ bool overflowed(const RunView& v) {
  return *reinterpret_cast<volatile const unsigned int*>(&v.hdr->overflow);
}

// Algorithm 1, insert loop, second pass: every candidate ORs its in/out bases
// (or the sentinel bit) into the exact table entry of its k-mer. Reads the
// candidate list and keeps the slot of each listed candidate for the probe
// loop; if the list overflowed, walks C_temp instead. AFTER_PARTS: of a run whose
// pass 2 goes on the records; this kernel then has the rounds that did not fit and
// those with a full part.
template <int KW, int TS, bool AFTER_PARTS = false>
__global__ void __launch_bounds__(kBlock) pass2_insert_kernel(RunView v) {
  if (pass2_done(v)) return;
  const uint64_t cap = *(volatile unsigned long long*)&v.hdr->table_slots;
  uint64_t tries = cap;
  if (AFTER_PARTS && ordered_round(v)) tries = min(cap, kWholeTries);
  if (list_complete(v)) {
    for_listed(v, [&](uint64_t i) {
      bool sent;
      const uint64_t g = list_at(v, i, &sent, false);
      OccT<KW> oc;
      read_listed<KW>(v, g, sent, &oc);
      uint64_t slot = kNoSlot;
      if (!AFTER_PARTS || !overflowed(v)) slot = insert_occurrence<KW, TS>(v, cap, oc, g, tries);
      if (slot == kNoSlot) v.hdr->overflow = 1;
      if (v.cand_slot) v.cand_slot[i] = slot == kNoSlot ? 0xFFFFFFFFu : (uint32_t)slot;
    });
    return;
  }
  const uint64_t stride = (uint64_t)gridDim.x * kBlock;
  for (uint64_t g = v.p_begin + (uint64_t)blockIdx.x * kBlock + threadIdx.x; g < v.p_end; g += stride) {
    if (!((__ldg(v.ctemp + (g >> 5)) >> (g & 31)) & 1u)) continue;
    if (AFTER_PARTS && overflowed(v)) return;
    OccT<KW> oc;
    if (!read_occurrence<KW>(v, g, &oc)) continue;
    if (insert_occurrence<KW, TS>(v, cap, oc, g, tries) == kNoSlot) v.hdr->overflow = 1;
  }
}

// Algorithm 1, probe loop, second pass: a candidate is a junction iff its
// k-mer is a sentinel or has more than one distinct in- or out-base. Sets
// the junction's bit of C_final (cleared before the first round). A listed
// candidate reads its mask from the slot the insert loop kept (or looks its
// k-mer up when no slots were kept). Records are read one row ahead; two or four rows at a
// time, with a row's bits combined into one atomic per bitmap word, measured
// slower (43 -> 49 us for 5.5 M candidates, 47 -> 62 with 16-byte slots).
template <int KW, int TS>
__global__ void __launch_bounds__(kBlock) pass2_classify_kernel(RunView v) {
  if (pass2_done(v)) return;
  if (v.o_fused && __syncthreads_or(overflowed(v))) return;  // no table to go by
  const uint64_t cap = *(volatile unsigned long long*)&v.hdr->table_slots;
  unsigned long long found = 0;
  auto mark = [&](uint64_t g, int mk) {
    if (mk < 0) v.hdr->overflow = 1;
    if (mk < 0 || is_junction_mask(mk)) {
      atomicOr(v.cfinal + (g >> 5), 1u << (g & 31));
      ++found;
    }
  };
  if (list_complete(v)) {
    auto classify_one = [&](uint64_t, uint64_t g, bool sent, uint32_t slot) {
      if (v.cand_slot) {
        mark(g, slot == 0xFFFFFFFFu ? -1 : table_mask<TS>(v, slot));
      } else {
        OccT<KW> oc;
        read_listed<KW>(v, g, sent, &oc);
        mark(g, find_occurrence<KW, TS>(v, cap, oc));
      }
    };
    if (v.cand_slot) for_listed_ahead<true>(v, true, classify_one);
    else for_listed_ahead<false>(v, true, classify_one);
  } else {
    const uint64_t stride = (uint64_t)gridDim.x * kBlock;
    for (uint64_t g = v.p_begin + (uint64_t)blockIdx.x * kBlock + threadIdx.x; g < v.p_end; g += stride) {
      if (!((__ldg(v.ctemp + (g >> 5)) >> (g & 31)) & 1u)) continue;
      OccT<KW> oc;
      if (!read_occurrence<KW>(v, g, &oc)) continue;
      mark(g, find_occurrence<KW, TS>(v, cap, oc));
    }
  }
  block_add(found, &v.hdr->pass2_kept);
}

// Partition counters (section "Multiple Rounds"): a Bloom pre-pass over all
// k-mers; counter f(k-mer) grows when the k-mer was not yet in the filter. On
// large inputs only a hash-chosen sample of the k-mers of some of the chunks is
// counted (bits of H that neither the bin nor the filter block uses): every bin's
// count then shrinks by the same factor in expectation, which keeps the cut's balance
// while the random filter accesses drop by that factor. What balances the cut is
// the number of k-mers counted, and what a chunk holds is the input's choice: the
// second launch (all) counts the rest where the sample came short of kPartMin k-mers
// a class (1024: a class to 3%), and returns at once otherwise.
template <int KW, int HB>
__global__ void __launch_bounds__(kBlock) partition_count_kernel(RunView v, int all) {
  if (all && __ldcg(&v.hdr->part_counted) >= kPartMin * (unsigned long long)v.rounds) return;
  const uint32_t chunks = all ? v.part_chunks_all : v.part_chunks;
  const uint64_t sample = all ? v.part_sample_all : v.part_sample;
  const uint64_t stride = (uint64_t)gridDim.x * kBlock * kR;
  uint32_t counted = 0;
  for (uint64_t p0 = ((uint64_t)blockIdx.x * kBlock + threadIdx.x) * kR; p0 < v.m; p0 += stride) {
    if ((uint32_t)(p0 >> 16) & chunks) continue;  // a sample of the 64K-position chunks
    walk<KW, kR, true>(v, p0, [&](int, uint64_t, bool valid, const auto& oc) {
      if (!valid || (oc.H & sample)) return;
      const uint64_t G = second_hash(oc.H);
      const uint64_t m = item_bits<HB>(G, 17u, v.hashes);
      unsigned long long* w = filter_word(v, oc.H, G);
      if ((__ldcg(w) & m) == m) return;
      const unsigned long long old = atomicOr(w, (unsigned long long)m);
      if ((old & m) != m) {
        atomicAdd(v.bins + ((uint32_t)oc.H & v.qmask), 1u);
        ++counted;
      }
    });
  }
  if (!all) block_add((unsigned long long)counted, &v.hdr->part_counted);
}

// Greedy class cut over the q counters: class r takes a maximal run of bins
// whose sum stays within (sum of all counters) / rounds, at least one bin,
// leaving one bin for every later class; the last class takes the rest.
__global__ void __launch_bounds__(1024) partition_cut_kernel(RunView v, int rounds, uint64_t* prefix) {
  const uint32_t q = v.qmask + 1u;
  // each thread sums and then scans its own run of bins: one block scan, not one
  // per 1024 bins; the runs' starts stay in shared memory for the search
  __shared__ unsigned long long wsum[32], start_s[1025];
  const uint32_t per = (q + 1023u) / 1024u, i0 = min(q, threadIdx.x * per), i1 = min(q, i0 + per);
  const bool vec = per % 4 == 0;  // whole 16-byte groups (q is a power of two)
  unsigned long long x = 0;
  if (vec) {
#pragma unroll 8
    for (uint32_t i = i0; i < i1; i += 4) {
      const uint4 e = *reinterpret_cast<const uint4*>(v.bins + i);
      x += (unsigned long long)e.x + e.y + e.z + e.w;
    }
  } else {
    for (uint32_t i = i0; i < i1; ++i) x += v.bins[i];
  }
  unsigned long long inc = x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  unsigned long long at = inc - x;
  for (int w = 0; w < wid; ++w) at += wsum[w];
  start_s[threadIdx.x] = at;
  if (threadIdx.x == 1023) start_s[1024] = at + x;
#pragma unroll 8
  for (uint32_t i = i0; i < i1; ++i) {
    prefix[i] = at;
    at += v.bins[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long total = start_s[1024];
    prefix[q] = total;
    const unsigned long long L = (unsigned long long)rounds;
    uint32_t j = 0;
    unsigned long long before = 0;  // prefix[j]
    v.cuts[0] = 0;
    for (int r = 0; r < rounds - 1; ++r) {
      const uint32_t limit = q - (uint32_t)(rounds - 1 - r);
      // largest e in [j + 1, limit] with (prefix[e] - prefix[j]) * L <= total (at least
      // j + 1): first the last run of bins that starts within it, then inside that run
      uint32_t a = 0, z = 1024;  // run a starts within it (or is j's), run z does not or is past the end
      while (z - a > 1) {
        const uint32_t mid = (a + z) / 2;
        if ((uint64_t)mid * per <= j || (start_s[mid] - before) * L <= total) a = mid; else z = mid;
      }
      uint32_t lo = max(j + 1, min(a * per, limit)), hi = min(limit, (a + 1) * per), best = j + 1;
      while (lo <= hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if ((prefix[mid] - before) * L <= total) {
          best = mid;
          lo = mid + 1;
        } else {
          hi = mid - 1;
        }
      }
      j = best;
      before = prefix[j];
      v.cuts[r + 1] = j;
    }
    v.cuts[rounds] = q;
  }
}

// Emit (single pass): tiles of kEmitTileWords bitmap words are claimed in
// order from a ticket; each publishes its junction count, looks back over its
// predecessors for the exclusive prefix (decoupled look-back, Merrill &
// Garland 2016), publishes its inclusive prefix and writes the position of
// every junction within its string, in ascending order (C_final of
// Algorithm 3). Tiles are claimed in order, so every wait is on a block that
// is already running; a wait that exceeds kSpinLimit polls sets the timeout
// flag and gives up (the result is then reported as invalid).
constexpr unsigned long long kFlagAgg = 1ull << 62, kFlagPrefix = 2ull << 62;
constexpr unsigned long long kValMask = (1ull << 62) - 1;
constexpr uint32_t kSpinLimit = 1u << 22;

__global__ void __launch_bounds__(kBlock) emit_kernel(RunView v) {
  __shared__ unsigned long long tile_s, prefix_s, total_s;
  __shared__ uint32_t before_s[kEmitTileWords];  // junctions of the tile before each of its words
  __shared__ uint32_t warp_s[kBlock / 32];
  __shared__ uint16_t stage_s[kBlock / 32][32 * 32];  // one batch's junctions: bit offsets within the tile
  __shared__ uint64_t t_lo_s, t_hi_s;
  volatile unsigned long long* status =
      reinterpret_cast<volatile unsigned long long*>(v.tile_prefix);  // n_tiles entries, zeroed per run
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (;;) {
    if (threadIdx.x == 0) tile_s = atomicAdd(&v.hdr->emit_ticket, 1ull);
    __syncthreads();
    const uint64_t tile = tile_s;
    if (tile >= v.n_tiles) break;
    // warp w takes the tile's words [256 w, 256 w + 256) in kEmitWordsPerThread
    // batches of 32 consecutive words, one word per lane
    const uint64_t tile_base = tile * kEmitTileWords;
    const uint32_t wbase = (uint32_t)wid * 32 * kEmitWordsPerThread;
    uint32_t words[kEmitWordsPerThread];
    uint32_t c = 0;
#pragma unroll
    for (int q = 0; q < kEmitWordsPerThread; ++q) {
      const uint64_t w = tile_base + wbase + 32 * q + lane;
      words[q] = w < v.bitmap_words ? __ldcg(v.cfinal + w) : 0u;
      c += __popc(words[q]);
    }
    c = warp_sum(c);
    if (lane == 0) warp_s[wid] = c;
    __syncthreads();
    if (wid == 0) {
      uint32_t tot = 0, mine = 0;
#pragma unroll
      for (int w = 0; w < kBlock / 32; ++w) {
        const uint32_t x = warp_s[w];
        if (lane == w) mine = tot;
        tot += x;
      }
      __syncwarp();
      if (lane < kBlock / 32) warp_s[lane] = mine;
      // the look-back, 32 tiles at a time: a lane per tile, down to the nearest
      // one that has published its prefix (one tile at a time, the last tiles of
      // a short run walked hundreds of round trips: 30 us for 35 M positions, 25
      // so; 128 tiles at a time waited for more of them and took 33)
      unsigned long long prefix = 0;
      if (lane == 0) {
        if (tile == 0) status[0] = kFlagPrefix | tot;
        else status[tile] = kFlagAgg | tot;
      }
      uint32_t spins = 0;
      for (int64_t j = (int64_t)tile - 1; j >= 0;) {
        const int64_t i = j - lane;
        unsigned long long st = kFlagPrefix;  // before tile 0: an empty prefix
        if (i >= 0) st = status[i];
        const uint32_t done_m = __ballot_sync(0xffffffffu, (st & kFlagPrefix) != 0);
        const uint32_t none_m = __ballot_sync(0xffffffffu, st == 0);
        const int p = done_m ? __ffs(done_m) - 1 : 31;  // the nearest prefix ends the walk
        if (none_m & ((2u << p) - 1u)) {  // a tile up to there has not published yet
          if (++spins > kSpinLimit) {
            if (lane == 0) v.hdr->timeout = 1;
            break;
          }
          __nanosleep(32);
          continue;
        }
        unsigned long long x = lane <= p ? st & kValMask : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        prefix += x;
        if (done_m) break;
        j -= 32;
      }
      if (lane == 0) {
        if (tile) status[tile] = kFlagPrefix | (prefix + tot);
        total_s = tot;
        prefix_s = prefix;
      }
    } else if (wid == 1 && lane < 2) {
      // meanwhile, the strings that start in this tile (the last tile also takes t = n_seqs)
      const uint64_t g = lane == 0 ? tile_base * 32
                                   : (tile + 1 == v.n_tiles ? ~0ull : (tile_base + kEmitTileWords) * 32);
      uint64_t lo = 0, hi = (uint64_t)v.n_seqs + 1;  // first t in [0, n_seqs + 1) with offsets[t] >= g
      while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (__ldg(v.offsets + mid) < g) lo = mid + 1; else hi = mid;
      }
      if (lane == 0) t_lo_s = lo;
      else t_hi_s = lo;
    }
    __syncthreads();
    // batch by batch: every lane expands its word into the warp's stage at its
    // exclusive prefix, then the warp writes the batch with consecutive lanes
    // on consecutive entries
    uint32_t at = warp_s[wid];  // junctions of the tile before this batch
    uint16_t* stage = stage_s[wid];
    Bounds bd{1, 0};
#pragma unroll
    for (int q = 0; q < kEmitWordsPerThread; ++q) {
      const uint32_t n = __popc(words[q]);
      uint32_t inc = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      const uint32_t word_at = wbase + 32 * q + lane;  // the word's index within the tile
      before_s[word_at] = at + inc - n;
      uint32_t bits = words[q], i = inc - n;
      while (bits) {
        const uint32_t b = __ffs(bits) - 1;
        bits &= bits - 1;
        stage[i++] = (uint16_t)(word_at * 32 + b);  // below 2^16: a tile is 65536 positions
      }
      const uint32_t batch = __shfl_sync(0xffffffffu, inc, 31);
      __syncwarp();
      const uint64_t o0 = prefix_s + at;
      for (uint32_t e = lane; e < batch; e += 32) {
        const uint64_t g = tile_base * 32 + stage[e];
        if (g < bd.start || g >= bd.end) bd = seq_bounds(v, g);
        if (o0 + e < v.out_capacity) v.out_positions[o0 + e] = g - bd.start;
      }
      __syncwarp();
      at += batch;
    }
    // out_offsets[t] (junctions before string t) for the strings that start in
    // this tile; the last tile also takes t = n_seqs (start m: the total)
    __syncthreads();
    for (uint64_t t = t_lo_s + threadIdx.x; t < t_hi_s; t += kBlock) {
      const uint64_t g = __ldg(v.offsets + t), w = g >> 5, j = w - tile_base;
      unsigned long long cnt = prefix_s + (j < (uint64_t)kEmitTileWords ? before_s[j] : total_s);
      if ((g & 31) && w < v.bitmap_words) cnt += __popc(__ldcg(v.cfinal + w) & ((1u << (g & 31)) - 1u));
      v.out_offsets[t] = cnt;
      if (t == v.n_seqs && cnt > v.out_capacity) v.hdr->out_overflow = 1;
    }
    __syncthreads();
  }
}

// offsets[t] = junctions in strings before t (one block per string); the
// last entry is the total, checked against the output's capacity. Only runs
// without input use it: otherwise the emit kernel writes the offsets.
__global__ void __launch_bounds__(kBlock) emit_offsets_kernel(RunView v) {
  const uint64_t t = blockIdx.x;
  const uint64_t g = (t == v.n_seqs) ? v.m : __ldg(v.offsets + t);
  const uint64_t w = g >> 5;
  const uint64_t tile = w / kEmitTileWords;
  unsigned long long cnt = 0;
  for (uint64_t x = tile * kEmitTileWords + threadIdx.x; x < w; x += kBlock) cnt += __popc(__ldcg(v.cfinal + x));
  __shared__ unsigned long long part[kBlock / 32];
  cnt = warp_sum(cnt);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    cnt = 0;
    for (int i = 0; i < kBlock / 32; ++i) cnt += part[i];
    if (tile > 0) cnt += __ldcg(reinterpret_cast<const unsigned long long*>(v.tile_prefix) + (tile - 1)) & kValMask;
    if (g & 31) cnt += __popc(__ldcg(v.cfinal + w) & ((1u << (g & 31)) - 1u));
    v.out_offsets[t] = cnt;
    if (t == v.n_seqs && cnt > v.out_capacity) v.hdr->out_overflow = 1;
  }
}

// ---------------------------------------------------------------------------
// Compacted-graph edges (section "Reduction to the Problem of Finding
// Junction Positions"): consecutive junction positions of a string.
// ---------------------------------------------------------------------------

struct EdgeOut {  // layout of twopaco_edge
  unsigned long long from_hi, from_lo, to_hi, to_lo, start, length;
  unsigned int from_rc, to_rc;
};

// With N splitting no edge crosses an N. Every piece of at least k bases
// holds a junction (its first k-mer is a sentinel), so a string with j
// junctions spread over r such pieces has j - r edges: one fewer per piece.
// run_rank[j] = pieces of at least k bases among runs[0 .. j) (one block).
__global__ void __launch_bounds__(1024) runs_rank_kernel(const DevHeader* hdr) {
  __shared__ unsigned int wsum[32];
  __shared__ unsigned int carry_s;
  if (!hdr->nmask) return;  // the run did not split at N
  const uint64_t n = hdr->n_runs;
  const uint64_t* runs = hdr->runs;
  const uint32_t* nmask = hdr->nmask;
  uint32_t* rank = hdr->run_rank;
  const uint64_t k = (uint64_t)hdr->k;
  if (threadIdx.x == 0) carry_s = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (uint64_t base = 0; base < n; base += 1024) {
    const uint64_t j = base + threadIdx.x;
    unsigned int x = 0;
    if (j < n) {
      const uint64_t a = runs[j], b = runs[j + 1];
      x = (!((nmask[a >> 5] >> (a & 31)) & 1u) && b - a >= k) ? 1u : 0u;
    }
    unsigned int inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    unsigned int before = 0, all = 0;
    for (int w = 0; w < 32; ++w) {
      before += (w < wid) ? wsum[w] : 0u;
      all += wsum[w];
    }
    const unsigned int c0 = carry_s;
    if (j < n) rank[j] = c0 + before + inc - x;
    __syncthreads();
    if (threadIdx.x == 0) carry_s = c0 + all;
    __syncthreads();
  }
  if (threadIdx.x == 0) rank[n] = carry_s;
}

// First j in [0, n] with runs[j] >= g (runs[n] = m).
__device__ __forceinline__ uint64_t runs_lower_bound(const uint64_t* runs, uint64_t n, uint64_t g) {
  uint64_t lo = 0, hi = n;
  while (lo < hi) {
    const uint64_t mid = (lo + hi) >> 1;
    if (runs[mid] < g) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Pieces of at least k bases in string t (N splitting).
__device__ __forceinline__ uint64_t long_pieces(const DevHeader* hdr, const uint64_t* offsets, uint64_t t) {
  const uint64_t n = hdr->n_runs;
  const uint64_t lo = runs_lower_bound(hdr->runs, n, offsets[t]);
  const uint64_t hi = runs_lower_bound(hdr->runs, n, offsets[t + 1]);
  return (uint64_t)hdr->run_rank[hi] - hdr->run_rank[lo];
}

// edge_offsets[t] = sum over strings before t of their edges: junctions - 1
// (none for a string without junctions), or junctions - pieces with N splitting.
__global__ void __launch_bounds__(1024) edge_offsets_kernel(const DevHeader* hdr, const uint64_t* offsets,
                                                            const uint64_t* out_off, uint64_t n_seqs,
                                                            uint64_t* edge_off, uint64_t capacity) {
  __shared__ unsigned long long wsum[32];
  __shared__ unsigned long long carry_s;
  if (threadIdx.x == 0) carry_s = 0;
  __syncthreads();
  const bool split = hdr->nmask != nullptr;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (uint64_t base = 0; base < n_seqs; base += 1024) {
    const uint64_t t = base + threadIdx.x;
    unsigned long long x = 0;
    if (t < n_seqs) {
      const unsigned long long j = out_off[t + 1] - out_off[t];
      if (split) x = j - long_pieces(hdr, offsets, t);
      else x = j ? j - 1 : 0;
    }
    unsigned long long inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    unsigned long long before = 0, all = 0;
    for (int w = 0; w < 32; ++w) {
      before += (w < wid) ? wsum[w] : 0ull;
      all += wsum[w];
    }
    const unsigned long long c0 = carry_s;
    if (t < n_seqs) edge_off[t] = c0 + before + inc - x;
    __syncthreads();
    if (threadIdx.x == 0) carry_s = c0 + all;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    edge_off[n_seqs] = carry_s;
    if (carry_s > capacity) const_cast<DevHeader*>(hdr)->overflow = 1;
  }
}

// The normalized k-mer at g (for k > 63 its 128 least significant bits, the
// last 64 bases) and whether the string reads its reverse complement.
template <int KW>
__device__ __forceinline__ void edge_vertex(const uint32_t* packed, uint64_t g, int k, int both,
                                            unsigned long long* hi, unsigned long long* lo,
                                            unsigned int* rc) {
  const KeyT<KW> f = load_kmer<KW>(packed, g, k);
  const KeyT<KW> r = both ? revcomp<KW>(f, k) : f;
  const bool use_r = both && key_less(r, f);
  const KeyT<KW>& x = use_r ? r : f;
  if constexpr (KW == 4) {
    *hi = x.w[2];
    *lo = x.w[3];
  } else {
    *hi = x.hi;
    *lo = x.lo;
  }
  *rc = use_r ? 1u : 0u;
}

// One lane per junction: the edge from it to the next junction of its
// string (with N splitting: of its piece; the last junction of a piece has
// none, and the edges of later pieces move down by one per earlier piece).
// A junction's k-mer is read once: the edge's end is the next lane's start. A
// warp's edges go through shared memory and out word by word, consecutive lanes
// on consecutive words -- written by their own lanes, 56 bytes apart, each of the
// seven stores touched 32 sectors (84 us for 2.7 M edges, 150 MB).
constexpr int kEdgeWords = (int)(sizeof(EdgeOut) / 8);
static_assert(sizeof(EdgeOut) == 56, "seven words");

__device__ __forceinline__ void edge_vertex_of(const uint32_t* packed, uint64_t g, int k, int both,
                                               unsigned long long* hi, unsigned long long* lo, unsigned int* rc) {
  if (k <= 31) edge_vertex<1>(packed, g, k, both, hi, lo, rc);
  else if (k <= 63) edge_vertex<2>(packed, g, k, both, hi, lo, rc);
  else edge_vertex<4>(packed, g, k, both, hi, lo, rc);
}

__global__ void __launch_bounds__(kBlock) edges_kernel(const DevHeader* hdr, const uint64_t* offsets,
                                                      uint64_t n_seqs, const uint64_t* out_off,
                                                      const uint64_t* out_pos, const uint64_t* edge_off,
                                                      EdgeOut* edges, uint64_t capacity) {
  __shared__ unsigned long long word_s[kBlock / 32][32 * kEdgeWords];
  __shared__ unsigned long long at_s[kBlock / 32][32];  // the edge's index, or ~0
  const uint32_t* packed = hdr->packed;
  const int k = hdr->k, both = hdr->both;
  const bool split = hdr->nmask != nullptr;
  const uint64_t total = out_off[n_seqs];
  const uint64_t stride = (uint64_t)gridDim.x * kBlock;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (uint64_t i0 = (uint64_t)blockIdx.x * kBlock + (threadIdx.x & ~31u); i0 < total; i0 += stride) {
    const uint64_t i = i0 + lane;
    const bool here = i < total;
    // the largest t with out_off[t] <= i: the warp's first junction's, or a later string's
    uint64_t t = 0;
    {
      uint64_t lo = 0, hi = n_seqs;
      while (hi - lo > 1) {
        const uint64_t mid = (lo + hi) >> 1;
        if (__ldg(out_off + mid) <= i0) lo = mid; else hi = mid;
      }
      t = lo;
      if (here && __ldg(out_off + t + 1) <= i) {
        hi = n_seqs;
        while (hi - lo > 1) {
          const uint64_t mid = (lo + hi) >> 1;
          if (__ldg(out_off + mid) <= i) lo = mid; else hi = mid;
        }
        t = lo;
      }
    }
    EdgeOut o{};
    uint64_t e = ~0ull, p = 0, g0 = 0;
    if (here) {
      p = out_pos[i];
      g0 = __ldg(offsets + t);
      edge_vertex_of(packed, g0 + p, k, both, &o.from_hi, &o.from_lo, &o.from_rc);
    }
    // the next junction: the next lane's, or read for the last lane
    uint64_t q = __shfl_down_sync(0xffffffffu, p, 1);
    o.to_hi = __shfl_down_sync(0xffffffffu, o.from_hi, 1);
    o.to_lo = __shfl_down_sync(0xffffffffu, o.from_lo, 1);
    o.to_rc = __shfl_down_sync(0xffffffffu, o.from_rc, 1);
    if (here) {
      const uint64_t first = __ldg(out_off + t), a = i - first;
      if (a + 1 < __ldg(out_off + t + 1) - first) {  // not the string's last junction
        if (lane == 31) {
          q = out_pos[i + 1];
          edge_vertex_of(packed, g0 + q, k, both, &o.to_hi, &o.to_lo, &o.to_rc);
        }
        e = edge_off[t] + a;
        if (split) {
          const uint64_t n = hdr->n_runs;
          const uint64_t jr = runs_lower_bound(hdr->runs, n, g0 + p + 1) - 1;  // the piece holding p
          if (hdr->runs[jr + 1] < g0 + q + (uint64_t)k) {
            e = ~0ull;  // q lies in a later piece
          } else {
            const uint64_t run0 = runs_lower_bound(hdr->runs, n, g0);
            e -= (uint64_t)hdr->run_rank[jr] - hdr->run_rank[run0];
          }
        }
      }
    }
    o.start = p;
    o.length = q - p;
    at_s[wid][lane] = e < capacity ? e : ~0ull;
    unsigned long long* w = word_s[wid] + lane * kEdgeWords;
    w[0] = o.from_hi;
    w[1] = o.from_lo;
    w[2] = o.to_hi;
    w[3] = o.to_lo;
    w[4] = o.start;
    w[5] = o.length;
    w[6] = (unsigned long long)o.from_rc | ((unsigned long long)o.to_rc << 32);
    __syncwarp();
    unsigned long long* out = reinterpret_cast<unsigned long long*>(edges);
#pragma unroll
    for (int x = 0; x < kEdgeWords; ++x) {
      const int y = 32 * x + lane, row = y / kEdgeWords;
      const unsigned long long at = at_s[wid][row];
      if (at != ~0ull) out[at * kEdgeWords + (y - row * kEdgeWords)] = word_s[wid][y];
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Launch helpers
// ---------------------------------------------------------------------------

// SMs and resident blocks per SM of a kernel: asked for once per kernel and
// device (three runtime calls before every launch cost more host time than the
// launch). Packed as SMs << 32 | blocks; devices past the table ask every time.
template <typename K>
uint64_t resident_blocks(K kernel, int block, size_t dyn_smem) {
  struct Known {
    std::atomic<const void*> kernel{nullptr};
    std::atomic<uint64_t> value{0};
  };
  constexpr int kDevices = 16, kKernels = 64;
  static Known known[kDevices][kKernels];  // one table per kernel signature
  int dev = 0;
  cudaGetDevice(&dev);
  const void* key = reinterpret_cast<const void*>(kernel);
  Known* at = nullptr;
  if (dev >= 0 && dev < kDevices) {
    for (int i = 0; i < kKernels; ++i) {
      const void* k = known[dev][i].kernel.load(std::memory_order_acquire);
      if (k == key) {
        const uint64_t v = known[dev][i].value.load(std::memory_order_acquire);
        if (v) return v;
        at = &known[dev][i];
        break;
      }
      if (!k) {
        if (known[dev][i].kernel.compare_exchange_strong(k, key) || k == key) {
          at = &known[dev][i];
          break;
        }
      }
    }
  }
  int per_sm = 0, sms = 0;
  const bool known_now =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, dyn_smem) == cudaSuccess &&
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && per_sm > 0 && sms > 0;
  const uint64_t v = ((uint64_t)std::max(sms, 1) << 32) | (uint32_t)std::max(per_sm, 1);
  if (at && known_now) at->value.store(v, std::memory_order_release);  // the same from any thread
  return v;
}

// Grid of at most (SMs x resident blocks per SM) blocks for work_items threads.
// (A kernel is always launched with the same block size and dynamic memory.)
template <typename K>
unsigned grid_for(K kernel, int block, uint64_t work_items, int cap_per_sm = 0, size_t dyn_smem = 0) {
  const uint64_t known = resident_blocks(kernel, block, dyn_smem);
  int per_sm = (int)(uint32_t)known;
  if (cap_per_sm > 0 && per_sm > cap_per_sm) per_sm = cap_per_sm;  // a chosen launch shape
  const uint64_t full = (known >> 32) * per_sm;
  const uint64_t need = (work_items + block - 1) / block;
  return (unsigned)(need < full ? (need ? need : 1) : full);
}

int done(int n) {
  if (cudaPeekAtLastError() != cudaSuccess) return -1;
  count_launches(n);
  return n;
}

}  // namespace

#ifndef TWOPACO_PART
void count_launches(int n) { g_launches.fetch_add((unsigned long long)n); }
unsigned long long launches_so_far() { return g_launches.load(); }

int launch_init(const RunView& v, cudaStream_t s) {
  return cudaMemsetAsync(v.hdr, 0, sizeof(DevHeader), s) == cudaSuccess ? 0 : -1;
}

int launch_digest(DevHeader* hdr_dev, const uint32_t* packed, uint64_t words, const uint64_t* offsets,
                  uint64_t n_seqs, const uint32_t* nmask, uint64_t nmask_words, cudaStream_t s) {
  if (cudaMemsetAsync(&hdr_dev->input_digest, 0, sizeof(unsigned long long), s) != cudaSuccess) return -1;
  digest_kernel<<<grid_for(digest_kernel, kBlock, words), kBlock, 0, s>>>(hdr_dev, packed, words, offsets,
                                                                         n_seqs + 1, nmask, nmask_words);
  return done(1);
}

int launch_pack(const RunView& v, cudaStream_t s) {
  if (launch_pack_chunk(v, 0, v.packed_words, true, s) < 0) return -1;
  return launch_pack_finish(v, s);
}

int launch_pack_chunk(const RunView& v, uint64_t w_begin, uint64_t w_end, bool first, cudaStream_t s) {
  Timed t("pack", s);
  pack_kernel<<<grid_for(pack_kernel, kBlock, (w_end - w_begin + 3) / 4), kBlock, 0, s>>>(v, w_begin, w_end,
                                                                                          first ? 1 : 0);
  return done(1);
}

int launch_pack_finish(const RunView& v, cudaStream_t s) {
  if (!v.nmask || v.m == 0) return 0;
  {
    Timed t("runs", s);
    runs_mark_kernel<<<grid_for(runs_mark_kernel, kBlock, v.bitmap_words), kBlock, 0, s>>>(v);
    runs_starts_kernel<<<grid_for(runs_starts_kernel, kBlock, v.n_seqs), kBlock, 0, s>>>(v);
    const unsigned gc = grid_for(runs_count_kernel, kBlock, v.n_chunks * kBlock);
    runs_count_kernel<<<gc, kBlock, 0, s>>>(v);
    runs_scan_kernel<<<1, 1024, 0, s>>>(v);
    runs_write_kernel<<<grid_for(runs_write_kernel, kBlock, v.n_chunks * kBlock), kBlock, 0, s>>>(v);
  }
  return done(5);
}

#else   // TWOPACO_PART

constexpr int kPartKw = TWOPACO_PART == 5 ? 4 : (TWOPACO_PART <= 2 ? 1 : 2);
constexpr bool kPartHigh = TWOPACO_PART == 2 || TWOPACO_PART == 4;

// Run f with the filter's bits per item as a compile-time constant (0 at
// k > 63: a run-time value).
template <typename F>
static void with_hashes(int h, F&& f) {
  if constexpr (kPartKw == 4) {
    f(std::integral_constant<int, 0>{});
  } else {
    constexpr int B = kPartHigh ? 4 : 0;
    switch (h - B) {
      case 1: f(std::integral_constant<int, B + 1>{}); break;
      case 2: f(std::integral_constant<int, B + 2>{}); break;
      case 3: f(std::integral_constant<int, B + 3>{}); break;
      default: f(std::integral_constant<int, B + 4>{}); break;
    }
  }
}

// The pass-2 table of a round, sized and cleared.
template <int TS>
static void launch_table(const RunView& v, cudaStream_t s) {
  {
    Timed t("table_setup", s);
    table_setup_kernel<TS><<<1, 1024, 0, s>>>(v);
  }
  {
    Timed t("table_clear", s);
    table_clear_kernel<TS><<<grid_for(table_clear_kernel<TS>, kBlock, v.table_max_slots), kBlock, 0, s>>>(v);
  }
}

// A round's first pass in filter-region order, and its second on the records or
// bucket by bucket:
// launches every kernel of it up to the candidate list's pass 2; *pv gets the
// list segments. Kernels launched, or -1.
template <int KW, int HB, int TS>
static int ordered_round_impl(const RunView& v, int round, cudaStream_t s, RunView* pv) {
  const bool fused = KW == 1 && v.o_fused;
  {
    Timed t("ord_rooms", s);
    const uint64_t chunks = (v.o_tiles + kOrdScanTiles - 1) / kOrdScanTiles;
    ord_room_sum_kernel<<<(unsigned)chunks, kBlock, 0, s>>>(v, round);
    ord_room_prefix_kernel<<<v.o_regions, kBlock, 0, s>>>(v, chunks);
    ord_room_scan_kernel<<<(unsigned)chunks, kBlock, 0, s>>>(v, round);
    ord_setup_kernel<<<1, kBlock, 0, s>>>(v, round);
  }
  {
    Timed t("tile_scatter", s);
    auto kern = tile_scatter_kernel<KW, HB, false>;
    if constexpr (KW == 1)
      if (fused) kern = tile_scatter_kernel<KW, HB, true>;
    kern<<<grid_for(kern, kBlock, v.o_tiles * kBlock, v.blocks_per_sm), kBlock, 0, s>>>(v, round);
  }
  {
    Timed t("ord_or", s);
    auto kern = fused ? ord_or_kernel<HB, true> : ord_or_kernel<HB, false>;
    kern<<<grid_for(kern, kBlock, ~0ull >> 1), kBlock, 0, s>>>(v);
  }
  {
    Timed t("list_insert", s);
    auto kern = list_insert_kernel<KW, HB>;
    kern<<<grid_for(kern, kBlock, v.o_tiles * kBlock, v.blocks_per_sm), kBlock, 0, s>>>(v, round);
  }
  // one candidate-list segment per warp of the gather (and of the direct probe)
  unsigned grid = std::min(grid_for(tile_gather_kernel, kBlock, v.o_tiles * kBlock, v.blocks_per_sm),
                           grid_for(list_probe_kernel<KW, HB>, kBlock, v.o_tiles * kBlock, v.blocks_per_sm));
  grid = std::min(grid, (unsigned)(kMaxSegments / (kBlock / 32)));
  pv->n_segments = grid * (kBlock / 32);
  pv->seg_cap = (v.narrow ? 2 * v.cand_cap : v.cand_cap) / pv->n_segments;
  if (fused && cudaMemsetAsync(v.table, 0xFF, (uint64_t)v.o_tcap * v.o_regions * 8, s) != cudaSuccess)
    return -1;  // every fused table slot empty (all ones)
  {
    Timed t("ord_probe", s);
    auto kern = fused ? ord_probe_kernel<HB, true> : ord_probe_kernel<HB, false>;
    kern<<<grid_for(kern, kBlock, ~0ull >> 1), kBlock, 0, s>>>(v);
  }
  if (fused) {
    Timed t("ord_classify", s);
    ord_classify_kernel<<<grid_for(ord_classify_kernel, kBlock, ~0ull >> 1), kBlock, 0, s>>>(v);
  }
  {
    Timed t("list_probe", s);
    list_probe_kernel<KW, HB><<<grid, kBlock, 0, s>>>(*pv, round);
  }
  int launched = fused ? 10 : 9;
  if (!v.partial) {
    launch_table<TS>(*pv, s);
    launched += 2;
    if constexpr (KW == 2) {
      {
        Timed t("ord_insert2", s);
        auto kern = ord_insert2_kernel<KW, TS>;
        kern<<<grid_for(kern, kBlock, ~0ull >> 1), kBlock, 0, s>>>(*pv, round);
      }
      {
        Timed t("ord_classify2", s);
        auto kern = ord_classify2_kernel<TS>;
        kern<<<grid_for(kern, kBlock, ~0ull >> 1), kBlock, 0, s>>>(*pv);
      }
      launched += 2;
    }
  }
  {
    Timed t("tile_gather", s);
    tile_gather_kernel<<<grid, kBlock, 0, s>>>(*pv, round);
  }
  return launched + 1;
}

template <int KW, bool RD, int HB, int TS>
static int round_impl(const RunView& v, int round, cudaStream_t s, const Ranges* ranges) {
  // the pack kernel cleared the filter and the LC bitmap for round 0; the
  // partition pre-pass (rounds > 1) uses the filter before round 0
  if (RD && cudaMemsetAsync(v.filter, 0, v.filter_words64 * 8, s) != cudaSuccess) return -1;
  if (round > 0 && cudaMemsetAsync(v.lc_bits, 0, (1ull << v.lc_log2) / 8, s) != cudaSuccess) return -1;
  constexpr bool kDescOk = HB <= 6;
  constexpr bool kOrdOk = HB >= 1 && HB <= 6 && KW <= 2;  // a record carries the bit bases of up to 6 bits per item
  const bool ord = kOrdOk && v.o_regions > 0;  // region-ordered first pass, over the sorted tiles
  const bool cm = RD && v.cmap != nullptr;     // rounds visit only their class's positions
  const bool desc = !cm && !ord && kDescOk && v.use_desc;
  // every loop over all positions at once, or once per string (ranges)
  const Ranges whole{{v.p_begin, v.p_end}};
  const Ranges& rs = ranges ? *ranges : whole;
  auto part = [&](const std::pair<uint64_t, uint64_t>& r) {
    RunView x = v;
    x.p_begin = r.first;
    x.p_end = r.second;
    return x;
  };
  int launched = 0;
  RunView pv = v;
  // region buckets for the inserts alone, chunk by chunk
  constexpr bool kBktOk = HB <= 6;  // a record carries the bit bases of up to 6 bits per item
  constexpr int HBO = kBktOk ? HB : 1;
  const bool bkt = kBktOk && v.n_regions > 0;
  if constexpr (kOrdOk) {
    if (ord) {
      const int n = ordered_round_impl<KW, HB, TS>(v, round, s, &pv);
      if (n < 0) return -1;
      launched += n;
    }
  }
  if (!ord) {
    for (const auto& r : rs) {
      const uint64_t step = bkt ? v.bucket_chunk : r.second - r.first;
      for (uint64_t c0 = r.first; c0 < r.second; c0 += step) {
        const RunView x = part({c0, std::min(r.second, c0 + step)});
        const uint64_t threads = (x.p_end - x.p_begin + kInsertR - 1) / kInsertR;
        constexpr int kSmallR = !RD ? kInsertSmallR : kInsertR;  // one round
        const bool small = kSmallR < kInsertR && x.p_end - x.p_begin < kInsertSmall;
        auto launch_insert = [&](auto kern, int r) {
          const uint64_t n = (x.p_end - x.p_begin + r - 1) / r;
          kern<<<grid_for(kern, kBlock, n, v.blocks_per_sm), kBlock, 0, s>>>(x, round);
        };
        {
        Timed t("pass1_insert", s);
        if (bkt && cudaMemsetAsync(v.bucket_fill, 0, ((uint64_t)v.n_regions * v.n_sub + 1) * kFillStride * 4,
                                   s) != cudaSuccess)
          return -1;
        if (cm && bkt)
          pass1_insert_cm_kernel<KW, HB, kBktOk><<<grid_for(pass1_insert_cm_kernel<KW, HB, kBktOk>, kBlock, threads, v.blocks_per_sm),
                                                   kBlock, 0, s>>>(x, round);
        else if (cm)
          pass1_insert_cm_kernel<KW, HB><<<grid_for(pass1_insert_cm_kernel<KW, HB>, kBlock, threads, v.blocks_per_sm), kBlock, 0,
                                           s>>>(x, round);
        else if (desc && bkt)
          pass1_insert_kernel<KW, RD, HB, kDescOk, kBktOk>
              <<<grid_for(pass1_insert_kernel<KW, RD, HB, kDescOk, kBktOk>, kBlock, threads, v.blocks_per_sm), kBlock, 0, s>>>(x, round);
        else if (desc && small)
          launch_insert(pass1_insert_kernel<KW, RD, HB, kDescOk, false, kSmallR>, kSmallR);
        else if (desc)
          launch_insert(pass1_insert_kernel<KW, RD, HB, kDescOk>, kInsertR);
        else if (bkt)
          pass1_insert_kernel<KW, RD, HB, false, kBktOk>
              <<<grid_for(pass1_insert_kernel<KW, RD, HB, false, kBktOk>, kBlock, threads, v.blocks_per_sm), kBlock, 0, s>>>(x, round);
        else if (small)
          launch_insert(pass1_insert_kernel<KW, RD, HB, false, false, kSmallR>, kSmallR);
        else
          launch_insert(pass1_insert_kernel<KW, RD, HB, false>, kInsertR);
        }
        ++launched;
        if (bkt) {
          Timed ta("filter_apply", s);
          filter_apply_kernel<kBktOk ? HB : 1><<<grid_for(filter_apply_kernel<kBktOk ? HB : 1>, kBlock, ~0ull >> 1),
                                                 kBlock, 0, s>>>(v);
          ++launched;
        }
      }
    }
  }
  for (const auto& r : rs) {
    if (ord) break;  // its segments are laid out
    pv = part(r);
    const uint64_t threads = (r.second - r.first + kProbeR - 1) / kProbeR;
    // one candidate-list segment per probe warp
    unsigned grid = cm     ? grid_for(pass1_probe_cm_kernel<KW, HB>, kBlock, (r.second - r.first + 15) / 16, v.blocks_per_sm)
                    : desc ? grid_for(pass1_probe_desc_kernel<kDescOk ? HB : 1>, kBlock, threads, v.blocks_per_sm)
                           : grid_for(pass1_probe_kernel<KW, RD, HB>, kBlock, threads, v.blocks_per_sm);
    if (grid * (kBlock / 32) > kMaxSegments) grid = kMaxSegments / (kBlock / 32);
    pv.n_segments = grid * (kBlock / 32);
    // the list region holds cand_cap 8-byte records, or twice as many 32-bit
    // ones; launched per string there is no list (pass 2 walks C_temp)
    pv.seg_cap = ranges ? 0 : (v.narrow ? 2 * v.cand_cap : v.cand_cap) / pv.n_segments;
    Timed t("pass1_probe", s);
    if (cm) pass1_probe_cm_kernel<KW, HB><<<grid, kBlock, 0, s>>>(pv, round);
    else if (desc) pass1_probe_desc_kernel<kDescOk ? HB : 1><<<grid, kBlock, 0, s>>>(pv, round);
    else pass1_probe_kernel<KW, RD, HB><<<grid, kBlock, 0, s>>>(pv, round);
    ++launched;
  }
  if (v.partial) return done(launched);  // the partially compacted graph: no second pass
  if (!ord) {
    launch_table<TS>(pv, s);
    launched += 2;
  }
  // pass 2: one resident wave; the warps share out the list's segment parts
  auto insert = pass2_insert_kernel<KW, TS>;
  if constexpr (KW == 1 && kOrdOk)
    if (v.o_fused) insert = pass2_insert_kernel<KW, TS, true>;
  const unsigned g2 = grid_for(insert, kBlock, ~0ull >> 1, v.blocks_per_sm);
  const unsigned g3 = grid_for(pass2_classify_kernel<KW, TS>, kBlock, ~0ull >> 1, v.blocks_per_sm);
  {
    Timed t("pass2_insert", s);
    for (const auto& r : rs) {
      RunView x = part(r);
      x.n_segments = pv.n_segments;
      x.seg_cap = pv.seg_cap;
      insert<<<g2, kBlock, 0, s>>>(x);
      ++launched;
    }
  }
  {
    Timed t("pass2_classify", s);
    for (const auto& r : rs) {
      RunView x = part(r);
      x.n_segments = pv.n_segments;
      x.seg_cap = pv.seg_cap;
      pass2_classify_kernel<KW, TS><<<g3, kBlock, 0, s>>>(x);
      ++launched;
    }
  }
  return done(launched);
}

static int part_round(const RunView& v, int round, int rounds, cudaStream_t s, const Ranges* ranges) {
  int rc = 0;
  with_hashes(v.hashes, [&](auto hb) {
    constexpr int HB = decltype(hb)::value;
    auto go = [&](auto ts) {
      constexpr int TS = decltype(ts)::value;
      rc = rounds > 1 ? round_impl<kPartKw, true, HB, TS>(v, round, s, ranges)
                      : round_impl<kPartKw, false, HB, TS>(v, round, s, ranges);
    };
    if constexpr (kPartKw == 1) {
      if (table_slot_kind(v.k) == 0) go(std::integral_constant<int, 0>{});
      else go(std::integral_constant<int, 1>{});
    } else {
      go(std::integral_constant<int, kPartKw == 2 ? 2 : 3>{});
    }
  });
  return rc;
}

static int part_count(const RunView& v, cudaStream_t s) {
  const uint64_t threads = (v.m + kR - 1) / kR;
  const bool sampled = v.part_chunks || v.part_sample;
  with_hashes(v.hashes, [&](auto hb) {
    auto kern = partition_count_kernel<kPartKw, decltype(hb)::value>;
    const unsigned grid = grid_for(kern, kBlock, threads);
    kern<<<grid, kBlock, 0, s>>>(v, 0);
    if (sampled) kern<<<grid, kBlock, 0, s>>>(v, 1);
  });
  return cudaPeekAtLastError() == cudaSuccess ? (sampled ? 2 : 1) : -1;
}

// The parts' entry points, one set per translation unit.
#define TWOPACO_PART_NAME2(f, p) f##p
#define TWOPACO_PART_NAME(f, p) TWOPACO_PART_NAME2(f, p)
int TWOPACO_PART_NAME(launch_round_, TWOPACO_PART)(const RunView& v, int round, int rounds, cudaStream_t s,
                                                   const Ranges* ranges) {
  return part_round(v, round, rounds, s, ranges);
}
int TWOPACO_PART_NAME(launch_count_, TWOPACO_PART)(const RunView& v, cudaStream_t s) { return part_count(v, s); }

#if TWOPACO_PART == 1 || TWOPACO_PART == 3 || TWOPACO_PART == 5
// The class map of this k-mer width.
int TWOPACO_PART_NAME(launch_map_, TWOPACO_PART)(const RunView& v, cudaStream_t s) {
  Timed t(v.o_regions ? "class_sort" : "class_map", s);
  if constexpr (kPartKw < 4) {
    if (v.o_regions) {  // the sorted tiles instead
      auto kern = class_sort_kernel<kPartKw>;
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortBytes) != cudaSuccess)
        return -1;
      kern<<<grid_for(kern, kSortBlock, v.o_tiles * kSortBlock, 0, kSortBytes), kSortBlock, kSortBytes, s>>>(v);
      return done(1);
    }
  }
  auto kern = class_map_kernel<kPartKw>;
  kern<<<grid_for(kern, kBlock, (v.m + kInsertR - 1) / kInsertR), kBlock, 0, s>>>(v);
  return done(1);
}
#endif

#endif  // TWOPACO_PART

#ifndef TWOPACO_PART
// The part that holds the instances of this run: by k-mer width, then by bits per item.
int part_of(const RunView& v) {
  if (v.k > 63) return 5;
  return (v.k <= 31 ? 1 : 3) + (v.hashes > 4 ? 1 : 0);
}

int launch_round(const RunView& v, int round, int rounds, cudaStream_t s, const Ranges* ranges) {
  if (v.m == 0) return 0;
  switch (part_of(v)) {
    case 1: return launch_round_1(v, round, rounds, s, ranges);
    case 2: return launch_round_2(v, round, rounds, s, ranges);
    case 3: return launch_round_3(v, round, rounds, s, ranges);
    case 4: return launch_round_4(v, round, rounds, s, ranges);
    default: return launch_round_5(v, round, rounds, s, ranges);
  }
}

int launch_partition(const RunView& v, int rounds, cudaStream_t s) {
  if (v.m == 0) return 0;
  // the filter is clear (pack kernel); the pre-pass uses it, round 0 clears it again
  if (cudaMemsetAsync(v.bins, 0, (uint64_t)(v.qmask + 1u) * 4, s) != cudaSuccess) return -1;
  int counts;
  {
    Timed t("partition_count", s);
    const int part = part_of(v);
    counts = part == 1   ? launch_count_1(v, s)
             : part == 2 ? launch_count_2(v, s)
             : part == 3 ? launch_count_3(v, s)
             : part == 4 ? launch_count_4(v, s)
                         : launch_count_5(v, s);
    if (counts < 0) return -1;
  }
  uint64_t* prefix = reinterpret_cast<uint64_t*>(v.bins + (v.qmask + 1u));
  {
    Timed t("partition_cut", s);
    partition_cut_kernel<<<1, 1024, 0, s>>>(v, rounds, prefix);
  }
  return done(counts + 1);
}

int launch_class_map(const RunView& v, cudaStream_t s) {
  if ((!v.cmap && !v.o_regions) || v.m == 0) return 0;
  return v.k <= 31 ? launch_map_1(v, s) : (v.k <= 63 ? launch_map_3(v, s) : launch_map_5(v, s));
}

int launch_emit(const RunView& v, cudaStream_t s, bool again) {
  // again: a second emit of the same run (into a larger output): its tile
  // tickets, tile status and output flag start over
  if (again && (cudaMemsetAsync(v.tile_prefix, 0, (v.n_tiles + 1) * 8, s) != cudaSuccess ||
                cudaMemsetAsync(&v.hdr->emit_ticket, 0, sizeof(unsigned long long), s) != cudaSuccess ||
                cudaMemsetAsync(&v.hdr->out_overflow, 0, sizeof(unsigned int), s) != cudaSuccess))
    return -1;
  if (v.n_tiles) {  // tile status cleared by the pack kernel; writes the offsets too
    Timed t("emit", s);
    emit_kernel<<<grid_for(emit_kernel, kBlock, v.n_tiles * kBlock), kBlock, 0, s>>>(v);
  } else {  // no input: every offset is 0
    Timed t("emit_offsets", s);
    emit_offsets_kernel<<<(unsigned)(v.n_seqs + 1), kBlock, 0, s>>>(v);
  }
  return done(1);
}

int launch_edges(const DevHeader* hdr_dev, const uint64_t* d_offsets, uint64_t n_seqs,
                 const uint64_t* d_out_offsets, const uint64_t* d_out_positions,
                 uint64_t* d_edge_offsets, void* d_edges, uint64_t edge_capacity, cudaStream_t s) {
  // the piece ranks, when the run split its strings at N (the kernel reads the
  // header and returns at once otherwise)
  {
    Timed t("edge_offsets", s);
    runs_rank_kernel<<<1, 1024, 0, s>>>(hdr_dev);
    edge_offsets_kernel<<<1, 1024, 0, s>>>(hdr_dev, d_offsets, d_out_offsets, n_seqs, d_edge_offsets,
                                           edge_capacity);
  }
  {
    Timed t("edges", s);
    edges_kernel<<<grid_for(edges_kernel, kBlock, 1ull << 30), kBlock, 0, s>>>(
        hdr_dev, d_offsets, n_seqs, d_out_offsets, d_out_positions, d_edge_offsets,
        static_cast<EdgeOut*>(d_edges), edge_capacity);
  }
  return done(3);
}

#endif  // TWOPACO_PART

}  // namespace twopaco

#ifndef TWOPACO_PART

extern "C" unsigned long long twopaco_kernel_launches(void) {
  return twopaco::g_launches.load();
}

extern "C" int twopaco_profile_enable(int on) {
  using namespace twopaco;
  std::lock_guard<std::mutex> g(g_prof_mu);
  for (auto& r : g_prof) {
    g_event_pool.push_back(r.start);
    g_event_pool.push_back(r.stop);
  }
  g_prof.clear();
  g_prof_on = on != 0;
  return 0;
}

extern "C" int twopaco_profile_kernels(const char** names, unsigned long long* launches,
                                       double* total_ms, int capacity) {
  using namespace twopaco;
  std::lock_guard<std::mutex> g(g_prof_mu);
  std::vector<std::string> seen;
  std::vector<unsigned long long> cnt;
  std::vector<double> ms;
  std::vector<const char*> ptr;
  for (auto& r : g_prof) {
    if (cudaEventSynchronize(r.stop) != cudaSuccess) return -5;
    float t = 0.f;
    if (cudaEventElapsedTime(&t, r.start, r.stop) != cudaSuccess) return -5;
    size_t i = 0;
    while (i < seen.size() && seen[i] != r.name) ++i;
    if (i == seen.size()) {
      seen.push_back(r.name);
      ptr.push_back(r.name);
      cnt.push_back(0);
      ms.push_back(0.0);
    }
    cnt[i] += 1;
    ms[i] += t;
  }
  const int n = (int)seen.size();
  for (int i = 0; i < n && i < capacity; ++i) {
    if (names) names[i] = ptr[i];
    if (launches) launches[i] = cnt[i];
    if (total_ms) total_ms[i] = ms[i];
  }
  return n;
}

#endif  // TWOPACO_PART
