// pcz_retrieve.cu -- fused reconstruction kernel: Algorithm 2 (Magri &
// Lindstrom, Sec. 4.2) on the 4x4x4 bricks that meet a box.
//
// For each brick the kernel decodes components k0+1..k and adds them, in
// ascending order, into the partial sum x~ held in registers; x~ starts at 0
// or, to continue a refinement (Sec. 4.2), at the caller's x~_k0.  Only the
// bricks meeting the box are touched: zfp-style blocks decode on their own
// (Sec. 6.1).
//
// A launch runs a list of box jobs (one box of one field each; a single
// retrieval is a list of one, a batch of queries a longer one), each cut into
// units of consecutive bricks of its box.  A job may carry a cache of partial
// sums with, per brick, the k it holds: a brick whose cached k is at most the
// job's k starts from the cached x~ and decodes only the components above it
// (Algorithm 2's partial sums are the same whichever way they are reached).
//
// Layout: persistent CTAs of 4 warps, each taking units of 32 or more consecutive
// bricks of a job's box, up to 6 components at a time.  Parse: the warps take
// tasks of 32 blocks of one component, a block per lane, plane by plane (the
// blocks of a task are neighbours, so they are of alike length and their index
// entries are adjacent); the plane words of all blocks lie one after another in
// shared memory, those that do not fit in global memory.  Rebuild: each warp takes
// 8 bricks at a time, 4 lanes each.  Lane q of a brick reads the planes' bits of
// the 16 coefficients q, transposes them back in registers, 8 or 16 planes at
// once, and hands the digits over through shared memory, each lane taking its
// y-plane of coefficients; two inverse lifting passes run in registers after one
// exchange (in float where 8 planes hold a brick's digits: fewer operations, on
// the otherwise idle pipe), and x_j is added into the lane's z-plane of x~.
//
// Bound by instruction issue.  With 16 lanes per brick in the rebuild, CTAs of
// 512 blocks sorted by length for the parse and an index pass of its own it took
// 190 (float32, k = 6) and 229 (float64, k = 8) warp instructions per brick and
// component, now 107 and 127; 512^3 float32: k = 6 2.87 -> 1.71 ms, k = 1 0.86 ->
// 0.44 ms; 256 x 384 x 384 float64: k = 8 1.29 -> 0.89 ms; refinement from k = 1 to
// 8 in place 7.06 -> 3.39 and 3.13 -> 1.75 ms (nearly half of it had gone to the
// index pass and the sort).  With what most streams' bricks do not need (more than
// 16 planes of a component, RAW) out of line, nothing spills and the common path is shorter to fetch: 512^3 float32 k =
// 6 1.72 -> 1.68 ms, 252 x 380 x 384 float64 k = 1 204 -> 185 us, refinement by one
// component 198 -> 183 us.  (Code that does not even run costs here: a prefetch
// behind a condition that is never true made k = 6 7 % slower.)
#include <algorithm>
#include <type_traits>

#include "pcz_device.cuh"
#include "pcz_kernels.h"

namespace pcz {

static __constant__ PermTable kRank3r = make_rank();

constexpr int kRWarps = 4;
constexpr int kRThreads = 32 * kRWarps;
constexpr int kRoundTasks = 6;                 // warp tasks (32 blocks of one component) parsed at a time, at most
constexpr int kBlocks = 32 * kRoundTasks;      // their blocks
constexpr int kPool = 1792;                    // plane words kept in shared memory (a round of the 512^3
                                               // workload's blocks has 900 to 1730)
constexpr int kPoolPad = 16;                   // words before and after them that may be read (and are masked)

struct BlockMeta {
  uint64_t off;   // first bit of the brick in the component's payload
  int16_t s;      // scale exponent (R6), within [-1100, 1100]
  int8_t p;       // lowest coded plane, 0..64
  int8_t top;     // highest non-empty plane, p - 1 if none
  uint8_t mode;
  uint8_t pad_;
  uint16_t at;    // first plane word, from the top plane down: below kPool in shared memory, else spilled
};
static_assert(sizeof(BlockMeta) == 16, "block header size");

// A warp's work area, in 16-byte vectors: the exchange of the inverse lifting
// (LineSet), or the digits in coded order (brick b from byte 80 b, 144 b, 272 b
// or 528 b for 1, 2, 4 or 8 bytes each).
template <typename T>
struct AreaR {
  static constexpr int kVectors = LineSet::kVectors * (int)(sizeof(T) / 4);
  static_assert(kVectors * 16 >= 8 * (64 * (int)sizeof(T) + 16), "digits fit");
};

template <typename T>
__host__ __device__ constexpr size_t retrieve_smem3() {
  return (size_t)(kPool + 2 * kPoolPad) * sizeof(uint64_t)        // plane words
         + (size_t)kBlocks * sizeof(BlockMeta)                    // block headers
         + (size_t)kRWarps * AreaR<T>::kVectors * 16              // work areas
         + (size_t)kTokLut * sizeof(uint32_t)                     // group-test byte table
         + (size_t)kBlocks / 8;                                   // decoding of every 8 blocks
}

// Plane words of a round that may not fit: all of the blocks' planes but the
// pool's, and one block's that straddles the pool's end.
template <typename T>
__host__ __device__ constexpr size_t spill_words_per_cta() {
  return (size_t)kBlocks * Fmt<T>::P - kPool + Fmt<T>::P;
}

// The place of the block whose plane words start at index `at` of the round.
template <typename T>
__device__ __forceinline__ uint64_t* words_at(uint64_t* pool, uint64_t* spill, int at, int nw) {
  return at + nw <= kPool ? pool + at : spill + (at - (kPool - Fmt<T>::P));
}
// Whether its nw words lie in one of the two (debug builds check it).
template <typename T>
__device__ __forceinline__ bool words_in(int at, int nw) {
  const int64_t end = (int64_t)at - (kPool - Fmt<T>::P) + nw;
  return at >= 0 && nw >= 0 && nw <= Fmt<T>::P && (at + nw <= kPool || end <= (int64_t)spill_words_per_cta<T>());
}

// A plane in which coefficients may turn significant (R11): n < 64 verbatim bits
// at pos, then the group-test part, a byte at a time through the table.  The
// plane word is gathered at the top of 64 bits, each byte's coefficient bits
// funnelled in from above, and moved down at the end.  When a byte would carry the
// count to 64, the last coefficient turns significant in it (after which no
// closing test bit follows) or the block is malformed; the part's end then
// follows from the byte's entry in closed form.  A valid part is at most
// 2 (64 - n) + 1 <= 129 bits.
__device__ __forceinline__ bool parse_group_plane(BlockBits& br, uint32_t& pos, int& n, uint64_t& W,
                                                  const uint32_t* lut) {
  const uint64_t v = (br.peek(pos) << 1) << (63 - n);
  uint32_t wlo = (uint32_t)v, whi = (uint32_t)(v >> 32), e = 0, idx = 0;
  pos += (uint32_t)n;
  int c = n, cnt = 0;
  bool end = false;
  // 4 bytes at a time without branches (a lane whose part has ended shifts by 0):
  // code at the exits of a loop over bytes would run once for every byte at which
  // some lane ends.  A byte that does not end the part holds at least 4
  // coefficients, which bounds the loop.
#pragma unroll 1
  for (;;) {
    const uint64_t g64 = br.peek(pos);
    auto word = [&](uint32_t g) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t i1 = token_index(e, g, j), e1 = lut[i1];
        const int c1 = token_count(e1);
        if (!end) {
          idx = i1;
          e = e1;
          cnt = c1;
        }
        end = end || c + cnt >= 64 || (int32_t)e < 0;  // the part ends in this byte
        const int add = end ? 0 : cnt;
        wlo = __funnelshift_r(wlo, whi, add);
        whi = __funnelshift_r(whi, e, add);
        c += add;
        pos += end ? 0u : 8u;
      }
    };
    word((uint32_t)g64);
    if (!end) word((uint32_t)(g64 >> 32));
    if (end) break;
  }
  const int k = min(64 - c, cnt);  // of its coefficients
  wlo = __funnelshift_r(wlo, whi, k);
  whi = __funnelshift_r(whi, e, k);
  c += k;
  W = (((uint64_t)whi << 32) | wlo) >> (64 - c);
  n = c;
  if (c == 64) {
    // bits used through the last coefficient's 1: its byte's first k coefficient
    // bits and the test bits before them (the byte's first bit in the test state,
    // and one after each earlier 1)
    pos += (uint32_t)k + (idx < 256u ? 1u : 0u) + (uint32_t)__popc(e & ((1u << (k - 1)) - 1u));
    return whi >> 31;  // (0: a run past the last coefficient)
  }
  pos += ((e >> 24) & 7u) + 1u;
  return true;
}

// R11 decoding of planes top .. p of one block (top: the highest non-empty one,
// whose test bit 1 is at bit pos), ending exactly at end, into out[0 .. top - p].
// Returns false on a malformed block; every loop is bounded.
__device__ __forceinline__ bool parse_planes(BlockBits& br, uint32_t pos, uint32_t end, int nw, uint64_t* out,
                                             const uint32_t* lut) {
  int n = 0;
  for (int k = 0; k < nw; ++k) {
    uint64_t W;
    if (n == 64) {
      W = br.peek(pos);
      pos += 64;
    } else if (!parse_group_plane(br, pos, n, W, lut)) {
      return false;
    }
    if (pos > end) return false;
    out[k] = W;
  }
  return pos == end;
}

// Level of brick b's cached partial sum that a job at k may start from (0:
// none): components up to it are already summed in the cache.
__device__ __forceinline__ int cached_level(const BoxJob& J, int64_t b) {
  if (!J.level) return 0;
  const int lv = J.level[b];
  return lv <= J.k ? lv : 0;
}

// Whether a block has planes, of which a short decoding reads the word at
// `last` and the `more` before it: within the pool and its pads (debug builds check it).
__device__ __forceinline__ bool from_pool(int nw, int last, int more) {
  return nw > 0 && PCZ_CHECK(last - more >= -kPoolPad && last < kPool + kPoolPad, 3);
}

// How 8 blocks (one component of a rebuild's bricks) are decoded: the largest of
// theirs, and whether one is RAW.
enum : int { kDecodeNone = 0, kDecodeFloat8 = 1, kDecodeInt16 = 2, kDecodeAny = 3, kHasRaw = 4 };

// One warp task: each lane parses component comp's block of box brick g into
// the round's plane words and its header.  A brick past the box, or a component
// the brick takes from the cache, has nothing to parse.  Every lane of the warp
// calls it.
template <typename T>
__device__ __forceinline__ void parse_task(const BoxJob& J, unsigned int* err, int64_t g, int comp, BlockMeta* meta,
                                           uint8_t* how, uint64_t* pool, uint64_t* spill, int* used,
                                           const uint32_t* lut) {
  using F = Fmt<T>;
  constexpr int N = 64;
  constexpr int Q = F::P - 2 - Geo<3>::G;
  constexpr int C = Geo<3>::C;
  constexpr int HDR = 2 + 3 + F::EBITS;
  constexpr int EMAXT = (1 << (F::EXPW - 1));  // frexp exponent of the largest finite T
  const int lane = threadIdx.x & 31;
  int mode = kModeZero, s = 0, p = 0, top = -1;
  uint64_t off = 0;
  uint32_t pos = 0, end = 0;
  bool ok = true;
  BlockBits br;  // positions from the start of the block's first word
  br.init(nullptr, 0, 0);
  int64_t bx, by, bz;
  if (g < J.nbox) {
    brick_of(J, g, &bx, &by, &bz);
    const int64_t b = bx + J.nb[0] * (by + J.nb[1] * bz);
    if (comp >= cached_level(J, b)) {
      const CompDesc& cd = J.comp[comp];
      off = cd.chunk_word[b / kChunk] * 64ull + cd.brick_off[b];
      const uint32_t len = cd.brick_len[b];
      br.init(cd.payload, cd.nwords, off);
      pos = (uint32_t)(off & 63u);
      end = pos + len;
      const uint64_t v = br.peek(pos);
      mode = (int)(v & 3ull);
      if (mode == kModeCoded) {
        const int esc = (int)((v >> 2) & 7ull);
        const int emax = (int)((v >> 5) & ((1ull << F::EBITS) - 1)) - F::EBIAS;
        ok = emax >= F::EMIN && emax <= EMAXT;
        if (ok) {
          s = Q - emax;
          p = min(max(cd.L + s - C - esc, 0), F::P);
          pos += HDR;
          // planes above the first significant coefficient are single 0 test bits
          top = F::P - 1;
          while (top >= p) {
            const uint64_t t = br.peek(pos);
            const int z = t ? __ffsll((long long)t) - 1 : 64;
            const int skip = min(z, top - p + 1);
            pos += (uint32_t)skip;
            top -= skip;
            if (z < 64) break;  // the bit after the zeros is the first significant plane's test 1
          }
          ok = pos <= end;
        }
      } else if (mode == kModeZero) {
        ok = len == 2;
      } else {
        ok = mode == kModeRaw && len == 2 + N * F::P;
      }
    }
  }
  // places of the lanes' plane words: a warp scan, and one atomic per task
  const bool coded = ok && mode == kModeCoded;
  const int nw = coded ? top - p + 1 : 0;
  int incl = nw;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  int at = 0;
  if (lane == 31) at = atomicAdd(used, incl);
  at = __shfl_sync(0xffffffffu, at, 31) + incl - nw;
  if (coded)
    ok = PCZ_CHECK(words_in<T>(at, nw), 3) &&
         parse_planes(br, pos, end, nw, words_at<T>(pool, spill, at, nw), lut);
  if (!ok) {
    atomicOr(err, 1u);
    mode = kModeZero;
  }
  BlockMeta bm;
  bm.off = off;
  bm.s = (int16_t)s;
  bm.p = (int8_t)p;
  bm.top = (int8_t)top;
  bm.mode = (uint8_t)mode;
  bm.pad_ = 0;
  bm.at = (uint16_t)at;
  *meta = bm;
  // Exactness of the two short decodings (see add_component): no value of the
  // inverse lifting is odd where it is halved (p >= 6), and none reaches 2^31
  // (planes up to 26) or 2^63 (up to 58) -- 2^(top + 1) * 2/3 * 2.75^3, with
  // 2.75 the largest row sum of the inverse lifting's coefficients.  Float64
  // blocks with higher planes (the first component's, mostly) take the decoding
  // of 16 planes after a look at their coefficients.
  int h = kDecodeNone;
  if (mode == kModeCoded && nw > 0) {
    const bool common = sizeof(T) == 8 ? s >= -960 && s <= 1022 : s >= -96 && s <= 126;
    const bool scaled = p >= 6 && common, low = top <= (sizeof(T) == 8 ? 58 : 26);
    h = at + nw > kPool || nw > 16 || (sizeof(T) == 8 && !scaled) ? kDecodeAny
        : nw <= 8 && scaled && low                                ? kDecodeFloat8
                                                                  : kDecodeInt16;
  }
#pragma unroll
  for (int o = 1; o <= 4; o <<= 1) h = max(h, __shfl_xor_sync(0xffffffffu, h, o));
  const unsigned raw = __ballot_sync(0xffffffffu, mode == kModeRaw);
  if ((lane & 7) == 0) *how = (uint8_t)(h | ((raw >> lane) & 0xffu ? kHasRaw : 0));
}

// A lane's share of a brick: z-plane q, values x + 4 y.  Which of them lie in
// the box, and where they are in the output and in the field.
struct BrickLane {
  bool have;
  int x0, x1, y0, y1;  // values [x0, x1) of rows [y0, y1); y1 = 0 where the plane is outside
  int64_t b, out, field;
};

__device__ __forceinline__ BrickLane brick_lane(const BoxJob& J, int64_t g, int q) {
  BrickLane L;
  L.have = g < J.nbox;
  int64_t bx = 0, by = 0, bz = 0;
  if (L.have) brick_of(J, g, &bx, &by, &bz);
  L.b = bx + J.nb[0] * (by + J.nb[1] * bz);
  const int64_t gy = 4 * by, gz = 4 * bz + q;
  L.x0 = (int)max(J.lo[0] - 4 * bx, (int64_t)0);
  L.x1 = (int)min(J.hi[0] - 4 * bx, (int64_t)4);
  L.y0 = (int)max(J.lo[1] - gy, (int64_t)0);
  L.y1 = L.have && gz >= J.lo[2] && gz < J.hi[2] ? (int)min(J.hi[1] - gy, (int64_t)4) : 0;
  const int64_t ext0 = J.hi[0] - J.lo[0], ext1 = J.hi[1] - J.lo[1];
  L.out = ((gz - J.lo[2]) * ext1 + (gy - J.lo[1])) * ext0 + 4 * bx - J.lo[0];
  L.field = (gz * J.dims[1] + gy) * J.dims[0] + 4 * bx;
  return L;
}

// x~ of the lane's values at the start of a job: 0, the caller's partial sum
// x~_k0 (refinement), or the cache.  -0 is read as +0, which is what adding a
// component makes of it even where the component is zero.  Returns whether the
// sum starts from 0.
template <typename T>
__device__ __forceinline__ bool start_sum(const BoxJob& J, int write, const BrickLane& L, T* xt) {
  using F = Fmt<T>;
#pragma unroll
  for (int v = 0; v < 16; ++v) xt[v] = T(0);
  const int lv = L.have ? cached_level(J, L.b) : 0;
  if (lv == 0 && !(write && J.k0 > 0)) return true;
  const T* src = lv > 0 ? reinterpret_cast<const T*>(J.cache) + L.field : reinterpret_cast<const T*>(J.out) + L.out;
  const int64_t row = lv > 0 ? J.dims[0] : J.hi[0] - J.lo[0];
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    if (y < L.y0 || y >= L.y1) continue;
    const T* line = src + y * row;
    if (L.x0 == 0 && L.x1 == 4) {
      load_line<T>(line, 4, xt + 4 * y);
    } else {
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if (x >= L.x0 && x < L.x1) xt[x + 4 * y] = line[x];
    }
  }
#pragma unroll
  for (int v = 0; v < 16; ++v)
    if (F::bits(xt[v]) == F::SIGN) xt[v] = T(0);
  return false;
}

// The lane's values into the output: whole aligned lines with 16-byte stores.
template <typename T>
__device__ __forceinline__ void store_lines(const BoxJob& J, const BrickLane& L, const T* xt) {
  T* out = reinterpret_cast<T*>(J.out) + L.out;
  const int64_t row = J.hi[0] - J.lo[0];
  const bool whole = L.x0 == 0 && L.x1 == 4 && (((uintptr_t)out | ((uintptr_t)row * sizeof(T))) & 15) == 0;
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    if (y < L.y0 || y >= L.y1) continue;
    T* line = out + y * row;
    if (whole) {
      constexpr bool all[4] = {true, true, true, true};
      store_line<T>(line, xt + 4 * y, all);
    } else {
#pragma unroll
      for (int x = 0; x < 4; ++x)
        if (x >= L.x0 && x < L.x1) line[x] = xt[4 * y + x];
    }
  }
}

// Float64 partial sums in fixed point.  As long as every partial sum of a brick
// is a multiple of some 2^e below 2^(e + 51), no addition rounds, and the sums can
// be kept as 64-bit integers in units of 2^e: the FP64 pipe (2 lanes per SM and
// clock, 16 clocks for a warp's addition) then sees one operation per value
// instead of one per component.  `lead` is the first coded component's highest
// plane, as an exponent (each component is below 2^(lead + 5)), depth = 46 -
// ceil(log2 k) the bits below it, e = lead - depth.  A component that does not
// fit (deeper, larger, RAW) ends it: the sums so far become doubles.  256 x 384 x
// 384, k = 8: 1070 -> 888 us.
struct FixedSum {
  bool on;    // (the same in the whole warp)
  int lead;   // kNoLead before the brick's first coded component
  int depth;
};
constexpr int kNoLead = -(1 << 20);

// units of 2^ue (|v| below 2^51, the result normal or 0) as a double
__device__ __forceinline__ double fixed_to_f64(double v, int ue) {
  const double m = __dsub_rn(__longlong_as_double(__double_as_longlong(v) + 0x4338000000000000ll), 6755399441055744.0);
  const int hi = __double2hiint(m);
  return __hiloint2double(hi ? hi + ue * (1 << 20) : 0, __double2loint(m));
}

__device__ __forceinline__ void end_fixed(FixedSum& fx, double* xt) {
  const int ue = fx.lead == kNoLead ? 0 : fx.lead - fx.depth;
#pragma unroll
  for (int k = 0; k < 16; ++k) xt[k] = fixed_to_f64(xt[k], ue);
  fx.on = false;
}

// i * 2^sh into a fixed-point sum: sh is at most 33, |i| below 2^27 (in the
// decoding of 16 planes) and |i| * 2^3 below 2^31.
__device__ __forceinline__ double fixed_add(double sum, int32_t i, int sh) {
  const int32_t hi = i * (1 << max(sh - 30, 0));
  return __longlong_as_double(__double_as_longlong(sum) + (int64_t)hi * (int64_t)(1 << min(sh, 30)));
}

// The decoding of any planes, out of line, so that the common path stays short.  xt:
// the lane's partial sums.  Components of more than 16 planes (steps of 12 bits and
// more) come here with every brick.  Two aligned windows instead of four, and 32-bit
// integers up to 20 planes: 256^3 float64, 2 components of 20 and 17 words a brick
// 347 -> 312 us, of 17 and 13 290 -> 235.
template <typename T>
__device__ __noinline__ void add_any(const BlockMeta* bm, uint64_t* pool, uint64_t* spill, uint4* area, int lane, T* xt) {
  using F = Fmt<T>;
  using U = typename F::U;
  using S = typename F::S;
  constexpr bool WIDE = F::P == 64;
  constexpr unsigned FULL = 0xffffffffu;
  const BlockMeta m = *bm;
  const int bq = lane >> 2, q = lane & 3;
  const bool coded = m.mode == kModeCoded;
  const int p = m.p, top = m.top, s = coded ? (int)m.s : 0;
  const int nw = coded && PCZ_CHECK(words_in<T>(m.at, top - p + 1), 3) ? top - p + 1 : 0;
  uint4* zw = area + LineSet::at(bq, 0, q);
  uint4* yw = area + LineSet::at(bq, q, 0);
  uint32_t place[4];
#pragma unroll
  for (int z = 0; z < 4; ++z) place[z] = coded_places(kRank3r.pos, q, z);
  // 16 planes at a time from plane `base`, 16 digits a half-word of the coefficients
  // in coded order.  Float64 blocks of at most 32 planes, aligned to the highest, take
  // two such windows and 32-bit digits: d stands for ((d ^ M) - M) * 2^base with M =
  // NBM >> base (as in add_component; 32 bits of M suffice).
  const bool two = WIDE && __all_sync(FULL, nw <= 32);
  const int base = two ? max(top, 31) - 31 : 0;
  const int bytes = two ? 4 : (int)sizeof(T);
  unsigned char* dig = reinterpret_cast<unsigned char*>(area) + (64 * bytes + 16) * bq;
  const uint64_t* words = words_at<T>(pool, spill, m.at, nw);
#pragma unroll 1
  for (int h = 0; h < 8 * bytes / 16; ++h) {
    auto plane = [&](int pl) {
      if (nw <= 0 || pl < p || pl > top) return 0u;
      return (uint32_t)reinterpret_cast<const uint16_t*>(words + (top - pl))[q];
    };
    uint32_t a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = plane(base + 16 * h + j) | (plane(base + 16 * h + j + 8) << 16);
    untranspose16(a);
#pragma unroll
    for (int i = 0; i < 8; ++i) {  // ranks i and i + 8 of the lane's 16, at their places
      uint16_t* e = reinterpret_cast<uint16_t*>(dig + (16 * q + 4 * (i & 3) + 2 * (i >> 2)) * bytes) + h;
      e[0] = (uint16_t)a[i];
      e[bytes / 2] = (uint16_t)(a[i] >> 16);
    }
  }
  __syncwarp();
  auto digits = [&](int k) { return dig + ((place[k >> 2] >> (8 * (k & 3))) & 0xffu) * bytes; };
  const bool common = __all_sync(FULL, WIDE ? s >= -960 && s <= 1022 : s >= -127 && s <= 126);
  if constexpr (WIDE) {
    // at most 20 planes: in 32-bit integers, as add_component's 16
    if (common && __all_sync(FULL, nw <= 0 || (nw <= 20 && p >= 6 && top <= 58))) {
      const int low = max(top, 19) - 19;
      const uint32_t M = (uint32_t)(F::NBM >> low);
      int32_t r[16];
#pragma unroll
      for (int k = 0; k < 16; ++k)
        r[k] = (int32_t)((((*reinterpret_cast<const uint32_t*>(digits(k)) >> (low - base)) ^ M) - M) << 6);
      __syncwarp();
      lift_inv_bricks<int32_t>(r, zw, yw, LineSet::kVectors);
      const uint32_t eb = (uint32_t)(1053 + (low - 6) - s) << 20;
#pragma unroll
      for (int k = 0; k < 16; ++k) xt[k] = F::add(xt[k], scaled_i32_to_f64(r[k], eb));
      return;
    }
  }
  S r[16];
  if (two) {
    const uint32_t M = (uint32_t)(F::NBM >> base);
#pragma unroll
    for (int k = 0; k < 16; ++k)
      r[k] = (S)(((int64_t)(*reinterpret_cast<const uint32_t*>(digits(k)) ^ M) - (int64_t)M) << base);
  } else {
#pragma unroll
    for (int k = 0; k < 16; ++k) r[k] = nb_inv<T>(*reinterpret_cast<const U*>(digits(k)));
  }
  __syncwarp();
  lift_inv_bricks<S>(r, zw, yw, LineSet::kVectors);
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    T xi[4];
    if (common) {
      dequantize_line<T, true>(r + 4 * y, s, xi);
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) xi[k] = F::val(dequantize_any<T>(r[4 * y + k], s));
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) xt[4 * y + k] = F::add(xt[4 * y + k], xi[k]);
  }
}

// A RAW block of the lane's brick into its sums: the words that hold its 16 values,
// each requested once and all together (200^3 float64, every block RAW, k = 1: 194
// -> 108 us, 114 before the 4-lane layout).
template <typename T>
__device__ __noinline__ void add_raw(const BlockMeta* bm, const CompDesc* cd, int q, T* xt) {
  using F = Fmt<T>;
  using U = typename F::U;
  constexpr int N = 16 * F::P / 64;  // words of values
  const uint64_t off = bm->off + 2 + (uint64_t)F::P * 16 * q;
  const uint64_t* w = cd->payload;
  const uint64_t nw = cd->nwords, i = off >> 6;
  const int sh = (int)(off & 63);
  uint64_t v[N + 1];
#pragma unroll
  for (int k = 0; k <= N; ++k) v[k] = i + k < nw ? __ldg(w + i + k) : 0ull;
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = sh ? (v[k] >> sh) | (v[k + 1] << (64 - sh)) : v[k];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const uint64_t b = v[k * F::P / 64] >> (k * F::P % 64);
    xt[k] = F::add(xt[k], F::val((U)b));
  }
}

// Adds one component into the z-planes of a warp's 8 bricks.  how: kDecode* and
// kHasRaw of the 8; m: header of the lane's brick; pool, spill: the round's plane
// words; zw, yw: the lane's lines of the exchange; place: the coded places of its
// coefficients.
template <typename T>
__device__ __forceinline__ void add_component(int how, const BlockMeta* bm, const CompDesc* cd, uint64_t* pool,
                                              uint64_t* spill, uint4* area, uint4* zw, uint4* yw,
                                              const uint32_t* place, int lane, T* xt, FixedSum& fx) {
  using F = Fmt<T>;
  using U = typename F::U;
  using S = typename F::S;
  constexpr bool WIDE = F::P == 64;
  constexpr unsigned FULL = 0xffffffffu;
  const BlockMeta m = *bm;
  const int bq = lane >> 2, q = lane & 3;
  const int p = m.p, top = m.top;
  const int nw = m.mode == kModeCoded ? top - p + 1 : 0;  // planes with digits
  const int s = nw > 0 ? (int)m.s : 0;  // (a CODED block without any may have a scale outside the others' range)
  const uint32_t areas = smem_addr(area);
  bool any = (how & 3) == kDecodeAny;
  if constexpr (WIDE) {
    if (fx.on) {
      bool fits = !any && !(how & kHasRaw);
      if (nw > 0) {
        if (fx.lead == kNoLead) {
          fx.lead = top - s;
          fits = fits && fx.lead >= -900 && fx.lead <= 900;
        }
        const int H = (how & 3) == kDecodeFloat8 ? 8 : 16;  // the decoding's units: 2^(base - 6 - s)
        fits = fits && top - s <= fx.lead && max(top, H - 1) - (H - 1) - 6 - s >= fx.lead - fx.depth;
      }
      if (!__all_sync(FULL, fits)) end_fixed(fx, xt);
    }
  }
  // The short decodings take the planes top .. top - H + 1 of the lane's 16
  // coefficients, transposed to digits: bit i of a digit is plane base + i.  What
  // lies outside [p, top] (other blocks' words) is masked off.
  if ((how & 3) == kDecodeFloat8) {
    const int base = max(top, 7) - 7;
    const uint32_t keep = nw > 0 ? ((1u << nw) - 1u) << (p - base) : 0u;
    const int last = m.at + top - base;  // word of plane base
    const uint16_t* pc = reinterpret_cast<const uint16_t*>(pool + (from_pool(nw, last, 7) ? last : 7)) + q;
    uint32_t a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = (uint32_t)pc[-4 * j] | ((uint32_t)pc[-4 * (j + 4)] << 16);
    untranspose8(a);
    area[5 * bq + q] = make_uint4(a[0], a[1], a[2], a[3]);
    __syncwarp();
    // R9: with M = NBM >> base (8 bits), digits d stand for (d ^ M) - M in units of
    // 2^base.  With 2^23's bit pattern in M, the difference of two floats.
    const uint32_t M = (uint32_t)(F::NBM >> base) & 0xffu | 0x4B000000u;
    const uint32_t get = areas + 80u * bq;
    float r[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      uint32_t d;  // the address: get + byte k & 3 of place
      asm volatile("ld.shared.u8 %0, [%1];" : "=r"(d) : "r"(__dp4a(place[k >> 2], 1u << (8 * (k & 3)), get)) : "memory");
      r[k] = __fsub_rn(__uint_as_float((d & keep) ^ M), __uint_as_float(M));
    }
    __syncwarp();
    // values below 2^12.8 units and multiples of 2^-6: 19 bits
    lift_inv_bricks<float>(r, zw, yw, LineSet::kVectors);
    if constexpr (WIDE) {
      if (fx.on) {  // r in units of 2^-6: the float sum with 1.5 * 2^17 holds it in its low bits
        const int sh = nw > 0 ? (base - 6 - s) - (fx.lead - fx.depth) : 0;
#pragma unroll
        for (int k = 0; k < 16; ++k)
          xt[k] = fixed_add(xt[k], __float_as_int(__fadd_rn(r[k], 196608.0f)) - 0x48400000, sh);
      } else {
        const uint32_t adj = (uint32_t)(896 + base - s) << 20;
#pragma unroll
        for (int k = 0; k < 16; ++k) xt[k] = F::add(xt[k], scaled_f32_to_f64(r[k], adj));
      }
    } else {
      const float sc = __uint_as_float((uint32_t)(127 + base - s) << 23);  // x_j = r * sc exactly
#pragma unroll
      for (int k = 0; k < 16; ++k) xt[k] = __fmaf_rn(r[k], sc, xt[k]);
    }
  } else if ((how & 3) == kDecodeInt16) {
    const int base = max(top, 15) - 15;
    const uint32_t keep = nw > 0 ? ((1u << nw) - 1u) << (p - base) : 0u;
    const int last = m.at + top - base;
    const uint16_t* pc = reinterpret_cast<const uint16_t*>(pool + (from_pool(nw, last, 15) ? last : 15)) + q;
    uint32_t a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = (uint32_t)pc[-4 * j] | ((uint32_t)pc[-4 * (j + 8)] << 16);
    untranspose16(a);
    area[9 * bq + 2 * q] = make_uint4(a[0], a[4], a[1], a[5]);
    area[9 * bq + 2 * q + 1] = make_uint4(a[2], a[6], a[3], a[7]);
    __syncwarp();
    const uint32_t M = (uint32_t)(F::NBM >> base);
    const uint32_t unit = WIDE ? 64u : 1u << base;  // float64: units of 2^(base - 6), values below 2^27
    const uint32_t get = areas + 144u * bq;
    int32_t r[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      uint16_t d;
      asm volatile("ld.shared.u16 %0, [%1];" : "=h"(d) : "r"(__dp4a(place[k >> 2], 2u << (8 * (k & 3)), get)) : "memory");
      r[k] = (int32_t)((((uint32_t)d & keep) ^ M) * unit - M * unit);
    }
    if constexpr (WIDE) {
      // planes above 58: no value of the inverse lifting is larger than the sum of
      // the brick's 64 coefficients' magnitudes (its matrix has no entry above 1)
      if (__any_sync(FULL, nw > 0 && top > 58)) {
        uint32_t sum = 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) sum += (uint32_t)abs(r[k]);  // each below 2^22
        sum += __shfl_xor_sync(FULL, sum, 1);
        sum += __shfl_xor_sync(FULL, sum, 2);
        any = __any_sync(FULL, nw > 0 && top > 58 && sum >= 1u << (69 - base));
      }
    }
    __syncwarp();
    if (!any) lift_inv_bricks<int32_t>(r, zw, yw, LineSet::kVectors);
    if constexpr (WIDE) {
      if (any) {
        if (fx.on) end_fixed(fx, xt);
      } else if (fx.on) {
        const int sh = nw > 0 ? (base - 6 - s) - (fx.lead - fx.depth) : 0;
#pragma unroll
        for (int k = 0; k < 16; ++k) xt[k] = fixed_add(xt[k], r[k], sh);
      } else {
        const uint32_t eb = (uint32_t)(1053 + (base - 6) - s) << 20;
#pragma unroll
        for (int k = 0; k < 16; ++k) xt[k] = F::add(xt[k], scaled_i32_to_f64(r[k], eb));
      }
    } else if (__all_sync(FULL, s >= -96 && s <= 126)) {
      // one rounding to float; the product by 2^-s is exact (normal, and below
      // 2^127 for s >= -96), so one fused add is x~ + x_j
      const float sc = __uint_as_float((uint32_t)(127 - s) << 23);
#pragma unroll
      for (int k = 0; k < 16; ++k) xt[k] = __fmaf_rn(__int2float_rn(r[k]), sc, xt[k]);
    } else {
#pragma unroll
      for (int k = 0; k < 16; ++k) xt[k] = F::add(xt[k], F::val(dequantize_any<T>(r[k], s)));
    }
  }
  if (any) {
    T t[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) t[k] = xt[k];
    add_any<T>(bm, pool, spill, area, lane, t);
#pragma unroll
    for (int k = 0; k < 16; ++k) xt[k] = t[k];
  }
  if ((how & kHasRaw) && m.mode == kModeRaw) {
    T t[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) t[k] = xt[k];
    add_raw<T>(bm, cd, q, t);
#pragma unroll
    for (int k = 0; k < 16; ++k) xt[k] = t[k];
  }
}

// CTAs that share an SM, as their shared memory allows: 31 KB for float32, 40 KB
// for float64 (6 and 4 measured 2 and 7 % slower).
template <typename T>
constexpr int kRetrieveCtas3 = sizeof(T) == 4 ? 7 : 5;

template <typename T>
__global__ void __launch_bounds__(kRThreads, kRetrieveCtas3<T>) k_retrieve3(const RetrieveParams R) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint64_t* pool = reinterpret_cast<uint64_t*>(smem) + kPoolPad;                // [kPool]
  BlockMeta* meta = reinterpret_cast<BlockMeta*>(pool + kPool + kPoolPad);     // [kBlocks]
  uint4* areas = reinterpret_cast<uint4*>(meta + kBlocks);                     // [kRWarps]
  uint32_t* lut = reinterpret_cast<uint32_t*>(areas + kRWarps * AreaR<T>::kVectors);
  uint8_t* how = reinterpret_cast<uint8_t*>(lut + kTokLut);                    // [kBlocks / 8]
  load_tokens<kRThreads>(lut);  // read after the loop's first barrier
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, bq = lane >> 2, q = lane & 3;
  uint4* area = areas + warp * AreaR<T>::kVectors;
  uint4* zw = area + LineSet::at(bq, 0, q);  // + 2 y: line (y, z = q)
  uint4* yw = area + LineSet::at(bq, q, 0);  // + 10 z: line (y = q, z)
  uint64_t* spill = R.spill + (size_t)blockIdx.x * spill_words_per_cta<T>();
  uint32_t place[4];  // coded places of the lane's coefficients x + 4 z (y = q)
#pragma unroll
  for (int z = 0; z < 4; ++z) place[z] = coded_places(kRank3r.pos, q, z);

  __shared__ BoxJob sJ;
  __shared__ int s_task, s_used;  // the round's next warp task, and its plane words so far
  const BoxJob& J = sJ;
  constexpr int JW = (int)(sizeof(BoxJob) / 8);
  static_assert(sizeof(BoxJob) % 8 == 0 && JW <= kRThreads, "job copy");
  if (tid == 0) s_task = s_used = 0;
  int64_t job_end = 0;  // the units of the job in sJ end here
  for (int64_t unit = blockIdx.x; unit < R.nunits; unit += gridDim.x) {
    if (unit >= job_end) {  // the job whose units contain this one
      __syncthreads();      // the previous unit is done with sJ
      if (!R.jobs) {
        if (tid == 0) sJ = R.job0;
        job_end = R.nunits;
      } else {
        int lo = 0, hi = R.njobs - 1;
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (R.jobs[mid].unit_begin <= unit)
            lo = mid;
          else
            hi = mid - 1;
        }
        if (tid < JW) reinterpret_cast<uint64_t*>(&sJ)[tid] = reinterpret_cast<const uint64_t*>(R.jobs + lo)[tid];
        job_end = lo + 1 < R.njobs ? R.jobs[lo + 1].unit_begin : R.nunits;
      }
      __syncthreads();
    }
    const int ub = J.unit_bricks, sets = ub / 32;  // bricks of a unit; sets of 32
    const int64_t unit0 = (unit - J.unit_begin) * ub;
    T xt[16];
    BrickLane BL;
    FixedSum fx;
    for (int c0 = J.k0; c0 < J.k; c0 += J.round) {
      const int nc = min(J.round, J.k - c0), ntask = nc * sets;
      for (;;) {  // the warps take tasks, the first component's (mostly the longest) first
        int t = 0;
        if (lane == 0) t = atomicAdd(&s_task, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntask) break;
        const int c = t / sets, u = 32 * (t - c * sets) + lane;
        const int blk = c * ub + u;
        parse_task<T>(J, R.err, unit0 + u, c0 + c, meta + blk, how + blk / 8, pool, spill, &s_used, lut);
      }
      __syncthreads();
      if (tid == 0) s_task = s_used = 0;
      if (R.write) {
        // (more than one set: the unit's components are all in this round)
        for (int g = 0; g < sets; ++g) {
          const int u = 8 * (kRWarps * g + warp) + bq;
          if (c0 == J.k0) {
            BL = brick_lane(J, unit0 + u, q);
            const bool zero = start_sum<T>(J, R.write, BL, xt);
            fx.on = sizeof(T) == 8 && __all_sync(0xffffffffu, zero) && J.k > 1;
            fx.lead = kNoLead;
            fx.depth = 46 - (32 - __clz(J.k - 1));
          }
          for (int c = 0; c < nc; ++c) {  // Algorithm 2, components in ascending order
            const int blk = c * ub + u, h = how[blk / 8];
            if (h == kDecodeNone) continue;
            add_component<T>(h, meta + blk, &J.comp[c0 + c], pool, spill, area, zw, yw, place, lane, xt, fx);
          }
          if (c0 + nc >= J.k) {
            if constexpr (sizeof(T) == 8)
              if (fx.on) end_fixed(fx, xt);
            store_lines<T>(J, BL, xt);
          }
        }
      }
      __syncthreads();  // the next blocks take the places
    }
  }
}

template <typename T>
static int retrieve_grid_t(int64_t nunits) {
  // CTAs that fit on the GPU at once, queried once per type (a function-local
  // static: initialised once even when several host threads get here first)
  static const int64_t g = [] {
    int dev = 0, sms = 0, ps = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(k_retrieve3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)retrieve_smem3<T>());
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, k_retrieve3<T>, kRThreads, retrieve_smem3<T>()) !=
        cudaSuccess) {
      cudaGetLastError();
      ps = 1;
    }
    return (int64_t)(ps < 1 ? 1 : ps) * (sms < 1 ? 1 : sms);
  }();
  return (int)(nunits < g ? (nunits > 0 ? nunits : 1) : g);
}

// How a job of ncomp components is decoded: in rounds of equal size of at most
// kRoundTasks components, units of so many bricks that a round has up to
// kRoundTasks warp tasks (4 where there is one component: its first planes are
// many).  Two or three components take fewer bricks, but no fewer than 3 tasks,
// where their blocks' plane words -- nearly the payload's words a brick -- would
// otherwise not fit in the pool: blocks past it take the decoding of any planes
// (192^3 float64, 2 components of 17 and 13 words 169 -> 139 us, 3 of 17, 13 and 13
// 211 -> 161; float32, 2 of 21 and 10 113 -> 87).  One component gains or loses
// little (0 to 10 %).
void retrieve_split(const uint64_t* words, int ncomp, int64_t nbricks, int* round, int* unit_bricks) {
  const int rounds = std::max((ncomp + kRoundTasks - 1) / kRoundTasks, 1);
  *round = std::max((ncomp + rounds - 1) / rounds, 1);
  int sets = *round == 1 ? 4 : std::max(kRoundTasks / *round, 1);
  if (rounds > 1) sets = 1;
  if (*round > 1) {
    uint64_t all = 0;  // the first round's words
    for (int i = 0; i < *round; ++i) all += words[i];
    while ((sets - 1) * *round >= 3 && 32.0 * sets * (double)all > (double)kPool * (double)nbricks) --sets;
  }
  *unit_bricks = 32 * sets;
}

// The unit of a job in a launch of `bricks` bricks: smaller ones where the units
// would otherwise not fill the GPU.
int retrieve_unit(int dtype, int unit_bricks, int64_t bricks) {
  const int64_t fit = dtype == 1 ? retrieve_grid_t<float>(INT64_MAX) : retrieve_grid_t<double>(INT64_MAX);
  while (unit_bricks > 32 && bricks < fit * unit_bricks) unit_bricks -= 32;
  return unit_bricks;
}

int retrieve_grid(int dtype, int ndims, int64_t nunits) {
  if (ndims != 3) return 1;  // the 1D/2D kernel is not persistent
  return dtype == 1 ? retrieve_grid_t<float>(nunits) : retrieve_grid_t<double>(nunits);
}

size_t retrieve_spill_words(int dtype, int ndims, int grid) {
  if (ndims != 3) return 0;
  return (dtype == 1 ? spill_words_per_cta<float>() : spill_words_per_cta<double>()) * (size_t)grid;
}

template <typename T>
static cudaError_t launch_retrieve_t(const RetrieveParams& p, cudaStream_t s) {
  const size_t smem = retrieve_smem3<T>();
  cudaError_t e = cudaFuncSetAttribute(k_retrieve3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (p.nunits == 0) return cudaSuccess;
  k_retrieve3<T><<<(unsigned)p.grid, kRThreads, smem, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_retrieve(int dtype, int ndims, const RetrieveParams& p, cudaStream_t s) {
  if (ndims == 1 || ndims == 2) return launch_retrieve_small(dtype, ndims, p, s);
  if (ndims != 3) return cudaErrorNotSupported;
  return dtype == 1 ? launch_retrieve_t<float>(p, s) : launch_retrieve_t<double>(p, s);
}

uint32_t check_word_retrieve(int reset) { return read_check_word(reset); }

}  // namespace pcz
