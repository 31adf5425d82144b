// pcz_chunk_small.cuh -- Algorithms 1 and 2 (Magri & Lindstrom, Sec. 4.1,
// 4.2) for 1D and 2D fields, whose bricks hold 4 and 16 values: one warp
// codes an index chunk of 32 bricks (a brick per lane, entirely in
// registers), one thread retrieves a brick.  Shared by the stand-alone
// kernels (pcz_small.cu) and the batched persistent kernel (pcz_batch.cu).
#pragma once

#include <type_traits>

#include "pcz_device.cuh"
#include "pcz_kernels.h"

namespace pcz {

constexpr int kSmallWarps = 4;  // chunks per CTA
constexpr int kSmallThreads = 32 * kSmallWarps;

// Largest coded block: the header, at most one verbatim or run bit per
// coefficient and plane, and at most one test bit per coefficient plus one
// closing test bit per plane (R11); RAW is shorter still.
template <typename T, int D>
__host__ __device__ constexpr int max_brick_bits_small() {
  return 2 + 3 + Fmt<T>::EBITS + Geo<D>::N * Fmt<T>::P + Geo<D>::N + Fmt<T>::P;
}

template <typename T, int D>
__host__ __device__ constexpr int chunk_words_small() {  // u32 words of one chunk buffer, whole 16-byte vectors
  return ((kChunk * max_brick_bits_small<T, D>() + 127) / 128) * 4;
}

// A warp's shared memory, in u32 words: the chunk's bits, each lane's own code
// before it is placed in the chunk (word w of lane l at 32 w + l) and the
// lanes' values (16-byte part h of lane l at vector 32 h + l).
template <typename T, int D>
struct SmallArea {
  static constexpr int kStageWords = max_brick_bits_small<T, D>() / 32 + 2;
  static constexpr int kStage = chunk_words_small<T, D>();
  static constexpr int kValues = (kStage + 32 * kStageWords + 3) / 4 * 4;
  static constexpr int kWords = kValues + 32 * Geo<D>::N * (int)(sizeof(T) / 4);
};

// Bytes of a CTA of `warps` warps: the warps' areas and the group-test table.
template <typename T, int D>
__host__ __device__ constexpr size_t small_smem(int warps) {
  return (size_t)warps * SmallArea<T, D>::kWords * 4 + kSpreadBytes;
}

// The CTA's copy of the group-test table, in shared memory; read after the next
// barrier.
template <int THREADS>
__device__ __forceinline__ const uint16_t* load_spread(void* at) {
  uint32_t* w = reinterpret_cast<uint32_t*>(at);
  for (int i = threadIdx.x; i < kSpreadBytes / 4; i += THREADS) w[i] = reinterpret_cast<const uint32_t*>(kSpread.code)[i];
  return reinterpret_cast<const uint16_t*>(at);
}

// R8: brick position (x + 4y) of the r-th coded coefficient.  The table is a
// compile-time constant, so with r known after unrolling the lookup folds
// away and the coefficient arrays stay in registers.
template <int D>
__device__ __forceinline__ int perm_small(int r) {
  if constexpr (D == 1) {
    return r;
  } else {
    constexpr PermTable t = make_perm(16);
    return t.pos[r];
  }
}

// lifting of the brick in registers: along x, then y (D = 2)
template <int D, typename S>
__device__ __forceinline__ void lift_fwd_brick(S* v) {
  constexpr int NY = D == 2 ? 4 : 1;
#pragma unroll
  for (int y = 0; y < NY; ++y) lift_fwd(v[4 * y], v[4 * y + 1], v[4 * y + 2], v[4 * y + 3]);
  if constexpr (D == 2) {
#pragma unroll
    for (int x = 0; x < 4; ++x) lift_fwd(v[x], v[x + 4], v[x + 8], v[x + 12]);
  }
}

template <int D, typename S>
__device__ __forceinline__ void lift_inv_brick(S* v) {
  constexpr int NY = D == 2 ? 4 : 1;
  if constexpr (D == 2) {
#pragma unroll
    for (int x = 0; x < 4; ++x) lift_inv(v[x], v[x + 4], v[x + 8], v[x + 12]);
  }
#pragma unroll
  for (int y = 0; y < NY; ++y) lift_inv(v[4 * y], v[4 * y + 1], v[4 * y + 2], v[4 * y + 3]);
}

// A lane's code under construction: bits are gathered in 64 and moved to the
// lane's column of the warp's stage 32 at a time.
struct LaneCode {
  uint32_t* col;  // word w of the column at col[32 w]
  int words, fill;
  uint64_t acc;
  int cap;  // words of the column
  __device__ __forceinline__ void drain() {
    while (fill >= 32) {
      if (PCZ_CHECK(words < cap, 2)) col[32 * words] = (uint32_t)acc;
      ++words;
      acc >>= 32;
      fill -= 32;
    }
  }
  __device__ __forceinline__ void put(uint64_t v, int nbits) {  // nbits <= 33
    acc |= v << fill;
    fill += nbits;
    drain();
  }
  __device__ __forceinline__ int finish() {  // the code's length in bits
    if (fill && PCZ_CHECK(words < cap, 2)) col[32 * words] = (uint32_t)acc;
    return 32 * words + fill;
  }
};

// Algorithm 1 on index chunk `chunk` (below the field's chunk count) of a 1D or
// 2D field, all components, by one warp: lane l codes brick 32 * chunk + l.
// area is the warp's own shared memory (SmallArea<T, D>), spread the CTA's
// group-test table.
//
// Everything of a brick is in its lane's registers.  The planes come from 8 x
// 16-bit transposes of the digits, aligned to the brick's highest plane that is
// not empty, so that step k of every lane is a plane of the same register; a
// plane's bits are formed at once (verbatim bits, and the group-test code
// through a byte table).  Bound by instruction issue.  With plane words gathered
// bit by bit, twice, and a loop over tokens it took 3932 warp instructions per
// 32 float32 2D bricks and component, now 1461; 4096^2 float32, 6
// components: 1.09 -> 0.35 ms.
template <typename T, int D>
__device__ __forceinline__ void compress_small_chunk(const CompressParams& P, int64_t chunk, uint32_t* area,
                                                     const uint16_t* spread) {
  using F = Fmt<T>;
  using U = typename F::U;
  using S = typename F::S;
  using A = SmallArea<T, D>;
  constexpr bool WIDE = F::P == 64;
  constexpr int N = Geo<D>::N;
  constexpr int Q = F::P - 2 - Geo<D>::G;
  constexpr int C = Geo<D>::C;
  constexpr int HDR = 2 + 3 + F::EBITS;
  constexpr int LEN_RAW = 2 + N * F::P;
  [[maybe_unused]] constexpr uint32_t CAP = (uint32_t)A::kStage * 32;  // bits of the chunk buffer
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int XV = 16 / (int)sizeof(T);

  const int lane = threadIdx.x & 31;
  const int64_t b = chunk * kChunk + lane;
  const bool have = b < P.nbricks;
  uint32_t* cbuf = area;
  uint32_t* col = area + A::kStage + lane;
  uint4* s_x = reinterpret_cast<uint4*>(area + A::kValues) + lane;
  for (int w = lane; w < A::kStage / 4; w += 32) reinterpret_cast<uint4*>(cbuf)[w] = make_uint4(0, 0, 0, 0);
  __syncwarp();

  // the values, with edge replication (R4)
  int64_t bx = 0, by = 0;
  if (have) {
    bx = b % P.nb[0];
    by = b / P.nb[0];
  }
  const int nvx = have ? (int)(P.dims[0] - 4 * bx < 4 ? P.dims[0] - 4 * bx : 4) : 4;
  const int nvy = (D == 2 && have) ? (int)(P.dims[1] - 4 * by < 4 ? P.dims[1] - 4 * by : 4) : (D == 2 ? 4 : 1);
  const bool any_partial = __any_sync(FULL, nvx < 4 || (D == 2 && nvy < 4));
  T xt[N], e[N];
  {
    const T* field = reinterpret_cast<const T*>(P.field);
#pragma unroll
    for (int j = 0; j < N / 4; ++j) {  // one x-line per row, rows past the field repeat the last
      if (have) {
        load_line<T>(field + (4 * by + min(j, nvy - 1)) * P.dims[0] + 4 * bx, nvx, &e[4 * j]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) e[4 * j + i] = T(0);
      }
    }
  }
  union Part {
    uint4 w;
    T v[XV];
    __device__ Part() {}
  };
#pragma unroll
  for (int h = 0; h < N / XV; ++h) {
    Part t;
#pragma unroll
    for (int o = 0; o < XV; ++o) t.v[o] = e[XV * h + o];
    s_x[32 * h] = t.w;
  }
  // r = x - a on the in-field values; padded ones copy the nearest in-field one
  // along x, then along y (R4)
  auto residual_of = [&](const T* a, T* r) {
#pragma unroll
    for (int h = 0; h < N / XV; ++h) {
      Part t;
      t.w = s_x[32 * h];
#pragma unroll
      for (int o = 0; o < XV; ++o) r[XV * h + o] = F::sub(t.v[o], a[XV * h + o]);
    }
    if (any_partial) {
#pragma unroll
      for (int j = 0; j < N / 4; ++j)
#pragma unroll
        for (int i = 1; i < 4; ++i)
          if (i >= nvx) r[i + 4 * j] = r[i - 1 + 4 * j];
#pragma unroll
      for (int j = 1; j < N / 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (j >= nvy) r[i + 4 * j] = r[i + 4 * (j - 1)];
    }
  };
#pragma unroll
  for (int k = 0; k < N; ++k) xt[k] = T(0);  // Algorithm 1 starts from x~ = 0: the first residual is x
  U m = lane_max<T, N>(e);
  if (__any_sync(FULL, m >= F::INF) && lane == 0) atomicOr(P.flags, kFlagNonFinite);

  for (int i = 0; i < P.n; ++i) {  // one component per tolerance
    const U tb = (U)P.tau_bits[i];
    const int L = P.L[i];
    const bool zero_blk = !have || m <= tb;  // R5
    const int be = (int)(m >> (F::MANT - 1));
    const bool coded = !zero_blk && be != (1 << F::EXPW) - 1;  // an infinite or NaN residual is RAW
    const int emax = block_emax_from_be<T>(be);
    const int s = coded ? Q - emax : 0;
    int esc = 0, p, top, nw;
    U u[N];
    T xtn[N], en[N];
    U mn;
    bool pass;
    for (;;) {  // again, with more planes in some brick, while Eq. 1 fails (R13): at most 8 times
      const bool common = __all_sync(FULL, WIDE ? s >= -960 && s <= 1000 : s >= -96 && s <= 126);
      S v[N];
      if (common) {  // R6, in the short forms of blocks with a common scale (as in pcz_chunk3.cuh)
        if constexpr (!WIDE) {
          const float sc = coded ? __uint_as_float((uint32_t)(127 + s) << 23) : 0.0f;
#pragma unroll
          for (int k = 0; k < N; ++k) v[k] = __float2int_rz(__fmul_rn(e[k], sc));
        } else {
          const int c = coded ? 1022 + Q - s : 4096;
#pragma unroll
          for (int k = 0; k < N; ++k) v[k] = quantize_f64_normal<Q - 53>(e[k], c);
        }
      } else {
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = coded ? quantize_any<T>(F::bits(e[k]), s) : S(0);
      }
      lift_fwd_brick<D>(v);  // R7
      U any = 0;
#pragma unroll
      for (int r = 0; r < N; ++r) {  // R8, R9
        u[r] = nb_fwd<T>(v[perm_small<D>(r)]);
        any |= u[r];
      }
      p = coded ? min(max(L + s - C - esc, 0), F::P) : F::P;  // R10
      top = any ? F::P - 1 - F::clz(any) : -1;
      nw = top - p + 1;  // planes from the highest that is not empty down to p
      // R13: decode-back, the candidate x~ + x_i and the residual it leaves;
      // bricks that are not coded decode to 0
      if constexpr (!WIDE) {
        S r[N];
        const U keep = __funnelshift_lc(0u, ~0u, p);
#pragma unroll
        for (int k = 0; k < N; ++k) r[perm_small<D>(k)] = nb_inv<T>(u[k] & keep);
        lift_inv_brick<D>(r);
        if (common) {
          const float sc = __uint_as_float((uint32_t)(127 - s) << 23);
#pragma unroll
          for (int k = 0; k < N; ++k) xtn[k] = __fmaf_rn(__int2float_rn(r[k]), sc, xt[k]);
        } else {
#pragma unroll
          for (int k = 0; k < N; ++k) xtn[k] = F::add(xt[k], F::val(dequantize_any<T>(r[k], s)));
        }
      } else {
        // 32-bit decode-back of digits within 20 planes from plane p in 32..57,
        // in units of 2^(p - 2 D): exact and without wrapping as in
        // pcz_chunk3.cuh, with D lifting passes for 3
        constexpr int SH = 2 * D;
        if (common && __all_sync(FULL, !coded || (nw <= 20 && p >= 32 && p <= 57))) {
          int32_t r[N];
          const uint32_t M = (uint32_t)(F::NBM >> min(p, 63));
#pragma unroll
          for (int k = 0; k < N; ++k) {
            const uint32_t w = __funnelshift_rc((uint32_t)(u[k] >> 32), 0u, p - 32);
            r[perm_small<D>(k)] = (int32_t)(((w ^ M) << SH) - (M << SH));
          }
          lift_inv_brick<D>(r);
          const uint32_t eb = (uint32_t)(1053 + (p - SH) - s) << 20;
#pragma unroll
          for (int k = 0; k < N; ++k) xtn[k] = F::add(xt[k], scaled_i32_to_f64(r[k], eb));
        } else {
          S r[N];
          const U keep = p >= F::P ? U(0) : ~U(0) << p;
#pragma unroll
          for (int k = 0; k < N; ++k) r[perm_small<D>(k)] = nb_inv<T>(u[k] & keep);
          lift_inv_brick<D>(r);
#pragma unroll
          for (int k = 0; k < N; ++k)
            xtn[k] = F::add(xt[k], F::val(common ? dequantize_f64_normal(r[k], s) : dequantize_any<T>(r[k], s)));
        }
      }
      residual_of(xtn, en);
      mn = lane_max<T, N>(en);
      pass = coded && mn <= tb;
      const bool again = coded && !pass && p > 0 && esc < 7;
      if (!__any_sync(FULL, again)) break;
      if (again) ++esc;
      residual_of(xt, e);
    }

    // R11: the brick's code, planes from the top down.  The planes above `top`
    // are one 0 test bit each.
    const int span = (int)__reduce_max_sync(FULL, (unsigned)(pass ? max(nw, 0) : 0));
    LaneCode code{col, 0, HDR, (uint64_t)kModeCoded | ((uint64_t)esc << 2) | ((uint64_t)(emax + F::EBIAS) << 5),
                  A::kStageWords};
    code.fill += F::P - max(top + 1, p);
    code.drain();
    const int lead = F::P - 1 - top;
    int n = 0;  // coefficients significant so far
    for (int half = 0; half <= (WIDE && span > 32 ? 1 : 0); ++half) {
      uint32_t al[N];  // 32 planes of each coefficient, the highest at bit 31
#pragma unroll
      for (int r = 0; r < N; ++r) {
        if constexpr (!WIDE) {
          al[r] = u[r] << (lead & 31);
        } else {
          const uint32_t lo = (uint32_t)u[r], hi = (uint32_t)(u[r] >> 32);
          const uint32_t w1 = lead < 32 ? hi : lo, w0 = lead < 32 ? lo : 0u;
          al[r] = half ? w0 << (lead & 31) : __funnelshift_l(w0, w1, lead & 31);
        }
      }
      const int end = min(span - 32 * half, 32);
      for (int k0 = 0; k0 < end; k0 += 8) {
        const uint32_t by8 = 3u - (uint32_t)(k0 >> 3), sel = 0x40u + 0x11u * by8;
        uint32_t a[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          if constexpr (N == 16)
            a[w] = __byte_perm(__byte_perm(al[w], al[w + 8], sel), __byte_perm(al[w + 4], al[w + 12], sel), 0x5410);
          else
            a[w] = __byte_perm(al[w], 0u, 0x4440u + by8);
        }
        transpose8(a);
        const int left = nw - 32 * half - k0, steps = min(end - k0, 8);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          if (kk >= steps) break;
          const uint32_t W = kk < 4 ? a[3 - kk] >> 16 : a[7 - kk] & 0xffffu;
          if (kk < left && pass) {
            const uint32_t rest = W >> n;
            uint64_t bits = W & ((1u << n) - 1u);
            int len = n;
            if (rest) {  // a first test 1, then the positions from n on through the byte table
              const uint32_t b0 = rest & 0xffu, b1 = rest >> 8;
              uint32_t c = spread[b0];
              if constexpr (N == 16) c |= (uint32_t)spread[b1] << (8 + __popc(b0));
              c ^= 0x80000000u >> __clz((int)c);  // no test 1 after the plane's last 1
              bits |= (uint64_t)(2u * c + 1u) << n;  // at most N - n coefficients: c is below 2^31
              n = 32 - __clz((int)W);
              len = n + __popc(rest);
            }
            code.put(bits, len + (n < N ? 1 : 0));
          }
        }
      }
    }
    const int lenC = code.finish();

    int mode = zero_blk ? kModeZero : pass ? kModeCoded : kModeRaw;
    int viol = 0;  // Eq. 1 failures left (only a RAW brick can have them)
    if (__any_sync(FULL, mode == kModeRaw || (pass && lenC > LEN_RAW))) {  // R14
      T eo[N], xr[N], er[N];
      residual_of(xt, eo);
#pragma unroll
      for (int k = 0; k < N; ++k) xr[k] = F::add(xt[k], eo[k]);
      residual_of(xr, er);
      const U mr = lane_max<T, N>(er);
      if (pass && lenC > LEN_RAW && mr <= tb) mode = kModeRaw;
      if (mode == kModeRaw) {
        mn = mr;
        LaneCode raw{col, 0, 2, (uint64_t)kModeRaw, A::kStageWords};
#pragma unroll
        for (int k = 0; k < N; ++k) {
          raw.put((uint32_t)F::bits(eo[k]), 32);
          if constexpr (WIDE) raw.put((uint32_t)(F::bits(eo[k]) >> 32), 32);
          xtn[k] = xr[k];
          en[k] = er[k];
          if ((k & 3) < nvx && (k >> 2) < nvy && magnitude(er[k]) > tb) ++viol;
        }
        raw.finish();
      }
    }
    if (mode == kModeZero) col[0] = 0u;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      xt[k] = xtn[k];
      e[k] = en[k];
    }
    m = mn;
    const int len = !have ? 0 : mode == kModeZero ? 2 : mode == kModeRaw ? LEN_RAW : lenC;

    // chunk layout: this brick's offset, pool space, index entries
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(FULL, incl, 31);
    const unsigned cw = (unsigned)((total + 63) >> 6);
    unsigned long long base = 0;
    if (lane == 0) base = cw ? atomicAdd(P.pool_used, (unsigned long long)cw) : 0ull;
    const uint32_t off = (uint32_t)(incl - len);
    if (have) {
      P.brick_len[(int64_t)i * P.nbricks + b] = (uint16_t)len;
      if (P.brick_off) P.brick_off[(int64_t)i * P.nbricks + b] = off;
    }
    // the brick's code, shifted to its place in the chunk
    const int words = (len + 31) >> 5, most = (int)__reduce_max_sync(FULL, (unsigned)words);
    uint32_t prev = 0;
    uint32_t* to = cbuf + (off >> 5);
    for (int w = 0; w <= most; ++w) {
      uint32_t x = w < words ? col[32 * w] : 0u;
      const uint32_t o = __funnelshift_l(prev, x, off);
      prev = x;
      if (o && PCZ_CHECK((off & ~31u) + 32u * (uint32_t)w < CAP, 2)) atomicOr(to + w, o);
    }
    // counters and the largest error (Sec. 4.3: the computed tolerance)
    const unsigned cz = __popc(__ballot_sync(FULL, have && mode == kModeZero));
    const unsigned cc = __popc(__ballot_sync(FULL, have && mode == kModeCoded));
    const unsigned cr = __popc(__ballot_sync(FULL, have && mode == kModeRaw));
    const unsigned se = __reduce_add_sync(FULL, have && mode == kModeCoded ? (unsigned)esc : 0u);
    const unsigned sv = __reduce_add_sync(FULL, have ? (unsigned)viol : 0u);
    unsigned long long me = have ? (unsigned long long)mn : 0ull;
    if constexpr (!WIDE)
      me = __reduce_max_sync(FULL, (unsigned)me);
    else
      me = warp_max_u64(FULL, me);
    if (lane == 0) {
      if (base + cw > P.pool_words) {
        atomicOr(P.flags, kFlagPoolOverflow);
        base = ~0ull;
      }
      const int64_t ci = (int64_t)i * P.nchunks + chunk;
      P.chunk_nwords[ci] = cw;
      P.chunk_pool[ci] = base;
      uint32_t* cnt = P.chunk_counts + ci * 5;
      cnt[0] = cz;
      cnt[1] = cc;
      cnt[2] = cr;
      cnt[3] = se;
      cnt[4] = sv;
      if (P.chunk_maxerr) P.chunk_maxerr[ci] = me;
    }
    base = __shfl_sync(FULL, base, 0);
    __syncwarp();
    uint64_t* b64 = reinterpret_cast<uint64_t*>(cbuf);
    for (unsigned wd = lane; wd < cw; wd += 32) {
      if (base != ~0ull) P.pool[base + wd] = b64[wd];
      b64[wd] = 0ull;
    }
    __syncwarp();
  }
}

// Retrieval of brick g (box order) of job J by one thread: components
// k0+1..k (at least one) parsed and rebuilt in ascending order and summed into x~
// (Algorithm 2).  No warp-collective operations.  tokens: the CTA's byte table of the
// group-test part (kTokens), there once ready() returns (false: this thread has no
// brick of its own); 1D requests the first block's bits before.
//
// A plane takes one look at the stream (at most 33 bits) and, while
// coefficients turn significant, a table step per byte; 8 planes at a time are
// transposed back into digits in registers, aligned to the brick's highest
// plane.  With planes scattered bit by bit into the coefficients and a loop over
// tokens it took 2877 warp instructions per 32 float32 2D bricks and component,
// now 1244; 4096^2 float32, k = 6: 659 -> 284 us.
template <typename T, int D, typename Ready>
__device__ __forceinline__ void retrieve_small_brick(const BoxJob& J, int write, unsigned int* err, int64_t g,
                                                     const uint32_t* tokens, Ready ready) {
  using F = Fmt<T>;
  using U = typename F::U;
  using S = typename F::S;
  constexpr bool WIDE = F::P == 64;
  constexpr int N = Geo<D>::N;
  constexpr int Q = F::P - 2 - Geo<D>::G;
  constexpr int C = Geo<D>::C;
  constexpr int HDR = 2 + 3 + F::EBITS;
  constexpr int EMAXT = (1 << (F::EXPW - 1));
  const int64_t bx = J.bl[0] + g % J.bn[0];
  const int64_t by = D == 2 ? J.bl[1] + g / J.bn[0] : 0;
  const int64_t b = bx + J.nb[0] * by;
  const int64_t ext0 = J.hi[0] - J.lo[0];
  // values [x0, x1) of rows [y0, y1) of the brick lie in the box (and the field)
  const int x0 = (int)max(J.lo[0] - 4 * bx, (int64_t)0), x1 = (int)min(J.hi[0] - 4 * bx, (int64_t)4);
  const int y0 = D == 2 ? (int)max(J.lo[1] - 4 * by, (int64_t)0) : 0;
  const int y1 = D == 2 ? (int)min(J.hi[1] - 4 * by, (int64_t)4) : 1;
  T* out = reinterpret_cast<T*>(J.out) + (4 * by - J.lo[1]) * ext0 + (4 * bx - J.lo[0]);
  T xt[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    xt[k] = T(0);
    if (write && J.k0 > 0 && (k & 3) >= x0 && (k & 3) < x1 && (k >> 2) >= y0 && (k >> 2) < y1)
      xt[k] = out[(k >> 2) * ext0 + (k & 3)];  // the partial sum so far
  }
  const int64_t chunk = b / kChunk;
  uint32_t blen, pos;
  BlockBits br;  // positions from the start of the block's first word
  auto block = [&](const CompDesc& cd) {
    const uint64_t off = cd.chunk_word[chunk] * 64ull + cd.brick_off[b];
    blen = cd.brick_len[b];
    br.init(cd.payload, cd.nwords, off);
    pos = (uint32_t)(off & 63u);
  };
  if constexpr (D == 1) block(J.comp[J.k0]);  // (2D has no registers for it: k = 6 2 % slower)
  if (!ready()) return;
  for (int j = J.k0; j < J.k; ++j) {  // Algorithm 2: x~ += D(y_j)
    if (D == 2 || j > J.k0) block(J.comp[j]);
    const uint32_t end = pos + blen;
    const uint64_t v = br.peek(pos);
    const int mode = (int)(v & 3ull);
    T xi[N];
#pragma unroll
    for (int k = 0; k < N; ++k) xi[k] = T(0);
    bool ok = true;
    if (mode == kModeZero) {
      ok = blen == 2;
    } else if (mode == kModeRaw) {
      ok = blen == 2 + N * F::P;
      if (ok) {
#pragma unroll
        for (int k = 0; k < N; ++k) xi[k] = F::val((U)br.peek(pos + 2 + F::P * k));
      }
    } else if (mode == kModeCoded) {
      const int esc = (int)((v >> 2) & 7ull);
      const int emax = (int)((v >> 5) & ((1ull << F::EBITS) - 1)) - F::EBIAS;
      ok = emax >= F::EMIN && emax <= EMAXT;
      if (ok) {
        const int s = Q - emax;
        const int p = min(max(J.comp[j].L + s - C - esc, 0), F::P);
        pos += HDR;
        int top = F::P - 1;  // highest plane with a significant coefficient; planes above it are a 0 test bit each
        while (top >= p) {
          const uint64_t t = br.peek(pos);
          const int z = t ? __ffsll((long long)t) - 1 : 64;
          const int skip = min(z, top - p + 1);
          pos += (uint32_t)skip;
          top -= skip;
          if (z < 64) break;
        }
        const int nw = top - p + 1;
        uint32_t al[N], al2[N];  // digits, plane top at bit 31 of al; al2 (float64): the 32 planes below
#pragma unroll
        for (int r = 0; r < N; ++r) al[r] = al2[r] = 0u;
        int n = 0;
        uint32_t q3 = 0, q2 = 0, q1 = 0, q0 = 0;  // the last 8 planes, the first in q3's upper half
        for (int k0 = 0; k0 < nw; k0 += 8) {
#pragma unroll 1
          for (int k = k0; k < k0 + 8; ++k) {
            uint32_t W = 0;
            if (k < nw && ok) {  // R11
              const uint64_t w64 = br.peek(pos);
              W = (uint32_t)w64 & ((1u << n) - 1u);
              uint32_t used = (uint32_t)n;
              if (n < N) {
                const uint64_t gb = w64 >> n;
                uint32_t gl = (uint32_t)gb, gh = (uint32_t)(gb >> 32), e = 0, idx = 0, o = 0;
                int cnt = 0;
                // a valid part is at most 2 (N - n) + 1 bits; left at one place for
                // all lanes (see pcz_retrieve.cu)
#pragma unroll 1
                for (int t = N == 16 ? 5 : 2; t > 0; --t) {
                  idx = token_index(e, gl, 0);
                  e = tokens[idx];
                  cnt = token_count(e);
                  o = e & 0xffu;
                  W |= o << n;
                  if (n + cnt >= N || (int32_t)e < 0) break;
                  n += cnt;
                  cnt = 0;
                  used += 8;
                  gl = __funnelshift_r(gl, gh, 8);
                  gh >>= 8;
                }
                if (n + cnt >= N) {  // the last coefficient's 1 ends it, with no closing test bit
                  const int l = N - 1 - n;
                  ok = (o >> l) & 1u;
                  W &= (1u << N) - 1u;
                  used += (uint32_t)(l + 1) + (idx < 256u ? 1u : 0u) + (uint32_t)__popc(o & ((1u << l) - 1u));
                  n = N;
                } else {
                  ok = (int32_t)e < 0;
                  used += ((e >> 24) & 7u) + 1u;
                  n += cnt;
                }
              }
              pos += used;
              if (pos > end) ok = false;
            }
            q3 = __funnelshift_l(q2, q3, 16);
            q2 = __funnelshift_l(q1, q2, 16);
            q1 = __funnelshift_l(q0, q1, 16);
            q0 = (q0 << 16) | W;
          }
          // back to a byte per coefficient
          uint32_t a[4] = {__byte_perm(q0, q2, 0x5410), __byte_perm(q0, q2, 0x7632), __byte_perm(q1, q3, 0x5410),
                           __byte_perm(q1, q3, 0x7632)};
          untranspose8(a);
          const uint32_t to = 12u - ((uint32_t)k0 >> 1 & 12u);  // selector nibble of the bytes' place: 3, 2, 1, 0
#pragma unroll
          for (int r = 0; r < N; ++r) {  // byte of rank r: word r & 3, byte (r >> 3) + 2 ((r >> 2) & 1)
            const uint32_t from = (uint32_t)((r >> 3) + 2 * ((r >> 2) & 1));
            const uint32_t d = __byte_perm(a[r & 3], 0u, 0x4444u ^ ((4u ^ from) << to));
            if (!WIDE || k0 < 32)
              al[r] |= d;
            else
              al2[r] |= d;
          }
        }
        if (ok && pos != end) ok = false;
        const int lead = F::P - 1 - top;
        bool done = false;
        if constexpr (WIDE) {
          // digits within 20 planes: decoded in 32-bit integers in units of
          // 2^(p - 2 D) (exact and without wrapping: see pcz_retrieve.cu, with D
          // lifting passes for 3)
          constexpr int SH = 2 * D;
          if (nw <= 20 && p >= SH && top <= 58 && s >= -960 && s <= 1022) {
            int32_t q[N];
            const uint32_t M = (uint32_t)(F::NBM >> min(p, 63));
#pragma unroll
            for (int r = 0; r < N; ++r) {
              const uint32_t w = __funnelshift_rc(al[r], 0u, 32 - nw);
              q[perm_small<D>(r)] = (int32_t)(((w ^ M) << SH) - (M << SH));
            }
            lift_inv_brick<D>(q);
            const uint32_t eb = (uint32_t)(1053 + (p - SH) - s) << 20;
#pragma unroll
            for (int k = 0; k < N; ++k) xi[k] = scaled_i32_to_f64(q[k], eb);
            done = true;
          }
        }
        if (!done) {
          S q[N];
#pragma unroll
          for (int r = 0; r < N; ++r) {
            U u;
            if constexpr (WIDE)
              u = lead < 64 ? (((U)al[r] << 32) | al2[r]) >> lead : U(0);
            else
              u = __funnelshift_rc(al[r], 0u, lead);
            q[perm_small<D>(r)] = nb_inv<T>(u);
          }
          lift_inv_brick<D>(q);
          const bool common = WIDE ? s >= -960 && s <= 1022 : s >= -127 && s <= 126;
          if (common) {
#pragma unroll
            for (int l = 0; l < N / 4; ++l) dequantize_line<T, true>(q + 4 * l, s, xi + 4 * l);
          } else {
#pragma unroll
            for (int k = 0; k < N; ++k) xi[k] = F::val(dequantize_any<T>(q[k], s));
          }
        }
      }
    } else {
      ok = false;
    }
    if (!ok) {
      atomicOr(err, 1u);
#pragma unroll
      for (int k = 0; k < N; ++k) xi[k] = T(0);
    }
#pragma unroll
    for (int k = 0; k < N; ++k) xt[k] = F::add(xt[k], xi[k]);
  }
  if (write) {
#pragma unroll
    for (int l = 0; l < N / 4; ++l) {
      bool vm[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) vm[k] = k >= x0 && k < x1 && l >= y0 && l < y1;
      store_line<T>(out + l * ext0, &xt[4 * l], vm);
    }
  }
}

}  // namespace pcz
