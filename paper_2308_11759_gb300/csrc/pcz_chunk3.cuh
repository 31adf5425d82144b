// pcz_chunk3.cuh -- Algorithm 1 (Magri & Lindstrom, Sec. 4.1) on one index
// chunk of 32 bricks of a 3D field, all components, by one CTA: the body of
// the construction kernel (pcz_compress.cu) and of the batched persistent
// kernel (pcz_batch.cu).  The layout and the coding steps are described in
// pcz_compress.cu.
#pragma once

#include <climits>
#include <type_traits>

#include <cuda.h>  // CUtensorMap (the type only; the library links no driver API)

#include "pcz_device.cuh"
#include "pcz_kernels.h"

namespace pcz {

static __constant__ PermTable kRank3 = make_rank();

// Largest bit string of one brick and component: the header, at most one
// verbatim or run bit per coefficient and plane, and at most one test bit per
// coefficient plus one closing test bit per plane (R11); RAW is shorter still.
template <typename T>
__host__ __device__ constexpr int max_brick_bits3() {
  return 2 + 3 + Fmt<T>::EBITS + 64 * Fmt<T>::P + 64 + Fmt<T>::P;
}

template <typename T>
__host__ __device__ constexpr int chunk_buf_words3() {  // u32 words, whole 16-byte vectors
  return ((kChunk * max_brick_bits3<T>() + 127) / 128) * 4;
}

constexpr int kCompressThreads3 = 128;  // threads that code a chunk: 4 warps of 8 bricks
constexpr int kWarps3 = kCompressThreads3 / 32;

// A warp's work area in shared memory, in u32 words.  Three uses follow one
// another within a component:
//  (a) the exchanges of the lifting passes (LineSet; float64: two sets);
//  (b) the digits in coded order, brick b from word 72 b (36 b as halves, 20 b
//      as bytes);
//  (c) the plane words, brick b from word b * kPlaneStride: word j of the
//      lane's 16 coefficients q at 4 j + q; a RAW brick's residual in their place.
template <typename T>
struct Area3 {
  static constexpr int kWords = LineSet::kVectors * 4 * (int)(sizeof(T) / 4);
  static constexpr int kPlaneStride = 16 * (int)sizeof(T) + 4;
  static constexpr int kInfoStride = Fmt<T>::P + 4;                       // plane table, words per brick
};

// Bytes of the staging area in front of the rest (TMA-staged form only).
template <typename T>
__host__ __device__ constexpr size_t staging_bytes3(bool staged) {
  return staged ? (size_t)kChunk * 64 * sizeof(T) + 16 : 0;  // the chunk's field values and a barrier
}

template <typename T>
__host__ __device__ constexpr size_t compress_smem3(bool staged = false) {
  return staging_bytes3<T>(staged)
         + (size_t)chunk_buf_words3<T>() * 4                        // chunk bit buffer
         + (size_t)kWarps3 * Area3<T>::kWords * 4                   // work areas
         + (size_t)kChunk * Area3<T>::kInfoStride * 4               // plane offsets and counts
         + (size_t)kChunk * 64 * sizeof(T)                          // the chunk's values
         + kSpreadBytes                                             // group-test code table
         + 4 * 32 * 4                                               // lengths, modes, escalations, violations
         + 32 * 8                                                   // per brick: bits of max |x - x~_i|
         + 16;                                                      // pool base and chunk bits
}

// The barrier of the 4 warps that code a chunk (id 0 in CTAs of 4 warps).
__device__ __forceinline__ void group_sync(int id) {
  asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory");
}

// The largest magnitude of a brick: over a lane's 16 values, then its 4 lanes.
template <typename T>
__device__ __forceinline__ typename Fmt<T>::U brick_max(const T* e) {
  using U = typename Fmt<T>::U;
  U m = lane_max<T, 16>(e);
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    const U a = __shfl_xor_sync(0xffffffffu, m, o);
    m = a > m ? a : m;
  }
  return m;
}

// R4 padding of a brick in a lane's layout (value x + 4 y, plane z = q):
// values past the field repeat the nearest in-field value along x, then y,
// then z.  Every lane of the warp calls it.
template <typename T>
__device__ __forceinline__ void pad_brick(T* e, int nvx, int nvy, int nvz, int lane) {
#pragma unroll
  for (int y = 0; y < 4; ++y)
#pragma unroll
    for (int x = 1; x < 4; ++x)
      if (x >= nvx) e[x + 4 * y] = e[x - 1 + 4 * y];
#pragma unroll
  for (int y = 1; y < 4; ++y)
#pragma unroll
    for (int x = 0; x < 4; ++x)
      if (y >= nvy) e[x + 4 * y] = e[x + 4 * (y - 1)];
  const int src = (lane & ~3) | min(lane & 3, nvz - 1);
#pragma unroll
  for (int v = 0; v < 16; ++v) e[v] = __shfl_sync(0xffffffffu, e[v], src);
}

// Bits 0 .. n - 1 of a 64-bit mask, n in 0..64.
__device__ __forceinline__ void low_mask(int n, uint32_t* lo, uint32_t* hi) {
  asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(*lo) : "r"(n));
  asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(*hi) : "r"(max(n - 32, 0)));
}

// OR of the three words that 64 bits hi:lo span from bit pos of a bit buffer.
__device__ __forceinline__ void or_words(uint32_t* buf, uint32_t pos, uint32_t lo, uint32_t hi) {
  uint32_t* w = buf + (pos >> 5);
  const uint32_t a = lo << (pos & 31u), b = __funnelshift_l(lo, hi, pos), c = __funnelshift_l(hi, 0u, pos);
  if (a) atomicOr(w, a);
  if (b) atomicOr(w + 1, b);
  if (c) atomicOr(w + 2, c);
}

// The plane word at plane p + j of a brick (layout of Area3's use (c)): its two
// halves, from the 4 lanes' 16 coefficients each; 0 for j < 0.
template <bool WIDE>
__device__ __forceinline__ void plane_at(const uint32_t* planes, int j, int H, uint32_t* lo, uint32_t* hi) {
  const int at = 4 * (j & (H - 1)) + (WIDE && j >= 32 ? 64 : 0);
  const uint4 r = *reinterpret_cast<const uint4*>(planes + at);
  const uint32_t sel = j & H ? 0x7632u : 0x5410u;
  *lo = j >= 0 ? __byte_perm(r.x, r.y, sel) : 0u;
  *hi = j >= 0 ? __byte_perm(r.z, r.w, sel) : 0u;
}

// Staging of a chunk's field values in shared memory with TMA (the
// persistent construction kernel, pcz_compress.cu): when the field's rows of
// bricks are whole chunks (bricks per row a multiple of 32), a chunk is one
// 128x4x4 box of the field, copied with one TMA tile copy ("row" layout: value
// (x, y, z) of the box at xs + 512 z + 128 y + x); otherwise one tile copy per
// brick of 4x4x4 boxes ("brick" layout: brick slot j at xs + 64 j, x
// fastest).  The copies signal an mbarrier by their bytes.  Values past the
// field's end arrive as zeros and are never used: readers clamp to the last
// in-field line and value (rule R4).
// Waits for the barrier's phase with parity `parity` to complete, at most
// `limit` polls (each poll may itself suspend the thread for a while); false
// when it gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int limit) {
  const uint32_t a = smem_addr(bar);
  for (int it = 0; it < limit; ++it) {
    uint32_t done = 0;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Issued by one thread: the copies of chunk `chunk` into xs, completing the
// barrier's current phase.
template <typename T>
__device__ __forceinline__ void issue_chunk_copy(const CompressParams& P, const CUtensorMap* map, bool row_box,
                                                 int64_t chunk, T* xs, uint64_t* bar) {
  const int64_t b0 = chunk * kChunk;
  const int nb = (int)(P.nbricks - b0 < kChunk ? P.nbricks - b0 : kChunk);
  const uint32_t bytes = (uint32_t)(row_box ? kChunk : nb) * 64u * (uint32_t)sizeof(T);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
  for (int j = 0; j < (row_box ? 1 : nb); ++j) {
    const int64_t b = b0 + j;
    const int64_t cx = b % P.nb[0], r = b / P.nb[0];
    const int x = (int)(4 * cx), y = (int)(4 * (r % P.nb[1])), z = (int)(4 * (r / P.nb[1]));
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
        "%4}], [%5];" ::"r"(smem_addr(xs + 64 * j)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
        : "memory");
  }
}

// This lane's x-line of its brick from the staged values (R4: the nearest
// in-field line and, along x, the last in-field value).
template <typename T>
__device__ __forceinline__ void staged_line(const T* xs, bool row_box, int slot, int ly, int lz, int nvx, int nvy,
                                            int nvz, T* v) {
  const int y = min(ly, nvy - 1), z = min(lz, nvz - 1);
  const T* src = row_box ? xs + 512 * z + 128 * y + 4 * slot : xs + 64 * slot + 16 * z + 4 * y;
  if (nvx == 4) {
    if constexpr (sizeof(T) == 4) {
      const float4 a = *reinterpret_cast<const float4*>(src);
      v[0] = a.x;
      v[1] = a.y;
      v[2] = a.z;
      v[3] = a.w;
    } else {
      const double2 a = reinterpret_cast<const double2*>(src)[0];
      const double2 b = reinterpret_cast<const double2*>(src)[1];
      v[0] = a.x;
      v[1] = a.y;
      v[2] = b.x;
      v[3] = b.y;
    }
    return;
  }
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = src[min(m, nvx - 1)];
}

// Copies a component's finished chunk from its shared buffer to the pool
// (base ~0: the pool was too small) and clears the buffer for reuse.
__device__ __forceinline__ void append_chunk(const CompressParams& P, uint32_t* buf, unsigned long long base,
                                             int chunk_bits, int tid) {
  const int nw = (chunk_bits + 63) >> 6;
  uint64_t* b64 = reinterpret_cast<uint64_t*>(buf);
  for (int w = tid; w < nw; w += kCompressThreads3) {
    if (base != ~0ull) P.pool[base + w] = b64[w];
    b64[w] = 0ull;
  }
}

// r = x - a, padded: x in shared memory, part h of the lane's at s_x[h * threads].
template <typename T>
__device__ __forceinline__ void residual_from(const uint4* s_x, bool any_partial, int nvx, int nvy, int nvz, int lane,
                                              const T* a, T* r) {
  constexpr int XV = 16 / (int)sizeof(T);  // values of a 16-byte part
  union Part {
    uint4 w;
    T v[XV];
    __device__ Part() {}
  };
#pragma unroll
  for (int h = 0; h < 16 / XV; ++h) {
    Part t;
    t.w = s_x[h * kCompressThreads3];
#pragma unroll
    for (int o = 0; o < XV; ++o) r[XV * h + o] = Fmt<T>::sub(t.v[o], a[XV * h + o]);
  }
  if (any_partial) pad_brick<T>(r, nvx, nvy, nvz, lane);
}

// A RAW block's outcome (R14), out of line: a holds x~ and receives the residual
// that is stored, xr x~ and er the residual after it; returns the brick's largest
// |er|.  (In line it made float64 spill 520 bytes a thread, now 12: 256 x 384 x
// 384, 12 components, 3.21 -> 3.10 ms.)
template <typename T>
static __device__ __noinline__ typename Fmt<T>::U raw_form(const uint4* s_x, bool any_partial, int nvx, int nvy, int nvz,
                                                           int lane, T* a, T* xr, T* er) {
  T e[16], x[16], r[16];
  residual_from<T>(s_x, any_partial, nvx, nvy, nvz, lane, a, e);
#pragma unroll
  for (int k = 0; k < 16; ++k) x[k] = Fmt<T>::add(a[k], e[k]);
  residual_from<T>(s_x, any_partial, nvx, nvy, nvz, lane, x, r);
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    a[k] = e[k];
    xr[k] = x[k];
    er[k] = r[k];
  }
  return brick_max<T>(r);
}

// Algorithm 1 on every brick of index chunk `chunk` of a 3D field, all
// components, by 4 warps (barrier `bar_id`); smem holds compress_smem3<T>(map
// != nullptr) bytes, 128-byte aligned.  With a tensor map, xs (= smem) holds
// the chunk's field values staged by TMA (row layout when row_box, brick layout
// otherwise): each lane reads its lines from there, and after a barrier thread
// 0 starts the copy of chunk `next` (if below nchunks) into xs on barrier
// `bar`, so that it lands while this chunk is coded.  Without a tensor map each
// lane loads its lines from the field with vector loads.  Every thread of the
// 4 warps must call it.
//
// A warp codes 8 bricks, 4 lanes each; lane q of a brick holds the z-plane q
// (16 values), and after the forward transform the coefficients of the y-plane
// q.  The kernel is bound by instruction issue, and this split spends the
// fewest: both in-plane lifting passes run in registers, the bits are
// transposed in registers, reductions over a brick take two shuffles, and what
// a component costs per warp (votes, scans, the barrier) is shared by 512
// values.  With 16 lanes per brick and 4 values per lane it took 582 (float32)
// and 997 (float64) warp instructions per brick and component, now 187 and 270;
// 512^3 float32, 8 components: 10.16 -> 3.52 ms, 256 x 384 x 384 float64, 12
// components: 8.77 -> 3.10 ms.  It runs at 0.71 (float32; ALU pipe 0.67) and
// 0.47 (float64) of the issue peak.
template <typename T>
__device__ __forceinline__ void compress3_chunk(const CompressParams& P, int64_t chunk, unsigned char* smem,
                                                int bar_id = 0, const CUtensorMap* map = nullptr,
                                                bool row_box = false, uint64_t* bar = nullptr, int64_t next = -1) {
  using F = Fmt<T>;
  using U = typename F::U;
  using S = typename F::S;
  using A3 = Area3<T>;
  constexpr bool WIDE = F::P == 64;
  constexpr int XV = 16 / (int)sizeof(T);  // values of a 16-byte part
  constexpr int Q = F::P - 2 - Geo<3>::G;  // quantisation bits (R6)
  constexpr int C = Geo<3>::C;             // guard planes (R10)
  constexpr int HDR = 2 + 3 + F::EBITS;    // mode, escalation, block exponent
  constexpr int LEN_RAW = 2 + 64 * F::P;
  constexpr int BUFW = chunk_buf_words3<T>();
  constexpr uint32_t CAP = (uint32_t)BUFW * 32;  // bits of the chunk buffer
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int SET = LineSet::kVectors;

  uint32_t* cbuf = reinterpret_cast<uint32_t*>(smem + staging_bytes3<T>(map != nullptr));
  uint32_t* areas = cbuf + BUFW;
  uint32_t* infos = areas + kWarps3 * A3::kWords;  // [brick][k]: plane offset << 8 | n
  uint4* s_x = reinterpret_cast<uint4*>(infos + kChunk * A3::kInfoStride);  // [16-byte part][thread]
  uint16_t* s_spread = reinterpret_cast<uint16_t*>(s_x + kChunk * 64 * sizeof(T) / 16);
  int* s_len = reinterpret_cast<int*>(s_spread + 256);
  int* s_mode = s_len + 32;
  int* s_esc = s_mode + 32;
  int* s_viol = s_esc + 32;
  uint64_t* s_merr = reinterpret_cast<uint64_t*>(s_viol + 32);
  unsigned long long* s_base = reinterpret_cast<unsigned long long*>(s_merr + 32);
  int* s_cbits = reinterpret_cast<int*>(s_base + 1);

  const int tid = threadIdx.x & (kCompressThreads3 - 1), warp = tid >> 5, lane = tid & 31;
  const int bq = lane >> 2, q = lane & 3;  // brick of the warp, z- or y-plane of the brick
  const int slot = warp * 8 + bq;
  const int64_t b = chunk * kChunk + slot;
  const bool have = b < P.nbricks;

  for (int w = tid; w < BUFW / 4; w += kCompressThreads3) reinterpret_cast<uint4*>(cbuf)[w] = make_uint4(0, 0, 0, 0);
  reinterpret_cast<uint32_t*>(s_spread)[tid] = reinterpret_cast<const uint32_t*>(kSpread.code)[tid];
  static_assert(kSpreadBytes == 4 * kCompressThreads3, "one word per thread");

  int64_t bx = 0, by = 0, bz = 0;
  if (have) {
    bx = b % P.nb[0];
    const int64_t r = b / P.nb[0];
    by = r % P.nb[1];
    bz = r / P.nb[1];
  }
  int nvx = 4, nvy = 4, nvz = 4;  // in-field extent of the brick per axis
  if (have) {
    nvx = (int)(P.dims[0] - 4 * bx < 4 ? P.dims[0] - 4 * bx : 4);
    nvy = (int)(P.dims[1] - 4 * by < 4 ? P.dims[1] - 4 * by : 4);
    nvz = (int)(P.dims[2] - 4 * bz < 4 ? P.dims[2] - 4 * bz : 4);
  }
  const bool any_partial = __any_sync(FULL, nvx < 4 || nvy < 4 || nvz < 4);

  // The values, padded (R4), are kept in shared memory, each lane's own, and
  // read back once per component: that leaves float32 the registers for 6 CTAs
  // per SM instead of 4 (512^3, 8 components: 3.98 -> 3.55 ms).  Algorithm 1
  // starts from x~ = 0, so the first residual is x itself (x - 0 in IEEE
  // arithmetic, -0 included).
  T xt[16], e[16];
  if (have) {
    const T* field = reinterpret_cast<const T*>(P.field);
    const int64_t gz = 4 * bz + min(q, nvz - 1);
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      if (map)
        staged_line<T>(reinterpret_cast<const T*>(smem), row_box, slot, y, q, nvx, nvy, nvz, e + 4 * y);
      else
        load_line<T>(field + (gz * P.dims[1] + 4 * by + min(y, nvy - 1)) * P.dims[0] + 4 * bx, nvx, e + 4 * y);
    }
  } else {
#pragma unroll
    for (int v = 0; v < 16; ++v) e[v] = T(0);
  }
  if (map) {
    group_sync(bar_id);  // every lane has its values: xs is free for the next chunk
    if (tid == 0 && next >= 0 && next < P.nchunks) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the reads above before the copy's writes
      issue_chunk_copy<T>(P, map, row_box, next, reinterpret_cast<T*>(smem), bar);
    }
  }
#pragma unroll
  for (int v = 0; v < 16; ++v) xt[v] = T(0);
  union Part {
    uint4 w;
    T v[XV];
    __device__ Part() {}
  };
#pragma unroll
  for (int h = 0; h < 16 / XV; ++h) {
    Part t;
#pragma unroll
    for (int o = 0; o < XV; ++o) t.v[o] = e[XV * h + o];
    s_x[h * kCompressThreads3 + tid] = t.w;
  }
  // r = x - a, padded
  auto residual_of = [&](const T* a, T* r) { residual_from<T>(s_x + tid, any_partial, nvx, nvy, nvz, lane, a, r); };
  U m = brick_max<T>(e);  // the largest magnitude of the residual, by brick
  if (__any_sync(FULL, m >= F::INF) && lane == 0) atomicOr(P.flags, kFlagNonFinite);

  uint32_t* area = areas + warp * A3::kWords;
  uint4* zw = reinterpret_cast<uint4*>(area) + LineSet::at(bq, 0, q);  // + 2 y: line (y, z = q)
  uint4* yw = reinterpret_cast<uint4*>(area) + LineSet::at(bq, q, 0);  // + 10 z: line (y = q, z)
  uint32_t* planes = area + bq * A3::kPlaneStride;
  uint32_t* info = infos + slot * A3::kInfoStride;
  uint32_t place[4];  // coded places of the lane's coefficients x + 4 z (y = q)
#pragma unroll
  for (int z = 0; z < 4; ++z) place[z] = coded_places(kRank3.pos, q, z);

  for (int i = 0; i < P.n; ++i) {  // one component per tau_i
    const U tb = (U)P.tau_bits[i];
    const int L = P.L[i];
    // R5: a brick whose residual meets tau_i is ZERO.  R6: the block exponent
    // comes from the largest magnitude; an infinite or NaN residual forces RAW.
    const bool zero_blk = !have || m <= tb;
    const int be = (int)(m >> (F::MANT - 1));
    const bool coded = !zero_blk && be != (1 << F::EXPW) - 1;
    const int emax = block_emax_from_be<T>(be);
    const int s = coded ? Q - emax : 0;
    int esc = 0;
    for (;;) {  // again, with more planes in some brick, while Eq. 1 fails (R13): at most 8 times
      // The blocks' common scales let every value take the short forms of R6
      // and R13; other scales take the general ones.
      const bool common = __all_sync(FULL, WIDE ? s >= -960 && s <= 1000 : s >= -96 && s <= 126);
      S v[16];
      if constexpr (!WIDE) {
        if (common) {
          // e * 2^s is exact whenever |q| >= 1 (at most 2^Q, no overflow; a
          // product below the normal range truncates to 0 either way), so
          // truncating the product is the R6 quantisation.  0 where not coded.
          const float sc = coded ? __uint_as_float((uint32_t)(127 + s) << 23) : 0.0f;
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = __float2int_rz(__fmul_rn(e[k], sc));
        } else {
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = coded ? quantize_any<T>(F::bits(e[k]), s) : S(0);
        }
      } else {
        if (common) {
          const int c = coded ? 1022 + Q - s : 4096;
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = quantize_f64_normal<Q - 53>(e[k], c);
        } else {
#pragma unroll
          for (int k = 0; k < 16; ++k) v[k] = coded ? quantize_any<T>(F::bits(e[k]), s) : S(0);
        }
      }
      lift_fwd_bricks<S>(v, zw, yw, SET);  // R7
      // R9, and the highest plane that is not empty.  Float64 takes it from the
      // high words; where they are empty in a coded brick, from the low ones.
      uint32_t any = 0;
      int top = -1;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const U u = nb_fwd<T>(v[k]);
        any |= (uint32_t)(u >> (F::P - 32));
        v[k] = (S)u;
      }
      any |= __shfl_xor_sync(FULL, any, 1);
      any |= __shfl_xor_sync(FULL, any, 2);
      if (any) top = F::P - 1 - __clz((int)any);
      if constexpr (WIDE) {
        if (__any_sync(FULL, coded && !any)) {
          uint32_t low = 0;
#pragma unroll
          for (int k = 0; k < 16; ++k) low |= (uint32_t)v[k];
          low |= __shfl_xor_sync(FULL, low, 1);
          low |= __shfl_xor_sync(FULL, low, 2);
          if (!any && low) top = 31 - __clz((int)low);
        }
      }
      // R10: the lowest coded plane
      const int p = coded ? min(max(L + s - C - esc, 0), F::P) : F::P;
      const int nw = top - p + 1;  // planes from the highest that is not empty down to p
      const int span = (int)__reduce_max_sync(FULL, (unsigned)max(nw, 0));

      // the coded digits, from plane p up: 32 of them (float64 where p >= 32 ...)
      auto digits = [&](int k) {
        if constexpr (WIDE)
          return __funnelshift_rc((uint32_t)((U)v[k] >> 32), 0u, p - 32);
        else
          return __funnelshift_rc((uint32_t)v[k], 0u, p);
      };
      auto digits64 = [&](int k) { return p >= F::P ? U(0) : (U)v[k] >> (p & (F::P - 1)); };  // (... and all)

      // the digits in coded order (R8), 16 ranks per lane, and their transpose:
      // plane words from word 4 j + q of the brick's plane area
      auto planes8 = [&](const uint32_t* w) {
        const uint32_t put = smem_addr(area + 20 * bq);
#pragma unroll
        for (int k = 0; k < 16; ++k)  // the address: put + byte k & 3 of place
          asm volatile("st.shared.u8 [%0], %1;" ::"r"(__dp4a(place[k >> 2], 1u << (8 * (k & 3)), put)), "r"(w[k])
                       : "memory");
        __syncwarp();
        const uint4 r = *reinterpret_cast<const uint4*>(area + 20 * bq + 4 * q);
        uint32_t a[4] = {r.x, r.y, r.z, r.w};
        __syncwarp();
        transpose8(a);
#pragma unroll
        for (int j = 0; j < 4; ++j) planes[4 * j + q] = a[j];
        __syncwarp();
      };
      auto planes16 = [&](const uint32_t* w) {
        const uint32_t put = smem_addr(area + 36 * bq);
#pragma unroll
        for (int k = 0; k < 16; ++k)
          asm volatile("st.shared.u16 [%0], %1;" ::"r"(__dp4a(place[k >> 2], 2u << (8 * (k & 3)), put)),
                       "h"((uint16_t)w[k])
                       : "memory");
        __syncwarp();
        uint32_t a[8];
        const uint4* get = reinterpret_cast<const uint4*>(area + 36 * bq + 8 * q);
#pragma unroll
        for (int k = 0; k < 2; ++k) {  // ranks 2k, 2k + 4, 2k + 1, 2k + 5, each with the one 8 above it
          const uint4 r = get[k];
          a[2 * k] = r.x;
          a[2 * k + 4] = r.y;
          a[2 * k + 1] = r.z;
          a[2 * k + 5] = r.w;
        }
        __syncwarp();
        transpose16(a);
#pragma unroll
        for (int j = 0; j < 8; ++j) planes[4 * j + q] = a[j];
        __syncwarp();
      };
      // 32 planes: the digits of 16 ranks, then (half 0: planes p + j) their words
      auto ranks32 = [&](const uint32_t* w, uint32_t (&a)[16]) {
        const uint32_t put = smem_addr(area + 72 * bq);
#pragma unroll
        for (int k = 0; k < 16; ++k)
          asm volatile("st.shared.u32 [%0], %1;" ::"r"(__dp4a(place[k >> 2], 4u << (8 * (k & 3)), put)), "r"(w[k])
                       : "memory");
        __syncwarp();
        const uint4* get = reinterpret_cast<const uint4*>(area + 72 * bq + 16 * q);
#pragma unroll
        for (int k = 0; k < 4; ++k) {  // ranks k, k + 8, k + 4, k + 12
          const uint4 r = get[k];
          a[k] = r.x;
          a[k + 8] = r.y;
          a[k + 4] = r.z;
          a[k + 12] = r.w;
        }
        __syncwarp();
      };
      auto words32 = [&](uint32_t (&a)[16], int half) {
        transpose32_lane(a);
#pragma unroll
        for (int j = 0; j < 16; ++j) planes[64 * half + 4 * j + q] = a[j];
      };
      auto planes32 = [&](const uint32_t* w) {
        uint32_t a[16];
        ranks32(w, a);
        words32(a, 0);
        __syncwarp();
      };

      // the plane words of at most 32 planes; returns how many words hold planes
      auto planes_of = [&](const uint32_t* w) {
        if (span <= 8) {
          planes8(w);
          return 4;
        }
        if (span <= 16) {
          planes16(w);
          return 8;
        }
        planes32(w);
        return 16;
      };

      // R13: decode-back x_i = D(y_i), the candidate x~ + x_i and the residual
      // it leaves.  Bricks that are not coded decode to 0, which leaves x~ and
      // the residual as they are.
      T xtn[16], en[16];
      int H;  // plane p + j is in half (j / H) & 1 of word j mod H
      if constexpr (!WIDE) {
        {
          S r[16];
          const U keep = __funnelshift_lc(0u, ~0u, p);  // planes p and up
#pragma unroll
          for (int k = 0; k < 16; ++k) r[k] = nb_inv<T>((U)v[k] & keep);
          lift_inv_bricks<S>(r, zw, yw, SET);
          if (common) {
            // int -> float rounds once; the product by 2^-s is exact (normal, and
            // below 2^127 for s >= -96), so one fused add is x~ + x_i
            const float sc = __uint_as_float((uint32_t)(127 - s) << 23);
#pragma unroll
            for (int k = 0; k < 16; ++k) xtn[k] = __fmaf_rn(__int2float_rn(r[k]), sc, xt[k]);
          } else {
#pragma unroll
            for (int k = 0; k < 16; ++k) xtn[k] = F::add(xt[k], F::val(dequantize_any<T>(r[k], s)));
          }
        }
        residual_of(xtn, en);
        uint32_t w[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) w[k] = digits(k);
        H = planes_of(w);
      } else {
        // Digits within 20 planes from plane p in 32..57 on: decoded in 32-bit
        // integers in units of 2^(p - 6).  A coefficient with negabinary digits d
        // from plane p is ((d ^ M) - M) * 2^p with M = NBM >> p (M's bits above
        // d's do not matter).  In these units each inverse lifting pass turns
        // multiples of 2^a into multiples of 2^(a - 2), so from 2^6 on every
        // shift divides an even number exactly; |value| < 2^(19 + 6.42) * 2.75^3
        // < 2^30 (2.75: the largest row sum of the inverse lifting's
        // coefficients).  The 64-bit form does not wrap either: without the
        // truncation its values are the forward transform's, below 2^62, and the
        // truncation moves them by less than 2.75^3 * 2^p < 2^62.  So the result
        // is the 64-bit decoding's exactly, in half the instructions.
        const bool narrow = common && __all_sync(FULL, !coded || (nw <= 20 && p >= 32 && p <= 57));
        auto add = [&](int k, T xi) {  // x~ + x_i; the first component's +0 + x_i is x_i with -0 turned to +0
          if (i == 0)
            xtn[k] = F::val(F::bits(xi) == F::SIGN ? U(0) : F::bits(xi));
          else
            xtn[k] = F::add(xt[k], xi);
        };
        if (narrow) {
          uint32_t w[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) w[k] = digits(k);
          // Within 13 planes the same in float, in units of 2^p: d and M's 13 bits
          // with 2^23's bit pattern in front are floats whose difference is the
          // coefficient, and values below 2^(13 + 4.4) that are multiples of
          // 2^-6 need 24 bits.  8 operations a line instead of 11, off the ALU
          // pipe, and a shorter conversion: 256 x 384 x 384, 12 components, 3.35
          // -> 3.22 ms.  (Float32, whose conversion is one instruction, became 3 %
          // slower with both forms in the kernel and keeps the integers.)
          if (span <= 13) {
            float r[16];
            const uint32_t M = ((uint32_t)(F::NBM >> min(p, 63)) & 0x1fffu) | 0x4B000000u;
#pragma unroll
            for (int k = 0; k < 16; ++k) r[k] = __fsub_rn(__uint_as_float(w[k] ^ M), __uint_as_float(M));
            lift_inv_bricks<float>(r, zw, yw, SET);
            const uint32_t adj = (uint32_t)(896 + p - s) << 20;
#pragma unroll
            for (int k = 0; k < 16; ++k) add(k, scaled_f32_to_f64(r[k], adj));
          } else {
            int32_t r[16];
            const uint32_t M = (uint32_t)(F::NBM >> min(p, 63)), M64 = M << 6;
#pragma unroll
            for (int k = 0; k < 16; ++k) r[k] = (int32_t)(((w[k] ^ M) << 6) - M64);
            lift_inv_bricks<int32_t>(r, zw, yw, SET);
            const uint32_t eb = (uint32_t)(1053 + (p - 6) - s) << 20;
#pragma unroll
            for (int k = 0; k < 16; ++k) add(k, scaled_i32_to_f64(r[k], eb));
          }
          residual_of(xtn, en);
          H = planes_of(w);
        } else {
          S r[16];
          const U keep = p >= 64 ? U(0) : ~U(0) << p;  // planes p and up
#pragma unroll
          for (int k = 0; k < 16; ++k) r[k] = nb_inv<T>((U)v[k] & keep);
          lift_inv_bricks<S>(r, zw, yw, SET);
#pragma unroll
          for (int k = 0; k < 16; ++k)
            add(k, F::val(common ? dequantize_f64_normal(r[k], s) : dequantize_any<T>(r[k], s)));
          residual_of(xtn, en);
          H = 16;
          uint32_t w[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) w[k] = (uint32_t)digits64(k);
          if (span <= 32) {
            planes32(w);
          } else {  // both halves' digits are read before the words take their place
            uint32_t a0[16], a1[16];
            ranks32(w, a0);
#pragma unroll
            for (int k = 0; k < 16; ++k) w[k] = (uint32_t)(digits64(k) >> 32);
            ranks32(w, a1);
            words32(a0, 0);
            words32(a1, 1);
            __syncwarp();
          }
        }
      }
      const U mn = brick_max<T>(en);
      const bool pass = !zero_blk && coded && mn <= tb;
      const bool again = coded && !pass && p > 0 && esc < 7;
      if (__any_sync(FULL, again)) {  // rare: code the warp's bricks again from the same residual
        if (again) ++esc;
        residual_of(xt, e);
        continue;
      }

      // R11, lengths: the planes above `top` are one 0 test bit each; then 4
      // planes at a time, one per lane of the brick: the significance count n
      // before a plane is the largest one-past-highest position over the planes
      // above it, and the planes' offsets are a running sum of their lengths.
      const int nrow = (span + 3) >> 2;
      int lenC = HDR + F::P - max(top + 1, p);
      {
        int carry = 0;
        for (int k = 0; k < nrow; ++k) {
          const int j = nw - 1 - 4 * k - q;  // plane p + j
          uint32_t lo, hi;
          plane_at<WIDE>(planes, j, H, &lo, &hi);
          int n = (int)(31 - __clz((int)(hi ? hi : lo))) + 1 + (hi ? 32 : 0);  // one past the highest position
          int t = __shfl_up_sync(FULL, n, 1, 4);
          if (q >= 1) n = max(n, t);
          t = __shfl_up_sync(FULL, n, 2, 4);
          if (q >= 2) n = max(n, t);
          const int after = max(n, carry);  // significant after the plane
          t = __shfl_up_sync(FULL, after, 1, 4);
          n = q ? t : carry;  // and before it
          carry = __shfl_sync(FULL, after, 3, 4);
          // n verbatim bits, the positions and 1s from n on, the closing 0
          uint32_t mlo, mhi;
          low_mask(n, &mlo, &mhi);
          int len = after + __popc(lo & ~mlo) + __popc(hi & ~mhi) + (after < 64 ? 1 : 0);
          if (j < 0) len = 0;
          int sum = len;
          t = __shfl_up_sync(FULL, sum, 1, 4);
          if (q >= 1) sum += t;
          t = __shfl_up_sync(FULL, sum, 2, 4);
          if (q >= 2) sum += t;
          if (PCZ_CHECK(4 * k + q < A3::kInfoStride, 1)) info[4 * k + q] = (uint32_t)(lenC + sum - len) << 8 | (uint32_t)n;
          lenC += __shfl_sync(FULL, sum, 3, 4);
        }
      }

      // R14: RAW replaces a longer CODED brick only if it also meets tau_i
      int mode = zero_blk ? kModeZero : pass ? kModeCoded : kModeRaw;
      int viol = 0;  // Eq. 1 failures left (only a RAW brick can have them)
      U mnew = mn;
      if (__any_sync(FULL, mode == kModeRaw || (pass && lenC > LEN_RAW))) {
        T a[16], xr[16], er[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) a[k] = xt[k];
        const U mr = raw_form<T>(s_x + tid, any_partial, nvx, nvy, nvz, lane, a, xr, er);
        if (pass && lenC > LEN_RAW && mr <= tb) mode = kModeRaw;
        if (mode == kModeRaw) {
          S* raw = reinterpret_cast<S*>(planes);  // the residual, for the bit writes
          mnew = mr;
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            raw[16 * q + k] = (S)F::bits(a[k]);
            xtn[k] = xr[k];
            en[k] = er[k];
            if ((k & 3) < nvx && (k >> 2) < nvy && q < nvz && magnitude(er[k]) > tb) ++viol;
          }
        }
        viol += __shfl_xor_sync(FULL, viol, 1);
        viol += __shfl_xor_sync(FULL, viol, 2);
      }
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        xt[k] = xtn[k];
        e[k] = en[k];
      }
      m = mnew;
      const int blen = !have ? 0 : mode == kModeZero ? 2 : mode == kModeRaw ? LEN_RAW : lenC;
      if (q == 0) {
        s_len[slot] = blen;
        s_mode[slot] = have ? mode : -1;
        s_esc[slot] = mode == kModeCoded ? esc : 0;
        s_viol[slot] = have ? viol : 0;
        s_merr[slot] = have ? (uint64_t)mnew : 0ull;
      }
      group_sync(bar_id);  // (the previous component's chunk is appended)

      // chunk layout: every warp scans the 32 brick lengths
      const int l0 = s_len[lane];
      int incl = l0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += t;
      }
      const int total = __shfl_sync(FULL, incl, 31);
      const uint32_t boff = (uint32_t)__shfl_sync(FULL, incl - l0, slot);
      // bookkeeping, spread over the warps: warp 0 sizes the chunk and
      // reserves its pool space (the atomic's result is needed after the bit
      // writes), warp 1 gathers the block counters, warp 2 writes the index
      unsigned long long pool_base = 0;
      const unsigned cw = (unsigned)((total + 63) >> 6);
      if (tid == 0) {
        *s_cbits = total;
        pool_base = cw ? atomicAdd(P.pool_used, (unsigned long long)cw) : 0ull;
        P.chunk_nwords[(int64_t)i * P.nchunks + chunk] = cw;
      }
      if (warp == 1) {
        const int md = s_mode[lane];
        const unsigned cz = __popc(__ballot_sync(FULL, md == kModeZero));
        const unsigned cc = __popc(__ballot_sync(FULL, md == kModeCoded));
        const unsigned cr = __popc(__ballot_sync(FULL, md == kModeRaw));
        const unsigned se = __reduce_add_sync(FULL, (unsigned)s_esc[lane]);
        const unsigned sv = __reduce_add_sync(FULL, (unsigned)s_viol[lane]);
        const unsigned long long me = warp_max_u64(FULL, s_merr[lane]);
        if (lane == 0) {
          const int64_t ci = (int64_t)i * P.nchunks + chunk;
          uint32_t* cnt = P.chunk_counts + ci * 5;
          cnt[0] = cz;
          cnt[1] = cc;
          cnt[2] = cr;
          cnt[3] = se;
          cnt[4] = sv;
          if (P.chunk_maxerr) P.chunk_maxerr[ci] = me;
        }
      }
      if (warp == 2 && chunk * kChunk + lane < P.nbricks) {
        const int64_t at = (int64_t)i * P.nbricks + chunk * kChunk + lane;
        P.brick_len[at] = (uint16_t)l0;
        if (P.brick_off) P.brick_off[at] = (uint32_t)(incl - l0);
      }

      // the bits of the warp's bricks, into the chunk buffer
      if (have && mode == kModeRaw) {
        if (q == 0) or_bits_in(cbuf, boff, (uint64_t)kModeRaw, CAP, 0);
        const U* raw = reinterpret_cast<const U*>(planes) + 16 * q;
        for (int k = 0; k < 16; ++k)
          or_bits_in(cbuf, boff + 2 + (uint32_t)(F::P * (16 * q + k)), (uint64_t)raw[k], CAP, 0);
      }
      const bool emit = have && mode == kModeCoded;
      if (emit && q == 0)
        or_bits_in(cbuf, boff, (uint64_t)kModeCoded | ((uint64_t)esc << 2) | ((uint64_t)(emax + F::EBIAS) << 5), CAP, 0);
      // R11: each plane by a lane: its n verbatim bits and, if a coefficient
      // turns significant, the first test bit; then the group-test code, 16
      // coefficients at a time through the byte table.  The code of the last 16
      // drops the test 1 after the plane's last 1; zeros need no write.
      for (int k = 0; k < nrow; ++k) {
        const int j = nw - 1 - 4 * k - q;
        if (!emit || j < 0) continue;
        uint32_t lo, hi, mlo, mhi;
        plane_at<WIDE>(planes, j, H, &lo, &hi);
        if (!(lo | hi)) continue;
        const uint32_t nf = info[4 * k + q];
        const int n = (int)(nf & 0xffu);
        const uint32_t at = boff + (nf >> 8);
        low_mask(n, &mlo, &mhi);
        const uint32_t rlo = lo & ~mlo, rhi = hi & ~mhi;  // from position n on
        lo &= mlo;
        hi &= mhi;
        if (rlo | rhi) {  // the first test 1, at position n < 64
          lo |= mlo + 1u;  // bit n below 32: the mask's end (0 when the mask is full)
          hi |= mlo == ~0u ? mhi + 1u : 0u;
        }
        if (PCZ_CHECK(at + (hi ? 64u - (uint32_t)__clz((int)hi) : 32u - (uint32_t)__clz((int)lo)) <= CAP, 0))
          or_words(cbuf, at, lo, hi);
        uint64_t rest = n < 64 ? (((uint64_t)rhi << 32) | rlo) >> n : 0ull;
        uint32_t pos = at + (uint32_t)n + 1u;
        while (rest) {
          const uint32_t b0 = (uint32_t)rest & 0xffu, b1 = ((uint32_t)rest >> 8) & 0xffu;
          const uint32_t l0c = 8u + (uint32_t)__popc(b0);
          uint32_t code = s_spread[b0] | ((uint32_t)s_spread[b1] << l0c);
          rest >>= 16;
          if (!rest) code ^= 0x80000000u >> __clz((int)code);
          const uint32_t sh = pos & 31u, w0 = pos >> 5;
          const uint32_t clo = code << sh, chi = __funnelshift_l(code, 0u, sh);
          if (PCZ_CHECK(pos + 32u - (uint32_t)__clz((int)(code | 1u)) <= CAP, 0)) {
            if (clo) atomicOr(cbuf + w0, clo);
            if (chi) atomicOr(cbuf + w0 + 1, chi);
          }
          pos += l0c + 8u + (uint32_t)__popc(b1);
        }
      }
      if (tid == 0) {
        if (pool_base + cw > P.pool_words) {
          atomicOr(P.flags, kFlagPoolOverflow);
          pool_base = ~0ull;
        }
        *s_base = pool_base;
        P.chunk_pool[(int64_t)i * P.nchunks + chunk] = pool_base;
      }
      group_sync(bar_id);  // the chunk is complete, and its pool place known
      append_chunk(P, cbuf, *s_base, *s_cbits, tid);
      break;
    }
  }
}

}  // namespace pcz
