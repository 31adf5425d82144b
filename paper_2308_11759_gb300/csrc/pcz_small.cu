// pcz_small.cu -- Algorithms 1 and 2 (Magri & Lindstrom, Sec. 4.1, 4.2) for
// 1D and 2D fields, whose bricks hold 4 and 16 values.
//
// A brick this small fits one thread: each thread codes one brick entirely
// in registers (residual, alignment, lifting along x then y, sequency order,
// negabinary, bit planes from the top down, decode-back and verification),
// and one warp covers one index chunk of 32 bricks, so the bricks' bit
// offsets in the chunk come from a warp scan.  Each lane's code is formed in its
// own column of shared memory, shifted into the warp's chunk buffer and appended
// to the scratch pool like the 3D kernel's chunks; retrieval mirrors this with
// one thread per brick and component parsing and rebuilding a brick.
#include "pcz_chunk_small.cuh"

namespace pcz {

// CTAs of 4 warps that share an SM, measured on 2D fields (4096^2 float32, 4096 x
// 3000 float64, 6 components).  Construction: float32 5 (349 us; 4: 376, 6: 387),
// float64 3 (613; 2: 709, 4: 640).  Retrieval: float32 8 (284 us; 6 and 5
// 5 and 14 % slower), float64 5 (330; 4 6 % slower).
template <typename T>
constexpr int kCompressCtas = sizeof(T) == 4 ? 5 : 3;
template <typename T>
constexpr int kRetrieveCtas = sizeof(T) == 4 ? 8 : 5;

template <typename T, int D>
__global__ void __launch_bounds__(kSmallThreads, kCompressCtas<T>) k_compress_small(const CompressParams P) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5;
  uint32_t* area = reinterpret_cast<uint32_t*>(smem) + (size_t)warp * SmallArea<T, D>::kWords;
  const uint16_t* spread = load_spread<kSmallThreads>(smem + small_smem<T, D>(kSmallWarps) - kSpreadBytes);
  __syncthreads();
  const int64_t chunk = (int64_t)blockIdx.x * kSmallWarps + warp;
  if (chunk < P.nchunks) compress_small_chunk<T, D>(P, chunk, area, spread);
}

// One thread per brick: of the single job, or of a job list whose units are
// bricks (unit_begin = the job's first brick among all jobs' bricks).
template <typename T, int D>
__global__ void __launch_bounds__(kSmallThreads, kRetrieveCtas<T>) k_retrieve_small(const RetrieveParams R) {
  // The table lands while the threads of a 1D field look up their first blocks (with
  // a copy and a barrier before that, 100 float32 values took 8.3 us at k = 1, now 6.9;
  // 8 million ZERO ones 29.9, now 28.5).  Threads past the end stop at the barrier.
  __shared__ __align__(16) uint32_t tokens[kTokLut];
  static_assert(sizeof(tokens) == 16 * kSmallThreads, "16 bytes per thread");
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_addr(tokens + 4 * threadIdx.x)),
               "l"(__cvta_generic_to_global(kTokens.entry + 4 * threadIdx.x))
               : "memory");
  const int64_t at = (int64_t)blockIdx.x * kSmallThreads + threadIdx.x;
  const int64_t g = min(at, R.nunits - 1);
  auto ready = [&] {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    return at == g;
  };
  if (!R.jobs) {
    retrieve_small_brick<T, D>(R.job0, R.write, R.err, g, tokens, ready);
    return;
  }
  int lo = 0, hi = R.njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (R.jobs[mid].unit_begin <= g)
      lo = mid;
    else
      hi = mid - 1;
  }
  const BoxJob& J = R.jobs[lo];
  retrieve_small_brick<T, D>(J, R.write, R.err, g - J.unit_begin, tokens, ready);
}

template <typename T, int D>
static cudaError_t launch_compress_small_t(const CompressParams& p, cudaStream_t s) {
  const size_t smem = small_smem<T, D>(kSmallWarps);
  cudaError_t e = cudaFuncSetAttribute(k_compress_small<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if (p.nchunks == 0) return cudaSuccess;
  k_compress_small<T, D><<<(unsigned)((p.nchunks + kSmallWarps - 1) / kSmallWarps), kSmallThreads, smem, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_compress_small(int dtype, int ndims, const CompressParams& p, cudaStream_t s) {
  if (ndims == 1) return dtype == 1 ? launch_compress_small_t<float, 1>(p, s) : launch_compress_small_t<double, 1>(p, s);
  return dtype == 1 ? launch_compress_small_t<float, 2>(p, s) : launch_compress_small_t<double, 2>(p, s);
}

template <typename T, int D>
static cudaError_t launch_retrieve_small_t(const RetrieveParams& p, cudaStream_t s) {
  const int64_t work = p.jobs ? p.nunits : p.job0.nbox;
  if (work == 0) return cudaSuccess;
  k_retrieve_small<T, D><<<(unsigned)((work + kSmallThreads - 1) / kSmallThreads), kSmallThreads, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_retrieve_small(int dtype, int ndims, const RetrieveParams& p, cudaStream_t s) {
  if (ndims == 1) return dtype == 1 ? launch_retrieve_small_t<float, 1>(p, s) : launch_retrieve_small_t<double, 1>(p, s);
  return dtype == 1 ? launch_retrieve_small_t<float, 2>(p, s) : launch_retrieve_small_t<double, 2>(p, s);
}

uint32_t check_word_small(int reset) { return read_check_word(reset); }

}  // namespace pcz
