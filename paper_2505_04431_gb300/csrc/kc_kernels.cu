// kc_kernels.cu - the k-mer counting hot path on sm_103a.
//
// k_prepare                 clears the sketch, the histogram's totals and the status record,
//                           and finds the first read of every phase-1 tile.
// Phase 1 (Section III-C, Algorithm 3 first loop; Section V "Phase 1"):
//   pass A  k_pack_count    ASCII -> 2-bit codes + invalid mask (the paper's Encode),
//                           rolling forward / reverse-complement keys (Algorithm 1's
//                           kmer = (kmer << 2) OR Encode), owner partition of every
//                           valid window, per-tile partition histogram.  Its last block
//                           scans the totals to partition starts; a tile of pass B then
//                           reserves its run in each partition with one atomic add on that
//                           partition's cursor.
//   pass B  k_scatter       recomputes the keys from the packed codes and writes each
//                           key to its owner partition.  A tile's keys are first
//                           grouped per partition in shared memory (a counting sort)
//                           and leave in contiguous runs: this block-level staging is
//                           the GPU form of the per-destination L2 buffers of
//                           Section IV-C / Algorithm 4 (AddToL2Buffer), which exist to
//                           turn many small sends into few large ones.
// Phase 2 (Algorithm 3 after the barrier: Sort + Accumulate; Section V "Phase 2"):
//   k_fine_plan, k_fine_hist, k_fine_scan, k_fine_scatter   split every owner partition
//                           into fine partitions small enough for one shared-memory table
//                           (sized from a HyperLogLog estimate of the distinct keys).
//   k_count_emit            persistent; per fine partition: count every key in a hashed
//                           open-addressing table in shared memory (CAS claims a slot, a
//                           32-bit atomic add counts), order the occupied slots by a
//                           bucketed counting sort over the partition's key range, and
//                           write the sorted (key, count) run at the offset found by a
//                           decoupled look-back over the fine partitions, or in its own
//                           input region when that offset is not known in time.
//   k_scan_distinct, k_compact   output offsets of all runs; the runs written in place
//                           move to their offsets.
// Pass A also checks the read offsets; where they do not ascend from 0 to the base count, it
// records that, plans no partition, and the later kernels of the count find nothing to do.
// One level (small inputs, and larger ones whose repeats leave few fine partitions): pass A
// counts the windows of 2^10 .. 2^13 bins instead of the coarse partitions' and fills the
// sketch; its last block groups the bins into fine partitions, pass B writes these, and the
// fine split is left out.  k_finish_one then does k_scan_distinct's and k_compact's work.
// Variants: every kernel body also runs as a batched kernel (one launch for a group of
// counts, each thread block working for one count found through a block table); pass B
// without the shared-memory staging (DIRECT) and the count kernel with a warp-level merge
// of equal keys (the heavy-hitter pre-aggregation of Section IV-D; slower on GB300, so off
// by default) exist for the aggregation experiment of Section VI.
//
// Owner partitions are key ranges (not hashes) so that the per-partition outputs
// concatenate into one ascending array.  A monotone map u(key) of the top 32 key bits
// flattens the distribution of canonical keys (the min of two near-independent uniforms
// has density 2(1-x); u = 1 - (1-x)^2 is its distribution function); the coarse partition
// is the top bits of u and the fine partitions split each coarse range of u into equal
// parts, so both are non-decreasing in the key.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "kc_internal.h"

namespace kc {

typedef unsigned __int128 u128;

// The kernels of a single count are launched so that each may be set up while the one before it
// still runs (programmatic dependent launch); a kernel first waits for that one's end and its
// writes.  When it came in, a count of 21 M bases, then 10 launches 2 us apart, went from 547 to
// 533 us, one of 90 M from 1942 to 1913.  Letting the next kernel's blocks onto the SMs early,
// before the last one's have ended, cost more than it gave (50.9 -> 52.4 ms at 3 G bases), and
// so did this form for the batched launches (32 small samples 932 -> 951 us), which stay as they are.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P, class... A>
static void pdl_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Batched launches: each block finds its count (one table load), copies the count's
// descriptor to shared memory and runs the kernel body for that count.
__device__ __forceinline__ void batch_locate(const BatchTab& t, BatchDesc& d_s, uint32_t& bid_s, uint32_t& nblk_s) {
  __shared__ uint32_t i_s;
  const uint32_t tid = threadIdx.x + threadIdx.y * blockDim.x, nth = blockDim.x * blockDim.y;
  if (tid == 0) {
    const uint32_t i = t.blk2s[blockIdx.x];
    const uint32_t a = t.start[i];
    i_s = i;
    bid_s = blockIdx.x - a;
    nblk_s = t.start[i + 1] - a;
  }
  __syncthreads();
  const uint32_t* src = reinterpret_cast<const uint32_t*>(t.desc + i_s);
  uint32_t* dst = reinterpret_cast<uint32_t*>(&d_s);
  for (uint32_t w = tid; w < sizeof(BatchDesc) / 4; w += nth) dst[w] = src[w];
  __syncthreads();
}
#define KC_BATCH_PROLOGUE(t)                 \
  __shared__ BatchDesc d_s_;                 \
  __shared__ uint32_t bid_s_, nblk_s_;       \
  batch_locate(t, d_s_, bid_s_, nblk_s_);    \
  const BatchDesc& d = d_s_;                 \
  const uint32_t bid = bid_s_, nblk = nblk_s_; \
  (void)bid;                                 \
  (void)nblk

template <int KW> struct KeyT;
template <> struct KeyT<1> { typedef uint64_t T; };
template <> struct KeyT<2> { typedef u128 T; };

// ------------------------------------------------------------------ bit helpers
__device__ __forceinline__ uint64_t revpairs64(uint64_t x) {
  x = __brevll(x);
  return ((x >> 1) & 0x5555555555555555ull) | ((x & 0x5555555555555555ull) << 1);
}
__device__ __forceinline__ uint64_t key_mask(uint64_t, int k) { return k >= 32 ? ~0ull : ((1ull << (2 * k)) - 1); }
__device__ __forceinline__ u128 key_mask(u128, int k) { return k >= 64 ? ~(u128)0 : (((u128)1 << (2 * k)) - 1); }
// value of the reverse complement of the k-mer v (digit d -> 3 - d, digit order reversed)
__device__ __forceinline__ uint64_t revcomp(uint64_t v, int k) { return revpairs64(~v) >> (64 - 2 * k); }
__device__ __forceinline__ u128 revcomp(u128 v, int k) {
  u128 r = ((u128)revpairs64(~(uint64_t)v) << 64) | revpairs64(~(uint64_t)(v >> 64));
  return r >> (128 - 2 * k);
}
template <class K> __device__ __forceinline__ K all_ones() { return ~(K)0; }

__device__ __forceinline__ uint64_t shfl_key(uint64_t v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ u128 shfl_key(u128 v, int src) {
  uint64_t lo = __shfl_sync(0xffffffffu, (uint64_t)v, src);
  uint64_t hi = __shfl_sync(0xffffffffu, (uint64_t)(v >> 64), src);
  return ((u128)hi << 64) | lo;
}

// Asynchronous 4-, 8- and 16-byte copies from global to shared memory (cp.async); the issuing
// thread waits for all of its copies with cp_async_wait_all.
__device__ __forceinline__ void cp_async4(void* dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Look-back status words carry their own payload (flag and value in one 64-bit word) and
// guard no other data, so relaxed GPU-scope accesses are enough.
__device__ __forceinline__ void st_status(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_status(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ u128 cas128_shared(u128* p, u128 cmp, u128 val) {
  uint64_t clo = (uint64_t)cmp, chi = (uint64_t)(cmp >> 64), vlo = (uint64_t)val, vhi = (uint64_t)(val >> 64), olo, ohi;
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile(
      "{\n\t.reg .b128 d, c, v;\n\tmov.b128 c, {%2, %3};\n\tmov.b128 v, {%4, %5};\n\t"
      "atom.shared.cas.b128 d, [%6], c, v;\n\tmov.b128 {%0, %1}, d;\n\t}"
      : "=l"(olo), "=l"(ohi)
      : "l"(clo), "l"(chi), "l"(vlo), "l"(vhi), "r"(a)
      : "memory");
  return ((u128)ohi << 64) | olo;
}

__device__ __forceinline__ void store_key(uint64_t* dst, uint64_t i, uint64_t key) { dst[i] = key; }
__device__ __forceinline__ void store_key(uint64_t* dst, uint64_t i, u128 key) {
  reinterpret_cast<ulonglong2*>(dst)[i] = make_ulonglong2((uint64_t)key, (uint64_t)(key >> 64));
}
__device__ __forceinline__ void load_key(const uint64_t* src, uint64_t i, uint64_t& key) { key = src[i]; }
__device__ __forceinline__ void load_key(const uint64_t* src, uint64_t i, u128& key) {
  const ulonglong2 v = reinterpret_cast<const ulonglong2*>(src)[i];
  key = ((u128)v.y << 64) | v.x;
}

// Block-wide exclusive scan of n values in shared memory (in place); returns the total.
// All threads of the block must call it.  `warp_tmp` holds 32 entries.
template <typename T>
__device__ T block_exclusive_scan(T* data, int n, T* warp_tmp) {
  const int nt = blockDim.x, t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = (nt + 31) >> 5;
  const int per = (n + nt - 1) / nt;
  const int lo = min(n, t * per), hi = min(n, lo + per);
  T s = 0;
  for (int i = lo; i < hi; ++i) s += data[i];
  T x = s;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_tmp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    T w = lane < nw ? warp_tmp[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    if (lane < nw) warp_tmp[lane] = w;  // inclusive per warp
  }
  __syncthreads();
  T run = x - s + (wid ? warp_tmp[wid - 1] : 0);
  const T total = warp_tmp[nw - 1];
  for (int i = lo; i < hi; ++i) {
    T v = data[i];
    data[i] = run;
    run += v;
  }
  __syncthreads();
  return total;
}

// Shared arrays that are scanned by contiguous per-thread chunks are padded (one word per
// 32) so that those chunks fall in distinct banks.
__host__ __device__ __forceinline__ uint32_t PAD(uint32_t i) { return i + (i >> 5); }
__host__ __device__ __forceinline__ size_t padded_len(size_t n) { return n + (n >> 5) + 1; }

// block_exclusive_scan over a padded array (logical element i at data[PAD(i)]).
template <typename T>
__device__ T block_exclusive_scan_pad(T* data, int n, T* warp_tmp) {
  const int nt = blockDim.x, t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = (nt + 31) >> 5;
  const int per = (n + nt - 1) / nt;
  const int lo = min(n, t * per), hi = min(n, lo + per);
  T s = 0;
  for (int i = lo; i < hi; ++i) s += data[PAD(i)];
  T x = s;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_tmp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    T w = lane < nw ? warp_tmp[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    if (lane < nw) warp_tmp[lane] = w;
  }
  __syncthreads();
  T run = x - s + (wid ? warp_tmp[wid - 1] : 0);
  const T total = warp_tmp[nw - 1];
  for (int i = lo; i < hi; ++i) {
    T v = data[PAD(i)];
    data[PAD(i)] = run;
    run += v;
  }
  __syncthreads();
  return total;
}

// The last block of a launch (of a count's blocks, in a batched launch) to get here returns
// true, with every other block's writes visible to L2 reads; all threads call it.
__device__ __forceinline__ bool last_block(uint32_t* done, uint32_t nblk) {
  __shared__ uint32_t last_s;
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last_s = atomicAdd(done, 1u) == nblk - 1;
    __threadfence();
  }
  __syncthreads();
  return last_s != 0;
}

// ------------------------------------------------------------------ prepare
// What a count needs cleared (status record, fine histogram, look-back words, sketch,
// partition counts), and the first read whose start is >= the halo start of each tile (lower
// bound in offsets): one launch where there were five clears and a kernel.
__device__ __forceinline__ void prepare_body(const Shape& s, const Buffers& b, uint32_t bid, uint32_t nblk) {
  const uint64_t i0 = (uint64_t)bid * blockDim.x + threadIdx.x, stride = (uint64_t)nblk * blockDim.x;
  for (uint64_t i = i0; i < s.nf_max; i += stride) {
    b.fhist[i] = 0;
    b.look[i] = 0;
  }
  for (uint64_t i = i0; i < (uint64_t)kHllRegs; i += stride) b.hll[i] = 0;
  if (s.one_level) {
    for (uint64_t i = i0; i < (1ull << s.bb); i += stride) b.bins[i] = 0;
  } else {
    for (uint64_t i = i0; i <= (1ull << s.b1); i += stride) b.cstart[i] = 0;
  }
  for (uint64_t i = i0; i < sizeof(Meta) / 4; i += stride) reinterpret_cast<uint32_t*>(b.meta)[i] = 0;
  // a warp per tile, 32 offsets compared at a time: 4 round trips for 1 M reads, not 20
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t t = i0 >> 5; t < s.n_tiles; t += stride >> 5) {
    const uint64_t pos = t * s.tile_words * kWordBases;
    const uint64_t halo = pos >= 64 ? pos - 64 : 0;
    uint64_t lo = 0, hi = s.n_reads;
    while (lo < hi) {
      const uint64_t len = hi - lo, p = len <= 32 ? lo + lane : lo + len / 33 * (lane + 1);
      const uint32_t below = __popc(__ballot_sync(0xffffffffu, p < hi && b.offsets[p] < halo));
      const uint64_t step = len <= 32 ? 1 : len / 33;
      const uint64_t first = len <= 32 ? lo : lo + step;  // lane 0's position
      if (len <= 32) {
        lo = hi = lo + below;
      } else {
        if (below < 32) hi = first + step * below;
        if (below > 0) lo = first + step * (below - 1) + 1;
      }
    }
    if (lane == 0) {
      b.tile_first[t] = lo;
      if (s.one_level == kEitherLevel) b.tile_first2[t] = lo;
    }
  }
}
__global__ void __launch_bounds__(256) k_prepare(Shape s, Buffers b) { pdl_wait(); prepare_body(s, b, blockIdx.x, gridDim.x); }
__global__ void __launch_bounds__(256) k_prepare_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  prepare_body(d.s, d.b, bid, nblk);
}

// Offsets start at 0, do not decrease and end at L: a share for each block of pass A, which by
// itself stays in bounds whatever they hold.  Passes A and B mark the read starts of sub-steps
// of different lengths with a cursor that only ascending offsets move alike, so with others
// pass B would find windows that pass A has not counted and that no partition has room for:
// pass A's last block then plans nothing, and no later kernel works on such a count.
__device__ __forceinline__ void check_offsets(const Shape& s, const Buffers& b, uint32_t bid, uint32_t nblk) {
  const uint64_t share = (s.n_reads + nblk - 1) / nblk, lo = min(s.n_reads, bid * share), hi = min(s.n_reads, lo + share);
  bool bad = false;
  for (uint64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) bad |= b.offsets[i + 1] < b.offsets[i];
  if (bid == 0 && threadIdx.x == 0) bad |= b.offsets[0] != 0 || b.offsets[s.n_reads] != s.L;
  if (bad) atomicOr(&b.meta->status, ST_BAD_OFFSETS);
}
// Set by pass A only, so the same for every thread of a later kernel.
__device__ __forceinline__ bool bad_offsets(const Buffers& b) { return (__ldcg(&b.meta->status) & ST_BAD_OFFSETS) != 0; }

// ------------------------------------------------------------------ phase 1 helpers
// ASCII -> codes for 32 bytes given as 8 little-endian words.  The 2-bit codes of a word's four
// bytes are gathered by one multiplication (their products fall on bits of their own), and a
// byte is a base iff it is, in lower case, the letter of its code (looked up for four bytes by
// one byte permutation): a third of the instructions of comparing each byte with each letter.
// The bytes that are not are picked out only in words that have one.
__device__ __forceinline__ void pack32(const uint32_t w[8], uint64_t& code, uint32_t& inv) {
  uint32_t p[8], any = 0;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    const uint32_t x = w[m];
    const uint32_t c4 = ((x >> 1) ^ (x >> 2)) & 0x03030303u;  // A0 C1 G2 T3 (either case), one per byte
    p[m] = c4 * 0x40100401u;                                   // the four codes in the top byte, first base on top
    const uint32_t n4 = c4 | (c4 >> 4);                        // two selectors in bytes 0 and 2
    const uint32_t letters = __byte_perm(0x74676361u, 0, __byte_perm(n4, 0, 0x4420));  // "acgt"
    any |= letters ^ (x | 0x20202020u);
  }
  const uint32_t hi = __byte_perm(__byte_perm(p[3], p[2], 0x0073), __byte_perm(p[1], p[0], 0x0073), 0x5410);
  const uint32_t lo = __byte_perm(__byte_perm(p[7], p[6], 0x0073), __byte_perm(p[5], p[4], 0x0073), 0x5410);
  code = ((uint64_t)hi << 32) | lo;
  inv = 0;
  if (any) {
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const uint32_t x = w[m];
      const uint32_t c4 = ((x >> 1) ^ (x >> 2)) & 0x03030303u;
      const uint32_t n4 = c4 | (c4 >> 4);
      const uint32_t d = __byte_perm(0x74676361u, 0, __byte_perm(n4, 0, 0x4420)) ^ (x | 0x20202020u);
      const uint32_t bad = (((d & 0x7f7f7f7fu) + 0x7f7f7f7fu) | d) & 0x80808080u;  // top bit of each nonzero byte
      inv |= (((bad >> 7) & 1u) | ((bad >> 14) & 2u) | ((bad >> 21) & 4u) | ((bad >> 28) & 8u)) << (4 * m);
    }
  }
}

// Convert code word w (bases 32w .. 32w+31) straight from the reads.
__device__ __forceinline__ void convert_word(const uint8_t* reads, uint64_t L, uint64_t w, uint64_t& code, uint32_t& inv) {
  const uint64_t p = w * 32;
  uint32_t x[8];
  if (p + 32 <= L) {
    const uint4* src = reinterpret_cast<const uint4*>(reads + p);
    const uint4 a = __ldcs(src), b2 = __ldcs(src + 1);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b2.x; x[5] = b2.y; x[6] = b2.z; x[7] = b2.w;
    pack32(x, code, inv);
  } else {
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      uint32_t v = 0;
      for (int r = 0; r < 4; ++r) {
        const uint64_t q = p + 4 * m + r;
        v |= (uint32_t)(q < L ? reads[q] : 0) << (8 * r);
      }
      x[m] = v;
    }
    pack32(x, code, inv);  // byte 0 is not a base, so the tail past L is invalid
  }
}

// Mark read starts inside the slot window [j0-2, j0+nw) of a sub-step in st_s; advance *rcur
// to the first read whose start is >= the next sub-step's halo.  All threads call it.
__device__ void build_starts(const uint64_t* offsets, uint64_t n_reads, uint64_t j0, int nw, uint32_t* st_s,
                             uint64_t* rcur_s) {
  const int t = threadIdx.x, nt = blockDim.x;
  const int64_t st0 = (int64_t)j0 * 32 - 64;
  const uint64_t end = (j0 + nw) * 32;
  const int64_t next_halo = (int64_t)end - 64;
  uint64_t base = *rcur_s;
  uint64_t adv = 0;
  while (true) {
    const uint64_t i = base + t;
    const uint64_t p = i < n_reads ? offsets[i] : ~0ull;
    if (p < end) {
      const int64_t rel = (int64_t)p - st0;
      if (rel >= 0 && rel < (int64_t)(nw + 2) * 32) atomicOr(&st_s[rel >> 5], 1u << (rel & 31));
    }
    const int nb = __syncthreads_count(p != ~0ull && (int64_t)p < next_halo);
    const int ne = __syncthreads_count(p < end);
    adv += nb;
    if (ne < nt) break;
    base += nt;
  }
  if (t == 0) *rcur_s += adv;
}

// Variants of the phase-1 kernels: canonical keys and forward keys of k >= 16, whose top 32
// bits need no mask, and any k < 16.
enum { V_SHORT, V_CANON, V_FORWARD };

// The range map: coarse partition, fine partition are bit fields of a 32-bit value u,
// non-decreasing in the key.  x = top 32 bits of the 2k-bit key; canonical keys are the
// min of two near-independent uniforms (density 2(1-x)), so u = 1 - (1-x)^2 (its
// distribution function) spreads them evenly.
__device__ __forceinline__ uint32_t top32_of(uint64_t key, int k) { return (uint32_t)((key << (64 - 2 * k)) >> 32); }
__device__ __forceinline__ uint32_t top32_of(u128 key, int k) { return (uint32_t)(key >> (2 * k - 32)); }
__device__ __forceinline__ uint32_t umap(uint32_t x, int canonical) {
  if (!canonical) return x;
  const uint32_t y = ~x;
  return ~__umulhi(y, y);
}
// x >> s, and 0 for s >= 32 (one clamping funnel shift)
__device__ __forceinline__ uint32_t shr_clamp(uint32_t x, uint32_t s) { return __funnelshift_rc(x, 0u, s); }
// the coarse field of u: its top b1 bits (none for b1 = 0)
__device__ __forceinline__ uint32_t coarse_field(uint32_t u, int b1) { return shr_clamp(u, 32 - b1); }
// The same field counted from its far end (2^b1 - 1 - field), one instruction cheaper: the
// order of the partitions inside one block's shared arrays.
__device__ __forceinline__ uint32_t coarse_field_rev(uint32_t x, int canonical, int b1) {
  const uint32_t y = ~x;
  return shr_clamp(canonical ? __umulhi(y, y) : y, 32 - b1);
}
template <class K>
__device__ __forceinline__ uint32_t coarse_of(K key, int k, int canonical, int b1) {
  return coarse_field(umap(top32_of(key, k), canonical), b1);
}

// floor(sqrt(v)) from 32-bit conversions and single-precision arithmetic (64-bit
// conversions and double precision are slow on this GPU): the single-precision root is
// within 2^32 * 2^-24 of the true one; one Newton step on the exact residual brings it
// within a few units, and exact integer comparisons finish.  The root is below 2^32, so
// every square fits in 64 bits.
__host__ __device__ __forceinline__ float u64_to_float(uint64_t v) {
  return (float)(uint32_t)(v >> 32) * 4294967296.0f + (float)(uint32_t)v;
}
__host__ __device__ __forceinline__ uint64_t isqrt64(uint64_t v) {
  const float f = sqrtf(u64_to_float(v));
  uint64_t y = f >= 4294967296.0f ? 0xffffffffull : (uint64_t)(uint32_t)f;
  if (y > 0) {
    const int64_t r = (int64_t)(v - y * y);  // |r| < 2^42
    const float rf = (float)(int32_t)(r >> 32) * 4294967296.0f + (float)(uint32_t)r;
    const int64_t z = (int64_t)y + (int32_t)(rf / (2.0f * (float)(uint32_t)y));  // step below 2^10
    y = z < 0 ? 0 : (z > 0xffffffffll ? 0xffffffffull : (uint64_t)z);
  }
  while (y > 0 && y * y > v) --y;
  while (y < 0xffffffffull && (y + 1) * (y + 1) <= v) ++y;
  return y;
}

// The top-32-bit values x whose range-map value lies in [ulo, uhi]: [xlo, xhi] (empty when
// xlo > xhi).  Canonical: umap(x) = 2^32 - 1 - floor(y^2 / 2^32) with y = 2^32 - 1 - x, so
// umap(x) >= ulo  <=>  y^2 < (2^32 - ulo) 2^32   and   umap(x) <= uhi  <=>  y^2 >= (2^32 - 1 - uhi) 2^32.
__host__ __device__ __forceinline__ void x_range(uint32_t ulo, uint32_t uhi, int canonical, uint32_t& xlo,
                                                 uint32_t& xhi) {
  if (!canonical) {
    xlo = ulo;
    xhi = uhi;
    return;
  }
  const uint64_t ymax = isqrt64(((uint64_t)(0x100000000ull - ulo) << 32) - 1);  // wraps to 2^64 - 1 for ulo = 0
  xlo = 0xffffffffu - (uint32_t)(ymax < 0xffffffffull ? ymax : 0xffffffffull);
  const uint64_t m = (uint64_t)(~uhi) << 32;
  const uint64_t ymin = m == 0 ? 0 : isqrt64(m - 1) + 1;  // ceil(sqrt(m))
  xhi = ymin > 0xffffffffull ? 0u : 0xffffffffu - (uint32_t)ymin;
  if (ymin > 0xffffffffull) xlo = 1;  // no x maps at or below uhi (only uhi = 0): empty
}

// Keys (2k bits) whose top 32 bits lie in [xlo, xhi].
__host__ __device__ __forceinline__ void key_range(uint32_t xlo, uint32_t xhi, int k, uint64_t& lo, uint64_t& hi) {
  lo = ((uint64_t)xlo << 32) >> (64 - 2 * k);
  hi = (((uint64_t)xhi << 32) | 0xffffffffull) >> (64 - 2 * k);
}
__host__ __device__ __forceinline__ void key_range(uint32_t xlo, uint32_t xhi, int k, u128& lo, u128& hi) {
  const int sh = 2 * k - 32;
  lo = (u128)xlo << sh;
  hi = ((u128)xhi << sh) | (((u128)1 << sh) - 1);
}

// Windows of one thread: WPT consecutive window ends starting at base q0 (q0 = 32j for
// WPT == 32; q0 = 32j + 16h for WPT == 16).  With the base stream S aligned so that window
// i's first base is S's base i, window i's forward key is the top 2k bits of S << 2i and
// its reverse complement the top 2k bits of R << 2(WPT-1-i), R being the complemented
// bases in reverse order.  Both shifts are compile-time constants once the loop over i is
// unrolled.  Values are kept top-aligned (key << (64 or 128) - 2k), so the top 32 bits
// that drive the range map come for free.
struct Win {
  uint64_t s0, s1, s2;  // S, left-aligned (192 bits; only s0, s1 used for k <= 32)
  uint64_t r0, r1, r2;  // R, left-aligned
  uint64_t m0, m1;      // mask of the top 2k bits (m1 used for k > 32)
  uint32_t valid;       // bit i: window i has k bases in ACGTacgt and no read start inside
};

__device__ __forceinline__ uint64_t shl128_hi(uint64_t a, uint64_t b, int sh) {  // top word of (a:b) << sh, 0 <= sh <= 64
  return sh == 0 ? a : (sh >= 64 ? b : (a << sh) | (b >> (64 - sh)));
}

// Mask of valid window ends for the 32 bases of word j: bit e (0..31) is set iff the k
// bases ending at 32j + e are all bases (inv clear) and no read starts at any of the last
// k - 1 of them.  inv / starts over words j-2, j-1, j as one 96-bit value, LSB = base 32j-64.
__device__ __forceinline__ uint32_t valid_mask(uint32_t i2, uint32_t i1, uint32_t i0, uint32_t t2, uint32_t t1,
                                               uint32_t t0, int k) {
  const u128 I = (u128)i2 | ((u128)i1 << 32) | ((u128)i0 << 64);
  const u128 S = (u128)t2 | ((u128)t1 << 32) | ((u128)t0 << 64);
  // a read start at base p forbids windows holding p-1 and p: mark base p-1 (C = I | S >> 1)
  // window [e-k+1, e] is valid iff C has no bit in [e-k+1, e-1] and I has no bit at e
  u128 bad = I;
  const int w = k - 1;
  if (w > 0) {
    const u128 C = I | (S >> 1);
    u128 Y = C;  // OR over a window of width 2^p ending at each bit
    int p = 1;
    while (2 * p <= w) {
      Y |= Y << p;
      p *= 2;
    }
    if (w > p) Y |= Y << (w - p);  // width w
    bad |= Y << 1;                 // windows ending at e look at C bits e-1 .. e-w
  }
  return ~(uint32_t)(bad >> 64);
}

template <int KW, int WPT>
__device__ __forceinline__ void win_setup(uint64_t w2, uint64_t w1, uint64_t w0, uint32_t vmask_word, int h, int k,
                                          Win& W) {
  // (w2 : w1 : w0) holds bases 32j-64 .. 32j+31; the first window's first base is
  // q0 - k + 1 = 32j + 16h - k + 1, at index 65 + 16h - k of that string.
  const int off = 65 + 16 * h - k;  // base index, >= 1
  const int sh = 2 * off;           // bits to drop from the top, 2 .. 162
  if (sh >= 128) {
    W.s0 = w0 << (sh - 128);
    W.s1 = 0;
    W.s2 = 0;
  } else if (sh >= 64) {
    W.s0 = shl128_hi(w1, w0, sh - 64);
    W.s1 = (sh - 64 == 0) ? w0 : w0 << (sh - 64);
    W.s2 = 0;
  } else {
    W.s0 = shl128_hi(w2, w1, sh);
    W.s1 = shl128_hi(w1, w0, sh);
    W.s2 = w0 << sh;
  }
  // R: complements of bases 32j+31 down to 32j-64; window i's reverse complement starts at
  // base q0 + i, i.e. at index 31 - 16h - i of R, so align R to index 31 - 16h - (WPT - 1).
  const uint64_t r0 = revpairs64(~w0), r1 = revpairs64(~w1), r2 = revpairs64(~w2);
  const int rsh = 2 * (32 - 16 * h - WPT);  // 0 (WPT 32 or h 1) or 32 (WPT 16, h 0)
  W.r0 = shl128_hi(r0, r1, rsh);
  W.r1 = shl128_hi(r1, r2, rsh);
  W.r2 = rsh ? r2 << rsh : r2;
  if (KW == 1) {
    W.m0 = k >= 32 ? ~0ull : ~(~0ull >> (2 * k));
    W.m1 = 0;
  } else {
    W.m0 = ~0ull;
    W.m1 = k >= 64 ? ~0ull : ~(~0ull >> (2 * k - 64));
  }
  W.valid = vmask_word >> (16 * h);
}

// Window i: the canonical value, top-aligned (top 64 bits in c0, next 64 in c1 for k > 32).
template <int KW, int WPT>
__device__ __forceinline__ void win_top(const Win& W, int i, int canonical, uint64_t& c0, uint64_t& c1) {
  const int fs = 2 * i, rs = 2 * (WPT - 1 - i);
  if constexpr (KW == 1) {
    const uint64_t f = shl128_hi(W.s0, W.s1, fs) & W.m0;
    const uint64_t r = shl128_hi(W.r0, W.r1, rs) & W.m0;
    c0 = (canonical && r < f) ? r : f;
    c1 = 0;
  } else {
    const uint64_t f0 = shl128_hi(W.s0, W.s1, fs), f1 = shl128_hi(W.s1, W.s2, fs) & W.m1;
    const uint64_t r0 = shl128_hi(W.r0, W.r1, rs), r1 = shl128_hi(W.r1, W.r2, rs) & W.m1;
    const bool rlt = canonical && ((r0 < f0) || (r0 == f0 && r1 < f1));
    c0 = rlt ? r0 : f0;
    c1 = rlt ? r1 : f1;
  }
}
// Top 32 bits of (a:b) << sh, 0 <= sh < 64 (a compile-time constant once unrolled).
__device__ __forceinline__ uint32_t top32_shl(uint64_t a, uint64_t b, int sh) {
  return sh < 32 ? __funnelshift_l((uint32_t)a, (uint32_t)(a >> 32), sh)
                 : __funnelshift_l((uint32_t)(b >> 32), (uint32_t)a, sh - 32);
}
// Window i: the top 32 bits of its canonical value only (the range-map input), from 32-bit
// shifts.  The smaller of the forward and reverse-complement top words is the canonical
// value's top word: where the top words differ they decide which value is smaller, and
// where they tie both values share them.
template <int KW, int WPT, int VAR>
__device__ __forceinline__ uint32_t win_top32(const Win& W, int i, int canonical, uint32_t& f, uint32_t& r) {
  const uint32_t m = VAR == V_SHORT ? (uint32_t)(W.m0 >> 32) : ~0u;
  f = top32_shl(W.s0, W.s1, 2 * i) & m;
  r = top32_shl(W.r0, W.r1, 2 * (WPT - 1 - i)) & m;
  return canonical ? min(f, r) : f;
}
__device__ __forceinline__ void top_to_key(uint64_t c0, uint64_t, int k, uint64_t& key) {
  key = k >= 32 ? c0 : c0 >> (64 - 2 * k);
}
__device__ __forceinline__ void top_to_key(uint64_t c0, uint64_t c1, int k, u128& key) {
  const u128 c = ((u128)c0 << 64) | c1;
  key = k >= 64 ? c : c >> (128 - 2 * k);
}

// ------------------------------------------------------------------ distinct-key sketch
__device__ __forceinline__ uint64_t key_hash(uint64_t key) { return key * 0x9E3779B97F4A7C15ull; }
__device__ __forceinline__ uint64_t key_hash(u128 key) {
  return ((uint64_t)key ^ ((uint64_t)(key >> 64) * 0xC2B2AE3D27D4EB4Full)) * 0x9E3779B97F4A7C15ull;
}

// A HyperLogLog over a 1/64 sample of the keys, chosen by the sum of the window's top forward
// and reverse-complement words (its first and its last 16 bases: the words that its partition
// is found from, the same on either strand).  The first bases alone would take or leave the
// variants of a repeat together: on the repeat genome that estimate was 11% low.  A register
// is read before it is raised: after the first few thousand keys hardly one still rises.
__device__ __forceinline__ bool sketch_sampled(uint32_t f, uint32_t r) {
  return ((f + r) * 0x9E3779B1u) >> (32 - kHllSampleLog2) == 0;
}
template <class K>
__device__ __forceinline__ void sketch_add(uint32_t* hll, K key) {
  const uint64_t h = key_hash(key);
  const uint32_t reg = (uint32_t)(h >> (64 - kHllLog2));
  const uint32_t v = (uint32_t)min(__clzll(h << kHllLog2) + 1, 64 - kHllLog2 + 1);
  if (v > hll[reg]) atomicMax(&hll[reg], v);
}
// The canonical (or forward) key of the window whose last base is s bases before the end of
// the 96 bases (w2 : w1 : w0); 0 <= s < 32.  For the few windows picked out by a run-time index.
__device__ __forceinline__ void window_key(uint64_t, uint64_t w1, uint64_t w0, uint32_t s, int k, int canonical,
                                           uint64_t& key) {
  const int x = 64 - 2 * k;
  const uint64_t f = (s ? (w0 >> (2 * s)) | (w1 << (64 - 2 * s)) : w0) << x >> x;
  const uint64_t r = revcomp(f, k);
  key = canonical && r < f ? r : f;
}
__device__ __forceinline__ void window_key(uint64_t w2, uint64_t w1, uint64_t w0, uint32_t s, int k, int canonical,
                                           u128& key) {
  const int x = 128 - 2 * k;
  u128 f = ((u128)w1 << 64 | w0) >> (2 * s);
  if (s) f |= (u128)(w2 << (64 - 2 * s)) << 64;
  f = f << x >> x;
  const u128 r = revcomp(f, k);
  key = canonical && r < f ? r : f;
}
// A thread's sampled windows (bit i of m: the window whose last base is last - i bases before
// the end of the words) go to the sketch after its loop over the windows.  Inside that loop
// two warps in five left it at every window for the one lane that had a sampled key. (Pass B of
// 2.4 G windows 11.93 -> 10.77 ms, of 59 M 128-bit windows 596 -> 565 us; pass A of 10 M bases,
// one level, 45 -> 40.)
template <class K>
__device__ __forceinline__ void sketch_windows(uint32_t* hll, uint32_t m, uint32_t last, uint64_t w2, uint64_t w1,
                                               uint64_t w0, int k, int canonical) {
  while (m) {
    const uint32_t i = __ffs(m) - 1;
    m &= m - 1;
    K key;
    window_key(w2, w1, w0, last - i, k, canonical, key);
    sketch_add(hll, key);
  }
}

// Estimated distinct keys D from the sketch's m = 1024 registers, each r (HyperLogLog, over one
// key in 64): 64 c / Z for Z = the sum of 2^-r, and 64 m log(m / zeros) (linear counting) while
// many registers are 0.  What a count needs is 9/10 of its windows per distinct key; the sketch
// gives it as an integer, 0.9 * 2^68 / D, to be multiplied by the windows.  Z is added up exactly
// (in units of 2^-53) and the quotients are constants, so that the way from the last key's
// register to the plan, on which every later kernel waits, has no division, logarithm or double
// precision on it.  (In double precision pass A of 0.2 M and of 10 M bases took 21.5 and 43 us
// instead of 17.5 and 38, and the calls 13 and 16 us more: its constants come from memory that is
// not in the caches between counts.  That holds for any constant that is not in the code: the two
// below as loads cost 5 to 11 us a call.)
constexpr double kTwo53 = 9007199254740992.0, kHllM = kHllRegs;
constexpr double kHllC = 0.7213 / (1.0 + 1.079 / kHllM) * kHllM * kHllM;
constexpr uint64_t kHllMul = (uint64_t)(0.9 / (kHllSample * kHllC) * 67108864.0 * kTwo53);  // times Z * 2^53: the top word
constexpr uint64_t kHllFew = (uint64_t)(kHllC / (2.5 * kHllM) * kTwo53);  // Z * 2^53 above which D is below 64 * 2.5 m
struct FewKeys {
  uint64_t at[kHllRegs + 1];  // [zeros]: linear counting (0 if every register is 0: no key seen)
};
constexpr double ln_series(double f) {  // log(f), f in [1, 2], by the series of atanh((f - 1) / (f + 1))
  const double t = (f - 1.0) / (f + 1.0);
  double p = t, sum = 0.0;
  for (int i = 1; i < 40; i += 2) {
    sum += p / i;
    p *= t * t;
  }
  return 2.0 * sum;
}
constexpr FewKeys few_keys() {
  FewKeys k{};
  const double ln2 = ln_series(2.0);
  for (int z = 1; z < kHllRegs; ++z) {
    double f = kHllM / z, l = 0.0;
    for (; f >= 2.0; f *= 0.5) l += ln2;
    l += ln_series(f);
    k.at[z] = (uint64_t)(0.9 / (kHllSample * kHllM * l) * 32768.0 * kTwo53);
  }
  return k;
}
static __device__ const FewKeys kFewKeys = few_keys();

// The keys a fine partition aims at, from the sketch of a count of K windows: fine_target
// distinct keys, i.e. fine_target * K / D keys (a tenth less, for the estimate's error, and at
// most 32 times as many); where that gives an SM few partitions, as much less as makes them a
// whole number (one partition too many for a last wave costs a small count a wave: 10 M bases
// had 497 for 152 SMs, and 0.2 M bases 11).  `extra`: partitions that come on top of K / target.
// All threads of the block call it.
__device__ uint32_t sketch_target(const uint32_t* hll, uint64_t K, const Shape& s, uint32_t extra) {
  __shared__ uint64_t zsum_s[32];
  __shared__ uint32_t zeros_s[32], target_s;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint64_t z = 0;  // in units of 2^-53 (at most 1024 registers of 1: below 2^64)
  uint32_t zeros = 0;
  for (int i = threadIdx.x; i < kHllRegs; i += blockDim.x) {  // (read from L2: written by every SM)
    const uint32_t r = __ldcg(&hll[i]);
    z += (1ull << 53) >> r;
    zeros += r == 0;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) z += __shfl_xor_sync(0xffffffffu, z, d);
  zeros = __reduce_add_sync(0xffffffffu, zeros);
  if (lane == 0) {
    zsum_s[wid] = z;
    zeros_s[wid] = zeros;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    z = zeros = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      z += zsum_s[w];
      zeros += zeros_s[w];
    }
    const uint64_t per_window = zeros && z > kHllFew ? kFewKeys.at[zeros] : __umul64hi(z, kHllMul);
    // 0.9 K / D in units of 2^-32, between 1 and 0.9 * 32
    const uint64_t hi = __umul64hi(K, per_window), lo = K * per_window, most = (uint64_t)(28.8 * 4294967296.0);
    const uint64_t dup = max((uint64_t)1 << 32, hi >= 512 ? most : min(most, (hi << 28) | (lo >> 36)));
    const uint64_t keys = s.fine_target * dup;
    uint32_t target = (uint32_t)((keys + 0xffffffffull) >> 32);
    const float per_sm = ceilf(((float)K / ((float)keys * 2.3283064e-10f) + (float)extra) / (float)s.n_sms);
    if (per_sm <= 16.0f) {  // (an empty count may have no partition left for keys: 0 / 0, which fmaxf drops)
      const float parts = per_sm * (float)s.n_sms - (float)extra;
      target = (uint32_t)fminf((float)target, ceilf(fmaxf((float)K / parts + 1.0f, (float)kMinFineKeys)));
    }
    target_s = target;
  }
  __syncthreads();
  return target_s;
}

// ------------------------------------------------------------------ pass A
// Add 1 to the shared word at address a if p is not 0.
__device__ __forceinline__ void red_shared_if(uint32_t a, uint32_t p) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q red.shared.add.u32 [%0], 1;\n\t}" ::"r"(a), "r"(p) : "memory");
}
// Partition starts (also pass B's cursors) from the partitions' totals (added up in cstart by
// all blocks), and the total number of windows.  One block; sc: P1 words.
__device__ __forceinline__ void bucket_scan(const Shape& s, const Buffers& b, uint64_t* sc) {
  __shared__ uint64_t wt[32];
  const int P1 = 1 << s.b1;
  for (int c = threadIdx.x; c < P1; c += blockDim.x) {
    const uint64_t n = __ldcg(&b.cstart[c]);
    sc[c] = n;
    if (n > 0xffffffffull) atomicOr(&b.meta->status, ST_PARTITION_OVERFLOW);  // (the fine split counts in 32 bits)
  }
  __syncthreads();
  const uint64_t K = block_exclusive_scan<uint64_t>(sc, P1, wt);
  for (int c = threadIdx.x; c < P1; c += blockDim.x) b.cstart[c] = b.fcur[c] = sc[c];
  if (threadIdx.x == 0) {
    b.cstart[P1] = K;
    b.meta->n_windows = K;
  }
}

// One-level partitioning: the bins, in order, are grouped into fine partitions of about T keys
// (T from the sketch): a bin belongs to the partition in which its first key falls when every
// partition takes T, so a partition takes T keys, give or take a bin.  Writes the bins' map and
// the partitions' starts (also pass B's cursors) and first range-map values; a partition that
// no bin starts in is left empty.  One block; sc: 2^bb words, padded.
__device__ __forceinline__ void one_level_plan(const Shape& s, const Buffers& b, uint32_t* sc) {
  __shared__ uint32_t wt[32];
  const int NB = 1 << s.bb;
  if (threadIdx.x <= kHllRegs / 16)  // linear counting's table, a line each, while the bins are added up
    asm volatile("prefetch.global.L2 [%0];" ::"l"(&kFewKeys.at[threadIdx.x * 16]));
#pragma unroll 8
  for (int i = threadIdx.x; i < NB; i += blockDim.x) sc[PAD(i)] = __ldcg(&b.bins[i]);
  __syncthreads();
  const uint32_t K = block_exclusive_scan_pad<uint32_t>(sc, NB, wt);  // below 2^26
  const uint32_t T = max(sketch_target(b.hll, K, s, 0), (uint32_t)(K / s.nf_max) + 1u);
  const uint32_t NF = sc[PAD(NB - 1)] / T + 1;  // the last bin's partition is the last: at most K / T + 1 <= nf_max
  const bool either = s.one_level == kEitherLevel;
  if (either && NF > kEitherFine) {  // two levels: the coarse partitions are the bins' top bits
    const int P1 = 1 << s.b1, per = NB >> s.b1;
    for (int i = threadIdx.x; i < NB; i += blockDim.x) b.bmap2[i] = (uint16_t)(i / per);
    for (int c = threadIdx.x; c < P1; c += blockDim.x) b.cstart[c] = b.fcur[c] = sc[PAD(c * per)];
    if (threadIdx.x == 0) {
      b.cstart[P1] = K;
      b.meta->n_windows = K;
    }
    return;
  }
  for (int i = threadIdx.x; i < NB; i += blockDim.x) {
    const uint32_t p = sc[PAD(i)];
    const int g = (int)(p / T), prev = i ? (int)(sc[PAD(i - 1)] / T) : -1;
    b.bmap[i] = (uint16_t)g;
    for (int q = prev + 1; q <= g; ++q) {
      b.foff[q] = p;
      b.fcur[q] = p;
      if (!either) b.flo[q] = (uint32_t)i << (32 - s.bb);  // (either: after pass B, in the codes' memory)
    }
  }
  if (threadIdx.x == 0) {
    b.foff[NF] = K;
    if (!either) b.flo[NF] = 0;  // so that the last partition ends at u = 2^32 - 1
    b.meta->one = 1;
    b.meta->n_windows = K;
    b.meta->n_fine = NF;
  }
}

// One code word per thread: convert, store, and histogram the partitions of its 32 windows
// (keys are computed in pass B, which needs the partition offsets first).  The last block turns
// the partitions' totals into their starts.  Bound by the ALU (86% busy at 2.4 G windows): a
// window takes two funnel shifts, a minimum, the range map and one predicated reduction, with
// no masks (variants by k and mode) and no select for invalid windows, and a word's bytes are
// converted by multiplications and byte permutations; 2.95 ms, where masks, selects and
// byte-by-byte comparisons took 4.44.
// ONE: the windows of every bin instead, and the distinct-key sketch, from which the last
// block plans the fine partitions.
template <int KW, bool ONE, int VAR>
__device__ __forceinline__ void pack_tile(const Shape& s, const Buffers& b, uint64_t tile, uint32_t* hist_s) {
  typedef typename KeyT<KW>::T K;
  __shared__ uint64_t code_s[kPackThreads + 2];
  __shared__ uint32_t inv_s[kPackThreads + 2];
  __shared__ uint32_t st_s[kPackThreads + 2];
  __shared__ uint64_t rcur_s, len_s;
  const int t = threadIdx.x;
  const int bits = ONE ? s.bb : s.b1;
  const int canonical = VAR == V_SHORT ? s.canonical : VAR == V_CANON;
  const uint32_t hist_a = (uint32_t)__cvta_generic_to_shared(hist_s);
  if (t == 0) {
    rcur_s = b.tile_first[tile];
    // bases read: never past the end the offsets give (a base count that disagrees with
    // them is reported by check_offsets; the reads buffer is not overrun meanwhile)
    const uint64_t e = b.offsets[s.n_reads];
    len_s = e < s.L ? e : s.L;
  }
  __syncthreads();
  const uint64_t len = len_s;
  for (int sub = 0; sub < (int)s.tile_words / kPackThreads; ++sub) {
    const uint64_t j0 = tile * s.tile_words + (uint64_t)sub * kPackThreads;
    if (j0 >= s.n_words) break;
    __syncthreads();
    if (t < 2) {
      if (sub > 0) {
        code_s[t] = code_s[kPackThreads + t];
        inv_s[t] = inv_s[kPackThreads + t];
      } else if (j0 + t >= 2) {
        convert_word(b.reads, len, j0 + t - 2, code_s[t], inv_s[t]);
      } else {
        code_s[t] = 0;
        inv_s[t] = ~0u;
      }
    }
    const uint64_t j = j0 + t;
    uint64_t code = 0;
    uint32_t inv = ~0u;
    if (j < s.n_words) {
      convert_word(b.reads, len, j, code, inv);
      b.codes64[j] = code;
      b.inv32[j] = inv;
    }
    __syncthreads();
    code_s[t + 2] = code;
    inv_s[t + 2] = inv;
    st_s[t + 2] = 0;
    if (t < 2) st_s[t] = 0;
    __syncthreads();
    build_starts(b.offsets, s.n_reads, j0, kPackThreads, st_s, &rcur_s);
    __syncthreads();
    if (j < s.n_words) {
      Win W;
      const uint32_t vm = valid_mask(inv_s[t], inv_s[t + 1], inv, st_s[t], st_s[t + 1], st_s[t + 2], s.k);
      win_setup<KW, 32>(code_s[t], code_s[t + 1], code, vm, 0, s.k, W);
      uint32_t picked = 0;  // windows for the sketch
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        uint32_t f, r;
        const uint32_t c = coarse_field_rev(win_top32<KW, 32, VAR>(W, i, canonical, f, r), canonical, bits);
        const uint32_t v = W.valid & (1u << i);
        red_shared_if(hist_a + 4 * c, v);  // predicated: no branch, no bin for the invalid windows
        if (ONE && sketch_sampled(f, r)) picked |= 1u << i;
      }
      if constexpr (ONE)
        sketch_windows<K>(b.hll, picked & W.valid, 31, code_s[t], code_s[t + 1], code_s[t + 2], s.k, canonical);
    }
  }
  __syncthreads();
}
template <int KW, bool ONE, int VAR>
__device__ __forceinline__ void pack_count_body(const Shape& s, const Buffers& b, uint32_t bid, uint32_t nblk) {
  extern __shared__ __align__(16) uint32_t hist_s[];  // [P1], partitions from the last to the first
  const int t = threadIdx.x, P1 = 1 << (ONE ? s.bb : s.b1);
  check_offsets(s, b, bid, nblk);
  if (bid < s.n_tiles) {  // (an empty input has a block and no tile; many short reads, blocks for their offsets only)
    for (int c = t; c < P1; c += kPackThreads) hist_s[c] = 0;
    if constexpr (ONE) {  // several tiles, so that the bins are added up less often
      for (uint64_t tile = bid; tile < s.n_tiles; tile += nblk) pack_tile<KW, true, VAR>(s, b, tile, hist_s);
      for (int i = t; i < P1; i += kPackThreads) {  // (each block starts elsewhere: all end together)
        const int c = (i + bid * 13 * kPackThreads) & (P1 - 1);
        if (hist_s[c]) atomicAdd(&b.bins[P1 - 1 - c], hist_s[c]);
      }
    } else {
      pack_tile<KW, false, VAR>(s, b, bid, hist_s);
      // the tile's counts, and the partitions' totals (cstart holds them until bucket_scan)
      for (int c = t; c < P1; c += kPackThreads) {
        const uint32_t n = hist_s[P1 - 1 - c];
        b.hist[(uint64_t)bid * P1 + c] = n;
        if (n) atomicAdd(reinterpret_cast<unsigned long long*>(&b.cstart[c]), (unsigned long long)n);
      }
    }
  }
  if (!last_block(&b.meta->done, nblk)) return;
  if (bad_offsets(b)) return;  // no windows, no fine partitions (both 0 since k_prepare)
  if constexpr (ONE) one_level_plan(s, b, hist_s);
  else bucket_scan(s, b, reinterpret_cast<uint64_t*>(hist_s));
}
template <int KW, bool ONE, int VAR>
__global__ void __launch_bounds__(kPackThreads, KW == 1 ? 4 : 2) k_pack_count(Shape s, Buffers b) {
  pdl_wait();
  pack_count_body<KW, ONE, VAR>(s, b, blockIdx.x, gridDim.x);
}
template <int KW, bool ONE, int VAR>
__global__ void __launch_bounds__(kPackThreads, KW == 1 ? 4 : 2) k_pack_count_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  pack_count_body<KW, ONE, VAR>(d.s, d.b, bid, nblk);
}

// Fine split of every coarse partition, after pass B: the distinct-key estimate (filled by pass
// B) gives the keys a fine partition aims at, and coarse partition c is cut into
// m_c = ceil(n_c / target).  One block per coarse partition; each finds the number of fine
// partitions before its own for itself (a block of one launch for all took 98 us for 100 K
// fine partitions and 219 us for 221 K, this takes 9 and 11).
__device__ __forceinline__ void fine_plan_body(const Shape& s, const Buffers& b, uint32_t c) {
  extern __shared__ uint32_t fsc[];  // [padded P1]
  __shared__ uint32_t wt[32];
  const int P1 = 1 << s.b1;
  if (bad_offsets(b)) return;
  if (s.one_level && b.meta->one) {  // planned before pass B; what is left is the partitions' first values
    for (int i = c * blockDim.x + threadIdx.x; i < (1 << s.bb); i += P1 * blockDim.x)
      for (int q = i ? b.bmap[i - 1] + 1 : 0; q <= b.bmap[i]; ++q) b.flo[q] = (uint32_t)i << (32 - s.bb);
    if (c == 0 && threadIdx.x == 0) b.flo[min(b.meta->n_fine, s.nf_max)] = 0;
    return;
  }
  const uint32_t T = sketch_target(b.hll, b.cstart[P1], s, P1);
  auto parts = [&](uint64_t n) -> uint32_t {  // (n is below 2^32)
    const uint32_t m = n ? ((uint32_t)n - 1) / T + 1 : 1;
    return m < (uint32_t)kMaxFine ? m : (uint32_t)kMaxFine;
  };
  for (int i = threadIdx.x; i < P1; i += blockDim.x) fsc[PAD(i)] = parts(b.cstart[i + 1] - b.cstart[i]);
  __syncthreads();
  const uint32_t NF = block_exclusive_scan_pad<uint32_t>(fsc, P1, wt);
  const uint32_t base = fsc[PAD(c)], nf_max = (uint32_t)s.nf_max;
  const uint64_t m = parts(b.cstart[c + 1] - b.cstart[c]);
  // fine partition f of c holds the values u of coarse field c whose low part v = u mod
  // 2^(32 - b1) has floor(v m / 2^(32 - b1)) = f, i.e. v >= ceil(f 2^(32 - b1) / m)
  const uint64_t w = 1ull << (32 - s.b1);
  for (uint64_t f = threadIdx.x; f < m && base + f < nf_max; f += blockDim.x)
    b.flo[base + f] = (uint32_t)((uint64_t)c << (32 - s.b1)) + (uint32_t)((f * w + m - 1) / m);
  if (threadIdx.x == 0) {
    b.fine_base[c] = base;
    b.fine_m[c] = (uint32_t)m;
    if ((int)c == P1 - 1) {
      if (NF <= nf_max) b.flo[NF] = 0;  // so that the last partition ends at u = 2^32 - 1
      b.fine_base[P1] = NF;
      b.meta->n_fine = NF <= nf_max ? NF : 0;  // later kernels never index past nf_max
      if (NF > nf_max) atomicOr(&b.meta->status, ST_INTERNAL);
    }
  }
}
__global__ void __launch_bounds__(256) k_fine_plan(Shape s, Buffers b) { pdl_wait(); fine_plan_body(s, b, blockIdx.x); }
__global__ void __launch_bounds__(256) k_fine_plan_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  fine_plan_body(d.s, d.b, bid);
}

// ------------------------------------------------------------------ pass B
// Per sub-step, NT threads x WPT windows.  A window's partition comes from the top 32 bits of
// its canonical value alone, and its rank inside the partition from a shared-memory atomic (a
// counting sort's first step); after the block scan of the partition histogram the whole keys
// are computed, go to their partition's run in the staging buffer, and the runs leave in
// order.  Bound by instruction issue and latency, not by HBM (19.2 GB written in 10.8 ms at 2.4 G
// windows): no key is kept in registers across the scan (each is computed once, after it) and
// a staged key's partition is found from the key again, so that three blocks fit an SM (80
// registers, 73 KB).  With the keys held and the partitions kept in shared memory there were
// two (128 registers) and it took 15.1 ms.
// SC_DIRECT (the aggregation ablation without per-block buckets): every valid window takes its
// slot with a global atomic on its partition's cursor and is written on its own.
// SC_ONE (one-level partitioning): the partitions are the fine ones, found through the bins'
// map, a sub-step reserves its run in each with one atomic, and the keys go to sbuf.
enum { SC_COARSE, SC_DIRECT, SC_ONE };
template <int KW, int NT, int MODE, int VAR>
__device__ __forceinline__ void scatter_body(const Shape& s, const Buffers& b, uint32_t bid) {
  typedef typename KeyT<KW>::T K;
  constexpr int WPT = KW == 1 ? 32 : 16;    // windows per thread
  constexpr int TPW = 32 / WPT;             // threads per code word
  constexpr int NW = NT / TPW;              // code words per sub-step
  constexpr int SUB = NT * WPT;             // windows per sub-step
  extern __shared__ __align__(16) uint8_t sm[];
  constexpr bool DIRECT = MODE == SC_DIRECT, ONE = MODE == SC_ONE;
  const bool refused = bad_offsets(b);
  const int canonical = VAR == V_SHORT ? s.canonical : VAR == V_CANON;
  const bool fine = ONE && b.meta->one;  // (ONE without: an either-level count that takes two)
  const int PM = ONE ? (s.one_level == kEitherLevel ? (int)kEitherFine : (int)s.nf_max) : 1 << s.b1;
  const int P1 = fine ? (int)min(b.meta->n_fine, (uint64_t)PM) : 1 << s.b1;
  K* stage = reinterpret_cast<K*>(sm);                                                // [SUB]
  unsigned long long* cursor = reinterpret_cast<unsigned long long*>(stage + SUB);   // [P1] absolute write positions
  uint32_t* hist = reinterpret_cast<uint32_t*>(cursor + (ONE ? 0 : P1));                // [padded PM + 32]
  uint32_t* soff = hist + padded_len(PM + 32);                                          // [padded PM + 32]
  uint16_t* map = reinterpret_cast<uint16_t*>(soff + padded_len(PM + 32));              // ONE: [2^bb]
  __shared__ uint64_t code_s[NW + 2];
  __shared__ uint32_t inv_s[NW + 2];
  __shared__ uint32_t st_s[NW + 2];
  __shared__ uint64_t rcur_s;
  __shared__ uint32_t wt[32];
  const int t = threadIdx.x;
  const int wl = t / TPW, h = t % TPW;  // code word of the thread within the sub-step, half
  const uint64_t tile = bid;
  for (int c = t; c < P1; c += NT) {
    // the tile's run in partition c, reserved at once (the order of the tiles' runs inside a
    // partition does not matter to any later step)
    if constexpr (!ONE) {
      const int p = P1 - 1 - c;  // shared arrays: partitions from the last to the first
      const uint32_t n = DIRECT ? 0u : b.hist[tile * P1 + p];
      cursor[c] = n ? atomicAdd(&b.fcur[p], (unsigned long long)n) : 0ull;
    }
    hist[PAD(c)] = 0;
  }
  if constexpr (ONE)
    for (int i = t; i < (1 << s.bb); i += NT) map[i] = (fine ? b.bmap : b.bmap2)[(1 << s.bb) - 1 - i];
  if (t == 0) rcur_s = (ONE && !fine ? b.tile_first2 : b.tile_first)[tile];
  if (refused) return;  // (here, so that the load's latency is shared with those above, all in bounds)
  for (int sub = 0; sub < (int)s.tile_words / NW; ++sub) {
    const uint64_t j0 = tile * s.tile_words + (uint64_t)sub * NW;
    if (j0 >= s.n_words) break;
    __syncthreads();
    if (t < 2) {  // the two words before: from memory again (the shared copies are being overwritten)
      const bool in = j0 + t >= 2;
      code_s[t] = in ? b.codes64[j0 + t - 2] : 0;
      inv_s[t] = in ? b.inv32[j0 + t - 2] : ~0u;
    }
    for (int w = t; w < NW; w += NT) {
      const uint64_t jw = j0 + w;
      code_s[w + 2] = jw < s.n_words ? b.codes64[jw] : 0;
      inv_s[w + 2] = jw < s.n_words ? b.inv32[jw] : ~0u;
      st_s[w + 2] = 0;
    }
    if (t < 2) st_s[t] = 0;
    __syncthreads();
    build_starts(b.offsets, s.n_reads, j0, NW, st_s, &rcur_s);
    __syncthreads();
    const int sw = wl + 2;
    const uint32_t vm = j0 + wl < s.n_words ? valid_mask(inv_s[sw - 2], inv_s[sw - 1], inv_s[sw], st_s[sw - 2],
                                                         st_s[sw - 1], st_s[sw], s.k)
                                            : 0u;
    Win W;
    win_setup<KW, WPT>(code_s[sw - 2], code_s[sw - 1], code_s[sw], vm, h, s.k, W);
    const uint32_t valid = W.valid & (WPT == 32 ? 0xffffffffu : 0xffffu);
    uint32_t cr[WPT];  // each window's partition and its rank there
    uint32_t picked = 0;  // windows for the sketch
    // every window is ranked without a branch (so that the windows' dependency chains
    // interleave): an invalid window is ranked in bin P1 + lane, which no scan reads (one such
    // bin per lane, so that a warp's invalid windows do not share an address), and the sketch's
    // windows are only noted
#pragma unroll
    for (int i = 0; i < WPT; ++i) {
      uint32_t f, r;
      const uint32_t x = win_top32<KW, WPT, VAR>(W, i, canonical, f, r);
      uint32_t c = coarse_field_rev(x, canonical, ONE ? s.bb : s.b1);
      if constexpr (ONE) c = map[c];
      const bool v = (valid >> i) & 1u;
      if constexpr (DIRECT) {
        if (v) {
          uint64_t c0, c1;
          K key;
          win_top<KW, WPT>(W, i, canonical, c0, c1);
          top_to_key(c0, c1, s.k, key);
          const unsigned long long pos = atomicAdd(&b.fcur[P1 - 1 - c], 1ull);
          if (pos < s.cap) store_key(b.kbuf, pos, key);
          else atomicOr(&b.meta->status, ST_INTERNAL);
        }
      } else {
        const uint32_t cc = v ? c : (uint32_t)P1 + (t & 31);
        cr[i] = (cc << 16) | atomicAdd(&hist[PAD(cc)], 1u);  // bin below 2^13, rank below 2^13
      }
      if (!ONE && sketch_sampled(f, r)) picked |= 1u << i;
    }
    if constexpr (!ONE)
      sketch_windows<K>(b.hll, picked & valid, 31 - 16 * h, code_s[sw - 2], code_s[sw - 1], code_s[sw], s.k, canonical);
    if constexpr (DIRECT) continue;
    __syncthreads();
    for (int c = t; c < P1; c += NT) soff[PAD(c)] = hist[PAD(c)];
    __syncthreads();
    const uint32_t n_sub = block_exclusive_scan_pad<uint32_t>(soff, P1, wt);
    // during the write-out cursor[c] holds cursor[c] - soff[c]: staged position i of partition c
    // goes to cursor[c] + i.  A run that would pass the end of the keys array (it cannot, if
    // pass A saw the same reads) is recorded and the sub-step not written.
    bool fits = true;
    for (int c = t; c < P1; c += NT) {
      if constexpr (ONE) {  // (positions are below 2^26; hist holds cursor - soff until it is cleared)
        const uint32_t n = hist[PAD(c)];
        if (n) {
          const uint64_t lim = (fine ? b.foff : b.cstart)[c + 1], at = atomicAdd(&b.fcur[c], (unsigned long long)n);
          fits = fits && at + n <= lim;
          hist[PAD(c)] = (uint32_t)at - soff[PAD(c)];
        }
      } else {
        fits = fits && cursor[c] + hist[PAD(c)] <= s.cap;
        cursor[c] -= soff[PAD(c)];
      }
    }
#pragma unroll
    for (int i = 0; i < WPT; ++i) {
      // an invalid window is staged at slot SUB - 1, which no valid window takes then (with
      // one window invalid, at most SUB - 1 are valid) and the write-out never reads
      uint64_t c0, c1;
      K key;
      win_top<KW, WPT>(W, i, canonical, c0, c1);
      top_to_key(c0, c1, s.k, key);
      const uint32_t pos = (valid & (1u << i)) ? soff[PAD(cr[i] >> 16)] + (cr[i] & 0xffffu) : (uint32_t)(SUB - 1);
      stage[pos] = key;
    }
    fits = __syncthreads_and(fits);
    if (fits) {
      for (uint32_t i = t; i < n_sub; i += NT) {
        const K key = stage[i];
        const uint32_t c = coarse_field_rev(top32_of(key, s.k), canonical, ONE ? s.bb : s.b1);  // as above, from the key
        if constexpr (ONE) store_key(fine ? b.sbuf : b.kbuf, (uint32_t)(hist[PAD(map[c])] + i), key);
        else store_key(b.kbuf, cursor[c] + i, key);
      }
    } else if (t == 0) {
      atomicOr(&b.meta->status, ST_INTERNAL);
    }
    __syncthreads();
    for (int c = t; c < P1; c += NT) {
      if constexpr (!ONE) cursor[c] += soff[PAD(c)] + hist[PAD(c)];
      hist[PAD(c)] = 0;
    }
  }
}
template <int KW, int NT, int MODE, int VAR>
__global__ void __launch_bounds__(NT, 3) k_scatter(Shape s, Buffers b) {
  pdl_wait();
  scatter_body<KW, NT, MODE, VAR>(s, b, blockIdx.x);
}
// Aggregation ablation: pass B writes every key on its own through the partition cursors.
template <int KW>
__global__ void __launch_bounds__(256, 2) k_scatter_direct(Shape s, Buffers b) {
  pdl_wait();
  scatter_body<KW, 256, SC_DIRECT, V_SHORT>(s, b, blockIdx.x);
}

template <int KW, int NT, int MODE, int VAR>
__global__ void __launch_bounds__(NT, 3) k_scatter_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  scatter_body<KW, NT, MODE, VAR>(d.s, d.b, bid);
}

// ------------------------------------------------------------------ phase 2: fine split
// Fine partition of a key: the coarse field c of u selects {first fine partition of c,
// m_c}; the fine index is floor(v m_c / 2^(32 - b1)) for the low part v of u (below the
// coarse field), taken as the high word of (v << b1) * m_c.  The m_c fine partitions of c
// split its range of u into near-equal parts.
struct FineMap {
  int k, canonical, b1;
};

template <class K>
__device__ __forceinline__ uint32_t fine_of(K key, const FineMap& x, const uint2* fmap) {
  const uint32_t u = umap(top32_of(key, x.k), x.canonical);
  const uint2 e = fmap[coarse_field(u, x.b1)];
  return e.x + __umulhi(u << x.b1, e.y);
}

// fmap[c] = {fine_base[c], fine_m[c]} for c < P1, fmap[P1].x = fine partition count.
__device__ __forceinline__ void load_fine_map(const Buffers& b, int P1, uint2* fmap) {
  for (int c = threadIdx.x; c <= P1; c += blockDim.x) fmap[c] = make_uint2(b.fine_base[c], c < P1 ? b.fine_m[c] : 0u);
}
__host__ __device__ inline FineMap make_fine_map(const Shape& s) { return FineMap{s.k, s.canonical, s.b1}; }

constexpr int kFineThreads = 512;
constexpr int kFinePer = 8;  // keys per thread per chunk (loaded as 16-byte pairs / single u128, all before use)
constexpr int kFineChunk = kFineThreads * kFinePer;

// Load this thread's keys of the chunk [c0, c1): pairs of words (read-only path, all
// loads issued before any use).  Key m of the thread is chunk key  (m / P) * P * T +
// threadIdx.x * P + m % P, P = 16 / (8 KW) keys per load, T = threads.
template <int KW>
__device__ __forceinline__ void load_chunk(const uint64_t* __restrict__ src, uint64_t c0, uint64_t c1,
                                           typename KeyT<KW>::T (&keys)[kFinePer], uint32_t& have) {
  typedef typename KeyT<KW>::T K;
  constexpr int P = KW == 1 ? 2 : 1;  // keys per 16-byte load
  have = 0;
  ulonglong2 v[kFinePer / P];
#pragma unroll
  for (int m = 0; m < kFinePer / P; ++m) {
    const uint64_t i = c0 + (uint64_t)m * P * kFineThreads + (uint64_t)threadIdx.x * P;
    v[m] = make_ulonglong2(0, 0);
    if (i + P <= c1) v[m] = __ldg(reinterpret_cast<const ulonglong2*>(src + i * KW));
    else if (i < c1) v[m].x = __ldg(src + i * KW);  // P == 2 and one key left
  }
#pragma unroll
  for (int m = 0; m < kFinePer / P; ++m) {
    const uint64_t i = c0 + (uint64_t)m * P * kFineThreads + (uint64_t)threadIdx.x * P;
    if constexpr (KW == 1) {
      keys[2 * m] = (K)v[m].x;
      keys[2 * m + 1] = (K)v[m].y;
      if (i < c1) have |= 1u << (2 * m);
      if (i + 1 < c1) have |= 1u << (2 * m + 1);
    } else {
      keys[m] = (K)(((u128)v[m].y << 64) | v[m].x);
      if (i < c1) have |= 1u << m;
    }
  }
}

// Chunks of the coarse-grouped keys are handed out round-robin.  A chunk's first and last
// keys bound the fine partitions it touches; they are fetched for the block's next chunk
// (cp.async into bnd_s[1 - cur]) while the current one is processed.
template <int KW>
__device__ __forceinline__ void fetch_bounds(const uint64_t* kbuf, uint64_t c0, uint64_t K_total,
                                             typename KeyT<KW>::T* bnd) {
  const uint64_t c1 = min(K_total, c0 + kFineChunk);
  if constexpr (KW == 1) {
    cp_async8(&bnd[0], kbuf + c0);
    cp_async8(&bnd[1], kbuf + c1 - 1);
  } else {
    cp_async16(&bnd[0], kbuf + 2 * c0);
    cp_async16(&bnd[1], kbuf + 2 * (c1 - 1));
  }
}

template <int KW>
__device__ __forceinline__ void fine_hist_body(const Shape& s, const Buffers& b, uint32_t bid, uint32_t nblk,
                                               bool redo = false) {
  typedef typename KeyT<KW>::T K;
  extern __shared__ __align__(16) uint8_t sm[];
  if (redo && !b.meta->fine_spill) return;  // the exact fine split runs again only after a spill
  if (s.one_level && b.meta->one) return;
  // a sampled layout counts one chunk in 2^kFineSampleLog2 (the exact split: every chunk)
  const uint64_t cstep = (s.fine_sampled && !redo) ? ((uint64_t)kFineChunk << kFineSampleLog2) : (uint64_t)kFineChunk;
  const int P1 = 1 << s.b1;
  uint2* fmap = reinterpret_cast<uint2*>(sm);                    // [P1 + 1]
  uint32_t* lh = reinterpret_cast<uint32_t*>(fmap + P1 + 1);     // [kFineLocalCap]
  __shared__ __align__(16) K bnd_s[2][2];
  load_fine_map(b, P1, fmap);
  for (int i = threadIdx.x; i < kFineLocalCap; i += kFineThreads) lh[i] = 0;
  const FineMap x = make_fine_map(s);
  const uint64_t K_total = min(b.meta->n_windows, s.cap);
  const uint64_t stride = (uint64_t)nblk * cstep;
  if (threadIdx.x == 0 && bid * cstep < K_total) {
    fetch_bounds<KW>(b.kbuf, bid * cstep, K_total, bnd_s[0]);
    cp_async_wait_all();
  }
  __syncthreads();
  int cur = 0;
  for (uint64_t c0 = bid * cstep; c0 < K_total; c0 += stride, cur ^= 1) {
    const uint64_t c1 = min(K_total, c0 + kFineChunk);
    const uint32_t g_lo = fmap[coarse_of(bnd_s[cur][0], s.k, s.canonical, s.b1)].x;
    const uint32_t span = fmap[coarse_of(bnd_s[cur][1], s.k, s.canonical, s.b1) + 1].x - g_lo;
    if (threadIdx.x == 0 && c0 + stride < K_total) fetch_bounds<KW>(b.kbuf, c0 + stride, K_total, bnd_s[cur ^ 1]);
    const bool local = span <= (uint32_t)kFineLocalCap;
    K keys[kFinePer];
    uint32_t have;
    load_chunk<KW>(b.kbuf, c0, c1, keys, have);
#pragma unroll
    for (int m = 0; m < kFinePer; ++m) {
      if ((have >> m) & 1u) {
        const uint32_t g = fine_of(keys[m], x, fmap);
        if (local && g - g_lo < span) atomicAdd(&lh[g - g_lo], 1u);
        else if (g < s.nf_max) atomicAdd(&b.fhist[g], 1u);
        else atomicOr(&b.meta->status, ST_INTERNAL);
      }
    }
    __syncthreads();
    if (local) {
      for (uint32_t i = threadIdx.x; i < span; i += kFineThreads) {
        const uint32_t v = lh[i];
        if (v) {
          if (g_lo + i < s.nf_max) atomicAdd(&b.fhist[g_lo + i], v);
          else atomicOr(&b.meta->status, ST_INTERNAL);
          lh[i] = 0;
        }
      }
    }
    if (threadIdx.x == 0) cp_async_wait_all();
    __syncthreads();
  }
}
template <int KW>
__global__ void __launch_bounds__(kFineThreads, 2) k_fine_hist(Shape s, Buffers b, int redo) {
  pdl_wait();
  fine_hist_body<KW>(s, b, blockIdx.x, gridDim.x, redo != 0);
}
template <int KW>
__global__ void __launch_bounds__(kFineThreads, 2) k_fine_hist_batch(BatchTab t, int redo) {
  KC_BATCH_PROLOGUE(t);
  fine_hist_body<KW>(d.s, d.b, bid, nblk, redo != 0);
}

// Keys at positions below x of the keys array that a sampled fine histogram counts: one
// kFineChunk-key chunk in 2^kFineSampleLog2.
__device__ __forceinline__ uint64_t sampled_below(uint64_t x) {
  const uint64_t per = (uint64_t)kFineChunk << kFineSampleLog2;
  const uint64_t r = x % per;
  return (x / per) * kFineChunk + (r < (uint64_t)kFineChunk ? r : (uint64_t)kFineChunk);
}

// Region of fine partition g of coarse partition c in a sampled layout: its estimated size (its
// sampled count scaled by c's n_c keys over its s_c sampled keys) plus 5.5 standard deviations
// of that estimate and 16 keys; never more than its coarse partition.  Too small a sample
// gives the whole coarse partition.
__device__ __forceinline__ uint64_t fine_region(const Shape& sh, const Buffers& b, uint64_t g, uint64_t n_c,
                                                uint64_t s_c, uint32_t m_c) {
  if (s_c < 1024) return n_c;
  const float f = (float)n_c / (float)s_c, cnt = (float)b.fhist[g];
  float slack = sh.tight_slack ? 0.f : 5.5f * f * sqrtf(cnt + 1.f) + 16.f;
  // a partition far above its coarse partition's average holds k-mers of tandem repeats, which
  // come many at a time (a read inside an array holds each of them 20 times and more), so its
  // sampled count varies more than a random sample's: an eighth on top.  (Without it, 72 M
  // windows with 3% satellite arrays took the exact split again in most counts, 225 to 350 us.)
  if (!sh.tight_slack && cnt * (float)m_c > 4.f * (float)s_c) slack += 0.125f * f * cnt;
  const uint64_t r = (uint64_t)(cnt * f + slack) + (sh.tight_slack ? 0 : 1);
  return r < n_c ? r : n_c;
}
// Room of a coarse partition in a sampled layout: its keys, a quarter and 64 per fine
// partition; as much as its regions take where the sample is too small.
__device__ __forceinline__ uint64_t coarse_room(uint64_t n_c, uint64_t s_c, uint32_t m_c) {
  return s_c < 1024 ? n_c * m_c : n_c + n_c / 4 + 64ull * m_c;
}

// Starts of the fine partitions of coarse partition c: an exclusive scan of their sizes (exact
// histogram) from c's own start, or of their regions (sampled layout) from the end of the room
// of the coarse partitions before.  One block of 256 threads per coarse partition (one block
// for all took 203 us for 100 K fine partitions and 430 us for 221 K, this takes 10 and 12).
// Regions that pass their coarse partition's room, or rooms that pass the keys arrays, are
// given up at once (the exact split follows).
__device__ __forceinline__ void fine_scan_body(const Shape& sh, const Buffers& b, uint32_t c, bool redo = false) {
  __shared__ uint64_t wt[32];
  if (redo && !b.meta->fine_spill) return;
  if (bad_offsets(b) || (sh.one_level && b.meta->one)) return;
  const bool sampled = sh.fine_sampled && !redo;
  const int P1 = 1 << sh.b1, t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = blockDim.x >> 5;
  const uint64_t NF = min(b.meta->n_fine, sh.nf_max);
  const uint64_t g0 = b.fine_base[c];
  const uint32_t m = b.fine_m[c];
  if (g0 + m > NF) return;  // (a plan that failed)
  auto block_sum = [&](uint64_t x, uint64_t& before) -> uint64_t {  // the total; `before`: of the threads before
    uint64_t y = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint64_t z = __shfl_up_sync(0xffffffffu, y, d);
      if (lane >= d) y += z;
    }
    __syncthreads();
    if (lane == 31) wt[wid] = y;
    __syncthreads();
    uint64_t total = 0, prev = 0;
    for (int w = 0; w < nw; ++w) {
      if (w < wid) prev += wt[w];
      total += wt[w];
    }
    before = prev + y - x;
    return total;
  };
  const uint64_t a = b.cstart[c], e = b.cstart[c + 1], n_c = e - a, s_c = sampled_below(e) - sampled_below(a);
  uint64_t base = a, room = n_c, skip;
  if (sampled) {
    uint64_t x = 0;
    for (uint32_t i = t; i < c; i += blockDim.x) {
      const uint64_t p = b.cstart[i], q = b.cstart[i + 1];
      x += coarse_room(q - p, sampled_below(q) - sampled_below(p), b.fine_m[i]);
    }
    base = block_sum(x, skip);
    room = coarse_room(n_c, s_c, m);
  }
  const uint32_t per = (m + blockDim.x - 1) / blockDim.x, lo = min(m, t * per), hi = min(m, lo + per);
  uint64_t sum = 0, run;
  for (uint32_t i = lo; i < hi; ++i)
    sum += sampled ? fine_region(sh, b, g0 + i, n_c, s_c, m) : (uint64_t)b.fhist[g0 + i];
  const uint64_t total = block_sum(sum, run);
  run += base;
  for (uint32_t i = lo; i < hi; ++i) {
    b.foff[g0 + i] = run;
    b.fcur[g0 + i] = run;
    run += sampled ? fine_region(sh, b, g0 + i, n_c, s_c, m) : (uint64_t)b.fhist[g0 + i];
  }
  if (t == 0) {
    if ((int)c == P1 - 1) b.foff[NF] = base + room;
    if (sampled && (total > room || base + room > sh.cap_kb)) b.meta->fine_unfit = b.meta->fine_spill = 1;
  }
}
__global__ void __launch_bounds__(256) k_fine_scan(Shape sh, Buffers b, int redo) {
  pdl_wait();
  fine_scan_body(sh, b, blockIdx.x, redo != 0);
}

// Before the exact fine split runs again (a sampled region overflowed): a fresh histogram.
__global__ void k_fine_redo_clear(Shape sh, Buffers b) {
  pdl_wait();
  if (!b.meta->fine_spill) return;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < sh.nf_max; i += (uint64_t)gridDim.x * blockDim.x)
    b.fhist[i] = 0;
}
__global__ void __launch_bounds__(256) k_fine_scan_batch(BatchTab t, int redo) {
  KC_BATCH_PROLOGUE(t);
  fine_scan_body(d.s, d.b, bid, redo != 0);
}
// (the fine scan's table: one block per coarse partition)
__global__ void k_fine_redo_clear_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  if (!d.b.meta->fine_spill) return;
  for (uint64_t i = bid * (uint64_t)blockDim.x + threadIdx.x; i < d.s.nf_max; i += (uint64_t)nblk * blockDim.x) d.b.fhist[i] = 0;
}

// Exclusive scan of in[0, n) into out[0, n) (all threads of the block, n <= 4 * blockDim);
// returns the total.
__device__ uint32_t block_scan_to(const uint32_t* in, uint32_t* out, int n, uint32_t* warp_tmp) {
  const int nt = blockDim.x, t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = (nt + 31) >> 5;
  const int per = (n + nt - 1) / nt;
  const int lo = min(n, t * per), hi = min(n, lo + per);
  uint32_t s = 0;
  for (int i = lo; i < hi; ++i) s += in[i];
  uint32_t x = s;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_tmp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    uint32_t w = lane < nw ? warp_tmp[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    if (lane < nw) warp_tmp[lane] = w;
  }
  __syncthreads();
  uint32_t run = x - s + (wid ? warp_tmp[wid - 1] : 0);
  const uint32_t total = warp_tmp[nw - 1];
  for (int i = lo; i < hi; ++i) {
    out[i] = run;
    run += in[i];
  }
  __syncthreads();
  return total;
}

// Split each chunk by fine partition: rank the keys in a shared histogram, bump each fine
// partition's global cursor once per chunk, stage the keys grouped by fine partition and
// write every group as one contiguous run.
template <int KW>
__device__ __forceinline__ void fine_scatter_body(const Shape& s, const Buffers& b, uint32_t bid, uint32_t nblk,
                                                  bool redo = false) {
  typedef typename KeyT<KW>::T K;
  extern __shared__ __align__(16) uint8_t sm[];
  // the exact split runs again only after a spill; a sampled layout given up by the scan is
  // not written at all.  In a sampled layout a run that would pass its region's end is not
  // written: the spill is recorded and the exact split follows.  (The first split is left by
  // fine_unfit, which only the scan sets: other blocks of this launch may be setting fine_spill
  // meanwhile, and warps of one block that read it on either side of that would part here.)
  if (redo ? !b.meta->fine_spill : (s.fine_sampled && b.meta->fine_unfit)) return;
  if (s.one_level && b.meta->one) return;
  const bool sampled = s.fine_sampled && !redo;
  constexpr uint64_t kSpilledRun = 1ull << 63;  // never a run's offset
  const int P1 = 1 << s.b1;
  K* stage = reinterpret_cast<K*>(sm);                                          // [kFineChunk]
  uint16_t* stage_g = reinterpret_cast<uint16_t*>(stage + kFineChunk);          // [kFineChunk]
  uint64_t* delta = reinterpret_cast<uint64_t*>(stage_g + kFineChunk);          // [kFineLocalCap]
  uint32_t* lh = reinterpret_cast<uint32_t*>(delta + kFineLocalCap);            // [kFineLocalCap]
  uint32_t* soff = lh + kFineLocalCap;                                          // [kFineLocalCap]
  uint2* fmap = reinterpret_cast<uint2*>(soff + kFineLocalCap);                 // [P1 + 1]
  __shared__ __align__(16) K bnd_s[2][2];
  __shared__ uint32_t wt[32];
  load_fine_map(b, P1, fmap);
  for (int i = threadIdx.x; i < kFineLocalCap; i += kFineThreads) lh[i] = 0;
  const FineMap x = make_fine_map(s);
  const uint64_t K_total = min(b.meta->n_windows, s.cap);
  const uint64_t stride = (uint64_t)nblk * kFineChunk;
  if (threadIdx.x == 0 && bid * (uint64_t)kFineChunk < K_total) {
    fetch_bounds<KW>(b.kbuf, bid * (uint64_t)kFineChunk, K_total, bnd_s[0]);
    cp_async_wait_all();
  }
  __syncthreads();
  int cur = 0;
  for (uint64_t c0 = bid * (uint64_t)kFineChunk; c0 < K_total; c0 += stride, cur ^= 1) {
    const uint64_t c1 = min(K_total, c0 + kFineChunk);
    const uint32_t g_lo = fmap[coarse_of(bnd_s[cur][0], s.k, s.canonical, s.b1)].x;
    const uint32_t span = fmap[coarse_of(bnd_s[cur][1], s.k, s.canonical, s.b1) + 1].x - g_lo;
    if (threadIdx.x == 0 && c0 + stride < K_total) fetch_bounds<KW>(b.kbuf, c0 + stride, K_total, bnd_s[cur ^ 1]);
    if (span == 0 || span > (uint32_t)kFineLocalCap) {
      // a chunk over very many tiny fine partitions: one global cursor bump per key
      for (int m = 0; m < kFinePer; ++m) {
        const uint64_t i = c0 + threadIdx.x + (uint64_t)m * kFineThreads;
        if (i < c1) {
          K key;
          load_key(b.kbuf, i, key);
          const uint32_t g = fine_of(key, x, fmap);
          const uint64_t pos = g < s.nf_max ? atomicAdd(&b.fcur[g], 1ull) : ~0ull;
          if (sampled && g < s.nf_max && pos >= b.foff[g + 1]) b.meta->fine_spill = 1;
          else if (pos < s.cap_kb) store_key(b.sbuf, pos, key);
          else atomicOr(&b.meta->status, ST_INTERNAL);
        }
      }
    } else {
      K keys[kFinePer];
      uint32_t gr[kFinePer];
      uint32_t have;
      load_chunk<KW>(b.kbuf, c0, c1, keys, have);
#pragma unroll
      for (int m = 0; m < kFinePer; ++m) {
        gr[m] = 0xffffffffu;
        if ((have >> m) & 1u) {
          const uint32_t lg = fine_of(keys[m], x, fmap) - g_lo;
          if (lg < span) gr[m] = (lg << 16) | atomicAdd(&lh[lg], 1u);  // span <= 2^10, rank < 2^16
          else atomicOr(&b.meta->status, ST_INTERNAL);
        }
      }
      __syncthreads();
      const uint32_t n_staged = block_scan_to(lh, soff, (int)span, wt);
      // one cursor bump per fine partition; delta[lg] + staged position = global position
      for (uint32_t i = threadIdx.x; i < span; i += kFineThreads) {
        const uint32_t v = lh[i];
        if (v) {
          uint64_t gb = s.cap_kb;  // positions at or past cap_kb are rejected below
          if (g_lo + i < s.nf_max) {
            const uint64_t lim = sampled ? b.foff[g_lo + i + 1] : ~0ull;  // loaded before the bump
            gb = atomicAdd(&b.fcur[g_lo + i], (unsigned long long)v);
            if (gb + v > lim) {  // the run passes its region's end
              b.meta->fine_spill = 1;
              gb = kSpilledRun;
            }
          } else {
            atomicOr(&b.meta->status, ST_INTERNAL);
          }
          delta[i] = gb == kSpilledRun ? kSpilledRun : gb - soff[i];
          lh[i] = 0;
        }
      }
#pragma unroll
      for (int m = 0; m < kFinePer; ++m) {
        if (gr[m] != 0xffffffffu) {
          const uint32_t lg = gr[m] >> 16;
          const uint32_t pos = soff[lg] + (gr[m] & 0xffffu);
          stage[pos] = keys[m];
          stage_g[pos] = (uint16_t)lg;
        }
      }
      __syncthreads();
      for (uint32_t i = threadIdx.x; i < n_staged; i += kFineThreads) {
        const uint64_t dl = delta[stage_g[i]];
        if (dl == kSpilledRun) continue;
        const uint64_t pos = dl + i;
        if (pos < s.cap_kb) store_key(b.sbuf, pos, stage[i]);
        else atomicOr(&b.meta->status, ST_INTERNAL);
      }
    }
    if (threadIdx.x == 0) cp_async_wait_all();
    __syncthreads();
  }
}
template <int KW>
__global__ void __launch_bounds__(kFineThreads, 2) k_fine_scatter(Shape s, Buffers b, int redo) {
  pdl_wait();
  fine_scatter_body<KW>(s, b, blockIdx.x, gridDim.x, redo != 0);
}
template <int KW>
__global__ void __launch_bounds__(kFineThreads, 2) k_fine_scatter_batch(BatchTab t, int redo) {
  KC_BATCH_PROLOGUE(t);
  fine_scatter_body<KW>(d.s, d.b, bid, nblk, redo != 0);
}

// ------------------------------------------------------------------ phase 2: count + emit
constexpr uint64_t kLookValue = (1ull << 62) - 1;
constexpr uint64_t kLookAgg = 1ull << 62;
constexpr uint64_t kLookIncl = 2ull << 62;

// Decoupled look-back (executed by one warp): sum of distinct counts of fine partitions < g.
// Each step reads the kLookPer * 32 status words before position j at once (lane l holds
// distance q * 32 + l); the nearest inclusive prefix among them ends the walk, and only
// unpublished words nearer than it are waited for (with a bounded spin).  With `abort`,
// the wait also ends as soon as *abort becomes nonzero, and kNoPrefix is returned.
constexpr int kLookPer = 8;
constexpr uint64_t kNoPrefix = ~0ull;
__device__ uint64_t lookback(unsigned long long* look, uint64_t g, uint32_t* status, uint32_t spin_limit,
                             const volatile uint32_t* abort = nullptr) {
  const int lane = threadIdx.x & 31;
  constexpr uint32_t kNone = kLookPer * 32;
  uint64_t excl = 0;
  int64_t j = (int64_t)g - 1;
  while (j >= 0) {
    uint64_t v[kLookPer];
#pragma unroll
    for (int q = 0; q < kLookPer; ++q) {
      const int64_t idx = j - (q * 32 + lane);
      v[q] = idx >= 0 ? ld_status(&look[idx]) : kLookIncl;  // before the first partition: inclusive 0
    }
    uint32_t stop = kNone, spins = 0;
    while (true) {
      stop = kNone;  // nearest inclusive distance
#pragma unroll
      for (int q = kLookPer - 1; q >= 0; --q) {
        const unsigned b = __ballot_sync(0xffffffffu, (v[q] >> 62) == 2);
        if (b) stop = q * 32 + __ffs(b) - 1;
      }
      bool wait = false;
#pragma unroll
      for (int q = 0; q < kLookPer; ++q) wait |= (uint32_t)(q * 32 + lane) < stop && (v[q] >> 62) == 0;
      if (!__any_sync(0xffffffffu, wait)) break;
      if (abort && *abort) return kNoPrefix;
      if (++spins > spin_limit) {
        if (lane == 0) atomicOr(status, ST_TIMEOUT);
        return excl;
      }
      __nanosleep(64);
#pragma unroll
      for (int q = 0; q < kLookPer; ++q) {
        const int64_t idx = j - (q * 32 + lane);
        if ((uint32_t)(q * 32 + lane) < stop && (v[q] >> 62) == 0) v[q] = ld_status(&look[idx]);
      }
    }
    uint64_t val = 0;
#pragma unroll
    for (int q = 0; q < kLookPer; ++q)
      if ((uint32_t)(q * 32 + lane) <= stop) val += v[q] & kLookValue;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) val += __shfl_xor_sync(0xffffffffu, val, d);
    excl += val;
    if (stop != kNone) break;
    j -= kNone;
  }
  return excl;
}

template <int KW>
struct Table {
  typedef typename KeyT<KW>::T K;
  K* keys;
  uint32_t* counts;
};

// Count kernel shared memory: a hash table of 2^bT_max slots (key + count), a bucket
// histogram of 16-bit entries (at most one bucket per slot, and the end of the last), and for
// up to 3/4 of the slots, grouped by bucket, the slot numbers and (64-bit keys) the keys.
constexpr int kTableLog2Cap = kCountThreads == 1024 ? 13 : 12;  // 8 slots per thread

size_t count_kernel_smem(int kw, int bT_max) {
  const size_t slots = (size_t)1 << bT_max;
  return slots * (size_t)(kw * 8 + 4) + slots * 2 + 16 + ((3 * slots) >> 2) * (kw == 1 ? 10 : 2) + 256;
}

// The largest table whose block (12 KB of static shared memory included) fits the opt-in
// limit, with kCountBlocksPerSM blocks on one SM (each also keeps 1 KB for the system).
int table_log2_max(int kw, size_t smem_optin, size_t smem_per_sm) {
  size_t budget = smem_optin;
  if (kCountBlocksPerSM > 1 && smem_per_sm) {
    const size_t per = smem_per_sm / kCountBlocksPerSM - 1024;
    budget = per < budget ? per : budget;
  }
  int best = 6;
  for (int bt = 6; bt <= kTableLog2Cap; ++bt)
    if (count_kernel_smem(kw, bt) + 12288 <= budget) best = bt;
  return best;
}

constexpr int kProbeLimit = 64;  // at the 3/4 load that a table is ordered with, 1 key in 10^8 probes longer
constexpr int kWorkers = kCountThreads - 32;  // warps 1.. load and sort while warp 0 looks back
constexpr int kSlotsPerWorker = ((1 << kTableLog2Cap) + kWorkers - 1) / kWorkers;


// Block barrier with the warp reconverged first: the count kernel reaches its barriers
// straight after branches taken by one thread or lane (ticket fetch, look-back bookkeeping).
__device__ __forceinline__ void block_sync() {
  __syncwarp();
  __syncthreads();
}

// Named barrier of the worker warps (1..31).  Its non-aligned form is used: a worker warp
// may arrive diverged (right after a branch taken by one of its threads, e.g. thread 32
// computing the key range), which the aligned form (bar.sync) does not allow.
__device__ __forceinline__ void bar_workers() {
  __syncwarp();
  asm volatile("barrier.sync 1, %0;" ::"r"(kWorkers) : "memory");
}

// The home slot is the top bits of a multiplicative hash (it spreads keys that share
// prefixes), the probe step an odd number from the bits below (every table is a power of two,
// so every slot is reached).  A warp probes until its unluckiest lane is done, so the tail of
// the probe lengths is what costs: with linear probing, whose runs of occupied slots grow
// long, the kernel took 21.7 ms on 2.4 G windows of 402 M distinct keys and 37.3 ms on 1.0 G
// nearly distinct 128-bit keys; stepping takes 20.8 and 34.4 ms.
//
// Add `inc` to the count of `key` (claiming a slot if new).  Returns 2 if the key claimed a
// new slot, 1 if it was already there, 0 if no slot was found within the probe limit.
template <int KW>
__device__ __forceinline__ int count_insert(Table<KW> tb, typename KeyT<KW>::T key, uint32_t inc, int bT, bool check,
                                            uint32_t limit, uint32_t* status) {
  typedef typename KeyT<KW>::T K;
  const K EMPTY = all_ones<K>();
  const uint32_t mask = (1u << bT) - 1;
  const uint32_t hh = (uint32_t)(key_hash(key) >> 32);
  uint32_t s = hh >> (32 - bT);
  const uint32_t step = (hh >> 5) | 1u;
  for (int probe = 0; probe < kProbeLimit; ++probe, s = (s + step) & mask) {
    int res = 0;
    if constexpr (KW == 1) {
      // read the slot; claim it only if empty (the claim's answer then replaces the read):
      // one exit test per probe instead of a branch per case
      uint64_t* p = reinterpret_cast<uint64_t*>(tb.keys) + s;
      unsigned long long old = *reinterpret_cast<volatile uint64_t*>(p);
      const bool emp = old == ~0ull;
      if (emp) old = atomicCAS(reinterpret_cast<unsigned long long*>(p), ~0ull, (unsigned long long)key);
      res = (emp && old == ~0ull) ? 2 : (old == (unsigned long long)key ? 1 : 0);
    } else {
      const K old = cas128_shared(reinterpret_cast<u128*>(tb.keys) + s, (u128)EMPTY, (u128)key);
      res = old == EMPTY ? 2 : (old == key ? 1 : 0);
    }
    if (res) {
      if (check) {
        const uint32_t o = atomicAdd(&tb.counts[s], inc);
        if (o > limit - inc) atomicOr(status, ST_COUNT_OVERFLOW);
      } else {
        atomicAdd(&tb.counts[s], inc);  // result unused: a reduction
      }
      return res;
    }
  }
  return 0;
}

// An empty table and an empty bucket histogram (at most one bucket per slot).
template <int KW>
__device__ __forceinline__ void table_clear(Table<KW> tb, uint32_t nslots, uint32_t* hist, uint32_t* big_n) {
  typedef typename KeyT<KW>::T K;
  for (uint32_t i = threadIdx.x; i < nslots; i += blockDim.x) {
    tb.keys[i] = all_ones<K>();
    tb.counts[i] = 0;
  }
  for (uint32_t i = threadIdx.x; i < nslots / 2; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x == 0) *big_n = 0;
}

// Clear the table and count the keys in[0, n) (only those in [lo, hi] when `ranged`).  The
// all-ones key is counted apart in *special (it marks empty slots); it exists only when the
// k-mer fills the key word (full_width).  Sets *ovf if a key found no slot.  Each thread's
// first keys are loaded before the table is cleared, and its next keys before the current ones
// are inserted, so that a load's latency is covered by the clearing or by the inserts.
// With MERGE, a warp whose active keys are all equal adds them with one atomic (the
// heavy-hitter merge of the paper's L3 layer); without it (the default) every key is added
// on its own: on GB300 the shared-memory atomics absorb equal keys faster than the merge's
// warp vote costs, even for a single key.
template <int KW, bool MERGE = false>
__device__ void count_all(Table<KW> tb, const uint64_t* in, uint64_t n, bool ranged, typename KeyT<KW>::T lo,
                          typename KeyT<KW>::T hi, int bT, bool full_width, uint32_t limit, uint32_t* hist,
                          uint32_t* big_n, uint32_t* n_new, uint32_t* ovf, uint32_t* special, uint32_t* status) {
  typedef typename KeyT<KW>::T K;
  constexpr int kIn = KW == 1 ? 4 : 2;  // keys per thread and batch (two batches held: register-bound at 64)
  const K EMPTY = all_ones<K>();
  const int lane = threadIdx.x & 31;
  const bool check = n > limit;  // a count can pass the limit only in a partition that large
  uint32_t claimed = 0;
  K nxt[kIn];
  auto load = [&](uint64_t base) {
#pragma unroll
    for (int m = 0; m < kIn; ++m) {
      const uint64_t i = base + (uint64_t)m * blockDim.x + threadIdx.x;
      nxt[m] = 0;
      if (i < n) load_key(in, i, nxt[m]);
    }
  };
  load(0);
  table_clear<KW>(tb, 1u << bT, hist, big_n);
  block_sync();
  for (uint64_t base = 0; base < n; base += kIn * (uint64_t)blockDim.x) {
    K kk[kIn];
#pragma unroll
    for (int m = 0; m < kIn; ++m) kk[m] = nxt[m];
    load(base + kIn * (uint64_t)blockDim.x);
    if (ranged) {  // a key without a slot: this part is counted again in smaller ones, so stop here
      bool stop = *reinterpret_cast<volatile uint32_t*>(ovf) != 0;
      if constexpr (MERGE) stop = __any_sync(0xffffffffu, stop);  // the merge below takes whole warps
      if (stop) break;
    }
#pragma unroll
    for (int m = 0; m < kIn; ++m) {
      const K key = kk[m];
      bool act = base + (uint64_t)m * blockDim.x + threadIdx.x < n;
      if (ranged) act = act && key >= lo && key <= hi && key != EMPTY;
      if constexpr (MERGE) {
        // a warp whose active keys all equal lane 0's key (a heavy hitter) adds them at once;
        // lane 0's own key counts only if it is active, so any inactive lane 0 is harmless
        const K k0 = shfl_key(key, 0);
        if (__all_sync(0xffffffffu, !act || key == k0)) {
          const unsigned am = __ballot_sync(0xffffffffu, act);
          if (am && lane == __ffs(am) - 1) {
            const uint32_t inc = __popc(am);
            if (full_width && k0 == EMPTY) {
              if (atomicAdd(special, inc) > limit - inc) atomicOr(status, ST_COUNT_OVERFLOW);
            } else {
              const int r = count_insert<KW>(tb, k0, inc, bT, check, limit, status);
              if (!r) atomicOr(ovf, 1u);
              claimed += r == 2;
            }
          }
          continue;
        }
      }
      if (act) {
        if (full_width && key == EMPTY) {
          if (atomicAdd(special, 1u) >= limit) atomicOr(status, ST_COUNT_OVERFLOW);
        } else {
          const int r = count_insert<KW>(tb, key, 1u, bT, check, limit, status);
          if (!r) atomicOr(ovf, 1u);
          claimed += r == 2;
        }
      }
    }
  }
  // the slots claimed, added once per warp (a shared counter bumped per new key would be
  // one address hit by every lane of a warp whose keys are all new)
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) claimed += __shfl_xor_sync(0xffffffffu, claimed, d);
  if (lane == 0 && claimed) atomicAdd(n_new, claimed);
}

template <class K> __device__ __forceinline__ int bitlen(K v);
template <> __device__ __forceinline__ int bitlen(uint64_t v) { return 64 - __clzll(v); }
template <> __device__ __forceinline__ int bitlen(u128 v) {
  const uint64_t hi = (uint64_t)(v >> 64);
  return hi ? 128 - __clzll(hi) : 64 - __clzll((uint64_t)v);
}

// The median of up to kSplitSample keys taken from a table's slots (all threads; at least two
// sampled keys lie in [lo, hi], else false): *out is in (lo, hi].  samp: kSplitSample entries.
constexpr int kSplitSample = 256;
// Ranges that wait while their lower neighbours are counted.  A table that overflows holds the
// keys that came first: where they come in falling order a median leaves half a table above it
// and everything else below, so that by medians alone a range would wait for every half table
// of the partition.  The blocks of pass B mix the order (1.5 M sorted reads of one prefix kept
// within 160 ranges), which is no bound.  From kMedianDepth ranges on, the range is halved
// instead, at most 128 times before it is a single key: never more than kMedianDepth + 1 + 128
// wait.  (Count kernel of 2.4 G windows 16.92 ms before, 16.96 with it; of 1.0 G 128-bit
// windows 32.5 and 32.1.)
constexpr int kMedianDepth = 24, kSplitStack = 160;
template <class K>
__device__ bool median_key(const K* keys, uint32_t nslots, K lo, K hi, K* samp, K* out) {
  const K EMPTY = all_ones<K>();
  const uint32_t step = nslots > kSplitSample ? nslots / kSplitSample : 1;
  const uint32_t n = min(nslots, (uint32_t)kSplitSample);
  block_sync();
  K mine = EMPTY;
  if (threadIdx.x < n) {
    mine = keys[threadIdx.x * step];
    if (mine < lo || mine > hi) mine = EMPTY;
    samp[threadIdx.x] = mine;
  }
  const uint32_t have = __syncthreads_count(mine != EMPTY);
  if (mine != EMPTY) {
    uint32_t below = 0;
    for (uint32_t i = 0; i < n; ++i) below += samp[i] < mine;
    if (below == have / 2) *out = mine;
  }
  block_sync();
  return have >= 2;
}

// Sort idx[a, a+c) by the keys the slots hold, by one warp: a bitonic network whose
// comparators all put the smaller key first, so positions past c act as +infinity.
template <class K>
__device__ void warp_sort_idx(const K* keys, uint16_t* idx, uint32_t a, uint32_t c) {
  const int lane = threadIdx.x & 31;
  uint32_t M = 1;
  while (M < c) M <<= 1;
  for (uint32_t size = 2; size <= M; size <<= 1) {
    for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
      for (uint32_t i = lane; i < M; i += 32) {
        const uint32_t j = (stride == (size >> 1)) ? (i ^ (size - 1)) : (i ^ stride);
        if (j > i && j < c) {
          const uint16_t x = idx[a + i], y = idx[a + j];
          if (keys[y] < keys[x]) {
            idx[a + i] = y;
            idx[a + j] = x;
          }
        }
      }
      __syncwarp();
    }
  }
}

// positions per worker thread: 7 * 992 >= 3/4 of 8192 slots, 7 * 480 >= 3/4 of 4096
constexpr int kRankPer = ((3 << kTableLog2Cap) / 4 + kWorkers - 1) / kWorkers;
static_assert(kRankPer == 7, "rank registers sized for 7 positions per worker");
constexpr int kRankRegs = (kRankPer + 1) / 2;  // ranks (< 2^13) are kept two per register
__device__ __forceinline__ uint32_t rank_get(const uint32_t (&rk)[kRankRegs], int m) {
  return (rk[m >> 1] >> (16 * (m & 1))) & 0xffffu;
}
// buckets above this are sorted by a warp, not ranked by counting
__host__ __device__ constexpr uint32_t big_bucket(int kw) { return kw == 1 ? 512 : 256; }
constexpr int kBigMax = 32;  // more than d / big_bucket <= 6144 / 257

// Exclusive scan of `words` words of two 16-bit counts each (worker warps; warp 0 is busy with
// the look-back meanwhile).  The total fits in 16 bits and goes behind the last word.
__device__ void workers_exclusive_scan16(uint32_t* data, int words, uint32_t* warp_tmp) {
  constexpr int nt = kWorkers, nw = kWorkers / 32;
  const int t = threadIdx.x - 32, lane = t & 31, wid = t >> 5;
  const int per = ((words + nt - 1) / nt) | 1;  // odd: the threads' words fall in distinct banks
  const int lo = min(words, t * per), hi = min(words, lo + per);
  uint32_t s = 0;
  for (int i = lo; i < hi; ++i) {
    const uint32_t v = data[i];
    s += (v & 0xffffu) + (v >> 16);
  }
  uint32_t x = s;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_tmp[wid] = x;
  bar_workers();
  // every warp adds up the warps before it (no second barrier for a scan by one warp)
  uint32_t before = lane < wid && lane < nw ? warp_tmp[lane] : 0;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
  uint32_t run = before + x - s;
  if (t == nt - 1) reinterpret_cast<uint16_t*>(data)[2 * words] = (uint16_t)(before + x);
  for (int i = lo; i < hi; ++i) {
    const uint32_t v = data[i], a = v & 0xffffu;
    data[i] = run | ((run + a) << 16);
    run += a + (v >> 16);
  }
  bar_workers();
}

// The buckets of a table's keys inside their range [lo, lo + width]: the top bB bits of
// (key - lo), aligned to the width of the range.
template <class K>
struct OrderMap {
  K lo, width;
  int rs, ls;  // w = low word of ((key - lo) >> rs), << ls
  int bs;      // bucket = w >> bs
};
template <class K>
__device__ __forceinline__ OrderMap<K> order_map(K lo, K hi, uint32_t NB) {
  OrderMap<K> o;
  o.lo = lo;
  o.width = hi - lo;
  const int nb = bitlen(o.width);
  o.rs = nb > 32 ? nb - 32 : 0;
  o.ls = nb >= 32 ? 0 : min(32 - nb, 31);  // nb = 0: the only offset is 0
  o.bs = 32 - (31 - __clz(NB));
  return o;
}
__device__ __forceinline__ uint32_t bucket_of(uint64_t off, const OrderMap<uint64_t>& o) {
  return (__funnelshift_rc((uint32_t)off, (uint32_t)(off >> 32), o.rs) << o.ls) >> o.bs;
}
__device__ __forceinline__ uint32_t bucket_of(u128 off, const OrderMap<u128>& o) {
  const uint32_t o0 = (uint32_t)off, o1 = (uint32_t)(off >> 32), o2 = (uint32_t)(off >> 64), o3 = (uint32_t)(off >> 96);
  const int q = o.rs >> 5;
  const uint32_t a = q == 0 ? o0 : (q == 1 ? o1 : (q == 2 ? o2 : o3));
  const uint32_t b = q == 0 ? o1 : (q == 1 ? o2 : (q == 2 ? o3 : 0u));
  return (__funnelshift_r(a, b, o.rs & 31) << o.ls) >> o.bs;
}

// Group the table's d occupied slots by bucket (worker warps only): an ordered counting sort
// of the slot numbers into idx[0, d) and, for 64-bit keys, of the keys into gkey[0, d), buckets
// ascending, slots unordered inside a bucket.  hist (cleared before) is left holding bucket
// b's first position in its b-th 16 bits, their number after the last; big_s[0, *big_n) lists
// the buckets above big_bucket entries.  Returns the number of entries placed: d, or the status
// says that the table does not hold what was counted (no more than these entries may be read).
template <int KW>
__device__ __forceinline__ uint32_t bucket_slots(Table<KW> tb, uint32_t nslots, uint32_t d, uint32_t NB,
                                             const OrderMap<typename KeyT<KW>::T>& o, uint32_t* hist, uint16_t* idx,
                                             uint64_t* gkey, uint32_t* wtmp, uint32_t* big_s, uint32_t* big_n,
                                             uint32_t* status, unsigned long long* prof = nullptr) {
  typedef typename KeyT<KW>::T K;
  const K EMPTY = all_ones<K>();
  long long tm = clock64();
  const int t = threadIdx.x - 32;
  auto mark = [&](int i) {
    if (prof && t == 0) {
      const long long now = clock64();
      atomicAdd(&prof[i], (unsigned long long)(now - tm));
      tm = now;
    }
  };
  uint32_t br[kSlotsPerWorker];
#pragma unroll
  for (int m = 0; m < kSlotsPerWorker; ++m) {
    const uint32_t s = t + m * kWorkers;
    br[m] = 0xffffffffu;
    if (s < nslots) {
      const K key = tb.keys[s];
      if (key != EMPTY) {
        const K off = key - o.lo;
        if (off > o.width) {  // cannot happen: the range holds every key of the table
          atomicOr(status, ST_INTERNAL);
        } else {
          const uint32_t bk = bucket_of(off, o);
          const uint32_t half = 16 * (bk & 1);
          const uint32_t r = (atomicAdd(&hist[bk >> 1], 1u << half) >> half) & 0xffffu;
          br[m] = (bk << 16) | r;  // bucket below 2^13, rank below 2^13
          if (r == big_bucket(KW)) {   // the entry that takes bucket bk past big_bucket
            const uint32_t q = atomicAdd(big_n, 1u);
            if (q < kBigMax) big_s[q] = bk;
            else atomicOr(status, ST_INTERNAL);
          }
        }
      }
    }
  }
  bar_workers();
  mark(5);
  workers_exclusive_scan16(hist, (int)(NB / 2), wtmp);
  mark(6);
  const uint16_t* start = reinterpret_cast<const uint16_t*>(hist);
  const uint32_t placed = start[NB];
  if (t == 0 && placed != d) atomicOr(status, ST_INTERNAL);
#pragma unroll
  for (int m = 0; m < kSlotsPerWorker; ++m)
    if (br[m] != 0xffffffffu) {
      const uint32_t pos = start[br[m] >> 16] + (br[m] & 0xffffu);
      idx[pos] = (uint16_t)(t + m * kWorkers);
      if constexpr (KW == 1) gkey[pos] = tb.keys[t + m * kWorkers];
    }
  bar_workers();
  mark(7);
  return placed;
}

// Worker warps: the rank of the entry at each bucket-grouped position j (its bucket's first
// position plus the number of smaller keys in the bucket).  64-bit keys are read in grouped
// order (consecutive words, no slot number first); 128-bit keys, for whose copies there is no
// room, through their slot numbers.  The rare bucket above big_bucket entries is first sorted
// in place by one warp and ranked by position (it pays above 512 keys: on the repeat genome,
// whose copies' variants share long prefixes, sorting from 256 up and reading every key through
// its slot number took 1147 M SM cycles of ranking and sorting, this takes 498 M).
template <int KW>
__device__ __forceinline__ void rank_slots(Table<KW> tb, uint16_t* idx, const uint64_t* gkey, uint32_t d,
                                           const uint32_t* hist, const OrderMap<typename KeyT<KW>::T>& o,
                                           const uint32_t* big_s, uint32_t n_big, uint32_t (&rank)[kRankRegs],
                                           unsigned long long* prof) {
  typedef typename KeyT<KW>::T K;
  const int t = threadIdx.x - 32, wid = t >> 5;
  const uint16_t* start = reinterpret_cast<const uint16_t*>(hist);
  long long tm = clock64();
  constexpr int kWarps = kWorkers / 32;
#pragma unroll
  for (int m = 0; m < kRankRegs; ++m) rank[m] = 0xffffffffu;
#pragma unroll
  for (int m = 0; m < kRankPer; ++m) {
    const uint32_t j = t + m * kWorkers;
    if (j < d) {
      K key;
      if constexpr (KW == 1) key = gkey[j];
      else key = tb.keys[idx[j]];
      const uint32_t bk = bucket_of((K)(key - o.lo), o);
      const uint32_t a = start[bk], e = start[bk + 1];
      uint32_t r = a;
      if (e - a > big_bucket(KW)) {
        r = j;
      } else {
        for (uint32_t q = a; q < e; ++q) {
          if constexpr (KW == 1) r += gkey[q] < key;
          else r += tb.keys[idx[q]] < key;
        }
      }
      const int sh = 16 * (m & 1);
      rank[m >> 1] = (rank[m >> 1] & ~(0xffffu << sh)) | (r << sh);
    }
  }
  if (prof && t == 0) {
    const long long now = clock64();
    atomicAdd(&prof[4], (unsigned long long)(now - tm));
    tm = now;
  }
  if (n_big) {  // rare: one warp per big bucket (none of whose entries was looked up above)
    bar_workers();
    for (uint32_t q = wid; q < min(n_big, (uint32_t)kBigMax); q += kWarps) {
      const uint32_t a = start[big_s[q]], e = start[big_s[q] + 1];
      warp_sort_idx<K>(tb.keys, idx, a, e - a);
    }
  }
  if (prof && t == 0) atomicAdd(&prof[3], (unsigned long long)(clock64() - tm));
}

// Worker threads: write the entry at each grouped position j to out[base + rank].  Ranks
// differ from j by less than a bucket, so the writes of a warp are nearly contiguous.
template <int KW>
__device__ __forceinline__ void emit_slots(Table<KW> tb, const uint16_t* idx, uint32_t d,
                                           const uint32_t (&rank)[kRankRegs], uint64_t base, uint64_t* out_keys,
                                           uint32_t* out_counts, uint64_t cap, uint32_t* status) {
  const int t = threadIdx.x - 32;
  if (base + d > cap) {
    if (t == 0) atomicOr(status, ST_INTERNAL);
    return;
  }
#pragma unroll
  for (int m = 0; m < kRankPer; ++m) {
    const uint32_t j = t + m * kWorkers;
    const uint32_t r = rank_get(rank, m);
    if (j < d && r < d) {
      const uint32_t s = idx[j];
      store_key(out_keys, base + r, tb.keys[s]);
      out_counts[base + r] = tb.counts[s];
    }
  }
}

__device__ __forceinline__ int ceil_log2_u32(uint32_t v) { return v <= 1 ? 0 : 32 - __clz(v - 1); }

template <int KW, bool MERGE = false>
__device__ __forceinline__ void count_emit_body(const Shape& s, const Buffers& b) {
  typedef typename KeyT<KW>::T K;
  extern __shared__ __align__(16) uint8_t sm[];
  const uint32_t cap_slots = 1u << s.bT_max;
  const uint32_t dcap = (3u * cap_slots) >> 2;  // most distinct keys a table is ordered with
  uint32_t* hist = reinterpret_cast<uint32_t*>(sm + (size_t)cap_slots * (KW * 8 + 4));  // [cap_slots / 2 + 4]
  uint64_t* gkey = reinterpret_cast<uint64_t*>(hist + cap_slots / 2 + 4);               // [dcap] (KW == 1)
  uint16_t* idx = reinterpret_cast<uint16_t*>(gkey + (KW == 1 ? dcap : 0));             // [dcap]
  __shared__ uint64_t excl_s, next_s[3];  // next ticket, its input range
  __shared__ volatile uint32_t ordered_s;  // the workers have ranked the current table
  __shared__ uint32_t next_u[2];          // its range-map interval: [next_u[0], next_u[1] - 1]
  __shared__ uint32_t ovf_s, special_s, nnew_s;
  __shared__ uint32_t wtmp[32];
  __shared__ K split_s, samp_s[kSplitSample];
  __shared__ K stk_lo[kSplitStack], stk_hi[kSplitStack];
  __shared__ K range_s[2];
  __shared__ uint32_t big_s[kBigMax], big_n;
  __shared__ int stk_n;
  const K EMPTY = all_ones<K>();
  const uint64_t NF = min(b.meta->n_fine, s.nf_max);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long* prof = s.profile ? reinterpret_cast<unsigned long long*>(b.meta->sub_cycles) : nullptr;
  unsigned long long* ticket = reinterpret_cast<unsigned long long*>(&b.meta->ticket);
  // profiled plans: thread 0 adds the cycles spent in each phase (0 -, 1 clear and count, 2 -,
  // 3 order, 4 look-back (warp 0, overlapped), 5 emit, 6 overflow path, 7 ticket + setup)
  long long t_mark = clock64();
  auto phase = [&](int i) {
    if (s.profile && threadIdx.x == 0) {
      const long long now = clock64();
      atomicAdd(reinterpret_cast<unsigned long long*>(&b.meta->phase_cycles[i]), (unsigned long long)(now - t_mark));
      t_mark = now;
    }
  };
  // The next partition's ticket, input range and range-map interval (next_s, next_u) are
  // fetched by thread 0 while the workers write the current partition out: the ticket is
  // taken as late as that, so that partitions start in ticket order and a look-back seldom
  // waits on a predecessor that started late; the rest arrives by asynchronous copies to
  // shared memory.  Tickets stay in increasing order within a block, so the block holding
  // the smallest unfinished ticket is always working on it and every look-back ends.
  auto fetch_next = [&](uint64_t nx) {  // one thread; completes at cp.async.wait_all
    next_s[0] = nx;
    if (nx < NF) {
      cp_async8(&next_s[1], &b.foff[nx]);
      cp_async8(&next_s[2], &b.fcur[nx]);  // the split's cursor: the partition's keys end there
      cp_async4(&next_u[0], &b.flo[nx]);
      cp_async4(&next_u[1], &b.flo[nx + 1]);
    }
  };
  if (threadIdx.x == 0) {
    ordered_s = 0;
    fetch_next(atomicAdd(ticket, 1ull));
    cp_async_wait_all();
  }
  while (true) {
    block_sync();
    const uint64_t g = next_s[0];
    if (g >= NF) break;
    const uint64_t f0 = next_s[1];
    uint64_t n = next_s[2] - f0;
    if (threadIdx.x == 0) {
      ovf_s = 0;
      special_s = 0;
      nnew_s = 0;
    }
    if (f0 > s.cap_kb || n > s.cap_kb - f0) {  // inconsistent scan: record it, count nothing
      if (threadIdx.x == 0) atomicOr(&b.meta->status, ST_INTERNAL);
      n = 0;
    }
    if (threadIdx.x == blockDim.x - 1) {
      // the partition's key range, from its range-map interval (flo[NF] = 0, so the last
      // interval ends at 2^32 - 1); by a thread of the warp with the fewest keys to count
      uint32_t xlo, xhi;
      x_range(next_u[0], next_u[1] - 1u, s.canonical, xlo, xhi);
      key_range(xlo, xhi, s.k, range_s[0], range_s[1]);
    }
    const uint64_t* in = b.sbuf + f0 * KW;
    // table: at least twice the keys (at most that many distinct), within the cap
    int bT = 6;
    while (bT < s.bT_max && ((uint64_t)1 << bT) < 2 * n) ++bT;
    Table<KW> tb;
    tb.keys = reinterpret_cast<K*>(sm);
    tb.counts = reinterpret_cast<uint32_t*>(tb.keys + (1u << bT));
    phase(7);
    count_all<KW, MERGE>(tb, in, n, false, K(0), K(0), bT, s.k == 32 * KW, s.count_limit, hist, &big_n, &nnew_s,
                         &ovf_s, &special_s, &b.meta->status);
    block_sync();
    phase(1);
    const uint32_t dn = nnew_s;
    if (!ovf_s && dn <= dcap) {
      const uint64_t d = (uint64_t)dn + (special_s ? 1 : 0);
      if (threadIdx.x == 0 && !(s.withhold && g == 0))
        st_status(&b.look[g], (g == 0 && !s.defer_all ? kLookIncl : kLookAgg) | d);
      // Warp 0 resolves the exclusive prefix (look-back) while the workers order the table,
      // waiting on unpublished predecessors only as long as the workers are busy.  Without a
      // prefix by then, the partition's run is written to its own input region instead
      // (deferred) and k_compact moves it once all counts are known.
      uint32_t rank[kRankRegs], placed = 0;
      if (wid == 0) {
        const long long lb0 = clock64();
        // (with a withheld prefix, a test that needs the wait to run out, it does not give up
        // when the ordering is done)
        const uint64_t ex = s.defer_all ? kNoPrefix
                            : g == 0    ? 0
                                        : lookback(b.look, g, &b.meta->status, s.spin_limit,
                                                   s.withhold ? nullptr : &ordered_s);
        if (lane == 0) {
          const bool direct = ex != kNoPrefix;
          if (direct && g > 0) st_status(&b.look[g], kLookIncl | (ex + d));
          b.fhist[g] = (uint32_t)d | (direct ? 0u : 0x80000000u);
          if (!direct) atomicAdd(reinterpret_cast<unsigned long long*>(&b.meta->n_deferred), 1ull);
          excl_s = ex;
          if (s.profile)
            atomicAdd(reinterpret_cast<unsigned long long*>(&b.meta->phase_cycles[4]), (unsigned long long)(clock64() - lb0));
        }
      } else {
        const long long tm = clock64();
        uint32_t NB = 2;
        while (NB < dn) NB <<= 1;
        const OrderMap<K> om = order_map<K>(range_s[0], range_s[1], NB);
        placed = bucket_slots<KW>(tb, 1u << bT, dn, NB, om, hist, idx, gkey, wtmp, big_s, &big_n, &b.meta->status, prof);
        if (prof && threadIdx.x == 32) atomicAdd(&prof[1], (unsigned long long)(clock64() - tm));
        rank_slots<KW>(tb, idx, gkey, placed, hist, om, big_s, big_n, rank, prof);
        bar_workers();
        if (threadIdx.x == 32) ordered_s = 1;
      }
      block_sync();
      phase(3);
      const uint64_t ex = excl_s;
      if (threadIdx.x == 0) {
        ordered_s = 0;
        fetch_next(atomicAdd(ticket, 1ull));
      }
      // direct: final positions; deferred: the partition's own input region
      const bool direct = ex != kNoPrefix;
      uint64_t* okeys = direct ? b.out_keys : b.sbuf;
      uint32_t* ocnts = direct ? b.out_counts : reinterpret_cast<uint32_t*>(b.kbuf);
      const uint64_t obase = direct ? ex : f0, olim = direct ? s.cap : f0 + n;
      if (wid > 0) emit_slots<KW>(tb, idx, placed, rank, obase, okeys, ocnts, olim, &b.meta->status);
      if (threadIdx.x == 0) {
        if (special_s) {
          if (obase + dn < olim) {
            store_key(okeys, obase + dn, EMPTY);
            ocnts[obase + dn] = special_s;
          } else {
            atomicOr(&b.meta->status, ST_INTERNAL);
          }
        }
        cp_async_wait_all();
      }
      phase(5);
    } else {
      // ---------------- overflow path: too many distinct keys for the table.  Split the
      // partition's key range into sub-ranges, each counted in its own table and ordered;
      // the exclusive prefix is resolved first because the partial outputs are written
      // before the total is known.  A sub-range narrower than the table holds fewer
      // distinct keys than slots, so the splitting ends.  The range is split at the median of a
      // sample of the keys in the table that overflowed, not in its middle: the keys that make
      // a partition overflow are mostly variants of a repeat and share long prefixes, so that
      // halving the range leaves them together for many passes over the partition's keys.
      // (72 M windows, 3% of them satellite arrays: count kernel 1271 -> 721 us.)
      if (threadIdx.x == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&b.meta->n_overflow), 1ull);
      bool have_prefix = false;
      {
        // the table just filled holds a sample of the partition's distinct keys (unless it was
        // a smaller table than the largest): the first split is at their median
        const K lo = range_s[0], hi = range_s[1];
        const bool split = bT == s.bT_max && median_key<K>(tb.keys, cap_slots, lo, hi, samp_s, &split_s);
        if (threadIdx.x == 0) {
          stk_lo[0] = split ? split_s : lo;
          stk_hi[0] = hi;
          stk_lo[1] = lo;
          stk_hi[1] = split ? split_s - 1 : hi;
          stk_n = split ? 2 : 1;
        }
      }
      block_sync();
      const int bTf = s.bT_max;
      tb.keys = reinterpret_cast<K*>(sm);
      tb.counts = reinterpret_cast<uint32_t*>(tb.keys + cap_slots);
      uint64_t written = 0;
      while (stk_n > 0) {
        const K lo = stk_lo[stk_n - 1], hi = stk_hi[stk_n - 1];
        block_sync();
        if (threadIdx.x == 0) {
          --stk_n;
          ovf_s = 0;
          special_s = 0;
          nnew_s = 0;
        }
        count_all<KW, MERGE>(tb, in, n, true, lo, hi, bTf, s.k == 32 * KW, s.count_limit, hist, &big_n, &nnew_s,
                             &ovf_s, &special_s, &b.meta->status);
        block_sync();
        const uint32_t dn2 = nnew_s;
        if (ovf_s || dn2 > dcap) {
          const bool median = median_key<K>(tb.keys, cap_slots, lo, hi, samp_s, &split_s);
          if (threadIdx.x == 0) {
            const K at = median && stk_n < kMedianDepth ? split_s : lo + ((hi - lo) >> 1) + 1;
            if (lo >= hi || stk_n + 2 > kSplitStack) {
              atomicOr(&b.meta->status, ST_INTERNAL);  // (a table that overflowed holds many keys)
            } else {
              stk_lo[stk_n] = at;
              stk_hi[stk_n] = hi;
              stk_lo[stk_n + 1] = lo;
              stk_hi[stk_n + 1] = at - 1;
              stk_n += 2;
            }
          }
          block_sync();
          continue;
        }
        {
          uint32_t rank2[kRankRegs], placed = 0;
          if (wid == 0) {  // the prefix is waited for while the first part is ordered
            if (!have_prefix) {
              const uint64_t ex = g == 0 ? 0 : lookback(b.look, g, &b.meta->status, s.spin_limit);
              if (lane == 0) excl_s = ex;
            }
          } else {
            uint32_t NB2 = 2;
            while (NB2 < dn2) NB2 <<= 1;
            const OrderMap<K> om = order_map<K>(lo, hi, NB2);
            placed = bucket_slots<KW>(tb, cap_slots, dn2, NB2, om, hist, idx, gkey, wtmp, big_s, &big_n, &b.meta->status);
            rank_slots<KW>(tb, idx, gkey, placed, hist, om, big_s, big_n, rank2, nullptr);
          }
          have_prefix = true;
          block_sync();
          const uint64_t base = excl_s + written;
          if (wid > 0) emit_slots<KW>(tb, idx, placed, rank2, base, b.out_keys, b.out_counts, s.cap, &b.meta->status);
        }
        written += dn2;
        block_sync();
      }
      // the all-ones key, if present, is the largest key of all
      uint32_t sp = 0;
      if (s.k == 32 * KW) {
        for (uint64_t i = threadIdx.x; i < n; i += blockDim.x) {
          K key;
          load_key(in, i, key);
          sp += key == EMPTY;
        }
      }
  #pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) sp += __shfl_xor_sync(0xffffffffu, sp, dd);
      if (lane == 0) wtmp[wid] = sp;
      block_sync();
      if (threadIdx.x == 0) {
        uint64_t tot = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += wtmp[w];
        if (tot) {
          if (tot > s.count_limit) atomicOr(&b.meta->status, ST_COUNT_OVERFLOW);
          if (excl_s + written < s.cap) {
            store_key(b.out_keys, excl_s + written, EMPTY);
            b.out_counts[excl_s + written] = (uint32_t)tot;
          } else {
            atomicOr(&b.meta->status, ST_INTERNAL);
          }
          ++written;
        }
        if (!(s.withhold && g == 0)) st_status(&b.look[g], kLookIncl | (excl_s + written));
        b.fhist[g] = (uint32_t)written;
        fetch_next(atomicAdd(ticket, 1ull));
        cp_async_wait_all();
      }
      phase(6);
    }
  }
}
template <int KW, bool MERGE = false>
__global__ void __launch_bounds__(kCountThreads, kCountBlocksPerSM) k_count_emit(Shape s, Buffers b) {
  pdl_wait();
  count_emit_body<KW, MERGE>(s, b);
}
template <int KW>
__global__ void __launch_bounds__(kCountThreads, kCountBlocksPerSM) k_count_emit_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  count_emit_body<KW>(d.s, d.b);
}

// ------------------------------------------------------------------ final: offsets of the runs
// Exclusive scan of the distinct counts of the fine partitions: fcur[g] = first output position
// of partition g, n_distinct = the total.  The look-back words are checked against it, and the
// deferred partitions are listed in flo (dead by now) for k_compact.  Every block adds up the
// counts before its own share for itself (they are read from L2; one block for all took 139 us
// for 100 K partitions and 214 us for 221 K, this takes 18 and 27).
__device__ __forceinline__ void scan_distinct_body(const Shape& sh, const Buffers& b, uint32_t bid, uint32_t nblk) {
  __shared__ uint64_t wt[32];
  __shared__ uint32_t wd[32];
  const uint64_t NF = min(b.meta->n_fine, sh.nf_max);
  const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, wid = t >> 5, nw = nt >> 5;
  const uint64_t share = (NF + nblk - 1) / nblk, start = min(NF, bid * share), end = min(NF, start + share);
  // sums over the block of (distinct, deferred), and the sums of the threads before
  auto block_sum = [&](uint64_t& x, uint32_t& y, uint64_t& before_x, uint32_t& before_y) {
    uint64_t p = x;
    uint32_t q = y;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint64_t xs = __shfl_up_sync(0xffffffffu, p, d);
      const uint32_t ys = __shfl_up_sync(0xffffffffu, q, d);
      if (lane >= d) {
        p += xs;
        q += ys;
      }
    }
    __syncthreads();
    if (lane == 31) {
      wt[wid] = p;
      wd[wid] = q;
    }
    __syncthreads();
    before_x = p - x;
    before_y = q - y;
    x = y = 0;
    for (int w = 0; w < nw; ++w) {
      if (w < wid) {
        before_x += wt[w];
        before_y += wd[w];
      }
      x += wt[w];
      y += wd[w];
    }
  };
  uint64_t carry = 0, skip_x;
  uint32_t dcarry = 0, skip_y;
  // the partitions before the share, four 16-byte loads in flight per thread
  const uint4* f4 = reinterpret_cast<const uint4*>(b.fhist);
  for (uint64_t i = t; i < start / 4; i += 4ull * nt) {
    uint4 v[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) v[m] = i + (uint64_t)m * nt < start / 4 ? f4[i + (uint64_t)m * nt] : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      carry += (uint64_t)(v[m].x & 0x7fffffffu) + (v[m].y & 0x7fffffffu) + (v[m].z & 0x7fffffffu) + (v[m].w & 0x7fffffffu);
      dcarry += (v[m].x >> 31) + (v[m].y >> 31) + (v[m].z >> 31) + (v[m].w >> 31);
    }
  }
  if (t < (int)(start & 3)) {  // an empty share after the last partition starts anywhere
    const uint32_t v = b.fhist[(start & ~3ull) + t];
    carry += v & 0x7fffffffu;
    dcarry += v >> 31;
  }
  block_sum(carry, dcarry, skip_x, skip_y);
  const uint64_t per = (end - start + nt - 1) / nt, lo = min(end, start + t * per), hi = min(end, lo + per);
  uint64_t s = 0, run;
  uint32_t nd = 0, drun;
  for (uint64_t i = lo; i < hi; ++i) {
    s += b.fhist[i] & 0x7fffffffu;
    nd += b.fhist[i] >> 31;
  }
  block_sum(s, nd, run, drun);
  run += carry;
  drun += dcarry;
  bool bad = false;
  for (uint64_t i = lo; i < hi; ++i) {
    const uint64_t d = b.fhist[i] & 0x7fffffffu;
    const bool deferred = b.fhist[i] >> 31;
    // a direct partition published its inclusive prefix, a deferred one its count
    bad |= ld_status(&b.look[i]) != (deferred ? (kLookAgg | d) : (kLookIncl | (run + d)));
    b.fcur[i] = run;
    if (deferred) b.flo[drun++] = (uint32_t)i;
    run += d;
  }
  if (bad) atomicOr(&b.meta->status, ST_INTERNAL);
  if (bid == nblk - 1 && t == 0) {
    b.meta->n_distinct = carry + s;
    if (dcarry + nd != b.meta->n_deferred) atomicOr(&b.meta->status, ST_INTERNAL);
  }
}
__global__ void __launch_bounds__(1024) k_scan_distinct(Shape sh, Buffers b) {
  pdl_wait();
  scan_distinct_body(sh, b, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(1024) k_scan_distinct_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  scan_distinct_body(d.s, d.b, bid, nblk);
}

// Move the runs of the deferred fine partitions from their input regions (keys in sbuf,
// counts in kbuf as 32-bit words) to their output positions: one block per partition.
template <int KW>
__device__ __forceinline__ void move_run(const Shape& s, const Buffers& b, uint64_t src, uint64_t dst, uint32_t d) {
  typedef typename KeyT<KW>::T K;
  const uint32_t* cnt_src = reinterpret_cast<const uint32_t*>(b.kbuf);
  if (src > s.cap_kb || d > s.cap_kb - src || dst > s.cap || d > s.cap - dst) {
    if (threadIdx.x == 0) atomicOr(&b.meta->status, ST_INTERNAL);
    return;
  }
  for (uint32_t i = threadIdx.x; i < d; i += blockDim.x) {
    K key;
    load_key(b.sbuf, src + i, key);
    store_key(b.out_keys, dst + i, key);
    b.out_counts[dst + i] = cnt_src[src + i];
  }
}
template <int KW>
__device__ __forceinline__ void compact_body(const Shape& s, const Buffers& b, uint32_t bid, uint32_t nblk) {
  const uint64_t n_def = min(b.meta->n_deferred, s.nf_max);
  for (uint64_t q = bid; q < n_def; q += nblk) {
    const uint64_t g = b.flo[q];
    if (g >= min(b.meta->n_fine, s.nf_max)) {
      if (threadIdx.x == 0) atomicOr(&b.meta->status, ST_INTERNAL);
      continue;
    }
    move_run<KW>(s, b, b.foff[g], b.fcur[g], b.fhist[g] & 0x7fffffffu);
  }
}
// One-level counts: the scan of the distinct counts and the moving of deferred runs in one
// launch.  There are at most kOneLevelFine partitions, so every block scans all of them for
// itself; the first one also checks the look-back words and records the total.
template <int KW>
__device__ __forceinline__ void finish_one_body(const Shape& s, const Buffers& b, uint32_t bid, uint32_t nblk) {
  __shared__ uint32_t pre[kOneLevelFine + kOneLevelFine / 32 + 1];
  __shared__ uint32_t wt[32];
  const int NF = (int)min(b.meta->n_fine, min(s.nf_max, kOneLevelFine));
  for (int g = threadIdx.x; g < NF; g += blockDim.x) pre[PAD(g)] = b.fhist[g] & 0x7fffffffu;
  __syncthreads();
  const uint32_t D = block_exclusive_scan_pad<uint32_t>(pre, NF, wt);  // below 2^24
  if (bid == 0) {
    bool bad = false;
    uint32_t n_def = 0;
    for (int g = threadIdx.x; g < NF; g += blockDim.x) {
      // a direct partition published its inclusive prefix, a deferred one its count
      const uint32_t v = b.fhist[g], d = v & 0x7fffffffu;
      bad |= ld_status(&b.look[g]) != (v >> 31 ? (kLookAgg | d) : (kLookIncl | ((uint64_t)pre[PAD(g)] + d)));
      n_def += v >> 31;
    }
    if (threadIdx.x == 0) wt[0] = 0;
    __syncthreads();
    if (n_def) atomicAdd(&wt[0], n_def);
    __syncthreads();
    bad |= wt[0] != b.meta->n_deferred;
    if (bad) atomicOr(&b.meta->status, ST_INTERNAL);
    if (threadIdx.x == 0) b.meta->n_distinct = D;
  }
  for (int g = bid; g < NF; g += nblk) {
    const uint32_t v = b.fhist[g];
    if (v >> 31) move_run<KW>(s, b, b.foff[g], pre[PAD(g)], v & 0x7fffffffu);
  }
}
template <int KW>
__global__ void __launch_bounds__(256) k_finish_one(Shape s, Buffers b) {
  pdl_wait();
  finish_one_body<KW>(s, b, blockIdx.x, gridDim.x);
}
template <int KW>
__global__ void __launch_bounds__(256) k_finish_one_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  finish_one_body<KW>(d.s, d.b, bid, nblk);
}
template <int KW>
__global__ void __launch_bounds__(256) k_compact(Shape s, Buffers b) {
  pdl_wait();
  compact_body<KW>(s, b, blockIdx.x, gridDim.x);
}
template <int KW>
__global__ void __launch_bounds__(256) k_compact_batch(BatchTab t) {
  KC_BATCH_PROLOGUE(t);
  compact_body<KW>(d.s, d.b, bid, nblk);
}

// ------------------------------------------------------------------ launches
constexpr size_t kScatterStaticSmem = 6144;  // pass B's static shared memory (batched form included), rounded up
static size_t scatter_smem(const Shape& s, int nt) {
  const size_t sub = (size_t)nt * (s.kw == 1 ? 32 : 16) * s.kw * 8;
  if (s.one_level) {
    const size_t most = s.one_level == kEitherLevel ? kEitherFine : s.nf_max;
    return sub + 2 * padded_len(most + 32) * 4 + ((size_t)2 << s.bb);
  }
  const size_t P1 = (size_t)1 << s.b1;
  return sub + P1 * 8 + 2 * padded_len(P1 + 32) * 4;
}
// clears (a thread per fine partition) and first reads (a warp per tile)
static uint32_t prepare_blocks(const Shape& s, uint64_t most) {
  const uint64_t want = std::max<uint64_t>((s.nf_max + 255) / 256, (s.n_tiles + 7) / 8) + 4;
  return (uint32_t)(want < most ? want : most);
}
// Pass A: a block per tile, or (one level) at most four per SM of 152, in a batch for each of its
// counts, each adding up the bins of several tiles (pass A of 10 M / 45 M bases: 608 blocks 40 /
// 93 us, 912 44 / 107, 1216 51 / 100; as few blocks as give each the same number of tiles, 407 /
// 550: 42 / 102).
// Many short or empty reads: more blocks than tiles, a share of the offsets each.
static uint32_t pack_blocks(const Shape& s) {
  const uint64_t tiles = s.one_level ? std::min<uint64_t>(s.n_tiles, 608) : s.n_tiles;
  return (uint32_t)std::max<uint64_t>(tiles, std::min<uint64_t>(s.n_reads / 8192 + 1, 608));
}
// the scan of the distinct counts: a share of about 4096 fine partitions each
static uint32_t scan_blocks(const Shape& s) {
  const uint64_t want = s.nf_max / 4096 + 1;
  return (uint32_t)(want < 128 ? want : 128);
}
// the last kernel: deferred runs to move (at most one per fine partition)
static uint32_t compact_blocks(const Shape& s, int n_sms) {
  const uint64_t want = s.nf_max / 8 + 1, most = (uint64_t)n_sms * 8;
  return (uint32_t)(want < most ? want : most);
}
// pass A: the histogram, and the last block's scan of the partitions' totals
static size_t pack_smem(const Shape& s) {
  const size_t P1 = (size_t)1 << s.b1;
  return s.one_level ? padded_len(((size_t)1 << s.bb) + 32) * 4 : (P1 + 16) * 8;
}
static size_t fine_hist_smem(int P1) { return (size_t)(P1 + 1) * 8 + kFineLocalCap * 4 + 16; }
static size_t fine_scatter_smem(int kw, int P1) {
  return (size_t)kFineChunk * (kw * 8 + 2) + kFineLocalCap * (8 + 4 + 4) + (size_t)(P1 + 1) * 8 + 16;
}

int configure_kernels(int device) {
  int optin = 0;
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e != cudaSuccess) return (int)e;
  // dynamic + static shared memory must fit the opt-in limit
#define KC_SET(fn)                                                                                          \
  {                                                                                                         \
    cudaFuncAttributes fa;                                                                                  \
    if ((e = cudaFuncGetAttributes(&fa, fn)) != cudaSuccess) return (int)e;                                 \
    const int dyn = optin - (int)fa.sharedSizeBytes;                                                        \
    if ((e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn)) != cudaSuccess) \
      return (int)e;                                                                                        \
  }
#define KC_SET_PHASE1(KW, VAR)                              \
  KC_SET((k_pack_count<KW, false, VAR>));                   \
  KC_SET((k_pack_count<KW, true, VAR>));                    \
  KC_SET((k_pack_count_batch<KW, false, VAR>));             \
  KC_SET((k_pack_count_batch<KW, true, VAR>));              \
  KC_SET((k_scatter<KW, 256, SC_COARSE, VAR>));             \
  KC_SET((k_scatter<KW, 256, SC_ONE, VAR>));                \
  KC_SET((k_scatter_batch<KW, 256, SC_COARSE, VAR>));       \
  KC_SET((k_scatter_batch<KW, 256, SC_ONE, VAR>))
  KC_SET_PHASE1(1, V_SHORT);
  KC_SET_PHASE1(1, V_CANON);
  KC_SET_PHASE1(1, V_FORWARD);
  KC_SET_PHASE1(2, V_CANON);
  KC_SET_PHASE1(2, V_FORWARD);
  KC_SET(k_scatter_direct<1>);
  KC_SET(k_scatter_direct<2>);
  KC_SET(k_fine_plan);
  KC_SET(k_fine_hist<1>);
  KC_SET(k_fine_hist<2>);
  KC_SET(k_fine_scatter<1>);
  KC_SET(k_fine_scatter<2>);
  KC_SET(k_count_emit<1>);
  KC_SET(k_count_emit<2>);
  KC_SET((k_count_emit<1, true>));
  KC_SET((k_count_emit<2, true>));
  KC_SET(k_fine_plan_batch);
  KC_SET(k_fine_hist_batch<1>);
  KC_SET(k_fine_hist_batch<2>);
  KC_SET(k_fine_scatter_batch<1>);
  KC_SET(k_fine_scatter_batch<2>);
  KC_SET(k_count_emit_batch<1>);
  KC_SET(k_count_emit_batch<2>);
#undef KC_SET
  return 0;
}

// After each launch: record the marker, and stop the sequence on a launch error so that
// no later kernel runs on buffers an earlier one did not fill (returns -cudaError_t).
#define KC_STEP(name)                                   \
  do {                                                  \
    const cudaError_t le = cudaGetLastError();          \
    if (le != cudaSuccess) return -(int)le;             \
    mark(name);                                         \
  } while (0)

// CALL(key words, variant) for a count's key width, k and mode.
#define KC_PHASE1_VARIANT(s, CALL)                         \
  do {                                                     \
    if ((s).kw == 2) {                                     \
      if ((s).canonical) { CALL(2, V_CANON); }             \
      else { CALL(2, V_FORWARD); }                         \
    } else if ((s).k < 16) {                               \
      CALL(1, V_SHORT);                                    \
    } else if ((s).canonical) {                            \
      CALL(1, V_CANON);                                    \
    } else {                                               \
      CALL(1, V_FORWARD);                                  \
    }                                                      \
  } while (0)

int launch_phase1(const Shape& s, const Buffers& b, int n_sms, void* stream, const Marker& mark) {
  cudaStream_t st = (cudaStream_t)stream;
  int launches = 0;
  pdl_launch(k_prepare, prepare_blocks(s, (uint64_t)n_sms * 8), 256, 0, st, s, b);
  ++launches;
  KC_STEP("k_prepare");
  const unsigned gt = pack_blocks(s);
  const size_t smA = pack_smem(s);
#define KC_PACK(KW, VAR)                                                                  \
  if (s.one_level) pdl_launch(k_pack_count<KW, true, VAR>, gt, kPackThreads, smA, st, s, b);      \
  else pdl_launch(k_pack_count<KW, false, VAR>, gt, kPackThreads, smA, st, s, b)
  KC_PHASE1_VARIANT(s, KC_PACK);
#undef KC_PACK
  ++launches;
  KC_STEP("k_pack_count");
  return launches;
}

int launch_phase2(const Shape& s, const Buffers& b, int n_sms, uint32_t nf_max, void* stream, const Marker& mark) {
  cudaStream_t st = (cudaStream_t)stream;
  const int P1 = 1 << s.b1;
  int launches = 0;
  if (s.n_tiles > 0) {
    const size_t smB = scatter_smem(s, 256);
    if (smB + kScatterStaticSmem > s.smem_budget) return -(int)cudaErrorInvalidConfiguration;
    const unsigned gt = (unsigned)s.n_tiles;
    if (s.aggr & kAggrNoSmemBuckets) {
      if (s.kw == 1) pdl_launch(k_scatter_direct<1>, gt, 256, smB, st, s, b);
      else pdl_launch(k_scatter_direct<2>, gt, 256, smB, st, s, b);
    } else {
#define KC_SCATTER(KW, VAR)                                                       \
  if (s.one_level) pdl_launch(k_scatter<KW, 256, SC_ONE, VAR>, gt, 256, smB, st, s, b);   \
  else pdl_launch(k_scatter<KW, 256, SC_COARSE, VAR>, gt, 256, smB, st, s, b)
      KC_PHASE1_VARIANT(s, KC_SCATTER);
#undef KC_SCATTER
    }
    ++launches;
    KC_STEP("k_scatter");
  }
  if (s.one_level != kOneLevel) {
    pdl_launch(k_fine_plan, P1, 256, padded_len(P1) * 4, st, s, b);
    ++launches;
    KC_STEP("k_fine_plan");
    const unsigned gf = (unsigned)(n_sms * 2);
    // the fine split (sampled layout or exact); after a sampled one, the exact split again,
    // whose kernels return at once unless a sampled region overflowed
    for (int redo = 0; redo <= (s.fine_sampled ? 1 : 0); ++redo) {
      if (redo) {
        pdl_launch(k_fine_redo_clear, (unsigned)n_sms, 1024, 0, st, s, b);
        ++launches;
        KC_STEP("k_fine_redo_clear");
      }
      if (s.kw == 1) pdl_launch(k_fine_hist<1>, gf, kFineThreads, fine_hist_smem(P1), st, s, b, redo);
      else pdl_launch(k_fine_hist<2>, gf, kFineThreads, fine_hist_smem(P1), st, s, b, redo);
      ++launches;
      KC_STEP(redo ? "k_fine_hist_redo" : "k_fine_hist");
      pdl_launch(k_fine_scan, P1, 256, 0, st, s, b, redo);
      ++launches;
      KC_STEP(redo ? "k_fine_scan_redo" : "k_fine_scan");
      if (s.kw == 1) pdl_launch(k_fine_scatter<1>, gf, kFineThreads, fine_scatter_smem(1, P1), st, s, b, redo);
      else pdl_launch(k_fine_scatter<2>, gf, kFineThreads, fine_scatter_smem(2, P1), st, s, b, redo);
      ++launches;
      KC_STEP(redo ? "k_fine_scatter_redo" : "k_fine_scatter");
    }
  }
  const size_t smC = count_kernel_smem(s.kw, s.bT_max);
  if (s.aggr & kAggrWarpMerge) {
    if (s.kw == 1) pdl_launch(k_count_emit<1, true>, (unsigned)(n_sms * kCountBlocksPerSM), kCountThreads, smC, st, s, b);
    else pdl_launch(k_count_emit<2, true>, (unsigned)(n_sms * kCountBlocksPerSM), kCountThreads, smC, st, s, b);
  } else if (s.kw == 1) {
    pdl_launch(k_count_emit<1>, (unsigned)(n_sms * kCountBlocksPerSM), kCountThreads, smC, st, s, b);
  } else {
    pdl_launch(k_count_emit<2>, (unsigned)(n_sms * kCountBlocksPerSM), kCountThreads, smC, st, s, b);
  }
  ++launches;
  KC_STEP("k_count_emit");
  if (s.one_level == kOneLevel) {
    if (s.kw == 1) pdl_launch(k_finish_one<1>, compact_blocks(s, n_sms), 256, 0, st, s, b);
    else pdl_launch(k_finish_one<2>, compact_blocks(s, n_sms), 256, 0, st, s, b);
    ++launches;
    KC_STEP("k_finish_one");
    return launches;
  }
  pdl_launch(k_scan_distinct, scan_blocks(s), 1024, 0, st, s, b);
  ++launches;
  KC_STEP("k_scan_distinct");
  if (s.kw == 1) pdl_launch(k_compact<1>, compact_blocks(s, n_sms), 256, 0, st, s, b);
  else pdl_launch(k_compact<2>, compact_blocks(s, n_sms), 256, 0, st, s, b);
  ++launches;
  KC_STEP("k_compact");
  return launches;
}

uint32_t batch_blocks(BatchKernel k, const Shape& s, int n_sms, uint64_t bases_total) {
  auto clampu = [](uint64_t v, uint64_t lo, uint64_t hi) { return (uint32_t)(v < lo ? lo : (v > hi ? hi : v)); };
  const uint64_t nsm = (uint64_t)n_sms;
  switch (k) {
    case BK_PREPARE: return prepare_blocks(s, 64);
    case BK_PACK: return s.one_level ? 0u : pack_blocks(s);
    case BK_PACK_ONE: return s.one_level ? pack_blocks(s) : 0u;
    case BK_SCATTER: return s.one_level ? 0u : (uint32_t)s.n_tiles;
    case BK_SCATTER_ONE: return s.one_level ? (uint32_t)s.n_tiles : 0u;
    case BK_FINE_PLAN:
    case BK_FINE_SCAN: return s.one_level == kOneLevel ? 0u : 1u << s.b1;
    case BK_FINE_HIST:
    case BK_FINE_SCATTER: return s.one_level == kOneLevel ? 0u : clampu((s.L + 4ull * kFineChunk - 1) / (4ull * kFineChunk), 1, 2 * nsm);
    case BK_COUNT: {
      const double share = bases_total ? (double)s.L / (double)bases_total : 1.0;
      return clampu((uint64_t)(2.0 * (double)nsm * share + 0.999), 1, nsm * kCountBlocksPerSM);
    }
    case BK_SCAN_DISTINCT: return s.one_level == kOneLevel ? 0u : scan_blocks(s);
    case BK_COMPACT: return s.one_level == kOneLevel ? 0u : compact_blocks(s, n_sms);
    case BK_FINISH_ONE: return s.one_level == kOneLevel ? compact_blocks(s, n_sms) : 0u;
    default: return 1u;
  }
}

// The launch sequence of launch_phase1 + launch_phase2, each kernel once for all counts of
// the batch (all with the same key width); a kernel that gives no count a block is skipped.
int launch_batch(const BatchPlan& bp, int n_sms, void* stream, const Marker& mark) {
  cudaStream_t st = (cudaStream_t)stream;
  const int P1 = bp.P1_max;
  const Shape& s0 = bp.host[0].s;
  int launches = 0;
  auto tab = [&](BatchKernel k) { return BatchTab{bp.desc, bp.blk2s[k], bp.start[k]}; };
#define KC_BLAUNCH(k, call, name) \
  if (bp.grid[k]) {               \
    call;                         \
    ++launches;                   \
    KC_STEP(name);                \
  }
  // shared memory: the most that any count of the launch asks for
  size_t smA[2] = {}, smB[2] = {};
  for (int q = 0; q < bp.n; ++q) {
    const Shape& s = bp.host[q].s;
    smA[s.one_level != 0] = std::max(smA[s.one_level != 0], pack_smem(s));
    smB[s.one_level != 0] = std::max(smB[s.one_level != 0], scatter_smem(s, 256));
  }
  if (std::max(smB[0], smB[1]) + kScatterStaticSmem > s0.smem_budget) return -(int)cudaErrorInvalidConfiguration;
  KC_BLAUNCH(BK_PREPARE, (k_prepare_batch<<<bp.grid[BK_PREPARE], 256, 0, st>>>(tab(BK_PREPARE))), "k_prepare");
#define KC_PHASE1(KW, VAR)                                                                                          \
  KC_BLAUNCH(BK_PACK, (k_pack_count_batch<KW, false, VAR><<<bp.grid[BK_PACK], kPackThreads, smA[0], st>>>(tab(BK_PACK))), \
             "k_pack_count");                                                                                      \
  KC_BLAUNCH(BK_PACK_ONE,                                                                                          \
             (k_pack_count_batch<KW, true, VAR><<<bp.grid[BK_PACK_ONE], kPackThreads, smA[1], st>>>(tab(BK_PACK_ONE))), \
             "k_pack_count");                                                                                      \
  KC_BLAUNCH(BK_SCATTER,                                                                                           \
             (k_scatter_batch<KW, 256, SC_COARSE, VAR><<<bp.grid[BK_SCATTER], 256, smB[0], st>>>(tab(BK_SCATTER))), \
             "k_scatter");                                                                                         \
  KC_BLAUNCH(BK_SCATTER_ONE,                                                                                       \
             (k_scatter_batch<KW, 256, SC_ONE, VAR><<<bp.grid[BK_SCATTER_ONE], 256, smB[1], st>>>(tab(BK_SCATTER_ONE))), \
             "k_scatter")
  KC_PHASE1_VARIANT(s0, KC_PHASE1);  // (all counts of a batch have the same k and mode)
#undef KC_PHASE1
  KC_BLAUNCH(BK_FINE_PLAN, (k_fine_plan_batch<<<bp.grid[BK_FINE_PLAN], 256, padded_len(P1) * 4, st>>>(tab(BK_FINE_PLAN))),
             "k_fine_plan");
  // the fine split; then, for counts with a sampled layout, the exact split again (each
  // count's blocks return at once unless its sampled regions overflowed)
  for (int redo = 0; redo <= (bp.sampled ? 1 : 0); ++redo) {
    if (redo)
      KC_BLAUNCH(BK_FINE_SCAN, (k_fine_redo_clear_batch<<<bp.grid[BK_FINE_SCAN], 1024, 0, st>>>(tab(BK_FINE_SCAN))),
                 "k_fine_redo_clear");
    if (bp.kw == 1) {
      KC_BLAUNCH(BK_FINE_HIST,
                 (k_fine_hist_batch<1><<<bp.grid[BK_FINE_HIST], kFineThreads, fine_hist_smem(P1), st>>>(
                     tab(BK_FINE_HIST), redo)),
                 redo ? "k_fine_hist_redo" : "k_fine_hist");
    } else {
      KC_BLAUNCH(BK_FINE_HIST,
                 (k_fine_hist_batch<2><<<bp.grid[BK_FINE_HIST], kFineThreads, fine_hist_smem(P1), st>>>(
                     tab(BK_FINE_HIST), redo)),
                 redo ? "k_fine_hist_redo" : "k_fine_hist");
    }
    KC_BLAUNCH(BK_FINE_SCAN, (k_fine_scan_batch<<<bp.grid[BK_FINE_SCAN], 256, 0, st>>>(tab(BK_FINE_SCAN), redo)),
               redo ? "k_fine_scan_redo" : "k_fine_scan");
    if (bp.kw == 1) {
      KC_BLAUNCH(BK_FINE_SCATTER,
                 (k_fine_scatter_batch<1><<<bp.grid[BK_FINE_SCATTER], kFineThreads, fine_scatter_smem(1, P1), st>>>(
                     tab(BK_FINE_SCATTER), redo)),
                 redo ? "k_fine_scatter_redo" : "k_fine_scatter");
    } else {
      KC_BLAUNCH(BK_FINE_SCATTER,
                 (k_fine_scatter_batch<2><<<bp.grid[BK_FINE_SCATTER], kFineThreads, fine_scatter_smem(2, P1), st>>>(
                     tab(BK_FINE_SCATTER), redo)),
                 redo ? "k_fine_scatter_redo" : "k_fine_scatter");
    }
  }
  const size_t smC = count_kernel_smem(bp.kw, s0.bT_max);
  if (bp.kw == 1) {
    KC_BLAUNCH(BK_COUNT, (k_count_emit_batch<1><<<bp.grid[BK_COUNT], kCountThreads, smC, st>>>(tab(BK_COUNT))),
               "k_count_emit");
  } else {
    KC_BLAUNCH(BK_COUNT, (k_count_emit_batch<2><<<bp.grid[BK_COUNT], kCountThreads, smC, st>>>(tab(BK_COUNT))),
               "k_count_emit");
  }
  KC_BLAUNCH(BK_SCAN_DISTINCT,
             (k_scan_distinct_batch<<<bp.grid[BK_SCAN_DISTINCT], 1024, 0, st>>>(tab(BK_SCAN_DISTINCT))),
             "k_scan_distinct");
  if (bp.kw == 1) {
    KC_BLAUNCH(BK_COMPACT, (k_compact_batch<1><<<bp.grid[BK_COMPACT], 256, 0, st>>>(tab(BK_COMPACT))), "k_compact");
    KC_BLAUNCH(BK_FINISH_ONE, (k_finish_one_batch<1><<<bp.grid[BK_FINISH_ONE], 256, 0, st>>>(tab(BK_FINISH_ONE))),
               "k_finish_one");
  } else {
    KC_BLAUNCH(BK_COMPACT, (k_compact_batch<2><<<bp.grid[BK_COMPACT], 256, 0, st>>>(tab(BK_COMPACT))), "k_compact");
    KC_BLAUNCH(BK_FINISH_ONE, (k_finish_one_batch<2><<<bp.grid[BK_FINISH_ONE], 256, 0, st>>>(tab(BK_FINISH_ONE))),
               "k_finish_one");
  }
#undef KC_BLAUNCH
  return launches;
}

}  // namespace kc
