// Exact-split BF16 products of FP64 or float-pair matrices on the fifth-generation
// tensor cores (tcgen05.mma, accumulators in tensor memory, operands staged in
// shared memory by tiled tensor copies).  Included by dqmc_device.cuh inside its
// namespace, after the float-pair arithmetic.
//
// Scheme (Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012, on BF16
// digits): every row i of op(A) and column j of op(B) is scaled by a power of
// two, rounded to a fixed-point integer and cut into ND balanced 8-bit digits,
//     x = 2^(e-8) sum_t q_t 2^(-8t),   q_t integer, |q_t| <= 128,
// ND = 7 for float pairs (|x| < 2^(e-1): 56 bits under the row's largest entry)
// and ND = 8 for FP64 (|x| < 2^(e-2): 63 bits).  The digit planes hold
// q_t 2^(-8t) as BF16 (exact), so the product of digits t and u carries the
// weight of its diagonal d = t + u:
//     (op(A) op(B))_ij = 2^(eA_i + eB_j - 16) sum_{t,u} sum_k qA_t qB_u 2^(-8(t+u)).
// Each diagonal d < ND has an FP32 tensor-memory accumulator of its own: its terms
// are multiples of 2^(-8d) below 2^(14-8d), so every partial sum is exact while
// (d+1) K <= 1024, for d <= 3 up to the segment length K = 256; later diagonals
// round at 2^-24 of terms already 2^-32 below the result.  Pairs with t + u >= ND
// are dropped (below 2^-56 and 2^-64 of the scale).  The diagonals are summed as
// float pairs, or for FP64 as one integer that is rounded once.
//
// Error: fixed-point under the largest entries of the row and the column, for FP64 at
// most K 2^-57 max|a| max|b| (the dropped pairs, all of one sign) and one rounding;
// an FP64 chain's is relative to each element's |A||B|, the smaller one where those
// largest entries do not meet.  Largest error over |A||B| against 80-bit sums (normal
// A, log-normal B): FP64 operands 1.0e-16 at N = 64 and 5.6e-16 at N = 144, where a chain
// of FP64 FMAs has 1.0e-15 and 1.4e-15.  Of the stable G with site potentials, sorted,
// that spread blocks of slices by 2^40 to 2^52 (N = 33, products of 63 bits and FP64
// chains emulated on the CPU, against 70-digit decimals): 3.0e-16 to 3.2e-15 and 2.3e-16
// to 6.8e-15.  Rows of G of the order of e^-28 have a relative error of 4e-10 where
// chains leave 5e-12, of e^-56 1e-6 where chains leave 4e-10 to 9e-10.
//
// Cost per product on GB300 (one CTA of two per SM, cycles): FP64 N = 64 44k, 72 69k,
// 144 298k, where the FP64 pipe's tiles need 159k, 280k and 1.8M per CTA and SM
// (half of it with one CTA); float pairs N = 144 274k (the float-pair register tiles
// 560k).  Cutting the operands and recombining the diagonals take about half of it,
// the chunk pipeline the rest.
//
// Tiles: 128 x 32 outputs (MMA M = 128).  The B digits of a tile are staged as one
// 32 ND-row operand, so digit t of A meets the digits 0..ND-1-t of B in one MMA of
// N = 32 (ND - t) whose accumulators t..ND-1 are adjacent columns: ND MMAs per
// 16-deep chunk instead of ND (ND+1) / 2, each reading A from shared memory once.
// A matrix of N rows is cut into ceil(N / 128) equal row tiles, rounded to 16 rows
// (rows past a tile read whatever follows it in the staging area: their outputs
// are not used).  The digit planes are laid out in global memory (per-chain
// scratch, L2-resident; the constant propagators' planes are prepared once per
// model) in the order (tile, k chunk, digit) with each 16-wide block in the
// canonical K-major layout without swizzle; a tensor map describes each plane
// buffer as 512-byte rows with a box of one whole (tile, k chunk), so one chunk is
// two tiled tensor copies (cp.async.bulk.tensor).  The chunks of all
// tiles form one sequence streamed through two or three stages: warp 1 issues the
// copies, warp 0 the MMAs, each through one elected thread (one thread doing both
// spent 1300 cycles a chunk on issue and bookkeeping, the MMAs take 450 - 580).
// Completion is tracked with mbarriers whose waits give up after ~1 s (the chain's
// error word records it).
#pragma once

constexpr int kUmmaNT = kPlaneRowsB;        // tile columns
constexpr int kUmmaK = kPlaneK;             // MMA K and staged chunk
constexpr int kUmmaM = kPlaneMaxRows;       // MMA M
constexpr int kUmmaKSeg = 256;              // k per exactly accumulated segment
constexpr int kUmmaCols = 256;              // tensor-memory columns allocated per CTA
constexpr int kUmmaStages = 3;              // copy pipeline depth (at most)
constexpr int kUmmaNonFinite = 1 << 20;     // exponent of a row that holds an Inf or NaN
constexpr long long kUmmaWaitCycles = 2000000000LL;        // default wait limit, ~1 s
static_assert(kPlaneDigits64 * kUmmaNT <= kUmmaCols && kPlaneDigits64 * kUmmaNT <= 256,
              "one MMA spans every diagonal's accumulator");

// digits of an operand type
template <typename T>
struct UmmaDigits { static constexpr int n = kPlaneDigits64; };
template <>
struct UmmaDigits<dd> { static constexpr int n = kPlaneDigits; };

__host__ __device__ inline int umma_pad(int n, int q) { return (n + q - 1) / q * q; }

// State of the tensor-core products of one CTA.  Nothing in it is indexed at
// run time (that would push the kernel's whole shared-memory descriptor into
// local memory): thread 0's bookkeeping lives in the 128-byte shared barrier area.
struct Umma {
  unsigned char* stage;   // staging area (nothing else is live there during a product)
  uint32_t stage_bytes;   // its bytes
  uint64_t* bar;          // shared, 128 bytes: [0, 48) the 2 kUmmaStages mbarriers (copies landed
                          // per stage, then MMAs done per stage); [48, 56) accumulators complete;
                          // [56, 64) a barrier that nothing arrives on (the test_stall hook);
                          // [64, 68) the parities of the seven barriers' next phases; [68, 76)
                          // chunks copied and multiplied by a product that gave up; [96, 100) the
                          // TMEM slot; [100, 104) the count of products
  uint32_t* tmem_slot;    // tcgen05.alloc writes the accumulator base here
  int* err;               // chain error word (nonzero: a wait gave up)
  long long limit;        // SM cycles after which a wait gives up
  int stall;              // test hook: the first wait of a product waits on the barrier at
                          // [56, 64), which gives up after `limit`
  int* where;             // [6] or null: the first wait that gave up (kind, chunk, chunks,
                          // product ordinal, barrier word)
};

__device__ __forceinline__ uint64_t* umma_acc(const Umma& U) { return U.bar + 2 * kUmmaStages; }
__device__ __forceinline__ uint64_t* umma_never(const Umma& U) { return U.bar + 2 * kUmmaStages + 1; }
__device__ __forceinline__ uint32_t* umma_book(const Umma& U) { return reinterpret_cast<uint32_t*>(U.bar + 8); }
__device__ __forceinline__ uint32_t* umma_calls(const Umma& U) { return U.tmem_slot + 1; }
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0u;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major operand without swizzle; lbo = byte
// distance of core matrices adjacent in K, sbo = in M / N.
__device__ __forceinline__ uint64_t umma_sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of this architecture
  return d;
}
// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Wait for the phase of the given parity to complete; false if it gave up
// after `limit` SM cycles.  Polls with the non-blocking test_wait, so that the
// limit holds however short it is.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit) {
  const uint32_t a = smem_u32(bar);
  const long long t0 = clock64();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}
// One block of digit planes (all digits of a tile x 16-wide K chunk, contiguous in
// the plane buffer) into shared memory: a tiled tensor copy of the block's rows of
// the buffer's 2D view [rows][kPlaneRowElems] the map describes.  The copy engine
// works row by row: 512-byte rows move a chunk in a third of the cycles that the
// 32-byte rows of a [digits][rows][16] view took (1400 a chunk of 25 KB).
__device__ __forceinline__ void tma_load_block(void* dst, const CUtensorMap* tm, int row, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(0), "r"(row), "r"(smem_u32(bar))
      : "memory");
}
// A tensor map in global memory that the host wrote (here by a copy, possibly over another
// map at the same address): ordered before the block's tiled copies that use it.
__device__ __forceinline__ void tensor_map_acquire(const CUtensorMap* tm) {
  asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(tm)) : "memory");
}
__device__ __forceinline__ void umma_bf16(uint32_t dtm, uint64_t ad, uint64_t bd, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtm),
      "l"(ad), "l"(bd), "r"(id), "r"(acc));
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* v) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = __uint_as_float(r[q]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// The tensor maps of a plane set, acquired by the warp that issues the copies: a plane set
// lies in memory that is written again (the adjoints' kept workspace, an arena that a
// context before this one had), and a descriptor cached from then describes other planes.
__device__ inline void umma_acquire_maps(const PlaneSet* ps) {
  if (ps == nullptr || (threadIdx.x >> 5) != 1) return;
  for (int q = 0; q < 2; ++q) tensor_map_acquire(&ps->tm_pl[q]);
  for (int q = 0; q < kCpSets; ++q) tensor_map_acquire(&ps->tm_cp[q]);
}

// Tensor memory of the CTA: warp 0 allocates kUmmaCols columns (at most two
// CTAs of a product kernel share an SM, so the 512 columns of an SM never run
// out) and gives up the right to allocate more; the base goes to *slot.
__device__ inline void umma_alloc(const Umma& U) {
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(U.tmem_slot)),
                 "r"(kUmmaCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the copy and MMA barriers live for the whole kernel: initialised once here,
  // never re-initialised while an arrival could still be on its way
  if (threadIdx.x == 0) {
    for (int q = 0; q < 2 * kUmmaStages + 2; ++q) mbar_init(U.bar + q);
    *umma_book(U) = 0u;
    *umma_calls(U) = 0u;
  }
  // tiled tensor copies need 128-byte aligned shared destinations: a staging
  // buffer that is not marks the products void (they are then skipped and the
  // call reports it) instead of issuing a copy the hardware would reject
  if (threadIdx.x == 0 && ((smem_u32(U.stage) & 127u) != 0u)) {
    if (U.where && U.where[0] == 0) U.where[0] = 9;
    if (U.err) atomicOr(U.err, 2);
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
}
// Every path out of a kernel that allocated calls this (all threads).
__device__ inline void umma_free(const Umma& U) {
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*U.tmem_slot), "r"(kUmmaCols)
                 : "memory");
}

// Offset (elements) of (r, k) inside a digit block of 16 k: core matrices of 8
// rows x 8 k (128 bytes, rows 16 bytes apart), k groups 128 bytes apart, row
// groups 256 bytes apart.
__device__ __forceinline__ int umma_core_off(int r, int k) { return (r >> 3) * 128 + (k >> 3) * 64 + (r & 7) * 8 + (k & 7); }

// ---- operands to digits -------------------------------------------------------
// |x| as an ordered integer whose top bits are the exponent, and the row exponent
// e from the largest one (|x| < 2^(e-2) FP64, 2^(e-1) float pairs; 0: a zero row)
__device__ __forceinline__ int umma_mag(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ int umma_mag(dd x) { return __float_as_int(x.hi) & 0x7fffffff; }
__device__ __forceinline__ int umma_exp_of(int mag, double) {
  const int ex = mag >> 20;
  return ex == 0x7ff ? kUmmaNonFinite : ex == 0 ? 0 : ex - 1023 + 3;
}
__device__ __forceinline__ int umma_exp_of(int mag, dd) {
  const int ex = mag >> 23;
  return ex == 0xff ? kUmmaNonFinite : ex == 0 ? 0 : ex - 127 + 2;
}
// x 2^(8 ND - e) rounded to an integer
__device__ __forceinline__ long long umma_fixed(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const int sh = (ex ? ex : 1) - 1075 + 64 - e;
  unsigned long long v = 0;
  if (sh >= 0) v = m << (sh & 63);
  else if (sh > -64) v = (m + (1ull << (-sh - 1))) >> (-sh);
  return (long long)b < 0 ? -(long long)v : (long long)v;
}
__device__ __forceinline__ long long umma_fixed_f(float x, int e) {
  const uint32_t b = __float_as_uint(x);
  const int ex = (int)(b >> 23) & 0xff;
  const uint32_t m = (b & 0x7fffffu) | (ex ? 0x800000u : 0u);
  const int sh = (ex ? ex : 1) - 150 + 56 - e;
  unsigned long long v = 0;
  if (sh >= 0) v = (unsigned long long)m << (sh & 63);
  else if (sh > -32) v = (m + (1u << (-sh - 1))) >> (-sh);
  return (int)b < 0 ? -(long long)v : (long long)v;
}
__device__ __forceinline__ long long umma_fixed(dd x, int e) { return umma_fixed_f(x.hi, e) + umma_fixed_f(x.lo, e); }

// Eight consecutive k of one row (or column) cut into digits: writes one 16-byte
// core row per digit, blocks `bstride` elements apart.  The balanced digits are the
// bytes of X + sum 128 256^b, less 128; a byte under the exponent bits of a power
// of two is a float after one subtraction, already scaled by 2^(-8t).
template <typename T>
__device__ __forceinline__ void umma_split8(const T* x, int e, __nv_bfloat16* out, size_t bstride) {
  constexpr int ND = UmmaDigits<T>::n;
  uint32_t lo[8], hi[8];
  const bool ok = e != kUmmaNonFinite;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const unsigned long long y = (unsigned long long)(ok ? umma_fixed(x[q], e) : 0ll) +
                                 (ND == 8 ? 0x8080808080808080ull : 0x0080808080808080ull);
    lo[q] = (uint32_t)y;
    hi[q] = (uint32_t)(y >> 32);
  }
#pragma unroll
  for (int t = 0; t < ND; ++t) {
    const int byte = ND - 1 - t;                       // of X: its top digit first
    const uint32_t magic = (uint32_t)(150 - 8 * t) << 23;
    // 2^23 2^(-8t) + byte 2^(-8t); the top digit of seven may need a ninth bit
    const uint32_t sel = (ND == 7 && t == 0) ? 0x7632u : (0x7640u | (uint32_t)(byte & 3));
    const float off = __uint_as_float(magic) * (1.0f + 128.0f / 8388608.0f);
    float dg[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) dg[q] = __uint_as_float(__byte_perm(byte >= 4 ? hi[q] : lo[q], magic, sel)) - off;
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const __nv_bfloat162 p2 = __floats2bfloat162_rn(dg[2 * q], dg[2 * q + 1]);  // exact: 8-bit digits
      w[q] = *reinterpret_cast<const uint32_t*>(&p2);
    }
    *reinterpret_cast<uint4*>(out + (size_t)t * bstride) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Exponents of the logical rows of an operand (R x Kd, padded to Rp rows).  TR:
// logical row r is column r of X (X[k * ldx + r]); else row r.  Ends with a barrier.
template <bool TR, typename T>
__device__ void umma_row_exponents(int R, int Kd, const T* X, int ldx, int Rp, int* ex) {
  const int tid = threadIdx.x, warp_id = tid >> 5, lane_id = tid & 31;
  constexpr int nw = kThreads / 32;
  if (!TR) {
    for (int r = warp_id; r < Rp; r += nw) {
      int mag = 0;
      if (r < R)
        for (int k = lane_id; k < Kd; k += 32) mag = max(mag, umma_mag(X[(size_t)r * ldx + k]));
      mag = __reduce_max_sync(0xffffffffu, mag);
      if (lane_id == 0) ex[r] = umma_exp_of(mag, T());
    }
  } else {
    if (Kd <= 32) {
      // few k (a rank-k update): one thread per row, no exchange between warps
      for (int r = tid; r < Rp; r += kThreads) {
        int mag = 0;
        if (r < R) {
#pragma unroll 8
          for (int k = 0; k < Kd; ++k) mag = max(mag, umma_mag(X[(size_t)k * ldx + r]));
        }
        ex[r] = umma_exp_of(mag, T());
      }
      __syncthreads();
      return;
    }
    // the warps share the k range, each thread one column of a 32-wide strip
    for (int r = tid; r < Rp; r += kThreads) ex[r] = 0;
    __syncthreads();
    for (int r0 = 0; r0 < R; r0 += 32) {
      const int r = r0 + lane_id;
      int mag = 0;
      if (r < R) {
        int k = warp_id;
        for (; k + 7 * nw < Kd; k += 8 * nw) {
          int m[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) m[q] = umma_mag(X[(size_t)(k + q * nw) * ldx + r]);
#pragma unroll
          for (int q = 0; q < 8; ++q) mag = max(mag, m[q]);
        }
#pragma unroll 4
        for (; k < Kd; k += nw) mag = max(mag, umma_mag(X[(size_t)k * ldx + r]));
        if (mag) atomicMax(ex + r, mag);
      }
    }
    __syncthreads();
    for (int r = tid; r < Rp; r += kThreads) ex[r] = umma_exp_of(ex[r], T());
  }
  __syncthreads();
}

// Digit planes of op(A) (row tiles of umma_rows(M) rows) or of op(B)^T (rows =
// columns of op(B), tiles of kUmmaNT): P[(tile * nkc + kc) * ND + t] is a block of
// `tile_rows` x 16.  TR: the logical row r of the operand is column r of X
// (X[k * ldx + r]); else row r (X[r * ldx + k]).  Eight neighbouring threads write
// one 128-byte core matrix.
template <bool TR, typename T>
__device__ void umma_planes(int R, int Kd, const T* X, int ldx, int Rp, int Kp, int tile_rows, const int* ex,
                            __nv_bfloat16* P) {
  constexpr int ND = UmmaDigits<T>::n;
  const int nkc = Kp / kUmmaK, kg8 = Kp / 8;
  const size_t blk = (size_t)tile_rows * kUmmaK;
  const int items = Rp * kg8;
  auto where = [&](int e, int& r, int& g) {
    if (TR) {
      g = e / Rp;
      r = e - g * Rp;
    } else {
      const int h = e >> 3;
      g = h % kg8;
      r = (h / kg8) * 8 + (e & 7);
    }
  };
  auto fetch = [&](int r, int g, T (&x)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = 8 * g + q;
      x[q] = (r < R && k < Kd) ? (TR ? X[(size_t)k * ldx + r] : X[(size_t)r * ldx + k]) : T{};
    }
  };
  // the next item's loads are in flight while this one is cut
  int e = threadIdx.x, r = 0, g = 0;
  T x[8];
  if (e < items) {
    where(e, r, g);
    fetch(r, g, x);
  }
  while (e < items) {
    T y[8];
    const int en = e + kThreads;
    int rn = 0, gn = 0;
    if (en < items) {
      where(en, rn, gn);
      fetch(rn, gn, y);
    }
    const int tile = r / tile_rows, rr = r - tile * tile_rows, kc = g >> 1;
    __nv_bfloat16* out = P + ((size_t)tile * nkc + kc) * ND * blk + umma_core_off(rr, (g & 1) * 8);
    umma_split8<T>(x, ex[r], out, blk);
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = y[q];
    e = en;
    r = rn;
    g = gn;
  }
}

// ---- diagonals to results ------------------------------------------------------
// sum_d v_d 2^e
__device__ __forceinline__ dd umma_combine(const float (&v)[kPlaneDigits], int e) {
  const dd s1 = two_sum(v[0], v[1]), s2 = two_sum(v[2], v[3]);
  const float tail = v[4] + (v[5] + v[6]);
  dd s = two_sum(s1.hi, s2.hi);
  s = two_sum(s.hi, s.lo + ((s1.lo + s2.lo) + tail));
  // 2^e as two float factors
  const int ec = max(-250, min(250, e)), e1 = ec / 2, e2 = ec - e1;
  const float f1 = __int_as_float((127 + e1) << 23), f2 = __int_as_float((127 + e2) << 23);
  s.hi = s.hi * f1 * f2;
  s.lo = s.lo * f1 * f2;
  if (e > 2000) s = {__int_as_float(0x7fc00000), 0.f};
  return s;
}
// For FP64 the eight diagonals make one integer T = sum_d V_d 2^(8 (7-d)), V_d =
// v_d 2^(8d), of at most 82 bits; it is normalised and rounded to 53 bits in
// integer arithmetic (a warp's FP64 instruction costs 65 cycles of its scheduler's
// FP64 unit, these thirty integer ones about as many issue slots).
__device__ __forceinline__ double umma_combine(const float (&v)[kPlaneDigits64], int e) {
  long long h = __float2int_rn(v[0]), l = __float2int_rn(v[4] * 4294967296.f);
  h = h * 256 + __float2int_rn(v[1] * 256.f);
  h = h * 256 + __float2int_rn(v[2] * 65536.f);
  h = h * 256 + __float2int_rn(v[3] * 16777216.f);
  l = l * 256 + __float2int_rn(v[5] * 1099511627776.f);
  l = l * 256 + __float2int_rn(v[6] * 281474976710656.f);
  l = l * 256 + __float2int_rn(v[7] * 72057594037927936.f);
  h += l >> 32;
  uint32_t w = (uint32_t)l;
  const bool neg = h < 0;
  if (neg) {
    h = ~h;
    w = 0u - w;
    if (w == 0u) ++h;
  }
  unsigned long long m = (unsigned long long)h;
  int ex = e - 56 + 32 + 63 + 1023;  // biased exponent of bit 63 of m
  if (!(m >> 32)) {
    m = (m << 32) | w;
    w = 0u;
    ex -= 32;
    if (!(m >> 32)) { m <<= 32; ex -= 32; }
  }
  const int s = __clz((int)(m >> 32));
  m = s ? (m << s) | (w >> (32 - s)) : m;
  ex -= s;
  m += 0x400ull;                        // round at bit 11
  if (m < 0x400ull) { m = 0x8000000000000000ull | (m >> 1); ++ex; }
  unsigned long long bits = ((unsigned long long)(uint32_t)ex << 52) | ((m >> 11) & 0xfffffffffffffull);
  if (ex <= 0 || !(m >> 63)) bits = 0ull;
  else if (ex >= 2047) bits = 0x7ff0000000000000ull;
  if (e > 8000) bits = 0x7ff8000000000000ull;
  return __longlong_as_double((long long)(bits | (neg ? 1ull << 63 : 0ull)));
}

__device__ __forceinline__ uint4 umma_pack(double a, double b) {
  return make_uint4((uint32_t)__double2loint(a), (uint32_t)__double2hiint(a), (uint32_t)__double2loint(b),
                    (uint32_t)__double2hiint(b));
}
__device__ __forceinline__ uint4 umma_pack(dd a, dd b) {
  return make_uint4(__float_as_uint(a.hi), __float_as_uint(a.lo), __float_as_uint(b.hi), __float_as_uint(b.lo));
}

// C (+)= op(A) op(B), M x Nc, inner dimension Kd, FP64 or float-pair operands
// (global, shared or L2-resident), on the tensor cores.  All threads of the CTA
// call it.  ps: the plane buffers and tensor maps, made for M rows; ca, cb: a
// prepared constant operand (kCpEA ...) or -1; expA, expB: shared, umma_pad'ed M and
// Nc ints.  C must not alias A or B.
template <typename T>
__device__ __noinline__ void gemm_umma(bool ta, bool tb, bool acc, int M, int Nc, int Kd, const T* A, int lda,
                                       const T* B, int ldb, T* C, int ldc, const PlaneSet* ps, int* expA_s,
                                       int* expB_s, Umma U, int ca, int cb) {
  constexpr int ND = UmmaDigits<T>::n;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  expA_s = as_shared(expA_s);
  expB_s = as_shared(expB_s);
  U.bar = as_shared(U.bar);
  U.tmem_slot = as_shared(U.tmem_slot);
  const int R = umma_rows(M), nmt = umma_row_tiles(M);
  const int Mp = R * nmt, Np = umma_pad(Nc, kUmmaNT), Kp = umma_pad(Kd, kUmmaK);
  const int nnt = Np / kUmmaNT, nkc = Kp / kUmmaK;
  const uint32_t blockA = (uint32_t)R * kUmmaK * 2, blockB = kUmmaNT * kUmmaK * 2;
  const uint32_t stage_bytes = ND * (blockA + blockB);
  const int nst = min(kUmmaStages, (int)(U.stage_bytes / stage_bytes));
  // after a wait gave up (in this or an earlier product of the kernel) the
  // products are skipped: the results are void and the host reports it
  // (the chain's error word is shared with the peer flavor's CTA: thread 0
  // reads it once for the whole CTA)
  if (tid == 0) *umma_calls(U) += 1u;
  if (__syncthreads_or(tid == 0 && U.err && (*(volatile int*)U.err & 2))) return;
  // earlier generic writes of the staging area (other products) before the
  // copies of this one
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  const CUtensorMap* tmA = ca >= 0 ? &ps->tm_cp[ca] : &ps->tm_pl[0];
  const CUtensorMap* tmB = cb >= 0 ? &ps->tm_cp[cb] : &ps->tm_pl[1];
  const int* expA = ca >= 0 ? ps->cex[ca] : expA_s;
  const int* expB = cb >= 0 ? ps->cex[cb] : expB_s;
  // both operands by the same code (a right operand's logical rows are its columns)
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    if ((side ? cb : ca) >= 0) continue;
    const T* X = side ? B : A;
    const int n = side ? Nc : M, ldx = side ? ldb : lda, np = side ? Np : Mp, tile = side ? kUmmaNT : R;
    int* ex = side ? expB_s : expA_s;
    __nv_bfloat16* P = (__nv_bfloat16*)ps->scratch + (side ? ps->boff : 0);
    if (side ? !tb : ta) {
      umma_row_exponents<true>(n, Kd, X, ldx, np, ex);
      umma_planes<true>(n, Kd, X, ldx, np, Kp, tile, ex, P);
    } else {
      umma_row_exponents<false>(n, Kd, X, ldx, np, ex);
      umma_planes<false>(n, Kd, X, ldx, np, Kp, tile, ex, P);
    }
  }
  // the planes are read by the bulk copies (async proxy)
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncthreads();
  const uint32_t tmem = *U.tmem_slot;
  // 16-byte stores of two neighbouring outputs where C's rows allow them
  const bool vec = ((reinterpret_cast<uintptr_t>(C) | ((uintptr_t)ldc * sizeof(T))) & 15) == 0;
  // Chunk sequence: tiles (mt, nt) in order, within a tile its k chunks; a tile's
  // chunks are accumulated in segments of kUmmaKSeg.  Chunk c uses stage c % nst for
  // the (c / nst)-th time in this product; every barrier has at most one phase in
  // flight when it is waited on (a stage is refilled only after its MMAs are done,
  // multiplied only after its copy landed), and a product ends with all of them
  // complete, so parity waits are sound.  par: the barriers' next parities (shared,
  // continued across products): bits 0..2 copies, 3..5 MMAs, 6 accumulators.
  const int segc = kUmmaKSeg / kUmmaK, nseg = (nkc + segc - 1) / segc;
  const int nch = nmt * nnt * nkc, n_seg = nmt * nnt * nseg;
  const uint32_t par = *umma_book(U);
  uint64_t* bar_full = U.bar;
  uint64_t* bar_mma = U.bar + kUmmaStages;
  bool live = true;  // no wait of this warp has given up
  auto gave_up = [&](int kind, int g, uint64_t* bar) {
    if (live && lane == 0 && U.where && atomicCAS(U.where, 0, kind) == 0) {
      unsigned long long w = 0;
      asm volatile("ld.shared.b64 %0, [%1];" : "=l"(w) : "r"(smem_u32(bar)));
      U.where[1] = g;
      U.where[2] = nch;
      U.where[3] = (int)*umma_calls(U);
      U.where[4] = (int)(w & 0xffffffffu);
      U.where[5] = (int)(w >> 32);
    }
    live = false;
  };
  int c = 0, cst = 0, cuse = 0;          // warp 1: next chunk to copy, its stage and use
  int crowA = 0, crowB = 0, ckc = 0, cnt = 0;  // ... its rows in the planes, k chunk and column tile
  int m = 0, mst = 0, muse = 0;          // warp 0: next chunk to multiply
  const int rowsA = (int)(ND * blockA / (2 * kPlaneRowElems)), rowsB = (int)(ND * blockB / (2 * kPlaneRowElems));
  const uint32_t stage0 = smem_u32(U.stage);
  bool dead = false;
  int mt = 0, nt = 0, seg = 0;
  for (int sg = 0; sg < n_seg && !dead; ++sg) {
    const int kc0 = seg * segc, kc1 = min(nkc, kc0 + segc);
    const int end = (mt * nnt + nt) * nkc + kc1;  // chunks up to the end of this segment
    if (warp == 1) {
      // copies of this segment and, while its MMAs drain, of the next one's first chunks
      const int ahead = min(nch, end + nst);
      while (live && c < ahead) {
        if (cuse > 0 && !mbar_wait(bar_mma + cst, ((par >> (3 + cst)) ^ (cuse - 1)) & 1, U.limit)) {
          gave_up(2, c, bar_mma + cst);
          break;
        }
        unsigned char* dst = U.stage + (size_t)cst * stage_bytes;
        if (elect_one()) {
          mbar_expect_tx(bar_full + cst, stage_bytes);
          tma_load_block(dst, tmA, crowA, bar_full + cst);
          tma_load_block(dst + ND * blockA, tmB, crowB, bar_full + cst);
        }
        __syncwarp();
        ++c;
        if (++cst == nst) { cst = 0; ++cuse; }
        crowA += rowsA;
        crowB += rowsB;
        if (++ckc == nkc) {
          ckc = 0;
          if (++cnt == nnt) { cnt = 0; crowB = 0; }
          else crowA -= nkc * rowsA;  // the next column tile reads the same row tile again
        }
      }
    } else if (warp == 0) {
      for (int kc = kc0; live && kc < kc1; ++kc) {
        bool landed = mbar_wait(bar_full + mst, ((par >> mst) ^ muse) & 1, U.limit);
        // test hook: a wait that cannot end (its barrier's phase 0 never completes)
        if (landed && U.stall && m == 0) landed = mbar_wait(umma_never(U), 0u, U.limit);
        if (!landed) {
          gave_up(1, m, bar_full + mst);
          break;
        }
        tc_fence_after();
        const uint32_t sa = stage0 + (uint32_t)mst * stage_bytes;
        const uint64_t ad = umma_sdesc(sa, 128, 256), bd = umma_sdesc(sa + ND * blockA, 128, 256);
        if (elect_one()) {
#pragma unroll
          for (int t = 0; t < ND; ++t)
            umma_bf16(tmem + t * kUmmaNT, ad + (uint64_t)(t * (blockA >> 4)), bd,
                      umma_idesc(kUmmaM, kUmmaNT * (ND - t)), !(kc == kc0 && t == 0));
          umma_commit(bar_mma + mst);
          if (kc + 1 == kc1) umma_commit(umma_acc(U));
        }
        __syncwarp();
        ++m;
        if (++mst == nst) { mst = 0; ++muse; }
      }
    }
    // epilogue of a tile segment: all its MMAs done
    if (live && !mbar_wait(umma_acc(U), ((par >> 6) ^ sg) & 1, U.limit)) gave_up(3, end - 1, umma_acc(U));
    tc_fence_after();
    if (live) {
      const bool add = acc || seg > 0;
      // warp w reads lanes 32 (w % 4) .. + 31 (tile rows) and the column half w / 4
      const int rloc = (warp & 3) * 32 + lane;
      const int row = mt * R + rloc;
      const bool live_row = rloc < R && row < M;
      if ((warp & 3) * 32 < R) {
        const int eA = live_row ? expA[row] : 0;
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
#pragma unroll 1
        for (int c0 = (warp >> 2) * (kUmmaNT / 2); c0 < (warp >> 2) * (kUmmaNT / 2) + kUmmaNT / 2; c0 += 4) {
          if (nt * kUmmaNT + c0 >= Nc) break;
          T* cp = C + (size_t)row * ldc + nt * kUmmaNT + c0;
          T old[4];
          if (add && live_row) {
#pragma unroll
            for (int q = 0; q < 4; ++q) old[q] = (nt * kUmmaNT + c0 + q < Nc) ? cp[q] : T{};
          }
          float v[ND][4];
#pragma unroll
          for (int d = 0; d < ND; ++d) tmem_ld4(tmem + lane_base + d * kUmmaNT + c0, v[d]);
          tmem_ld_wait();
          if (live_row) {
            T sum[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int col = nt * kUmmaNT + c0 + q;
              float d[ND];
#pragma unroll
              for (int t = 0; t < ND; ++t) d[t] = v[t][q];
              sum[q] = umma_combine(d, eA + expB[col] - 16);
              if (add) sum[q] = radd(old[q], sum[q]);
            }
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
              const int col = nt * kUmmaNT + c0 + q;
              if (vec && col + 1 < Nc) {
                *reinterpret_cast<uint4*>(cp + q) = umma_pack(sum[q], sum[q + 1]);
              } else {
                if (col < Nc) cp[q] = sum[q];
                if (col + 1 < Nc) cp[q + 1] = sum[q + 1];
              }
            }
          }
        }
      }
    }
    if (++seg == nseg) {
      seg = 0;
      if (++nt == nnt) { nt = 0; ++mt; }
    }
    // the accumulators are overwritten by the next segment's first MMAs
    tc_fence_before();
    dead = __syncthreads_or(!live);
    tc_fence_after();
  }
  // A wait gave up: what is in flight is drained (with the default limit) before the
  // staging buffers and the tensor memory are used again.
  if (dead) {
    uint32_t* book = umma_book(U);
    if (warp == 1 && lane == 0) book[1] = (uint32_t)c;
    if (warp == 0 && lane == 0) book[2] = (uint32_t)m;
    __syncthreads();
    if (tid == 0) {
      for (int q = max(0, (int)book[1] - nst); q < (int)book[1]; ++q)
        mbar_wait(bar_full + q % nst, ((par >> (q % nst)) ^ (q / nst)) & 1, kUmmaWaitCycles);
      for (int q = max(0, (int)book[2] - nst); q < (int)book[2]; ++q)
        mbar_wait(bar_mma + q % nst, ((par >> (3 + q % nst)) ^ (q / nst)) & 1, kUmmaWaitCycles);
      // the products after a wait gave up are skipped: the parities are not used again
      if (U.err) atomicOr(U.err, 2);
    }
  } else if (tid == 0) {
    // every copy and MMA of the product is complete: next parities
    uint32_t p = par ^ ((uint32_t)(n_seg & 1) << 6);
    bool done = true;
    for (int q = 0; q < nst && q < nch; ++q) {
      const uint32_t uses = (uint32_t)((nch - q + nst - 1) / nst);
      done = done && mbar_wait(bar_mma + q, ((par >> (3 + q)) ^ (uses - 1)) & 1, kUmmaWaitCycles);
      p ^= ((uses & 1u) << q) | ((uses & 1u) << (3 + q));
    }
    *umma_book(U) = p;
    if (!done && U.err) atomicOr(U.err, 2);
  }
  // the staging buffers are reused by generic loads and stores after the product
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
}
