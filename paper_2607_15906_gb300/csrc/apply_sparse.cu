// H psi (Eq. 3) with the energy epilogue (Eq. 1) for states with few
// nonzero amplitudes, by scattering from the nonzero source amplitudes.
//
// The staged kernel (apply_tiled.cu) gives every thread an output octet and
// walks the groups of a piece, skipping a group only where the whole source
// octet is zero; in a state confined to a particle-number sector (1.5 % of
// the amplitudes nonzero at 24 qubits, in 8.9 % of the octets) most lanes of
// a warp idle while a few work.  This kernel turns the loop around:
//
//  * a listing pass writes the nonzero amplitudes (index, value) in index
//    order, and the first entry of every tile;
//  * a block (one per SM) owns an output tile t of 2^kSpLB amplitudes and
//    accumulates it in shared memory.  Its work units are (piece, span of
//    chunks): 32 consecutive nonzero amplitudes, one per lane, of the piece's
//    source tile u = t ^ (x >> kSpLB), against the piece's groups.  Units are
//    numbered piece by piece from a per-tile scan and claimed by the warps;
//  * the host splits every LUT group into cases (see SpHead): a case applies
//    where up to three parities of the output index are zero.  A head of 32
//    cases has its 4 x 32 parities from three 16-byte table reads, and the
//    cases that apply to a lane's amplitude are one word, so a lane spends
//    instructions only on nonzero products: about a sixth of the (amplitude,
//    case) pairs of a sector-confined state.  Testing every (amplitude, group)
//    pair by population counts, as before, took two thirds of the issue slots;
//  * a case whose parities the tile's bits alone make one is dead in the whole
//    tile; pieces with only dead cases get no units there (half of the units
//    at 24 qubits, three fifths at 28);
//  * term-list groups take their weight from tables over index ranges (SpTab),
//    summed in integers; the diagonal group and the identity are units over
//    the own tile's amplitudes;
//  * a product is added to the accumulator, in fixed point, with shared-memory
//    integer atomics.  A warp whose amplitudes are all real (every state of a
//    real H and pool) forms no imaginary products;
//  * after the last unit, lanes over the nonzero amplitudes of the own tile
//    take the energy partials, and the whole tile (zeros included) is streamed
//    to H psi.
//
// The order in which products reach an accumulator element is not fixed, but
// integer addition does not depend on it: H psi, E and everything computed
// from them are reproducible bit for bit from run to run.
//
// What bounds it (24 qubits, 233,867 nonzero amplitudes, 2.3e8 nonzero
// products): the latency of the table reads and of a unit's start, with 54 % of
// the issue slots busy (7e8 warp instructions); the shared-memory atomics'
// wavefronts take 0.37 ms.  2.29 -> 1.1 ms (complex64), 6.2 -> 1.9 ms
// (complex128), 18 -> 9 ms at 28 qubits (where the tables of 32,768 tiles are a
// fifth), against the kernel that tested every pair.
//
// The kernel is launched with the staged one; each returns at once unless
// the count of nonzero amplitudes selects it, so the choice needs no host
// round trip.
#include <algorithm>
#include <cstdlib>
#include <mutex>
#include <vector>

#include "device.cuh"
#include "internal.h"

namespace gocp {

namespace {

constexpr int kAmpBlock = 256;   // listing passes: one amplitude word (4 octets) per thread
constexpr uint32_t kUnitBatch = 4;   // scatter work units per claim, at most

// One block of 1024 threads (64 registers) per SM in both precisions.
constexpr int kSpThreads = 1024;

template <typename R>
__device__ __forceinline__ void load_octet(const C_t<R>* __restrict__ psi, uint32_t octet, C_t<R> (&v)[kAmpsH]) {
  if (sizeof(R) == 4) {
    const float4* p = reinterpret_cast<const float4*>(psi) + (size_t)octet * 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 f = __ldg(p + q);
      v[2 * q] = cmake<R>((R)f.x, (R)f.y);
      v[2 * q + 1] = cmake<R>((R)f.z, (R)f.w);
    }
  } else {
    const double2* p = reinterpret_cast<const double2*>(psi) + (size_t)octet * 8;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const double2 f = __ldg(p + q);
      v[q] = cmake<R>((R)f.x, (R)f.y);
    }
  }
}

template <typename R>
__device__ __forceinline__ uint32_t nonzero_members(const C_t<R> (&v)[kAmpsH]) {
  uint32_t nz = 0;
#pragma unroll
  for (int m = 0; m < kAmpsH; ++m) nz |= (uint32_t)(v[m].x != R(0) || v[m].y != R(0)) << m;
  return nz;
}

// Members of octet o nonzero in psi or (when set) psi2.
template <typename R>
__device__ __forceinline__ uint32_t octet_nonzero2(const C_t<R>* __restrict__ psi, const C_t<R>* __restrict__ psi2,
                                                   uint32_t o) {
  C_t<R> v[kAmpsH];
  load_octet<R>(psi, o, v);
  uint32_t nz = nonzero_members<R>(v);
  if (psi2) {
    load_octet<R>(psi2, o, v);
    nz |= nonzero_members<R>(v);
  }
  return nz;
}

// Amplitude word w: bit 8j + i = member i of octet 4w + j nonzero in psi or
// (when set) psi2, read only from the octets the octet mask marks live.
template <typename R>
__device__ __forceinline__ uint32_t amp_word(const C_t<R>* __restrict__ psi, const C_t<R>* __restrict__ psi2,
                                             const uint32_t* __restrict__ mask, uint32_t w) {
  const uint32_t mb = (mask[w >> 3] >> ((w & 7u) * 4u)) & 0xFu;
  uint32_t word = 0;
#pragma unroll
  for (uint32_t j = 0; j < 4; ++j)
    if ((mb >> j) & 1u) word |= octet_nonzero2<R>(psi, psi2, 4u * w + j) << (8u * j);
  return word;
}

// counts[b] = the amplitudes nonzero in psi or psi2 in amplitude words
// kAmpBlock b .. kAmpBlock (b + 1) - 1 (one thread per word of 32).
template <typename R>
__global__ void __launch_bounds__(kAmpBlock)
k_amp_count(const C_t<R>* __restrict__ psi, const C_t<R>* __restrict__ psi2, const uint32_t* __restrict__ mask,
            uint32_t words, uint32_t* counts) {
  __shared__ uint32_t red[kAmpBlock / 32];
  const uint32_t w = blockIdx.x * kAmpBlock + threadIdx.x;
  uint32_t c = w < words ? __popc(amp_word<R>(psi, psi2, mask, w)) : 0u;
  for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int q = 0; q < kAmpBlock / 32; ++q) t += red[q];
    counts[blockIdx.x] = t;
  }
}

// counts[0..nb) -> exclusive prefix sums in place; *total = the sum (when
// set; and, when ring is set, the chain-list ring's base(slot) = the sum,
// count(slot) = count(first) = 0); sync (when set) = 0; *amax = 0 when set.  One block of 1024
// threads.  The sum reaches 2^32 only for a 32-qubit state with every
// amplitude nonzero; it is stored saturated at 2^32 - 1 (above every list
// capacity, so the list is not used), while every prefix, at most the sum
// less the last block's count, fits 32 bits.
__global__ void __launch_bounds__(1024)
k_amp_scan(uint32_t* counts, uint32_t nb, uint32_t* total, uint32_t* ring, uint32_t* sync, int slot, int first,
           unsigned long long* amax) {
  __shared__ uint32_t s[1024];
  __shared__ unsigned long long carry;
  if (threadIdx.x == 0) carry = 0;
  for (uint32_t base = 0; base < nb; base += 1024u) {
    const uint32_t i = base + threadIdx.x;
    const uint32_t v = i < nb ? counts[i] : 0u;
    s[threadIdx.x] = v;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {   // inclusive scan
      const uint32_t u = (int)threadIdx.x >= d ? s[threadIdx.x - d] : 0u;
      __syncthreads();
      s[threadIdx.x] += u;
      __syncthreads();
    }
    if (i < nb) counts[i] = (uint32_t)(carry + s[threadIdx.x] - v);
    __syncthreads();
    if (threadIdx.x == 0) carry += s[1023];
    __syncthreads();
  }
  if (sync)
    for (int w = threadIdx.x; w < kSyncWords; w += 1024) sync[w] = 0u;
  if (threadIdx.x == 0) {
    const uint32_t sum = carry > 0xffffffffull ? 0xffffffffu : (uint32_t)carry;
    if (total) *total = sum;
    if (amax) *amax = 0ull;
    if (ring) {
      ring[kRingBase(slot)] = sum;
      ring[kRingAdd(slot)] = 0u;
      ring[kRingAdd(first)] = 0u;
    }
  }
}

// Writes the index (and, when aval is set, the psi value) of every amplitude
// nonzero in psi or psi2, in index order, at the offsets of k_amp_scan;
// entries at or beyond cap are not stored.  With amask set, also writes
// amask[w] = amplitude word w (one bit per amplitude, zeros included).  With
// amax set, raises *amax to the largest |Re| or |Im| of the listed psi values
// (the bits of a non-negative double, which order as unsigned integers).
template <typename R>
__global__ void __launch_bounds__(kAmpBlock)
k_amp_list(const C_t<R>* __restrict__ psi, const C_t<R>* __restrict__ psi2, const uint32_t* __restrict__ mask,
           uint32_t words, const uint32_t* __restrict__ offs, uint32_t* aidx, C_t<R>* aval, uint32_t* amask,
           uint32_t cap, unsigned long long* amax) {
  __shared__ uint32_t red[kAmpBlock / 32];
  const uint32_t w = blockIdx.x * kAmpBlock + threadIdx.x;
  const uint32_t word = w < words ? amp_word<R>(psi, psi2, mask, w) : 0u;
  const uint32_t c = __popc(word);
  // exclusive scan over the block: lanes by shuffles, warps through red
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = c;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) red[warp] = incl;
  __syncthreads();
  uint32_t before = 0;
  for (int q = 0; q < warp; ++q) before += red[q];
  uint32_t at = offs[blockIdx.x] + before + incl - c;
  R big = R(0);
  for (uint32_t m = word; m; m &= m - 1u, ++at) {
    if (at >= cap) break;
    const uint32_t k = 32u * w + (uint32_t)(__ffs(m) - 1);
    aidx[at] = k;
    if (aval) {
      const C_t<R> v = psi[k];
      aval[at] = v;
      big = fmax(big, fmax(fabs(v.x), fabs(v.y)));
    }
  }
  if (amask && w < words) amask[w] = word;
  if (amax) {
    for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
    if (lane == 0 && big > R(0)) atomicMax(amax, (unsigned long long)__double_as_longlong((double)big));
  }
}

// off[u] = first stored entry with index >> shift >= u, u = 0 .. ntiles
// (off[ntiles] = the number of stored entries).
__global__ void __launch_bounds__(256)
k_tile_offsets(const uint32_t* __restrict__ idx, const uint32_t* __restrict__ len, uint32_t cap, uint32_t ntiles,
               int shift, uint32_t* off) {
  const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u > ntiles) return;
  uint32_t lo = 0, hi = min(*len, cap);
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if ((idx[mid] >> shift) < u) lo = mid + 1;
    else hi = mid;
  }
  off[u] = lo;
}

// Fixed-point accumulation.  A product p is added as the integer
// round(p 2^F) (the amplitudes are scaled by 2^F once, see below), so the
// sum is exact integer arithmetic: the same in any order of the atomics,
// and the result is bit-for-bit reproducible.  F is chosen per call so that
// the sum of the magnitudes of all contributions to one output component --
// at most hbound x 2 max(|Re psi|, |Im psi|) -- stays below 2^62 (in split form
// 2^46, see fx_put): no partial sum can overflow.  For complex64, F also keeps
// every off-diagonal product below 2^30, so that it converts with a 32-bit
// instruction; its rounding,
// at most 2^-(F+1), is then about 1e-9 of the largest possible product, and
// an entry of H psi collects it from at most a few thousand products.  For
// complex128 the rounding is at most 2^-(F+1) with F near 62 - log2 of the
// bound, far below the FP64 rounding of the products.
//
// The tile's accumulator is four planes of 32-bit words, one word per
// amplitude of the tile: low and high half of the real part, low and high
// half of the imaginary part.  An atomic's bank is then the amplitude's low
// five bits whatever the half, so a warp's 32 scattered adds spread over all
// 32 banks (64-bit words side by side would put the low halves on 16).
constexpr uint32_t kPlane = 4u * kSpTile;                                 // bytes of a plane
constexpr uint32_t kRe = 0u, kIm = 2u * kPlane;                           // low planes; the high plane follows each
constexpr uint32_t kAccBytes = 4u * kPlane;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory adds by 32-bit address and a constant offset.
template <uint32_t OFF>
__device__ __forceinline__ void red_add(uint32_t at, uint32_t v) {
  asm volatile("red.shared.add.u32 [%0+%2], %1;" ::"r"(at), "r"(v), "n"(OFF) : "memory");
}
template <uint32_t OFF>
__device__ __forceinline__ uint32_t atom_add(uint32_t at, uint32_t v) {
  uint32_t old;
  asm volatile("atom.shared.add.u32 %0, [%1+%3], %2;" : "=r"(old) : "r"(at), "r"(v), "n"(OFF) : "memory");
  return old;
}

// One 64-bit accumulator component at byte offset `at` of its low plane.
__device__ __forceinline__ long long acc_get(const uint8_t* acc, uint32_t at) {
  return (long long)(((unsigned long long)*reinterpret_cast<const uint32_t*>(acc + at + kPlane) << 32) |
                     *reinterpret_cast<const uint32_t*>(acc + at));
}
__device__ __forceinline__ void acc_set(uint8_t* acc, uint32_t at, long long v) {
  *reinterpret_cast<uint32_t*>(acc + at) = (uint32_t)(unsigned long long)v;
  *reinterpret_cast<uint32_t*>(acc + at + kPlane) = (uint32_t)((unsigned long long)v >> 32);
}

// Adds v to the component PL (kRe, kIm) of the amplitude at shared address at.
//
// Carry form (complex128): the low word's add, and the high word's plus the
// carry out of the low word, taken from the old value that atomic returns;
// exact modulo 2^64 in any order of the atomics (measured faster than one
// 64-bit atomic).
//
// Split form (complex64, products below 2^30): the low plane sums the low 16
// bits of each product (0 .. 65535) and the high plane the product shifted
// right by 16 (arithmetic, |.| <= 2^14), two independent adds with no carry
// between them.  With fewer than 65536 products per word (one per
// off-diagonal group, and the diagonal's) the low half cannot wrap,
// low < 2^16 * 65536 = 2^32, and the high half holds the word's total above
// bit 16, |high| < 2^31.  The value is high * 2^16 + low, formed exactly once every
// product has been added.
template <bool SPLIT, uint32_t PL>
__device__ __forceinline__ void fx_put(uint32_t at, long long v) {
  const uint32_t lo = (uint32_t)(unsigned long long)v;
  if constexpr (SPLIT) {
    red_add<PL>(at, lo & 0xFFFFu);
    red_add<PL + kPlane>(at, (uint32_t)((int)lo >> 16));
  } else {
    const uint32_t old = atom_add<PL>(at, lo);
    red_add<PL + kPlane>(at, (uint32_t)((unsigned long long)v >> 32) + (uint32_t)(old + lo < old));
  }
}

// A product of more than 32 bits (the diagonal's).  In split form: its low 16
// bits into the low plane, the bits above into the high plane modulo 2^32;
// only the word's total has to fit there, and it is below 2^46 by the choice
// of F.
template <bool SPLIT, uint32_t PL>
__device__ __forceinline__ void fx_put_wide(uint32_t at, long long v) {
  if constexpr (SPLIT) {
    red_add<PL>(at, (uint32_t)v & 0xFFFFu);
    red_add<PL + kPlane>(at, (uint32_t)(unsigned long long)(v >> 16));
  } else {
    fx_put<false, PL>(at, v);
  }
}

// A scaled product as an integer.  complex64: every off-diagonal product is
// below 2^30 by the choice of F, so a 32-bit conversion suffices (the 64-bit
// conversions run on the FP64 pipe, narrow on this part).
__device__ __forceinline__ long long fx_prod(float v) { return (long long)__float2int_rn(v); }

// An accumulator value back in R (zeros, most of a sector state's tile,
// skip the conversion).
template <typename R>
__device__ __forceinline__ R fx_val(long long a) {
  if (a == 0ll) return R(0);
  return sizeof(R) == 4 ? (R)__ll2float_rn(a) : (R)__ll2double_rn(a);
}

// complex128 products in integers.  The weights (LUT entries and term-list
// weights) are stored as d_q = round(d 2^Fd) (|d_q| < 2^62) and the lane's
// amplitude components as v_q = round(v 2^(F + 63 - Fd)) (|v_q| < 2^63:
// |v| 2^F < 2^61 / hbound and hbound >= dmax >= 2^(61 - Fd)); their product
// shifted right by 63 is round(d v 2^F), the fixed-point product, formed
// exactly and rounded once.  FP64 instructions run on a pipe about 1/64 the
// width of FP32 here; these are integer instructions.
__device__ __forceinline__ long long q_mul(long long a, long long b) {
  const unsigned long long hi = (unsigned long long)__mul64hi(a, b);
  const unsigned long long lo = (unsigned long long)a * (unsigned long long)b;
  return (long long)((hi << 1) + (lo >> 63) + ((lo >> 62) & 1ull));
}

// Not a number, or infinite (on the bits).
__device__ __forceinline__ bool not_finite(float v) { return (__float_as_uint(v) & 0x7F800000u) == 0x7F800000u; }
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7FF00000) == 0x7FF00000; }

// The lane's amplitude in the form its products take: scaled by 2^F
// (complex64), or as v_q (complex128, see q_mul).
template <typename R> struct SpVal;
template <> struct SpVal<float> { using T = float; };
template <> struct SpVal<double> { using T = long long; };

__device__ __forceinline__ long long sp_product(float d, float v) { return fx_prod(d * v); }
__device__ __forceinline__ long long sp_product(long long d, long long v) { return q_mul(d, v); }

// d negated by the top bit of s.
__device__ __forceinline__ float sp_signed(float d, uint32_t s) {
  return __uint_as_float(__float_as_uint(d) ^ (s & 0x80000000u));
}
__device__ __forceinline__ long long sp_signed(long long d, uint32_t s) {
  const long long m = (long long)((int)s >> 31);
  return (d ^ m) - m;
}

__device__ __forceinline__ SpItem<float> sp_item(const SpItem<float>* p) {
  const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
  return {__uint_as_float(v.x), v.y};
}
__device__ __forceinline__ SpItem<double> sp_item(const SpItem<double>* p) {
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
  return {(long long)(((unsigned long long)v.y << 32) | v.x), v.z, 0u};
}

// The cases `on` (bit 31 - g) of one head that apply to the lane's amplitude:
// weight and output offset, sign from sg, product, adds.  A lane walks its own
// cases, so no slot is spent on a case that does not apply to that lane.  CPLX
// false: every lane's amplitude has a zero imaginary part (checked by the
// warp), whose products are zero and are not formed.  acc_s: shared address
// of the accumulator.
template <typename R, bool SPLIT, bool CPLX>
__device__ __forceinline__ void sp_items(const SpItem<R>* __restrict__ it, uint32_t on, uint32_t sg, uint32_t k4,
                                         typename SpVal<R>::T vx, typename SpVal<R>::T vy, uint32_t acc_s) {
  while (on) {
    const int g = __clz(on);
    on &= ~(0x80000000u >> g);
    const SpItem<R> e = sp_item(it + g);
    const typename SpVal<R>::T d = sp_signed(e.w, sg << g);
    const uint32_t at = acc_s + (k4 ^ e.xo);
    fx_put<SPLIT, kRe>(at, sp_product(d, vx));
    if constexpr (CPLX) fx_put<SPLIT, kIm>(at, sp_product(d, vy));
  }
}

// The same for the term groups of one head: the weight from the tables (fixed
// point, summed in integers), s_tab the tile's parts of its groups.
template <typename R, bool SPLIT>
__device__ __forceinline__ void sp_tab_items(const SpTab<R>* __restrict__ tab, const typename SpWeight<R>::T* s_tab,
                                             const SpTables& T, uint32_t on, uint32_t sg, uint32_t kk,
                                             typename SpVal<R>::T vx, typename SpVal<R>::T vy, bool cplx,
                                             uint32_t acc_s) {
  using W = typename SpWeight<R>::T;
  const uint32_t klow = kk & (kSpTile - 1u);
  while (on) {
    const int g = __clz(on);
    on &= ~(0x80000000u >> g);
    const SpTab<R>* S = tab + g;
    W q = s_tab[g] + __ldg(S->fa + (klow & 31u)) + __ldg(S->fb + ((klow >> 5) & 15u)) + __ldg(S->fc + (klow >> 9));
    const uint4 h = __ldg(reinterpret_cast<const uint4*>(&S->xo));   // xo, x, rb, re
    for (uint32_t r = h.z; r < h.w; ++r) {
      const W v = __ldg(reinterpret_cast<const W*>(T.rw) + r);
      q += (__popc((kk ^ h.y) & __ldg(T.ry + r)) & 1) ? -v : v;
    }
    typename SpVal<R>::T d;
    if constexpr (sizeof(R) == 4) d = (float)q * __uint_as_float(h.x & 0xFFFF0000u);
    else d = q;
    d = sp_signed(d, sg << g);
    const uint32_t at = acc_s + ((4u * klow) ^ (h.x & 0xFFFFu));
    fx_put<SPLIT, kRe>(at, sp_product(d, vx));
    if (cplx) fx_put<SPLIT, kIm>(at, sp_product(d, vy));
  }
}

__device__ __forceinline__ uint4 xor4(const uint4 a, const uint4 b) {
  return make_uint4(a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w);
}

// The four parity words of head H at source index klow, with the tile's part
// b: for the head's 32 cases three loads and 12 XORs in place of 128
// population counts.
__device__ __forceinline__ uint4 head_words(const SpHead* __restrict__ H, uint32_t klow, const uint4 b) {
  return xor4(xor4(__ldg(H->ta + (klow & 31u)), __ldg(H->tb + ((klow >> 5) & 15u))),
              xor4(__ldg(H->tc + (klow >> 9)), b));
}

// The factor 0, 1 or 2 of a term-list group at output k (paired groups: 0 or 2).
__device__ __forceinline__ uint32_t pair_factor(uint32_t k, uint32_t delta, uint32_t neg) {
  if (!delta) return 1u;
  const uint32_t p = __popc(k & delta) & 1u;
  return (neg ? p : p ^ 1u) ? 2u : 0u;
}

// One term-list group: D(k) = sum_t w_t (-1)^popc(k & z_t), real terms
// [tb, tm), imaginary [tm, te); a paired group keeps one term of each pair
// and D = (1 + sigma (-1)^popc(k & delta)) E(k), the factor 0 or 2.  Called
// by every lane of the warp (the group is warp-uniform); kk = k'.
template <bool SPLIT>
__device__ __forceinline__ void sp_terms(const SpListGroup& G, const uint32_t* __restrict__ zs,
                                         const float* __restrict__ ws, uint32_t kk, float vx, float vy, bool valid,
                                         uint32_t acc_s) {
  const uint32_t k = kk ^ G.x, fz = pair_factor(k, G.delta, G.neg);
  if (!__any_sync(0xffffffffu, valid && fz != 0u)) return;
  float dr = 0.f, di = 0.f;
  for (uint32_t t = G.tb; t < G.tm; ++t) {
    const float w = __ldg(ws + t);
    dr += (__popc(k & __ldg(zs + t)) & 1) ? -w : w;
  }
  for (uint32_t t = G.tm; t < G.te; ++t) {
    const float w = __ldg(ws + t);
    di += (__popc(k & __ldg(zs + t)) & 1) ? -w : w;
  }
  const float f = fz == 2u ? 2.f : 1.f;
  const float a = dr * f, b = di * f;
  if (valid && fz != 0u && (a != 0.f || b != 0.f)) {
    const uint32_t at = acc_s + 4u * (k & (kSpTile - 1u));
    fx_put<SPLIT, kRe>(at, fx_prod(a * vx - b * vy));
    fx_put<SPLIT, kIm>(at, fx_prod(a * vy + b * vx));
  }
}

// complex128: the fixed-point weights wq summed exactly,
// D_q = (sum of all w_q) - 2 (sum of the w_q with odd parity), times the
// factor 0, 1 or 2, and the complex product in integers.
template <bool SPLIT>
__device__ __forceinline__ void sp_terms(const SpListGroup& G, const uint32_t* __restrict__ zs,
                                         const long long* __restrict__ wq, uint32_t kk, long long vx, long long vy,
                                         bool valid, uint32_t acc_s) {
  const uint32_t k = kk ^ G.x, fz = pair_factor(k, G.delta, G.neg);
  if (!__any_sync(0xffffffffu, valid && fz != 0u)) return;
  unsigned long long ar = 0ull, ai = 0ull, odr = 0ull, odi = 0ull;   // modulo 2^64; the results fit
  for (uint32_t t = G.tb; t < G.tm; ++t) {
    const unsigned long long w = (unsigned long long)__ldg(wq + t);
    ar += w;
    if (__popc(k & __ldg(zs + t)) & 1) odr += w;
  }
  for (uint32_t t = G.tm; t < G.te; ++t) {
    const unsigned long long w = (unsigned long long)__ldg(wq + t);
    ai += w;
    if (__popc(k & __ldg(zs + t)) & 1) odi += w;
  }
  const int sh = fz == 2u ? 1 : 0;
  const long long a = (long long)((ar - 2ull * odr) << sh), b = (long long)((ai - 2ull * odi) << sh);
  if (valid && fz != 0u && (a | b) != 0ll) {
    const uint32_t at = acc_s + 4u * (k & (kSpTile - 1u));
    fx_put<SPLIT, kRe>(at, q_mul(a, vx) - q_mul(b, vy));
    fx_put<SPLIT, kIm>(at, q_mul(a, vy) + q_mul(b, vx));
  }
}

// Terms [m0, m1) of the diagonal group at k (one lane's own amplitude): their
// sum in 64-bit fixed point times the amplitude as v_q, exact but for one
// rounding.
template <bool SPLIT>
__device__ __forceinline__ void sp_diag(const SpTables& T, uint32_t m0, uint32_t m1, bool imag, uint32_t k, bool on,
                                        long long vx, long long vy, uint32_t acc_s) {
  long long d = 0ll;
#pragma unroll 4
  for (uint32_t m = m0; m < m1; ++m) {
    const long long w = __ldg(T.dq + m);
    d += (__popc(k & __ldg(T.dz + m)) & 1) ? -w : w;
  }
  if (!on) return;
  const uint32_t at = acc_s + 4u * (k & (kSpTile - 1u));
  const long long pr = imag ? -q_mul(d, vy) : q_mul(d, vx), pi = imag ? q_mul(d, vx) : q_mul(d, vy);
  if (pr) fx_put_wide<SPLIT, kRe>(at, pr);
  if (pi) fx_put_wide<SPLIT, kIm>(at, pi);
}

// 2^e as R, for |e| beyond one float exponent split in two factors.
template <typename R>
__device__ __forceinline__ void pow2_split(int e, R* a, R* b) {
  const int lim = sizeof(R) == 4 ? 120 : 1000;
  const int e1 = e > lim ? lim : (e < -lim ? -lim : e);
  int e2 = e - e1;
  e2 = e2 > lim ? lim : (e2 < -lim ? -lim : e2);
  *a = sizeof(R) == 4 ? (R)ldexpf(1.0f, e1) : (R)ldexp(1.0, e1);
  *b = sizeof(R) == 4 ? (R)ldexpf(1.0f, e2) : (R)ldexp(1.0, e2);
}

// Shared memory: the accumulator planes, the term groups' tile parts, the
// first unit of each piece (n_pieces + 1 words) and, when they fit, the heads'
// tile words.
constexpr uint32_t kSpMaxSmem = 224u << 10;   // of the 227 KB a block can have

// The part of head q's words that tile t gives.
__device__ __forceinline__ uint4 tile_words(const SpTables& T, uint32_t q, uint32_t t) {
  uint4 w = __ldg(T.base + q);
  const uint4* h = T.hi + q;
  // four set bits at a time, their loads in flight together
  for (uint32_t m = t; m;) {
    uint4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[i] = make_uint4(0u, 0u, 0u, 0u);
      if (m) v[i] = __ldg(h + (size_t)(__ffs(m) - 1) * T.n_sub);
      m &= m - 1u;
    }
    w = xor4(w, xor4(xor4(v[0], v[1]), xor4(v[2], v[3])));
  }
  return w;
}

// Whether a case of head q can apply in a tile with words b: no parity that
// the tile decides is one.
__device__ __forceinline__ bool head_alive(const SpTables& T, uint32_t q, const uint4 b) {
  const uint4 f = __ldg(T.fix + q);
  return ~((b.x & f.x) | (b.y & f.y) | (b.z & f.z)) != 0u;
}

// SPLIT (complex64 only): products added to the accumulator in split form
// (fx_put), converted to 64-bit values before the epilogue.
template <typename R, bool SPLIT>
__global__ void __launch_bounds__(kSpThreads, 1) k_apply_h_sparse(const SparseArgs<R> a) {
  static_assert(!SPLIT || sizeof(R) == 4, "the split accumulator takes 32-bit products");
  constexpr int NT = kSpThreads;
  if (*a.alen > a.max_amps) return;           // the staged kernel takes this state
  using W = typename SpWeight<R>::T;
  extern __shared__ __align__(16) uint8_t sp_raw[];
  uint8_t* acc = sp_raw;
  const uint32_t acc_s = smem_u32(acc);
  const uint32_t P = (uint32_t)a.sp.n_pieces;
  uint4* s_base = reinterpret_cast<uint4*>(sp_raw + kAccBytes);
  W* s_tab = reinterpret_cast<W*>(s_base + (a.base_smem ? a.sp.n_sub : 0u));
  uint32_t* s_pre = reinterpret_cast<uint32_t*>(s_tab + a.sp.n_tab);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ uint32_t s_tile, s_unext;
  __shared__ uint32_t s_wsum[32];
  __shared__ double s_red[2][NT / 32];
  __shared__ bool s_last;
  const uint32_t ntiles = a.n > kSpLB ? 1u << (a.n - kSpLB) : 1u;
  const uint32_t n_oct = a.n > kSpLB ? kSpTile / 8u : 1u << (a.n - 3);   // octets of a tile
  const bool base_smem = a.base_smem;
  for (uint32_t j = threadIdx.x; j < kAccBytes / 16u; j += NT)
    reinterpret_cast<uint4*>(acc)[j] = make_uint4(0u, 0u, 0u, 0u);
  // fixed-point scale 2^F: every sum below 2^62 (split: 2^46, which binds for
  // no H that takes the split form), hbound x 2 max|component| x 2^F, and, for
  // complex64, every off-diagonal product below 2^30 (dmax x 2 max|component| x
  // 2^F <= 2^30)
  int F = 0;
  {
    const double m = __longlong_as_double((long long)*a.amax);
    const double bnd = 2.0 * a.hbound * m, bnd1 = 2.0 * a.dmax * m;
    if (bnd > 0.0) {
      int e;
      frexp(bnd, &e);   // bnd < 2^e
      F = (SPLIT ? 46 : 62) - e;
      if (sizeof(R) == 4 && bnd1 > 0.0) {
        frexp(bnd1, &e);
        F = min(F, 30 - e);
      }
    }
  }
  R up_a, up_b, dn_a, dn_b;          // 2^F and 2^-F, each as two factors
  pow2_split<R>(F, &up_a, &up_b);
  pow2_split<R>(-F, &dn_a, &dn_b);
  const double dn = ldexp(1.0, -F);
  const uint32_t K = a.parts;   // blocks per output tile
  for (;;) {
    if (threadIdx.x == 0) {
      s_tile = atomicAdd(a.tile_counter, 1u);
      s_unext = 0u;
    }
    __syncthreads();
    const uint32_t claim = s_tile;
    if (claim >= ntiles * K) break;
    // the claim is part `part` of output tile t: the part takes the tile's
    // unit batches part, part + K, part + 2K, ...
    const uint32_t t = claim / K, part = claim - t * K;
    // A tile none of whose source tiles holds an amplitude (its own among them,
    // for the diagonal) is all zero: no tables, no accumulator.  Few amplitudes
    // in a large state leave most tiles so.
    if (K == 1u) {
      bool any = false;
      for (uint32_t p = threadIdx.x; p < P && !any; p += NT) {
        const uint32_t u = t ^ a.sp.piece[p].xhi;
        any = a.toff[u + 1] != a.toff[u];
      }
      if (!__syncthreads_or(any || a.toff[t + 1] != a.toff[t])) {
        float4* d4 = reinterpret_cast<float4*>(a.out + (size_t)t * kSpTile);
        for (uint32_t q = threadIdx.x; q < n_oct * (8u * (uint32_t)sizeof(C_t<R>) / 16u); q += NT)
          __stcs(d4 + q, make_float4(0.f, 0.f, 0.f, 0.f));
        if (a.partials && threadIdx.x < 2) a.partials[2u * t + threadIdx.x] = 0.0;
        continue;
      }
    }
    // Work units are (piece p, span of chunks): 32 span consecutive nonzero
    // amplitudes of p's source tile u = t ^ (x >> LB) against p's groups,
    // numbered piece by piece (s_pre: a block scan of the unit counts).
    // A piece of few sub-blocks takes several chunks per unit, so that
    // finding and starting a unit stays small beside its work; small states
    // (K > 1), which have few units, take one.
    {
      // the tile's part of each head's parities and of each term group's weight
      if (base_smem)
        for (uint32_t q = threadIdx.x; q < a.sp.n_sub; q += NT) s_base[q] = tile_words(a.sp, q, t);
      for (uint32_t q = threadIdx.x; q < a.sp.n_tab; q += NT) {
        const SpTabTile<R> tt = reinterpret_cast<const SpTabTile<R>*>(a.sp.tile)[q];
        W f = tt.f0;
        for (uint32_t h = tt.hb; h < tt.he; ++h) {
          const W v = __ldg(reinterpret_cast<const W*>(a.sp.hw) + h);
          f += (__popc(t & __ldg(a.sp.hy + h)) & 1) ? -v : v;
        }
        s_tab[q] = f;
      }
      __syncthreads();
      const uint32_t per = (P + NT - 1) / NT, p0 = min(P, threadIdx.x * per), p1 = min(P, p0 + per);
      uint32_t mine = 0;
      for (uint32_t p = p0; p < p1; ++p) {
        const SpPiece pc = a.sp.piece[p];
        const uint32_t u = t ^ pc.xhi, cs = 32u * (K > 1u ? 1u : pc.span);
        uint32_t nu = (a.toff[u + 1] - a.toff[u] + cs - 1u) / cs;
        if (nu && pc.kind < 2) {   // a piece none of whose cases can apply in this tile has no units
          bool alive = false;
          for (uint32_t q = pc.sub0; q < pc.sub0 + pc.nsub && !alive; ++q)
            alive = head_alive(a.sp, q, base_smem ? s_base[q] : tile_words(a.sp, q, t));
          if (!alive) nu = 0u;
        }
        s_pre[p] = nu;
        mine += nu;
      }
      uint32_t incl = mine;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t q = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += q;
      }
      if (lane == 31) s_wsum[warp] = incl;
      __syncthreads();
      if (warp == 0) {
        uint32_t ws = s_wsum[lane], wi = ws;
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t q = __shfl_up_sync(0xffffffffu, wi, o);
          if (lane >= o) wi += q;
        }
        s_wsum[lane] = wi - ws;   // exclusive
        if (lane == 31) s_pre[P] = wi;
      }
      __syncthreads();
      uint32_t run = s_wsum[warp] + incl - mine;
      for (uint32_t p = p0; p < p1; ++p) {
        const uint32_t nu = s_pre[p];
        s_pre[p] = run;
        run += nu;
      }
    }
    __syncthreads();
    const uint32_t n_units = s_pre[P];
    // kUnitBatch consecutive units per claim (mostly of one piece, whose
    // tables then stay in L1), single ones towards the end of a tile and for
    // the few units of a small state (K > 1): a warp that starts a batch when
    // the others find none left keeps the whole block waiting
    uint32_t j0 = 0, p = 0;
    for (;;) {
      // units left when this warp claimed last decide how many it takes now
      const uint32_t batch = K == 1u && n_units - j0 > 8u * kUnitBatch * (uint32_t)(NT / 32) ? kUnitBatch : 1u;
      if (lane == 0) j0 = atomicAdd(&s_unext, batch) * K + part;
      j0 = __shfl_sync(0xffffffffu, j0, 0);
      if (j0 >= n_units) break;
      const uint32_t j1 = min(n_units, j0 + batch);
      // p = the last piece with s_pre[p] <= j0 (pieces without units share
      // their successor's start and are passed over), from the last claim's
      // piece on, then advanced along the batch
      if (s_pre[p + 1] <= j0) {
        uint32_t lo = p + 1, hi = P - 1;
        while (lo < hi) {
          const uint32_t mid = (lo + hi + 1) >> 1;
          if (s_pre[mid] <= j0) lo = mid;
          else hi = mid - 1;
        }
        p = lo;
      }
      for (uint32_t j = j0; j < j1; ++j) {
        while (p + 1 < P && s_pre[p + 1] <= j) ++p;
        const SpPiece pc = a.sp.piece[p];
        const uint32_t u = t ^ pc.xhi, cs = 32u * (K > 1u ? 1u : pc.span);
        const uint32_t l0 = a.toff[u] + (j - s_pre[p]) * cs, a1 = min(a.toff[u + 1], l0 + cs);
        for (uint32_t l = l0; l < a1; l += 32u) {
          const uint32_t li = l + (uint32_t)lane;
          const bool valid = li < a1;
          const uint32_t kk = a.aidx[valid ? li : l];
          const C_t<R> v = a.aval[valid ? li : l];
          typename SpVal<R>::T vx, vy;
          if constexpr (sizeof(R) == 4) {
            vx = v.x * up_a * up_b;
            vy = v.y * up_a * up_b;
          } else {
            vx = __double2ll_rn(v.x * up_a * up_b * a.sp.wscale);
            vy = __double2ll_rn(v.y * up_a * up_b * a.sp.wscale);
          }
          const bool cplx = __any_sync(0xffffffffu, valid && !rzero<R>(v.y));
          const uint32_t on = valid ? ~0u : 0u, klow = kk & (kSpTile - 1u);
          if (pc.kind < 2) {
            for (uint32_t q = pc.sub0; q < pc.sub0 + pc.nsub; ++q) {
              const uint4 w = head_words(a.sp.head + q, klow, base_smem ? s_base[q] : tile_words(a.sp, q, t));
              const uint32_t cases = ~(w.x | w.y | w.z) & on;
              if (pc.kind == 0) {
                const SpItem<R>* it = reinterpret_cast<const SpItem<R>*>(a.sp.item) + (size_t)kSpCases * q;
                if (cplx) sp_items<R, SPLIT, true>(it, cases, w.w, 4u * klow, vx, vy, acc_s);
                else sp_items<R, SPLIT, false>(it, cases, w.w, 4u * klow, vx, vy, acc_s);
              } else {
                const uint32_t slot = pc.tab0 + kSpCases * (q - pc.sub0);
                sp_tab_items<R, SPLIT>(reinterpret_cast<const SpTab<R>*>(a.sp.tab) + slot, s_tab + slot, a.sp, cases,
                                       w.w, kk, vx, vy, cplx, acc_s);
              }
              __syncwarp();   // the lanes' walks differ in length: the next head starts together
            }
          } else if (pc.kind != 2) {
            // the own tile's amplitudes (pc.xhi = 0) times diagonal terms
            const long long wx = __double2ll_rn((double)(v.x * up_a * up_b) * a.sp.dscale);
            const long long wy = __double2ll_rn((double)(v.y * up_a * up_b) * a.sp.dscale);
            sp_diag<SPLIT>(a.sp, pc.sub0, pc.sub0 + pc.nsub, pc.kind == 4, kk, valid, wx, wy, acc_s);
          } else {
            for (uint32_t g = pc.sub0; g < pc.sub0 + pc.nsub; ++g)
              sp_terms<SPLIT>(a.sp.list[g], a.sp.lz, reinterpret_cast<const typename SpVal<R>::T*>(a.sp.lw), kk, vx,
                              vy, valid, acc_s);
          }
        }
      }
    }
    __syncthreads();
    if constexpr (SPLIT) {
      // every product is in: the split halves become 64-bit values
      for (uint32_t j = threadIdx.x; j < 2u * kSpTile; j += NT) {
        const uint32_t at = 4u * (j & (kSpTile - 1u)) + (j & kSpTile ? kIm : kRe);
        const long long v = acc_get(acc, at);   // high half | low half
        if (v) acc_set(acc, at, (v >> 32) * 65536ll + (v & 0xffffffffll));
      }
      __syncthreads();
    }
    if (K > 1) {
      // several blocks per tile: each adds its nonzero accumulator entries
      // to the tile's global accumulator (64-bit integer atomics: the same
      // sum in any order), and the last to finish takes the total, clears
      // the global copy for the next call and runs the epilogue
      unsigned long long* g = a.gacc + (size_t)t * (2u * kSpTile);
      for (uint32_t j = threadIdx.x; j < 2u * kSpTile; j += NT) {
        const long long v = acc_get(acc, 4u * (j & (kSpTile - 1u)) + (j & kSpTile ? kIm : kRe));
        if (v) atomicAdd(g + j, (unsigned long long)v);
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) s_last = atomicAdd(a.tdone + t, 1u) == K - 1u;
      __syncthreads();
      if (!s_last) {
        for (uint32_t j = threadIdx.x; j < kAccBytes / 16u; j += NT)
          reinterpret_cast<uint4*>(acc)[j] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        continue;
      }
      __threadfence();
      for (uint32_t j = threadIdx.x; j < 2u * kSpTile; j += NT) {
        acc_set(acc, 4u * (j & (kSpTile - 1u)) + (j & kSpTile ? kIm : kRe), (long long)__ldcg(g + j));
        __stcg(g + j, 0ull);
      }
      if (threadIdx.x == 0) a.tdone[t] = 0u;
      __syncthreads();
    }
    // epilogue, first the energy partials over the nonzero amplitudes of the
    // own tile (zero amplitudes add nothing): one full warp of amplitudes at a
    // time, since the FP64 pipe is narrow here
    bool bad = false;   // an amplitude that fixed point cannot hold
    const uint32_t e0 = a.toff[t], e1 = a.toff[t + 1];
    {
      double2 w = make_double2(0.0, 0.0);   // this thread's |psi|^2 and Re<psi|H psi> partials
      for (uint32_t e = e0 + threadIdx.x; e < e1; e += NT) {
        const C_t<R> q = a.aval[e];
        bad = bad || not_finite(q.x) || not_finite(q.y);
        if (!a.partials) continue;
        const uint32_t at = 4u * (a.aidx[e] & (kSpTile - 1u));
        w.x += (double)q.x * q.x;
        w.y += (double)q.x * ((double)acc_get(acc, at + kRe) * dn);
        if (!rzero<R>(q.y)) {
          w.x += (double)q.y * q.y;
          w.y += (double)q.y * ((double)acc_get(acc, at + kIm) * dn);
        }
      }
      // the tile's energy partials, summed in a fixed order (warps that
      // hold no amplitude of the tile skip the FP64 shuffles)
      if (a.partials) {
        const bool any = __any_sync(0xffffffffu, w.x != 0.0 || w.y != 0.0);
        const double sx = any ? warp_sum(w.x) : 0.0, sy = any ? warp_sum(w.y) : 0.0;
        if (lane == 0) {
          s_red[0][warp] = sx;
          s_red[1][warp] = sy;
        }
      }
    }
    const bool bad_tile = __syncthreads_or(bad);
    if (a.partials && warp < 2) {
      const double sum = warp_sum(s_red[warp][lane]);
      if (lane == 0) a.partials[2u * t + warp] = sum;
    }
    // then the whole tile out (zeros included) and the accumulator cleared
    for (uint32_t o = threadIdx.x; o < n_oct; o += NT) {
      const uint32_t k0 = t * kSpTile + 8u * o;
      C_t<R> res[kAmpsH];
#pragma unroll
      for (int h = 0; h < kAmpsH; h += 4) {   // four amplitudes of each plane at a time
        const uint32_t at = 4u * (8u * o + h);
        uint4 pl[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint4* e = reinterpret_cast<uint4*>(acc + at + q * kPlane);
          pl[q] = *e;
          *e = make_uint4(0u, 0u, 0u, 0u);
        }
        const uint32_t rl[4] = {pl[0].x, pl[0].y, pl[0].z, pl[0].w}, rh[4] = {pl[1].x, pl[1].y, pl[1].z, pl[1].w};
        const uint32_t il[4] = {pl[2].x, pl[2].y, pl[2].z, pl[2].w}, ih[4] = {pl[3].x, pl[3].y, pl[3].z, pl[3].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const R re = fx_val<R>((long long)(((unsigned long long)rh[i] << 32) | rl[i]));
          const R im = fx_val<R>((long long)(((unsigned long long)ih[i] << 32) | il[i]));
          res[h + i] = cmake<R>(re * dn_a * dn_b, im * dn_a * dn_b);
        }
      }
      C_t<R>* dst = a.out + k0;
      if (sizeof(R) == 4) {
        float4* d4 = reinterpret_cast<float4*>(dst);
#pragma unroll
        for (int q = 0; q < kAmpsH / 2; ++q)
          __stcs(d4 + q, make_float4((float)res[2 * q].x, (float)res[2 * q].y, (float)res[2 * q + 1].x,
                                     (float)res[2 * q + 1].y));
      } else {
        double2* d2 = reinterpret_cast<double2*>(dst);
#pragma unroll
        for (int q = 0; q < kAmpsH; ++q) __stcs(d2 + q, make_double2((double)res[q].x, (double)res[q].y));
      }
    }
    __syncthreads();
    if (bad_tile)   // what is not finite shows at its own entry, as in a floating-point diagonal
      for (uint32_t e = e0 + threadIdx.x; e < e1; e += NT) {
        const C_t<R> q = a.aval[e];
        const R v = (q.x - q.x) + (q.y - q.y);
        if (not_finite(v)) a.out[a.aidx[e]] = cmake<R>(v, v);
      }
  }
  if (!a.partials) return;
  // the last block to finish adds the per-tile partials in tile order, so E
  // does not depend on which block took which tile
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double acc0 = 0.0, acc1 = 0.0;
  for (uint32_t u = threadIdx.x; u < ntiles; u += NT) {
    acc0 += ((volatile double*)a.partials)[2u * u];
    acc1 += ((volatile double*)a.partials)[2u * u + 1u];
  }
  acc0 = warp_sum(acc0);
  acc1 = warp_sum(acc1);
  if (lane == 0) {
    s_red[0][warp] = acc0;
    s_red[1][warp] = acc1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double n2 = 0.0, eh = 0.0;
    for (int q = 0; q < NT / 32; ++q) {
      n2 += s_red[0][q];
      eh += s_red[1][q];
    }
    a.scal[1] = n2;
    a.scal[2] = eh - a.identity * n2;
    a.scal[0] = eh / n2;
    *a.counter = 0u;
  }
}

}  // namespace

template <typename R>
int sparse_apply_h(SparseArgs<R> a, const LiveOctets& lv, int sm_count, cudaStream_t st) {
  if (!lv.toff || !lv.aidx || !lv.aval || !lv.alen || !lv.acounts || !lv.amax || a.max_amps > lv.acap || a.sp.n_pieces <= 0)
    return fail(GOCP_EINVAL, "scatter H psi needs the amplitude list and its tables");
  a.amax = lv.amax;
  a.aidx = lv.aidx;
  a.aval = reinterpret_cast<const C_t<R>*>(lv.aval);
  a.alen = lv.alen;
  a.toff = lv.toff;
  // complex64 adds its products in split form when every accumulator word
  // takes fewer than 65536 of them (at most one per off-diagonal group and
  // diagonal piece), and hbound is at most 2^15 times the largest weight, so
  // that totals below 2^46 cost the products no bits (a large constant beside
  // small couplings takes the carry form, whose totals have 62); the two
  // forms then give the same integers, so H psi does not depend on the choice
  // (GOCP_SCATTER_SPLIT=0 selects the carry form)
  bool split = sizeof(R) == 4 && a.n_offdiag + (uint32_t)a.sp.n_pieces < 65536u && a.hbound <= 0x1p15 * a.dmax;
  if (const char* ev = std::getenv("GOCP_SCATTER_SPLIT"))
    if (ev[0] == '0') split = false;
  auto kern = split ? k_apply_h_sparse<R, sizeof(R) == 4> : k_apply_h_sparse<R, false>;
  static std::mutex mu;
  static std::vector<bool> done;
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return cuda_status(e, "cudaGetDevice");
  {
    std::lock_guard<std::mutex> lk(mu);
    if (device >= (int)done.size()) done.resize(device + 1, false);
    if (!done[device]) {
      e = cudaFuncSetAttribute(k_apply_h_sparse<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kSpMaxSmem);
      if (e == cudaSuccess && sizeof(R) == 4)
        e = cudaFuncSetAttribute(k_apply_h_sparse<R, sizeof(R) == 4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kSpMaxSmem);
      if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute(k_apply_h_sparse)");
      done[device] = true;
    }
  }
  int rc = amp_list(sizeof(R) == 4 ? GOCP_C64 : GOCP_C128, a.psi, a.mask, a.n, lv, st);
  if (rc) return rc;
  const uint32_t ntiles = a.n > kSpLB ? 1u << (a.n - kSpLB) : 1u;
  k_tile_offsets<<<(ntiles + 256u) / 256u, 256, 0, st>>>(lv.aidx, lv.alen, lv.acap, ntiles, kSpLB, lv.toff);
  // tiles for fewer than half the SMs: K blocks share each tile (K a power
  // of two up to 64, or GOCP_SCATTER_PARTS, so that ntiles K reaches the SM
  // count), combining their fixed-point accumulators in global memory; the
  // sums are integer, so H psi and E do not depend on K.
  const uint32_t sms = (uint32_t)std::max(sm_count, 1);
  uint32_t kmax = 64u;
  if (const char* e = std::getenv("GOCP_SCATTER_PARTS")) {
    const long v = std::strtol(e, nullptr, 10);
    if (v >= 1) kmax = (uint32_t)std::min<long>(v, 64);
  }
  uint32_t K = 1;
  if (lv.gacc && lv.tdone && ntiles <= lv.gtiles && 2u * ntiles < sms)
    while (2u * K <= kmax && ntiles * K < sms) K *= 2u;
  a.parts = K;
  a.gacc = lv.gacc;
  a.tdone = lv.tdone;
  const int grid = (int)std::min<uint64_t>((uint64_t)ntiles * K, (uint64_t)sms);
  static_assert(kAccBytes + 8u * kSpMaxTab + 4u * (kSpMaxPieces + 1u) <= kSpMaxSmem, "the tables fit beside the planes");
  uint32_t smem = kAccBytes + (uint32_t)sizeof(typename SpWeight<R>::T) * a.sp.n_tab +
                  4u * ((uint32_t)a.sp.n_pieces + 1u);
  a.base_smem = (uint64_t)smem + 16ull * a.sp.n_sub <= kSpMaxSmem;
  if (a.base_smem) smem += 16u * a.sp.n_sub;
  kern<<<grid, kSpThreads, smem, st>>>(a);
  count_launches(2);
  return cuda_status(cudaGetLastError(), "k_apply_h_sparse");
}

int amp_list(int precision, const void* psi, const uint32_t* mask, int n, const LiveOctets& lv, cudaStream_t st) {
  if (n < 8 || !mask || !lv.aidx || !lv.aval || !lv.alen || !lv.acounts)
    return fail(GOCP_EINVAL, "amplitude list needs n >= 8 and its buffers");
  const uint32_t words = 1u << (n - 5);   // amplitude words
  const uint32_t nb = (words + kAmpBlock - 1u) / kAmpBlock;
  if (precision == GOCP_C64) {
    const float2* p = reinterpret_cast<const float2*>(psi);
    k_amp_count<float><<<nb, kAmpBlock, 0, st>>>(p, nullptr, mask, words, lv.acounts);
    k_amp_scan<<<1, 1024, 0, st>>>(lv.acounts, nb, lv.alen, nullptr, nullptr, 0, 0, lv.amax);
    k_amp_list<float><<<nb, kAmpBlock, 0, st>>>(p, nullptr, mask, words, lv.acounts, lv.aidx,
                                                reinterpret_cast<float2*>(lv.aval), nullptr, lv.acap, lv.amax);
  } else {
    const double2* p = reinterpret_cast<const double2*>(psi);
    k_amp_count<double><<<nb, kAmpBlock, 0, st>>>(p, nullptr, mask, words, lv.acounts);
    k_amp_scan<<<1, 1024, 0, st>>>(lv.acounts, nb, lv.alen, nullptr, nullptr, 0, 0, lv.amax);
    k_amp_list<double><<<nb, kAmpBlock, 0, st>>>(p, nullptr, mask, words, lv.acounts, lv.aidx,
                                                 reinterpret_cast<double2*>(lv.aval), nullptr, lv.acap, lv.amax);
  }
  count_launches(3);
  return cuda_status(cudaGetLastError(), "k_amp_list");
}

int chain_list(int precision, const void* psi, const void* lam, const uint32_t* mask, int n, const ChainList& cl,
               uint32_t* counts, int slot, int first, cudaStream_t st) {
  if (n < 8 || !mask || !cl.list || !cl.amask || !cl.cnt || !counts)
    return fail(GOCP_EINVAL, "chain list needs n >= 8 and its buffers");
  const uint32_t words = 1u << (n - 5);   // amplitude words
  const uint32_t nb = (words + kAmpBlock - 1u) / kAmpBlock;
  if (precision == GOCP_C64) {
    const float2* p = reinterpret_cast<const float2*>(psi);
    const float2* q = reinterpret_cast<const float2*>(lam);
    k_amp_count<float><<<nb, kAmpBlock, 0, st>>>(p, q, mask, words, counts);
    k_amp_scan<<<1, 1024, 0, st>>>(counts, nb, nullptr, cl.cnt, cl.sync, slot, first, nullptr);
    k_amp_list<float><<<nb, kAmpBlock, 0, st>>>(p, q, mask, words, counts, cl.list, nullptr, cl.amask, cl.cap,
                                                nullptr);
  } else {
    const double2* p = reinterpret_cast<const double2*>(psi);
    const double2* q = reinterpret_cast<const double2*>(lam);
    k_amp_count<double><<<nb, kAmpBlock, 0, st>>>(p, q, mask, words, counts);
    k_amp_scan<<<1, 1024, 0, st>>>(counts, nb, nullptr, cl.cnt, cl.sync, slot, first, nullptr);
    k_amp_list<double><<<nb, kAmpBlock, 0, st>>>(p, q, mask, words, counts, cl.list, nullptr, cl.amask, cl.cap,
                                                 nullptr);
  }
  count_launches(3);
  return cuda_status(cudaGetLastError(), "chain list");
}

template int sparse_apply_h<float>(SparseArgs<float>, const LiveOctets&, int, cudaStream_t);
template int sparse_apply_h<double>(SparseArgs<double>, const LiveOctets&, int, cudaStream_t);

}  // namespace gocp
