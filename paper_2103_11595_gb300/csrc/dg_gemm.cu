// GEMMs of the FP64 and FP32 modes on the fp16 tensor cores (sm_103a), as sums of exact digit
// products (digits.cuh), and the gathers that prepare their operands.
//
//   C[M][N] = X[M][K] . Y[N][K]^T   (FP64 or FP32 result, row-major, N contiguous)
//
// k_row_exp   the largest exponent of every operand row, for rows longer than a gather tile (the
//             digits of a row share one quantum; shorter rows are reduced inside the gather).
// k_digits    gathers a complex tensor into the digit form of a real, K-contiguous operand
//             (embedded [[Re, -Im], [Im, Re]] or plain [Re | Im], as k_perm).
// k_dg_gemm   the product.
//
// k_dg_gemm, arithmetic. With x = sum_i d_i 2^(-9 i) q_x and y likewise, the products of equal
// i + j = l share the weight q_x q_y 2^(-9 l): level l is one tensor-core accumulation of l + 1
// digit products over a chunk of 64 columns. Its value is an integer of at most
// (l + 1) 2^16 64 <= 2^24 for l <= 3, so the tensor core's FP32 accumulation (which truncates) is
// exact there -- but for the last digit, which carries the rest: with four digits level 3 is truncated to
// 2^-27 q_x q_y, 2^-41 of the row maxima's product. Levels 4 and up can pass 2^24 when nearly all digits
// are at their largest and of one sign; a truncation is then 2^-35 q_x q_y, 2^-49 of that product. The epilogue
// converts every level to an integer and adds it, shifted, into a 64-bit fixed-point register sum (unit
// q_x q_y 2^-sh0), which is rounded once, to FP64, at the end. An FP64 CUDA-core product rounds at every one of its K additions; both errors against exact
// products are compared in tests/test_gpu_dg_gemm.py. FP64 keeps 7 levels (26 digit products) at
// every K: without the seventh (about 2^-54 of the row maxima's product per column) the error was
// 1.5 to 2 times a CUDA-core sum's on normally distributed operands at K = 1024 .. 8192, and up to 15
// times on operands graded over 10^3; with it, 0.3 to 0.7 times (in the norm; digits.cuh says what that leaves
// open). The FP32 mode keeps 4 (10 products).
//
// k_dg_gemm, structure: persistent, one CTA per SM, 640 threads: bulk-copy producer warp, MMA issuer
// warp, two idle warps, sixteen epilogue warps. The M = 128 side of the MMA is Y's rows (the larger
// operand), its N side a row block of X (BC = 32, 64 or 128): with n on the TMEM lanes a warp stores
// 32 consecutive n of one C row, so C needs no staging and no tile is padded along X.
//  * Operand tiles are contiguous in memory, already swizzled: one 1-D bulk copy each. A chunk of
//    six 128 x 64 digit tiles of both sides is 192 KB for 26 products of 256 clocks, 30 bytes per
//    clock and SM.
//  * The digits of a chunk arrive highest first and a slot is released after its last product. The
//    first level's products start from the middle digits, so that they run before digit 0 -- the
//    last to be released and reloaded -- has arrived.
//  * A ring of TMEM buffers of BC columns holds one level each: the epilogue drains a level while
//    the next ones are computed. Its 64-bit sums (64 registers a thread) must not spill: the L1 left
//    beside 225 KB of shared memory does not hold the stack, and 50 bytes of it per thread cost a
//    third of the kernel's time. setmaxnreg gives the epilogue 104 of the launch's 96 registers
//    (64 x 128 + 104 x 512 = 96 x 640).
// Measured on GB300, 1024 x 32768 x 1024 (FP64): 1.40 ms, 1,270 TFLOP/s of fp16 products (67% of
// the measured bf16 burst), 49 TFLOP/s of FP64 products; the CUDA-core GEMM: 71 ms. What is left is
// the epilogue (7 levels of 128 x 128 values per 6,656 MMA clocks). 32 x 262144 x 32: 66 us, 2.3 TB/s
// of operands and result, bound by the result's conversion and stores.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "bodies.cuh"
#include "digits.cuh"
#include "kernels.h"
#include "tc_gemm_dev.cuh"

namespace ajf {
namespace {

using namespace dg;

// ------------------------------------------------------------------ operand gathers

constexpr int kTileElems = 2048;  // complex elements of a gather tile (at most)
constexpr int kDigThreads = 512;  // gather threads: 256 units of 8 elements per plane

// The exponent field (FP64 encoding) of a source value; zero and subnormal values give 0, infinities and
// NaN kNonFinite.
constexpr int kNonFinite = 0x7FF;
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ int exp_field(float x) {
  const int f = (__float_as_uint(x) >> 23) & 0xFF;
  return f == 0xFF ? kNonFinite : (f ? f + (1023 - 127) : 0);
}
__device__ __forceinline__ uint64_t f64_bits(double x) { return static_cast<uint64_t>(__double_as_longlong(x)); }
// exact, without the FP64 pipe
__device__ __forceinline__ uint64_t f64_bits(float x) {
  const uint32_t b = __float_as_uint(x);
  return (static_cast<uint64_t>(b >> 31) << 63) | (static_cast<uint64_t>(exp_field(x)) << 52) |
         (static_cast<uint64_t>(b & 0x7FFFFFu) << 29);
}

// Source offset and local index bits of thread `tid`'s elements (8 low bits of l), and of the up
// to 8 element groups q (the high bits).
struct TileMap {
  int64_t off;
  int loc;
  int nq;
  bool active;
};
__device__ __forceinline__ TileMap tile_map(const PermDev& p, int tid) {
  TileMap t{0, 0, 1, true};
  const int nb = p.tr + p.tk;
  const uint32_t* ws = reinterpret_cast<const uint32_t*>(p.tsrc);
  const uint32_t* wl = reinterpret_cast<const uint32_t*>(p.tloc);
  const uint32_t src[2] = {ws[0], ws[1]}, loc[2] = {wl[0], wl[1]};
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j < nb && ((tid >> j) & 1)) {
      t.off += int64_t(1) << ((src[j >> 2] >> (8 * (j & 3))) & 63);
      t.loc |= 1 << ((loc[j >> 2] >> (8 * (j & 3))) & 15);
    }
  t.active = nb >= 8 || tid < (1 << nb);
  t.nq = nb > 8 ? 1 << (nb - 8) : 1;
  return t;
}
// Offset and index bits of the element groups' three bits.
struct GroupMap {
  int64_t off[3];
  int loc[3];
  __device__ __forceinline__ explicit GroupMap(const PermDev& p) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      off[j] = int64_t(1) << p.tsrc[8 + j];
      loc[j] = 1 << p.tloc[8 + j];
    }
  }
  __device__ __forceinline__ int64_t offset(int q) const {
    return ((q & 1) ? off[0] : 0) + ((q & 2) ? off[1] : 0) + ((q & 4) ? off[2] : 0);
  }
  __device__ __forceinline__ int index(int q) const {
    return ((q & 1) ? loc[0] : 0) | ((q & 2) ? loc[1] : 0) | ((q & 4) ? loc[2] : 0);
  }
};

// Largest exponent field of every complex row over strips of its K (dst[2]: [strip][row]). Only
// the exponents are needed: one pass of reads, bound by HBM.
template <typename S>
__device__ __forceinline__ void row_exp_body(const PermDev& p, const S* src, char* base,
                                             int64_t* tab, int* rmax) {
  const int c_r = nchunks(p.rows.nbits), c_k = nchunks(p.cols.nbits);
  int64_t* t_r = tab;
  int64_t* t_k = tab + c_r * 256;
  build_table(p.rows, t_r);
  build_table(p.cols, t_k);
  chain_wait();
  __syncthreads();
  const int64_t R = int64_t(1) << p.rbits;
  const int TR = 1 << p.tr;
  const int64_t ntr = R >> p.tr, ntk = int64_t(1) << (p.kbits - p.tk), per = ntk / p.strips;
  const TileMap tm = tile_map(p, threadIdx.x);
  const GroupMap gm(p);
  int* out = reinterpret_cast<int*>(base + p.dst[2]);
  for (int64_t it = blockIdx.x; it < ntr * p.strips; it += gridDim.x) {
    const int64_t rt = it / p.strips, st = it % p.strips;
    for (int i = threadIdx.x; i < TR; i += kBodyThreads) rmax[i] = 0;
    __syncthreads();
    const int64_t orow = lookup(t_r, c_r, rt << p.tr) + tm.off;
    int m[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) m[q] = 0;
    if (tm.active) {
      for (int64_t kt = st * per; kt < (st + 1) * per; ++kt) {
        const S* s0 = src + orow + lookup(t_k, c_k, kt << p.tk);
        const S* s1 = s0 + p.plane;
        int a[8], b[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (q < tm.nq) {
            a[q] = exp_field(s0[gm.offset(q)]);
            b[q] = exp_field(s1[gm.offset(q)]);
          }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < tm.nq) m[q] = max(m[q], max(a[q], b[q]));
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q < tm.nq) {
          atomicMax(&rmax[(tm.loc | gm.index(q)) >> p.tk], m[q]);
        }
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < TR; i += kBodyThreads) out[st * R + (rt << p.tr) + i] = rmax[i];
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kBodyThreads, 4) k_row_exp(const PermDev* __restrict__ perms,
                                                             const double* arena, char* base) {
  extern __shared__ int64_t tab[];
  __shared__ int rmax[256];
  const PermDev& p = perms[blockIdx.y];
  if (p.strips == 0) return;
  if (p.src_f32) row_exp_body<float>(p, reinterpret_cast<const float*>(arena) + p.src, base, tab, rmax);
  else row_exp_body<double>(p, arena + p.src, base, tab, rmax);
}

// Place of local element `loc` (= row * 2^tk + k) in the staged tile: pairs of elements (16 bytes)
// XOR-permuted within 64-element groups, so that neither the stores (lanes along any bits of the
// index) nor the reads of 8 consecutive elements per thread pile up on one bank. Linear over XOR.
__device__ __forceinline__ int tile_place(int loc) {
  const int g = loc >> 6, c = ((loc >> 3) & 7) ^ ((g >> 2) & 7), m = ((loc >> 1) & 3) ^ ((c >> 1) & 3) ^ (g & 3);
  return (g << 6) | (c << 3) | (m << 1) | (loc & 1);
}

// Two digits (fields 0..512 = digit + 256) as packed fp16: 1024 + field has the field in its low
// mantissa bits, and subtracting 1280 is exact.
__device__ __forceinline__ uint32_t pack_digits(uint32_t f0, uint32_t f1) {
  const uint32_t v = (f0 | (f1 << 16)) + 0x64006400u;
  const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&v), __floats2half2_rn(1280.f, 1280.f));
  return *reinterpret_cast<const uint32_t*>(&r);
}

__device__ __forceinline__ uint4 neg_f16x8(uint4 v) {
  return make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u, v.w ^ 0x80008000u);
}

// Bound by memory traffic: 16 bytes (complex128) read per complex element and 12 (T = 6) or 8 bytes written
// per real operand element. All arithmetic is on the integer and fp16 pipes (an FP64 instruction
// per value would cost 32 times an integer one on GB300). Tiles of up to 2048 complex elements are
// staged in shared memory: loads follow the source order, whatever it is, and stores write whole
// 128-byte rows of the operand tiles, 16 bytes per thread. A thread has one plane's 8 values: with both
// planes in one thread a block's chain of some 1,000 instructions per tile took 24 us even alone.
template <typename S, int T>
__device__ __forceinline__ void digits_body(const PermDev& p, const S* src, char* base,
                                            int64_t* tab, S* tre, S* tim, bool early) {
  const int c_r = nchunks(p.rows.nbits), c_k = nchunks(p.cols.nbits);
  int64_t* t_r = tab;
  int64_t* t_k = tab + c_r * 256;
  build_table<kDigThreads>(p.rows, t_r);
  build_table<kDigThreads>(p.cols, t_k);
  const int64_t R = int64_t(1) << p.rbits, K = int64_t(1) << p.kbits;
  const int kt_bits = p.kbits - p.tk;              // log2 of the tiles along K
  const int64_t ntiles = int64_t(1) << (p.rbits - p.tr + kt_bits);
  const int ob = p.rbits + (p.embed ? 1 : 0);      // log2 of the operand's rows
  const int plane = threadIdx.x >> 8, u = threadIdx.x & 255;  // unit: 8 consecutive local elements of one plane
  const TileMap tm = tile_map(p, u);
  const GroupMap gm(p);
  const int ph = tile_place(tm.loc);
  char* dst = base + p.dst[0];
  int* exps = reinterpret_cast<int*>(base + p.dst[1]);
  const int* part = reinterpret_cast<const int*>(base + p.dst[2]);
  S* const mine = plane ? tim : tre;
  const bool unit = u < (1 << (p.tr + p.tk - 3));
  const int urow = (u << 3) >> p.tk, uk = (u << 3) & ((1 << p.tk) - 1);
  const int lanes = 1 << (p.tk - 3);               // units of one row of the tile
  chain_wait(early);
  __syncthreads();
  const unsigned units = __ballot_sync(0xffffffffu, unit);  // lanes that take part in a row's reduction
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t r0 = (tile >> kt_bits) << p.tr, k0 = (tile & ((int64_t(1) << kt_bits) - 1)) << p.tk;
    if (tm.active) {
      const S* s0 = src + lookup(t_r, c_r, r0) + lookup(t_k, c_k, k0) + tm.off + (plane ? p.plane : 0);
      S v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < tm.nq) v[q] = s0[gm.offset(q)];
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < tm.nq) mine[ph ^ tile_place(gm.index(q))] = v[q];
    }
    __syncthreads();
    if (unit) {
      int E = 0;
      const int64_t r = r0 + urow, k = k0 + uk;
      if (p.strips == 0) {  // the whole row is in this tile: reduce over its units (adjacent lanes)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int at = tile_place((u << 3) | j);
          E = max(E, max(exp_field(tre[at]), exp_field(tim[at])));
        }
        for (int o = 1; o < lanes; o <<= 1) E = max(E, __shfl_xor_sync(units, E, o));
      } else {
        for (int s = 0; s < p.strips; ++s) E = max(E, part[s * R + r]);
      }
      if (k == 0 && plane == 0) exps[r] = E;
      int64_t y[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) y[j] = biased_fixed(f64_bits(mine[tile_place((u << 3) | j)]), E, T);
      // embedded: Re at (s=0, t=0) and (s=1, t=1), Im at (s=1, t=0) and -Im at (s=0, t=1); plain: the
      // plane's columns
      const Piece p0(ob, p.kbits + 1, T, plane && p.embed ? R + r : r, plane && !p.embed ? K + k : k);
      const Piece p1(ob, p.kbits + 1, T, plane ? r : R + r, K + k);
#pragma unroll
      for (int t = 0; t < T; ++t) {
        uint32_t w[4];
        if (t == T - 1) {
          // the last digit with the rest: 18 bits, value (v - 2^17) 2^-9
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float f[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int v = static_cast<int>(static_cast<uint64_t>(y[2 * j + e]) >> (54 - 9 * t - 9)) & 0x3FFFF;
              f[e] = static_cast<float>(v - 0x20000) * (1.0f / 512.0f);
            }
            const __half2 h = __floats2half2_rn(f[0], f[1]);
            w[j] = *reinterpret_cast<const uint32_t*>(&h);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            uint32_t f[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              if (t == 0) f[e] = static_cast<uint32_t>(static_cast<int>(y[2 * j + e] >> 54) + 256);
              else f[e] = static_cast<uint32_t>(static_cast<uint64_t>(y[2 * j + e]) >> (54 - 9 * t)) & 511u;
            }
            w[j] = pack_digits(f[0], f[1]);
          }
        }
        const uint4 v = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(dst + p0.at(t)) = v;
        if (p.embed) *reinterpret_cast<uint4*>(dst + p1.at(t)) = plane ? neg_f16x8(v) : v;
      }
    }
    __syncthreads();
  }
}

template <int T>
__global__ void __launch_bounds__(kDigThreads, 2) k_digits(const PermDev* __restrict__ perms,
                                                           const double* arena, char* base,
                                                           bool early) {
  extern __shared__ int64_t tab[];
  __shared__ __align__(16) double tile[2 * kTileElems];
  const PermDev& p = perms[blockIdx.y];
  if (p.src_f32) {
    float* t = reinterpret_cast<float*>(tile);
    digits_body<float, T>(p, reinterpret_cast<const float*>(arena) + p.src, base, tab, t, t + kTileElems, early);
  } else {
    digits_body<double, T>(p, arena + p.src, base, tab, tile, tile + kTileElems, early);
  }
}

// ------------------------------------------------------------------ the product

constexpr int kEpiWarp0 = 4, kEpiWarps = 16;
constexpr int kThreads = 32 * (kEpiWarp0 + kEpiWarps);
constexpr int kDgMaxSlots = 12, kDgMaxBufs = 8;
constexpr uint32_t kDgSmemSlots = 224 * 1024;
constexpr uint32_t kDgControl = 512;
constexpr int kMaxChunksPerSplit = 32;

struct DgParams {
  const char* ya;                    // Y digits: the MMA's 128-row side
  const char* xb;                    // X digits: its BC-column side
  const int* ey;                     // row exponent fields of Y (N) and X (M / 2 complex rows)
  const int* ex;
  void* C;                           // [M][N], or with ksplit > 1
  double* ws;                        // [ksplit][M][N] partials (FP64)
  int* status;
  int64_t M, N;
  int32_t chunks, chunks_split, ksplit;
  int32_t pack;                      // digits per 128-byte row (log2)
  int32_t sh0;                       // weight 2^sh0 of the leading level in the fixed-point sums
  int32_t S, bufs;                   // ring sizes
  int32_t nty, ntx, group;           // tiles along Y and X, raster group
  int32_t yrows;                     // rows of a Y row block
  uint32_t idesc;
  int32_t early;
  unsigned long long wait_ns;
};

struct DgShared {
  uint8_t* slots;
  uint32_t full0, empty0, accf0, acce0, drain0;
  volatile int* abort_flag;
  uint32_t* tmem_slot;
};

__device__ __forceinline__ void dg_layout(uint8_t* slots, uint8_t* bars, DgShared& sh) {
  sh.slots = slots;
  sh.full0 = tc::smem_u32(bars);
  sh.empty0 = sh.full0 + 8 * kDgMaxSlots;
  sh.accf0 = sh.empty0 + 8 * kDgMaxSlots;
  sh.acce0 = sh.accf0 + 8 * kDgMaxBufs;
  sh.drain0 = sh.acce0 + 8 * kDgMaxBufs;
  sh.tmem_slot = reinterpret_cast<uint32_t*>(bars + 16 * kDgMaxSlots + 16 * kDgMaxBufs + 8);
  sh.abort_flag = reinterpret_cast<volatile int*>(sh.tmem_slot + 1);
}
static_assert(16 * kDgMaxSlots + 16 * kDgMaxBufs + 16 <= kDgControl, "control region");

// acc 2^(e) rounded to nearest (even) in FP64, e = exponent of acc's unit: integer arithmetic only
// (a 64-bit conversion instruction runs at the FP64 pipe's rate). Below the normal range: 0.
__device__ __forceinline__ double fixed_to_f64(int64_t acc, int e) {
  const uint64_t s = static_cast<uint64_t>(acc) & 0x8000000000000000ull;
  uint64_t u = acc < 0 ? static_cast<uint64_t>(-acc) : static_cast<uint64_t>(acc);
  if (u == 0) return 0.0;
  const int lz = __clzll(static_cast<long long>(u));
  u <<= lz;
  uint64_t m = u >> 11;
  m += ((u & 0x7FF) + (m & 1)) > 0x400 ? 1 : 0;
  const int f = 63 - lz + e + 1023;
  if (f <= 0) return 0.0;
  if (f >= 2047) return __longlong_as_double(static_cast<long long>(s | 0x7FF0000000000000ull));
  return __longlong_as_double(static_cast<long long>(s | ((static_cast<uint64_t>(f - 1) << 52) + m)));
}
__device__ __forceinline__ float fixed_to_f32(int64_t acc, int e) {
  const uint32_t s = acc < 0 ? 0x80000000u : 0u;
  uint64_t u = acc < 0 ? static_cast<uint64_t>(-acc) : static_cast<uint64_t>(acc);
  if (u == 0) return 0.0f;
  const int lz = __clzll(static_cast<long long>(u));
  u <<= lz;
  uint32_t m = static_cast<uint32_t>(u >> 40);
  const uint64_t rest = u & 0xFFFFFFFFFFull;
  m += (rest + (m & 1)) > 0x8000000000ull ? 1 : 0;
  const int f = 63 - lz + e + 127;
  if (f <= 0) return 0.0f;
  if (f >= 255) return __uint_as_float(s | 0x7F800000u);
  return __uint_as_float(s | ((static_cast<uint32_t>(f - 1) << 23) + m));
}

// acc += v * mul, and acc += (v * mul) 2^32: one multiply-add each
__device__ __forceinline__ void mad_wide(int64_t& acc, int v, int mul) { asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(v), "r"(mul)); }
__device__ __forceinline__ void mad_high(int64_t& acc, int v, int mul) { acc += static_cast<int64_t>(static_cast<uint64_t>(static_cast<uint32_t>(v * mul)) << 32); }

template <int BC, int T, int PACK, typename Out>
__global__ void __launch_bounds__(kThreads, 1) k_dg_gemm(const __grid_constant__ DgParams p) {
  constexpr int kLevels = T == 6 ? 7 : 4;
  constexpr int COLS = BC / 4;                 // columns per epilogue thread
  constexpr int CH = COLS < 16 ? COLS : 16;    // columns per TMEM load
  constexpr uint32_t kYBytes = kTileRows * 128, kXBytes = BC * 128, kSlotBytes = kYBytes + kXBytes;
  constexpr uint32_t kTmemCols = 512;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // the same value in every lane, and known to be: the roles' addresses and descriptors then live in
  // uniform registers, which is where the tensor and bulk-copy instructions take them from
  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int S = p.S, NB = p.bufs, NS = slots_of(T, PACK);
  DgShared sh;
  dg_layout(smem, smem + S * kSlotBytes, sh);
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(sh.full0 + 8 * s, 1);
      tc::mbar_init(sh.empty0 + 8 * s, 1);
    }
    for (int b = 0; b < NB; ++b) {
      tc::mbar_init(sh.accf0 + 8 * b, 1);
      tc::mbar_init(sh.acce0 + 8 * b, kEpiWarps);
    }
    tc::mbar_init(sh.drain0, 1);
    *sh.abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(sh.tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = __shfl_sync(0xffffffffu, *sh.tmem_slot, 0);
  chain_wait(p.early != 0);

  // work item wi: tile wi % tiles of K split wi / tiles; `group` Y blocks sweep the X blocks together
  const uint32_t tiles = static_cast<uint32_t>(p.nty) * static_cast<uint32_t>(p.ntx);
  const uint32_t nwork = tiles * static_cast<uint32_t>(p.ksplit);
  auto work_item = [&](uint32_t wi, int& ty, int& tx, int& c0, int& c1) {
    const uint32_t tile = wi % tiles, ks = wi / tiles;
    const uint32_t per_group = static_cast<uint32_t>(p.group) * static_cast<uint32_t>(p.ntx);
    const uint32_t g = tile / per_group, rr = tile % per_group;
    const uint32_t first = g * static_cast<uint32_t>(p.group);
    const uint32_t left = static_cast<uint32_t>(p.nty) - first;
    const uint32_t gm = left < static_cast<uint32_t>(p.group) ? left : static_cast<uint32_t>(p.group);
    ty = static_cast<int>(first + rr % gm);
    tx = static_cast<int>(rr / gm);
    c0 = static_cast<int>(ks) * p.chunks_split;
    c1 = c0 + p.chunks_split < p.chunks ? c0 + p.chunks_split : p.chunks;
  };
  bool ok = true;
  // producer and issuer: every lane waits, and the vote keeps the outcome (and the code that depends on
  // it) uniform
  auto warp_wait = [&](uint32_t bar, uint32_t parity, int code) {
    return __all_sync(0xffffffffu, !*sh.abort_flag && tc::mbar_wait(bar, parity, p.wait_ns, p.status, code)) != 0;
  };
  if (warp >= kEpiWarp0) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    // ---- epilogue: levels into 64-bit fixed-point sums, one rounding and store per tile
    const int q = warp & 3, h = (warp - kEpiWarp0) >> 2;
    const uint32_t lane_base = static_cast<uint32_t>(32 * q) << 16;
    const int half = static_cast<int>(p.M >> 1);  // complex rows of X
    int64_t acc[COLS];
    int buf = 0;
    uint32_t bphase = 0;
    // the next level's TMEM buffer, once its products are complete (ok = false when the wait expired)
    auto next_level = [&]() {
      const int b = buf;
      ok = __all_sync(0xffffffffu, tc::mbar_wait(sh.accf0 + 8 * b, bphase, p.wait_ns, p.status, 33)) != 0;
      if (++buf == NB) {
        buf = 0;
        bphase ^= 1u;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return b;
    };
    // the sums' shift, opaque to the compiler: values derived from it are not kept in registers
    auto scale = [&]() {
      int v = p.sh0;
      asm volatile("" : "+r"(v));
      return v;
    };
    auto column = [&](int b) { return tmem + lane_base + static_cast<uint32_t>(b * BC + h * COLS); };
    auto drained = [&](int b) {
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(sh.acce0 + 8 * b);
    };
    for (uint32_t wi = blockIdx.x; wi < nwork && ok; wi += gridDim.x) {
      int ty, tx, c0, c1;
      work_item(wi, ty, tx, c0, c1);
#pragma unroll
      for (int j = 0; j < COLS; ++j) acc[j] = 0;
      for (int c = c0; c < c1 && ok; ++c) {
        // levels 6, 5, 4: rounded in the sum's unit
#pragma unroll 1
        for (int l = kLevels - 1; l > 3; --l) {
          const int b = next_level();
          if (!ok) break;
          const uint32_t t = column(b);
          const float fs = pow2f(scale() - 9 * l);
#pragma unroll
          for (int j0 = 0; j0 < COLS; j0 += CH) {
            uint32_t r[CH];
            tc::tmem_ld<CH>(t + j0, r);
            tc::tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < CH; ++j) mad_wide(acc[j0 + j], __float2int_rn(__uint_as_float(r[j]) * fs), 1);
          }
          drained(b);
        }
        // exact integers: levels 3, 2 and, with a full chunk, 1 (shifts of 5 .. 30)
        constexpr int kHigh = PACK == 0 ? 0 : 1;  // levels 0 .. kHigh are shifted by 32 or more
#pragma unroll 1
        for (int l = 3; l > kHigh; --l) {
          const int b = next_level();
          if (!ok) break;
          const uint32_t t = column(b);
          const int mul = 1 << (scale() - 9 * l);
#pragma unroll
          for (int j0 = 0; j0 < COLS; j0 += CH) {
            uint32_t r[CH];
            tc::tmem_ld<CH>(t + j0, r);
            tc::tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < CH; ++j) mad_wide(acc[j0 + j], __float2int_rn(__uint_as_float(r[j])), mul);
          }
          drained(b);
        }
        // added to the high word
#pragma unroll 1
        for (int l = kHigh; l >= 0; --l) {
          if (!ok) break;
          const int b = next_level();
          if (!ok) break;
          const uint32_t t = column(b);
          const int mul = 1 << (scale() - 9 * l - 32);
#pragma unroll
          for (int j0 = 0; j0 < COLS; j0 += CH) {
            uint32_t r[CH];
            tc::tmem_ld<CH>(t + j0, r);
            tc::tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < CH; ++j) mad_high(acc[j0 + j], __float2int_rn(__uint_as_float(r[j])), mul);
          }
          drained(b);
        }
      }
      if (!ok) break;
      // lanes are consecutive n: a warp stores 32 consecutive elements of one C row at a time
      const int64_t n = static_cast<int64_t>(ty) * kTileRows + 32 * q + lane;
      const int m0 = tx * BC + h * COLS;
      if (n < p.N) {
        const int fy = p.ey[n];
        const int e0 = fy - 2 * (1023 + 7) - p.sh0;
        const bool part = p.ksplit > 1;
        const int64_t at = (part ? static_cast<int64_t>(wi / tiles) * p.M * p.N : 0) + m0 * p.N + n;
        double* wd = part ? p.ws + at : static_cast<double*>(p.C) + at;  // FP64 partials, or an FP64 result
        float* wf = static_cast<float*>(p.C) + at;
        const int* exm = p.ex + (m0 & (half - 1));  // COLS divides half: one run of X's row exponents
        int top = fy;  // largest exponent field of the rows multiplied
#pragma unroll
        for (int j = 0; j < COLS; ++j) {
          int e;
          // (volatile: hoisted above the loop, the loads would not leave enough registers)
          asm volatile("ld.global.s32 %0, [%1];" : "=r"(e) : "l"(exm + j));
          top = max(top, e);
          e += e0;
          if (sizeof(Out) == 8 || part) {
            *wd = fixed_to_f64(acc[j], e);
            wd += p.N;
          } else {
            *wf = fixed_to_f32(acc[j], e);
            wf += p.N;
          }
        }
        // a row with an infinity or a NaN has no digits: all of its products are NaN. (After the loop, and
        // not per element in it: tests there cost 2% of the n = 16 circuit, 4,142 -> 4,216 us.)
        if (top == kNonFinite) {
#pragma unroll 1
          for (int j = 0; j < COLS; ++j) {
            if (fy != kNonFinite && exm[j] != kNonFinite) continue;
            if (sizeof(Out) == 8 || part) wd[(j - COLS) * p.N] = __longlong_as_double(0x7FF8000000000000ll);
            else wf[(j - COLS) * p.N] = __uint_as_float(0x7FC00000u);
          }
        }
      }
    }
    if (!ok) *sh.abort_flag = 1;
    } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
  if (warp == 0) {
    // ---- producer: a chunk's slots, highest digits first (one lane issues)
    const bool leader = tc::elect_one();
    const uint32_t ybytes = static_cast<uint32_t>(p.yrows) * 128u;
    int slot = 0;
    uint32_t phase = 0, issued = 0;
    for (uint32_t wi = blockIdx.x; wi < nwork && ok; wi += gridDim.x) {
      int ty, tx, c0, c1;
      work_item(wi, ty, tx, c0, c1);
      for (int c = c0; c < c1 && ok; ++c) {
        const char* ysrc = p.ya + (static_cast<int64_t>(ty) * p.chunks + c) * NS * ybytes;
        const char* xsrc = p.xb + (static_cast<int64_t>(tx) * p.chunks + c) * NS * kXBytes;
        for (int s = NS - 1; s >= 0; --s) {
          ok = warp_wait(sh.empty0 + 8 * slot, phase ^ 1u, 31);
          if (!ok) break;
          const uint32_t dst = tc::smem_u32(sh.slots + slot * kSlotBytes);
          const uint32_t bar = sh.full0 + 8 * slot;
          if (leader) {
            tc::mbar_expect_tx(bar, ybytes + kXBytes);
            tc::bulk_load(dst, ysrc + static_cast<int64_t>(s) * ybytes, ybytes, bar);
            tc::bulk_load(dst + kYBytes, xsrc + static_cast<int64_t>(s) * kXBytes, kXBytes, bar);
          }
          ++issued;
          if (++slot == S) {
            slot = 0;
            phase ^= 1u;
          }
        }
      }
    }
    if (!ok) *sh.abort_flag = 1;
    if (*sh.abort_flag && leader) {
      // before the block gives its shared memory back: the last copies issued have landed (bounded)
      const uint32_t us = static_cast<uint32_t>(S);
      const uint32_t first = issued > us ? issued - us : 0u;
      for (uint32_t i = first; i < issued; ++i) tc::mbar_wait(sh.full0 + 8 * (i % us), (i / us) & 1u, p.wait_ns, p.status, 35);
    }
  } else if (warp == 1) {
    // ---- MMA issuer. One lane issues 104 MMAs of 64 clocks per chunk, so the instructions around them
    // count: the levels and products are unrolled, a chunk's operand descriptors are computed once
    // per digit (the low words; the high word is constant), and the whole warp runs the loop with
    // values that the compiler can see are uniform. (Run by a single lane of a diverged warp, each MMA
    // cost 120 to 220 clocks of issue, and the kernel took 1.9 to 3.0 ms on 1024 x 32768 x 1024.)
    const bool leader = tc::elect_one();
    int first = 0, buf = 0;
    uint32_t phase = 0, bphase = 0;
    bool any = false;
    constexpr int pack = PACK, steps = 4 >> PACK;
    const uint64_t desc0 = tc::smem_desc(tc::smem_u32(sh.slots));
    const uint32_t dlo0 = static_cast<uint32_t>(desc0), dhi = static_cast<uint32_t>(desc0 >> 32);
    for (uint32_t wi = blockIdx.x; wi < nwork && ok; wi += gridDim.x) {
      int ty, tx, c0, c1;
      work_item(wi, ty, tx, c0, c1);
      for (int c = c0; c < c1 && ok; ++c) {
        // slot s of the chunk (loaded in the order NS - 1 .. 0) is at ring position first + NS - 1 - s
        auto ring = [&](int s) {
          const int r = first + (NS - 1 - s);
          return r >= S ? r - S : r;
        };
        uint32_t yd[T];  // descriptor low words of the Y digits; X digits follow kYBytes behind
#pragma unroll
        for (int t = 0; t < T; ++t)
          yd[t] = dlo0 + static_cast<uint32_t>(ring(t >> pack)) * (kSlotBytes >> 4) +
                  static_cast<uint32_t>(t & ((1 << pack) - 1)) * (8u >> pack);
        int arrived = NS;  // slots arrived .. NS - 1 are resident
        auto need = [&](int s) {
          while (ok && arrived > s) {
            const int r = first + (NS - arrived);
            ok = warp_wait(sh.full0 + 8 * (r >= S ? r - S : r), r >= S ? phase ^ 1u : phase, 32);
            --arrived;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        };
#pragma unroll
        for (int l = kLevels - 1; l >= 0; --l) {
          if (!ok) break;
          const int b = buf;
          ok = warp_wait(sh.acce0 + 8 * b, bphase ^ 1u, 34);
          if (!ok) break;
          if (++buf == NB) {
            buf = 0;
            bphase ^= 1u;
          }
          const uint32_t dst = tmem + static_cast<uint32_t>(b * BC);
          bool fresh = true;
          auto product = [&](uint32_t y, uint32_t x) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              if (kk == 0 || kk < steps) {
                if (fresh && kk == 0) tc::mma<2, false>(dst, y, x, dhi, p.idesc);
                else tc::mma<2, true>(dst, y + 2 * kk, x + 2 * kk, dhi, p.idesc);
              }
            }
            fresh = false;
          };
          const int lo = l - (T - 1) > 0 ? l - (T - 1) : 0;
#pragma unroll
          for (int i = l >> 1; i >= lo; --i) {  // from the middle digits outward
            need(i >> pack);
            if (!ok) break;
            any = true;
            if (leader) {
              product(yd[i], yd[l - i] + (kYBytes >> 4));
              if (l - i != i) product(yd[l - i], yd[i] + (kYBytes >> 4));
            }
            fresh = false;
          }
          if (!ok) break;
          // the slots whose lowest digit is l have had their last product
          if (leader) {
            if ((l & ((1 << pack) - 1)) == 0 && (l >> pack) < NS) tc::mma_commit(sh.empty0 + 8 * ring(l >> pack));
            tc::mma_commit(sh.accf0 + 8 * b);
          }
        }
        first += NS;
        if (first >= S) {
          first -= S;
          phase ^= 1u;
        }
      }
    }
    if (!ok) *sh.abort_flag = 1;
    if (*sh.abort_flag && any && leader) {
      tc::mma_commit(sh.drain0);
      tc::mbar_wait(sh.drain0, 0u, p.wait_ns, p.status, 36);
    }
  }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// C[i] = sum over K splits (in order) of W[s][i]
template <typename Out>
__global__ void __launch_bounds__(kBodyThreads) k_dg_split_sum(const double* W, int ksplit, int64_t n,
                                                               Out* C) {
  chain_wait();
  for (int64_t i = int64_t(blockIdx.x) * kBodyThreads + threadIdx.x; i < n; i += int64_t(gridDim.x) * kBodyThreads) {
    double s = W[i];
    for (int k = 1; k < ksplit; ++k) s += W[k * n + i];
    C[i] = static_cast<Out>(s);
  }
}

int device_sms() {
  static int counts[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (counts[dev] == 0) cudaDeviceGetAttribute(&counts[dev], cudaDevAttrMultiProcessorCount, dev);
  return counts[dev];
}

int ceil_log2(int64_t x) {
  int b = 0;
  while ((int64_t(1) << b) < x) ++b;
  return b;
}

template <int BC, int T, int PACK, typename Out>
cudaError_t run_dg(DgParams& p, cudaStream_t s) {
  constexpr uint32_t slot_bytes = (kTileRows + BC) * 128;
  p.S = std::min<int>(kDgMaxSlots, kDgSmemSlots / slot_bytes);
  p.bufs = std::min<int>(kDgMaxBufs, 512 / BC);
  p.nty = static_cast<int32_t>((p.N + kTileRows - 1) / kTileRows);
  p.ntx = static_cast<int32_t>(p.M / BC);
  p.group = std::min<int32_t>(p.nty, 8);
  // D = FP32, A and B fp16, both K-major
  p.idesc = (1u << 4) | (static_cast<uint32_t>(BC >> 3) << 17) | (static_cast<uint32_t>(kTileRows >> 4) << 24);
  const size_t smem = size_t(p.S) * slot_bytes + kDgControl + 1024;
  // the shared-memory opt-in is a per-function attribute: set once per device
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !attr_set[dev]) {
    e = cudaFuncSetAttribute(k_dg_gemm<BC, T, PACK, Out>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) attr_set[dev] = true;
  }
  const int sms = device_sms();
  if (sms <= 0) return cudaErrorInvalidDevice;
  // as few CTAs as keep the number of rounds at its minimum (the SMs left over run other streams)
  const int64_t work = int64_t(p.nty) * p.ntx * p.ksplit;
  const int64_t rounds = (work + sms - 1) / sms;
  return launch_chained(k_dg_gemm<BC, T, PACK, Out>, dim3(static_cast<unsigned>((work + rounds - 1) / rounds)), kThreads, smem,
                        s, p);
}

template <int BC, int T, typename Out>
cudaError_t run_dg_p(DgParams& p, cudaStream_t s) {
  if (p.pack == 0) return run_dg<BC, T, 0, Out>(p, s);
  if (p.pack == 1) return run_dg<BC, T, 1, Out>(p, s);
  return run_dg<BC, T, 2, Out>(p, s);
}

template <int T, typename Out>
cudaError_t run_dg_t(DgParams& p, cudaStream_t s) {
  if (p.M >= 128) return run_dg_p<128, T, Out>(p, s);
  if (p.M >= 64) return run_dg_p<64, T, Out>(p, s);
  return run_dg_p<32, T, Out>(p, s);
}

}  // namespace

size_t dg_operand_bytes(int64_t rows, int64_t kcols, int mode) {
  return static_cast<size_t>(operand_bytes(rows, kcols, digit_terms(mode)));
}

bool dg_gemm_supported(int64_t M, int64_t N, int64_t K) {
  const bool pow2 = (M & (M - 1)) == 0 && (N & (N - 1)) == 0 && (K & (K - 1)) == 0;
  return pow2 && M >= 32 && N >= 16 && K >= 16 && M * N <= (int64_t(1) << 40) && K <= (int64_t(1) << 30);
}

int dg_gemm_splits(int64_t M, int64_t N, int64_t K) {
  constexpr int64_t sms = 152;
  const int64_t bc = std::min<int64_t>(M, 128);
  const int64_t tiles = (M / bc) * ((N + kTileRows - 1) / kTileRows), chunks = chunks_of(K);
  // accuracy: the fixed-point sum keeps 40 - log2(chunks) bits below the leading level's unit
  int64_t ks = (chunks + kMaxChunksPerSplit - 1) / kMaxChunksPerSplit;
  // parallelism: with fewer tiles than SMs, about one work item per SM of at least 2 chunks
  if (tiles < sms) ks = std::max(ks, std::min((sms + tiles - 1) / tiles, chunks / 2));
  // workspace of ksplit * M * N FP64 values: at most 8 GiB
  while (ks > 1 && ks * M * N * 8 > (int64_t(8) << 30) && (chunks + ks - 2) / (ks - 1) <= 256) --ks;
  if (ks <= 1) return 1;
  const int64_t per = (chunks + ks - 1) / ks;
  return static_cast<int>((chunks + per - 1) / per);
}

cudaError_t launch_row_exp(const PermDev* d_perms, int nperm, int grid_x, size_t smem, const void* arena, void* base,
                           cudaStream_t s) {
  return launch_chained(k_row_exp, dim3(grid_x, nperm), kBodyThreads, smem, s, d_perms, static_cast<const double*>(arena),
                        static_cast<char*>(base));
}

cudaError_t launch_digits(const PermDev* d_perms, int nperm, int grid_x, size_t smem, const void* arena, void* base,
                          int mode, cudaStream_t s, bool early) {
  return launch_chained(mode == OPM_DIG6 ? k_digits<6> : k_digits<4>, dim3(grid_x, nperm), kDigThreads, smem, s, d_perms,
                        static_cast<const double*>(arena), static_cast<char*>(base), early);
}

cudaError_t launch_dg_gemm(const DgGemm& g, cudaStream_t s) {
  if (!dg_gemm_supported(g.M, g.N, g.K) || g.ksplit < 1 || (g.ksplit > 1 && !g.ws)) return cudaErrorInvalidValue;
  DgParams p;
  std::memset(&p, 0, sizeof(p));
  p.ya = static_cast<const char*>(g.y);
  p.xb = static_cast<const char*>(g.x);
  p.ey = g.ey;
  p.ex = g.ex;
  p.C = g.C;
  p.ws = g.ws;
  p.status = g.status;
  p.M = g.M;
  p.N = g.N;
  p.chunks = static_cast<int32_t>(chunks_of(g.K));
  p.ksplit = g.ksplit;
  p.chunks_split = (p.chunks + g.ksplit - 1) / g.ksplit;
  if ((p.chunks + p.chunks_split - 1) / p.chunks_split != g.ksplit || p.chunks_split > 256) return cudaErrorInvalidValue;
  p.pack = pack_bits(g.K);
  // the sum's unit: |sum| <= chunks min(K, 64) 2^16 2^sh0 <= 2^62, and the shifts of levels 1 .. 3 at most
  // 30 or at least 32: 39 down to 32 for full chunks, 41 and 42 for K = 32 and 16
  p.sh0 = 46 - ceil_log2(int64_t(p.chunks_split) * std::min<int64_t>(g.K, 64));
  if (p.pack == 0) p.sh0 = std::min(p.sh0, 39);
  p.yrows = static_cast<int32_t>(block_rows(g.N));
  p.wait_ns = g.wait_ns;
  p.early = g.early ? 1 : 0;
  cudaError_t e;
  if (g.mode == OPM_DIG6) e = run_dg_t<6, double>(p, s);
  else e = run_dg_t<4, float>(p, s);
  if (e != cudaSuccess || g.ksplit == 1) return e;
  const int64_t n = g.M * g.N;
  const unsigned blocks = static_cast<unsigned>(std::min<int64_t>((n + 255) / 256, 4096));
  if (g.mode == OPM_DIG6)
    return launch_chained(k_dg_split_sum<double>, dim3(blocks), kBodyThreads, size_t(0), s, g.ws, g.ksplit, n,
                          static_cast<double*>(g.C));
  return launch_chained(k_dg_split_sum<float>, dim3(blocks), kBodyThreads, size_t(0), s, g.ws, g.ksplit, n,
                        static_cast<float*>(g.C));
}

cudaError_t set_dg_smem_limits() {
  const int big = 96 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k_row_exp, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_digits<6>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_digits<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  return e;
}

}  // namespace ajf
