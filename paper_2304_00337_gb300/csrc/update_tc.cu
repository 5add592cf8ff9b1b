// Block update Y = X C (+ Z) of the mixed policy on the tensor cores (tcgen05, accumulators in TMEM).
//
// With operand rows n = (output column, component) and 2 q real operand columns k = (trial column,
// component), Y is a real product of height `rows`.  k_block_update (dense.cu) did it on the FP64
// pipe, which takes 64 cycles per warp instruction, k_block_update_df with 20 FP32 operations per
// product.  Here each value of X is brought to a 62-bit fixed-point integer relative to a power of
// two that bounds its trial column's x- or y-edges (the exponents of gram_tc.cu, for the weighted
// edge values: with h2/h1 = r the fields differ by about r, and relative to one bound for both the
// smaller would lose log2 r of its bits), each coefficient likewise relative to the largest of its
// output column, and both are cut into eight signed 8-bit digits held as binary16 integers (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump, 2012).  The FP32 sums of digit products are
// exact (at most 64 x 7 x 2^14 < 2^23), digit pairs of equal i + j <= 7 share an accumulator, and the
// eight sums are put together in 64-bit integers.  Operands keep 2^-62 of
// their bound and the dropped pairs are below 7.1 2^-62 of the largest product, so what is left is the
// one rounding of the result to FP64 (by integers), and the addition of Z.  Largest error relative to
// the largest value of an output column's field, for columns of similar size: 1.0e-16, sums of FP64
// products 3e-16 to 5e-16; in general up to (2 q 16 2^-62 + 2^-57) of the bound, the largest |C_ij| 2^E_i.
//
// One persistent CTA per SM (each allocates the whole TMEM, and 544 threads of more than 60 registers leave
// no room for a second one, however little shared memory a narrow launch takes): 16 warps convert tiles of 128 rows into shared memory (a thread has one
// row and quadruples of trial columns: loads of 32 neighbouring rows, 16-byte stores in the MMA's
// K-major layout), one thread of a 17th warp issues the MMAs (A = one digit of X, M = 128; B = the
// first digits of C side by side, so that pair (i, j) lands in accumulator i + j), and the 16 warps
// read TMEM.  Two tiles are in flight in shared memory and TMEM (one in shared memory where two
// don't fit, more than 24 trial columns in a launch), and the next tile's loads are issued before a tile's sums are read.
#include <algorithm>

#include "internal.h"
#include "tc.cuh"

namespace pbs {

namespace {

constexpr int kWorkers = 512;              // conversion and read-out (16 warps)
constexpr int kThreads = kWorkers + 32;    // and the warp whose first lane issues the MMAs
constexpr int kTile = 128;                 // rows
constexpr int ND = 8;                      // digits per value
constexpr int kOctet = kTile * 16;         // bytes of 8 operand columns of a tile's digit
constexpr int kMaxSmem = 227 * 1024;
constexpr int kTail = 512;                 // barriers, flags and exponents after the operands
constexpr unsigned kTmemCols = 512;
constexpr unsigned long long kBias = 0x8080808080808080ull;

struct UpdateArgs {
  Roles X;
  int q;  // trial columns
  const double2* C;
  int ldc;
  long cgs;
  const int* E;  // exponent of trial column i of group g at E[g egs + 2 i]
  int egs;
  double2* Y;
  long ldy;
  bool more;  // added to what Y holds
  int p, pg;  // output columns of the launch, of a group
  int i0;     // first trial column of the launch
  const double2* Z;
  long ldz;
  long rows;
  int nbuf;
  int off;  // added to the exponents of X: values of column i are below 2^(E + off)
};

// v 2^{62 - E} truncated to an integer, for |v| < 2^E, E > kMinExp (zero and subnormals are shifted out)
__device__ __forceinline__ unsigned long long fixed62(double v, int E) {
  const int hi = __double2hiint(v), sh = min(max(E + 1023 - ((hi >> 20) & 0x7FF), 1), 63);
  const unsigned long long m = (((unsigned long long)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(v))
                               << 10 >> sh;
  const long long s = (long long)(hi >> 31);
  return (m ^ (unsigned long long)s) - (unsigned long long)s;
}

// Digit `s` (0 = top byte) of biased values a and b as two binary16 integers -128 .. 127: a byte next to
// the byte 0x64 is the binary16 number 1024 + byte.
__device__ __forceinline__ unsigned two_digits(unsigned bytes, unsigned sel) {
  const unsigned two = __byte_perm(bytes, 0x64646464u, sel);
  const __half2 bias = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));  // 1024 + 128
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&two), bias);
  return *reinterpret_cast<const unsigned*>(&d);
}

// V 2^{F - 56} rounded to nearest, by integers (conversions run on the FP64 pipe)
__device__ __forceinline__ double scaled(long long V, int F) {
  const unsigned sgn = (unsigned)((unsigned long long)V >> 32) & 0x80000000u;
  unsigned long long u = (unsigned long long)(V < 0 ? -V : V);
  const int lz = __clzll((long long)u), ex = F + 1030 - lz;  // F - 56 + 63 - lz + 1023
  u <<= lz & 63;
  unsigned long long r = ((unsigned long long)(unsigned)(ex - 1) << 52) + (u >> 11) + ((u >> 10) & 1);
  if (ex <= 0 || lz == 64) r = 0;
  if (ex > 2046) r = 0x7FF0000000000000ull;
  return __longlong_as_double((long long)(r | ((unsigned long long)sgn << 32)));
}

template <int N> __device__ __forceinline__ void tc_ld(unsigned addr, float (&v)[N]);
template <> __device__ __forceinline__ void tc_ld<4>(unsigned addr, float (&v)[4]) { tc_ld4(addr, v); }
template <> __device__ __forceinline__ void tc_ld<8>(unsigned addr, float (&v)[8]) { tc_ld8(addr, v); }

// QU: quadruples of trial columns per thread, 16 QU >= q; JW: output columns per group of four warps, 4 JW >= p
template <int QU, int JW>
__global__ void __launch_bounds__(kThreads, 1) k_update_tc(UpdateArgs A) {
  constexpr int NP = JW <= 2 ? 16 : 32;  // operand rows per digit of C
  constexpr int kRowsB = ND * NP, kOctetB = kRowsB * 16;
  extern __shared__ __align__(1024) unsigned char sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = blockIdx.y;
  const int ksteps = (2 * A.q + 15) / 16, octets = 2 * ksteps, quads = (A.q + 3) / 4;
  const int digit_bytes = octets * kOctet, buf_bytes = ND * digit_bytes, b_bytes = octets * kOctetB;
  const unsigned sB = smem_u32(sm), sA = sB + b_bytes;
  unsigned char* tail = sm + b_bytes + A.nbuf * buf_bytes;
  const unsigned full = smem_u32(tail), done = full + 16;  // two barriers each
  volatile int* abort = reinterpret_cast<volatile int*>(tail + 32);
  unsigned* tmem_slot = reinterpret_cast<unsigned*>(tail + 36);
  int* bad = reinterpret_cast<int*>(tail + 40);
  int* F = reinterpret_cast<int*>(tail + 64);   // exponents of the output columns
  int* Ex = reinterpret_cast<int*>(tail + 128);  // exponents of the trial columns
  const double2** Xp = reinterpret_cast<const double2**>(tail + 256);  // trial columns, null for those without values
  const double2* C = A.C + g * A.cgs;

  if (tid == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(full + 8 * b, kWorkers / 32);
      mbar_init(done + 8 * b, 1);
    }
    *abort = 0;
    *bad = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 16) F[tid] = -100000;
  if (tid < 32) {
    const int e = tid < A.q ? A.E[(long)g * A.egs + 2 * tid] : -kExpInf, i = A.i0 + tid, r = i / A.X.pr;
    const double2* base = r == 0 ? A.X.b[0] : (r == 1 ? A.X.b[1] : A.X.b[2]);
    const bool on = e > kMinExp && e < kExpInf;
    Ex[tid] = e;
    Xp[tid] = on ? base + ((long)g * A.X.pr + i % A.X.pr) * A.X.ld : nullptr;
  }
  // operand columns beyond 2 q and rows beyond 2 p stay zero
  for (int t = tid; t < (b_bytes + A.nbuf * buf_bytes) / 16; t += kThreads)
    reinterpret_cast<int4*>(sm)[t] = make_int4(0, 0, 0, 0);
  if (warp == kWorkers / 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // coefficients: c 2^{E_i} < 2^{F_j}
  for (int t = tid; t < A.p * A.q; t += kThreads) {
    const int j = t / A.q, i = t - j * A.q, e = Ex[i];
    if (e >= kExpInf) *bad = 1;
    if (e <= kMinExp || e >= kExpInf) continue;
    const double2 c = C[(long)j * A.ldc + i];
    const int hx = __double2hiint(c.x) >> 20 & 0x7FF, hy = __double2hiint(c.y) >> 20 & 0x7FF, h = max(hx, hy);
    if (h == 0x7FF) *bad = 1;
    if (h > 0) atomicMax(&F[j], h - 1022 + e);
  }
  __syncthreads();
  for (int t = tid; t < A.p * A.q; t += kThreads) {
    const int j = t / A.q, i = t - j * A.q, e = Ex[i];
    if (e <= kMinExp || e >= kExpInf || F[j] == -100000) continue;
    const double2 c = C[(long)j * A.ldc + i];
    const bool zx = (__double2hiint(c.x) & 0x7FF00000) == 0, zy = (__double2hiint(c.y) & 0x7FF00000) == 0;
    const unsigned long long x = zx ? 0 : fixed62(c.x, F[j] - e), y = zy ? 0 : fixed62(c.y, F[j] - e);
    // row 2 j: (re, -im), row 2 j + 1: (im, re)
    const unsigned long long row[2][2] = {{x + kBias, kBias - y}, {y + kBias, x + kBias}};
    unsigned char* base = sm + (i >> 2) * kOctetB + (i & 3) * 4;
#pragma unroll
    for (int c2 = 0; c2 < 2; ++c2)
#pragma unroll
      for (int s = 0; s < ND; ++s) {
        const unsigned b = (unsigned)(row[c2][0] >> (56 - 8 * s) & 0xFF) | (unsigned)(row[c2][1] >> (56 - 8 * s) & 0xFF) << 8;
        *reinterpret_cast<unsigned*>(base + (s * NP + 2 * j + c2) * 16) = two_digits(b, 0x4140);
      }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  // the exponents of the values from here on
  if (tid < 32) Ex[tid] = max(Ex[tid], kMinExp) + A.off;
  if (tid < 16) F[tid] += A.off;
  __syncthreads();
  const unsigned tmem = *tmem_slot;
  const long tiles = (A.rows + kTile - 1) / kTile;
  const int first = blockIdx.x, step = gridDim.x;
  const int mine = first < tiles ? (int)((tiles - first + step - 1) / step) : 0;

  if (warp == kWorkers / 32) {
    if (lane == 0) {
      for (int t = 0; t < mine; ++t) {
        const int b = t & 1;
        mbar_wait(full + 8 * b, (t >> 1) & 1, abort);
        tc_fence_after();
        const unsigned a0 = sA + (A.nbuf == 2 ? b : 0) * buf_bytes, d0 = tmem + 256 * b;
        for (int ks = 0; ks < ksteps; ++ks)
#pragma unroll
          for (int s = 0; s < ND; ++s)
            tc_mma(d0 + NP * s, tc_desc(a0 + s * digit_bytes + 2 * ks * kOctet, kOctet), tc_desc(sB + 2 * ks * kOctetB, kOctetB),
                   tc_idesc(NP * (ND - s)), !(ks == 0 && s == 0));
        tc_commit(done + 8 * b);
      }
      // the last commits have to land before the barriers' memory goes away
      for (int t = max(mine - 2, 0); t < mine; ++t) mbar_wait(done + 8 * (t & 1), (t >> 1) & 1, abort);
    }
    __syncwarp();
  } else {
    const int wg = warp >> 2, row = 32 * (warp & 3) + lane;
    double2 v[QU][4];
    auto load = [&](int t) {
      const long r = ((long)first + (long)t * step) * kTile + row;
#pragma unroll
      for (int u = 0; u < QU; ++u)
        if (wg + 4 * u < quads) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const double2* x = Xp[4 * (wg + 4 * u) + k];
            v[u][k] = x && r < A.rows ? x[r] : make_double2(0.0, 0.0);
          }
        }
    };
    auto convert = [&](int t) {
      const unsigned a0 = sA + (A.nbuf == 2 ? t & 1 : 0) * buf_bytes + row * 16;
#pragma unroll
      for (int u = 0; u < QU; ++u)
        if (wg + 4 * u < quads) {
          unsigned bytes[4][4];  // per column: digits (0, 1), (2, 3), (4, 5), (6, 7) of both components
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int e = Ex[4 * (wg + 4 * u) + k];
            const unsigned long long x = fixed62(v[u][k].x, e) + kBias, y = fixed62(v[u][k].y, e) + kBias;
            const unsigned xh = (unsigned)(x >> 32), xl = (unsigned)x, yh = (unsigned)(y >> 32), yl = (unsigned)y;
            bytes[k][0] = __byte_perm(xh, yh, 0x6273);  // x digit 0, y digit 0, x digit 1, y digit 1 from the low byte up
            bytes[k][1] = __byte_perm(xh, yh, 0x4051);
            bytes[k][2] = __byte_perm(xl, yl, 0x6273);
            bytes[k][3] = __byte_perm(xl, yl, 0x4051);
          }
          const unsigned at = a0 + (wg + 4 * u) * kOctet;
#pragma unroll
          for (int s = 0; s < ND; ++s) {
            const unsigned sel = s & 1 ? 0x4342u : 0x4140u;
            unsigned w[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = two_digits(bytes[k][s >> 1], sel);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + s * digit_bytes), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                         "r"(w[3])
                         : "memory");
          }
        }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(full + 8 * (t & 1));
    };
    const bool broken = *bad != 0;
    auto finish = [&](int t) {
      constexpr int NL = JW <= 2 ? 4 : 8;  // accumulator columns read (2 JW of them used)
      const int j0 = wg * JW;
      mbar_wait(done + 8 * (t & 1), (t >> 1) & 1, abort);
      __syncwarp();
      tc_fence_after();
      const unsigned ta = tmem + 256 * (t & 1) + ((unsigned)(warp & 3) << 21) + 2 * j0;
      if (j0 < A.p) {
        // sums of digit pairs i + j = t as integers, two of them in 32 bits, four in 64
        int hi[2 * JW], mid[2 * JW], lo0[2 * JW], lo1[2 * JW];
        auto pair = [&](int s, int (&out)[2 * JW]) {  // D_s 2^8 + D_{s+1}
          float a[NL], b[NL];
          tc_ld<NL>(ta + NP * s, a);
          tc_ld<NL>(ta + NP * (s + 1), b);
#pragma unroll
          for (int k = 0; k < 2 * JW; ++k) {
            if (QU == 2 && s >= 4) {  // above the 2^22 of the addition below when 2 q = 64
              out[k] = (__float2int_rn(a[k]) << 8) + __float2int_rn(b[k]);
            } else {  // an integer below 2^22 in magnitude plus 1.5 2^23 has it in the low bits
              constexpr unsigned kOff = 0x4B400000u;
              const unsigned x = __float_as_uint(a[k] + 12582912.0f), y = __float_as_uint(b[k] + 12582912.0f);
              out[k] = (int)(x * 256u + y - (kOff * 256u + kOff));
            }
          }
        };
        pair(0, hi);
        pair(2, mid);
        pair(4, lo0);
        pair(6, lo1);
        const long r = ((long)first + (long)t * step) * kTile + row;
        const bool give_up = broken || *abort != 0;
#pragma unroll
        for (int jj = 0; jj < JW; ++jj) {
          const int j = j0 + jj;
          double out[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const int k = 2 * jj + c;
            const long long top = (long long)hi[k] * 65536 + mid[k], low = (long long)lo0[k] * 65536 + lo1[k];
            const long long V = (long long)((unsigned long long)top << 20) + ((low + 2048) >> 12);
            out[c] = scaled(V, F[j & 15]);
          }
          if (j < A.p && r < A.rows) {
            double2 y = give_up ? make_double2(nan(""), nan("")) : make_double2(out[0], out[1]);
            double2* to = A.Y + ((long)g * A.pg + j) * A.ldy + r;
            if (A.more) y = y + *to;
            if (A.Z) y = y + A.Z[((long)g * A.pg + j) * A.ldz + r];
            *to = y;
          }
        }
      }
      tc_fence_before();
    };
    if (mine > 0) load(0);
    for (int t = 0; t < mine; ++t) {
      convert(t);
      if (t + 1 < mine) load(t + 1);
      if (A.nbuf == 2) {
        if (t > 0) finish(t - 1);
      } else {
        finish(t);
      }
    }
    if (A.nbuf == 2 && mine > 0) finish(mine - 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWorkers / 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

int smem_of(int np, int q, int nbuf) {
  const int octets = 2 * ((2 * q + 15) / 16);
  return octets * ND * np * 16 + nbuf * ND * octets * kOctet + kTail;
}

template <int QU, int JW> void launch(UpdateArgs a, int slices, int ngroups, cudaStream_t s) {
  static PerDeviceOnce once;
  once([] { PBS_CUDA(cudaFuncSetAttribute(k_update_tc<QU, JW>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem)); });
  const int np = JW <= 2 ? 16 : 32;
  a.nbuf = smem_of(np, a.q, 2) <= kMaxSmem ? 2 : 1;
  k_update_tc<QU, JW><<<dim3(slices, ngroups), kThreads, smem_of(np, a.q, a.nbuf), s>>>(a);
  PBS_LAUNCHED();
}

}  // namespace

void update_tc(Roles X, int q, const double2* C, int ldc, long cgs, const int* d_exps, int egs, double2* Y, long ldy, int p,
               const double2* Z, long ldz, long rows, int ngroups, int slices, cudaStream_t s, int ox, int oy) {
  if (ox != oy) {
    // the two fields of unequal exponents one after the other (an offset per row instead, for every
    // mesh, made the launch of square cells 11 % longer)
    const long half = rows / 2;
    for (int f = 0; f < 2; ++f) {
      const Roles Xf{{X.b[0] + f * half, X.b[1] + f * half, X.b[2] + f * half}, X.pr, X.ld};
      update_tc(Xf, q, C, ldc, cgs, d_exps, egs, Y + f * half, ldy, p, Z ? Z + f * half : nullptr, ldz, half, ngroups, slices, s,
                f ? oy : ox, f ? oy : ox);
    }
    return;
  }
  slices = (int)std::max<long>(1, std::min<long>(slices, (rows + kTile - 1) / kTile));
  // wide blocks (24 outputs of 72 trial columns, three groups at 128 x 128: 0.53 -> 0.17 ms per iteration)
  // in even parts: outputs of 16 at most (the accumulators of two tiles), trial columns of
  // 32 at most, each part after the first added to what is there, Z with the last
  const int np = (p + 15) / 16, nq = (q + 31) / 32;
  for (int jp = 0; jp < np; ++jp) {
    const int j0 = p * jp / np, pj = p * (jp + 1) / np - j0;
    for (int iq = 0; iq < nq; ++iq) {
      const int i0 = q * iq / nq, qi = q * (iq + 1) / nq - i0;
      UpdateArgs a{X, qi, C + (long)j0 * ldc + i0, ldc, cgs, d_exps + 2 * i0, egs, Y + j0 * ldy, ldy, iq > 0, pj, p, i0,
                   Z && iq == nq - 1 ? Z + j0 * ldz : nullptr, ldz, rows, 1, ox};
      if (qi <= 16) {
        if (pj <= 8) launch<1, 2>(a, slices, ngroups, s);
        else if (pj <= 12) launch<1, 3>(a, slices, ngroups, s);
        else launch<1, 4>(a, slices, ngroups, s);
      } else {
        if (pj <= 8) launch<2, 2>(a, slices, ngroups, s);
        else if (pj <= 12) launch<2, 3>(a, slices, ngroups, s);
        else launch<2, 4>(a, slices, ngroups, s);
      }
    }
  }
}

}  // namespace pbs
