// Float64-accurate triangle kernel on the FP32 pipe (Alg. 6 line 11, Eq. 34):
//   H^XYZ += sum_I (E_I^XY F_I^XZ + E_I^XZ F_I^XY) G_I^YZ.
//
// The step is not a product (every operand shares two of the three output
// indices), so it cannot use the tensor cores, and GB300's FP64 pipe delivers
// 1/64 of the FP32 rate.  Here every float64 operand is carried as an
// unevaluated sum of two floats x = x_h + x_l (x_h = fl32(x), x_l = fl32(x -
// x_h); 48 significant bits), and the arithmetic uses error-free
// transformations:
//   * TwoProduct with an FMA:  p = fl(a b),  e = fma(a, b, -p),  a b = p + e
//     exactly (Karp and Markstein; Ogita, Rump and Oishi 2005, Alg. 3.3);
//   * TwoSum (Knuth):  s = fl(a + b),  z = s - a,
//     e = (a - (s - z)) + (b - z),  a + b = s + e exactly.
// t^XYZ = E^XY F^XZ + E^XZ F^XY is formed as a float pair (th, tl) from two
// exact products of the high parts, their exact sum, and the four cross
// products of high and low parts; H accumulates t G as a float pair whose
// high word is updated by TwoSum, the rounding errors and the low-order
// product terms going to the low word.  Each term carries an error of about
// 2^-45 of |E F G| (2^-43 at worst, from the roundings of the low words;
// float64: 2^-53), far below the 1e-10 bound on the residual.
//
// Like the float64 kernel, a block takes a pair of mirror (Y, Z) tiles, since
// t is symmetric in (Y, Z): one t feeds H^XYZ (with G^YZ) and H^XZY (with
// G^ZY).  Two amplitude indices X run in the two lanes of packed f32x2
// instructions (add/sub/fma.rn.f32x2), which halves the issued
// instructions; E and F are stored with the two X rows of a pair interleaved
// ({h(x), h(x+1), l(x), l(x+1)}), so that one 16-byte load gives both lanes.
// Per (X pair, Y, Z) pair of mirror outputs: 19 packed operations for t and
// 12 for each accumulation, i.e. 21.5 float32 operations per (I, X, Y, Z) term.
#include "kernels.cuh"

namespace thc {
namespace {

typedef unsigned long long f2;   // two float32 lanes: low word = lane 0

__device__ __forceinline__ f2 pk(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
// -a in both lanes: a sign-bit flip on the integer pipe (the FMA pipe is the
// busy one here; -0 for a zero lane, which no later sum can tell from +0).
__device__ __forceinline__ f2 neg2(f2 a) {
    return a ^ 0x8000000080000000ull;
}
// The rounded product fl(a b), written as fma(a, b, +0).  ptxas contracts a
// packed mul.rn.f32x2 whose result feeds an add.rn.f32x2 into one fused
// operation, which would round a b + c once where TwoSum needs fl(a b)
// itself (measured on GB300: every case where the two differ); an FMA with
// a zero addend is left alone.
__device__ __forceinline__ f2 prod2(f2 a, f2 b) { return fma2(a, b, 0ull); }

// t = a b + c d for float pairs a = aH + aL etc.: (th, tl) with th + tl = t
// up to the dropped low*low products and the roundings of the cross terms.
__device__ __forceinline__ void df_dot2(f2 aH, f2 aL, f2 bH, f2 bL, f2 cH, f2 cL, f2 dH,
                                        f2 dL, f2& th, f2& tl) {
    const f2 p1 = prod2(aH, bH);
    const f2 e1 = fma2(aH, bH, neg2(p1));   // aH bH - p1, exact
    const f2 p2 = prod2(cH, dH);
    const f2 e2 = fma2(cH, dH, neg2(p2));
    const f2 s = add2(p1, p2);                     // TwoSum(p1, p2)
    const f2 z = sub2(s, p1);
    const f2 es = add2(sub2(p1, sub2(s, z)), sub2(p2, z));
    f2 lo = fma2(aH, bL, e1);
    lo = fma2(aL, bH, lo);
    lo = fma2(cH, dL, lo);
    lo = fma2(cL, dH, lo);
    lo = add2(lo, e2);
    th = s;
    tl = add2(lo, es);
}

// (Sh, Sl) -= t g, with thn = -th: the accumulator holds -H so that the
// negated rounded product qn = fl(-th gH) feeds both TwoProduct and TwoSum.
__device__ __forceinline__ void df_acc(f2& Sh, f2& Sl, f2 th, f2 tl, f2 thn, f2 gH, f2 gL) {
    const f2 qn = prod2(thn, gH);      // -fl(th gH)
    const f2 e = fma2(th, gH, qn);     // th gH - fl(th gH), exact
    f2 low = fma2(th, gL, e);
    low = fma2(tl, gH, low);           // t g - fl(th gH), to second order
    const f2 s = add2(Sh, qn);         // TwoSum(Sh, qn)
    const f2 z = sub2(s, Sh);
    const f2 es = add2(sub2(Sh, sub2(s, z)), sub2(qn, z));
    Sl = sub2(add2(Sl, es), low);
    Sh = s;
}

// ---------------------------------------------------------------------------
// The same sums with fewer operations: TwoSum (six operations, because it does
// not know which addend is larger) is replaced by additions to constants that
// are known to be larger.  For a bound b >= |x| and a power of two 2^k >= 2 b,
// c = 1.5 2^k:  s = fl(x + c) stays in [2^k, 2^(k+1)), so s - c is x rounded
// to a multiple of u = 2^(k-23), exactly, and x - (s - c) has at most u / 2
// (Rump, Ogita and Oishi's extraction).  With x = a b in an FMA:
//   h = fma(a, b, c),  z = c - h,  r = fma(a, b, z):   a b = -z + r
// up to the rounding of r (2^-25 of u / 2).  t = E^XY F^XZ + E^XZ F^XY is
// formed this way from its two products (12 packed operations instead of 16),
// and t G is added to the accumulator as an integer: the low bits of s are
// (s - c) / u, so the sum over grid points of the bits of s, minus those of c,
// is exact in 32 bits for up to 512 points and takes an integer addition per
// lane; the remainder and the low-order products t_h g_l + t_l g_h go to a
// float32 sum.  6 packed operations per accumulation instead of 12: 24 per
// (X pair, Y, Z) pair of mirror outputs instead of 40.
// The bounds come from the largest |E|, |F|, |G| of BC grid points at a time
// (k_split_pairs and k_chunk_max write them), for every (X, Y, Z) of its own;
// after BC points the integer and float32 sums are added to a float pair in
// shared memory.
// Accuracy: the error of a term is relative to the chunk's bound, not to the
// term or the running sum.  It does not grow with the number of grid points as
// the TwoSum form's does: on Gaussian operands, rms over W = sum_I |E F G|,
// 2^-46.2 / -46.8 / -47.2 for 256 / 512 / 1200 points against 2^-47.3 / -46.6 /
// -46.3.  But a bound is the product of three largest values, and where E, F
// or G vary over the 16 points, or are large at different ones, it lies far
// above the terms: 2^-36 with entries spread over 2^-40 .. 1, 2^-42.5 with
// operands that decay over the grid as exp(-I / 2) (TwoSum: 2^-44.7, 2^-46.8).
// So it is used where the data carry it: in launches of kBiasMinPoints grid
// points or more, and there for the tiles that k_bias_check finds even enough.
constexpr int BC = kBiasChunk;              // grid points per chunk of common bounds

// A block of 128 threads takes 8 rows X (4 lane pairs) and a pair of mirror 16
// x 16 (Y, Z) tiles; its two halves of 8 x 8 threads take two X pairs each, and
// a thread 2 x 2 (Y, Z) of both.  Two blocks share an SM, so that one computes
// while the other waits for its copies.  The tile is small because mirror pairs
// of tiles cover the diagonal and the ragged edge with work that counts for
// nothing: 32-wide tiles do 1.16 times the needed work at P = 400, 1.43 at 200
// and 2.0 at 100, 16-wide ones 1.04, 1.16 and 1.42.
constexpr int DT = 16;                      // Y and Z tile
constexpr int DP = 4;                       // X pairs per block
constexpr int DX = 2 * DP;
constexpr int DTH = 128;
constexpr int BS = 2;                       // grid points per pipeline stage
constexpr int BST = 3;                      // stages
static_assert(DTH == 2 * DP * DT && DTH == DT * DT / 2, "one copy per thread, array and grid point");
static_assert(BC % BS == 0 && BC <= 512, "chunks are whole stages; 512 x 2^22 fits 32 bits");

struct DfStage {
    // {h(x), h(x+1), l(x), l(x+1)} of E^{x,Y} of the Y tile etc.: [x pair][.]
    float4 ey[BS][DP][DT], ez[BS][DP][DT], fy[BS][DP][DT], fz[BS][DP][DT];
    // {h, l} of G^YZ, rows Y, and of G^ZY, rows Z: column c of row r at
    // 2 ((c / 2) ^ swz(r)) + c % 2, so that rows (16-byte copies), reads of
    // four rows by eight columns (G^YZ) and of eight by four (G^ZY) take no
    // more shared-memory cycles than their bytes
    float2 g1[BS][DT][DT];
    float2 g2[BS][DT][DT];
};
__device__ __forceinline__ int swz(int r) { return (r & 1) << 2 | (r >> 1 & 3); }

template <bool BIAS>
struct DfSmem {
    DfStage st[BST];
};
template <>
struct DfSmem<true> {
    DfStage st[BST];
    // bounds of a chunk (two chunks in flight)
    struct {
        uint2 ey[DP][DT], ez[DP][DT], fy[DP][DT], fz[DP][DT];    // [x pair][.]
        unsigned g1[DT][DT], g2[DT][DT];                         // G^YZ rows Y, G^ZY rows Z
    } mx[2];
    ulonglong2 sum[16][DTH];          // float pairs {high, low} of the thread's 16 accumulators
};

// 1.5 2^k with 2^(k-1) above b (a thousandth above the true bound).
__device__ __forceinline__ f2 bias_of(f2 b) {
    float x, y;
    upk(b, x, y);
    auto one = [](float v) {
        const unsigned e = min(__float_as_uint(v * 1.001f) & 0x7F800000u, 0x7D800000u);
        return __uint_as_float(e + 0x01400000u);
    };
    return pk(one(x), one(y));
}
// The bounds of a chunk are bf16 halves: {largest of x, of x + 1}, {means} of E and
// F, {largest, mean} of G.
__device__ __forceinline__ float bf_lo(unsigned v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(unsigned v) { return __uint_as_float(v & 0xFFFF0000u); }
__device__ __forceinline__ f2 bound2(uint2 v) { return pk(bf_lo(v.x), bf_hi(v.x)); }
__device__ __forceinline__ f2 max2(f2 a, f2 b) {
    float a0, a1, b0, b1;
    upk(a, a0, a1);
    upk(b, b0, b1);
    return pk(fmaxf(a0, b0), fmaxf(a1, b1));
}

// t = E^XY F^XZ + F^XY E^XZ for one Y and two Z (float pairs .x + .y), s the
// biases of both products.  Both Z are taken operation by operation:
// neighbours share an operand, which the register caches then keep (measured
// 5.14 -> 4.93 ms at P = 200, 200 X, 600 grid points).
__device__ __forceinline__ void bias_dot2(ulonglong2 ey, ulonglong2 fy, const ulonglong2 (&ez)[2],
                                          const ulonglong2 (&fz)[2], const f2 (&s)[2], f2 (&th)[2],
                                          f2 (&tl)[2]) {
    f2 z1[2], z2[2], r1[2], r2[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) z1[j] = fma2(ey.x, fz[j].x, s[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) z2[j] = fma2(fy.x, ez[j].x, s[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        z1[j] = sub2(s[j], z1[j]);
        z2[j] = sub2(s[j], z2[j]);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) r1[j] = fma2(ey.x, fz[j].x, z1[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) r2[j] = fma2(fy.x, ez[j].x, z2[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) r1[j] = fma2(ey.x, fz[j].y, r1[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) r2[j] = fma2(fy.x, ez[j].y, r2[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) r1[j] = fma2(ey.y, fz[j].x, r1[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) r2[j] = fma2(fy.y, ez[j].x, r2[j]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        th[j] = neg2(add2(z1[j], z2[j]));
        tl[j] = add2(r1[j], r2[j]);
    }
}

struct BiasAcc {
    unsigned i0, i1;   // sums of the bits of s, per lane
    f2 lo;             // remainders and low-order products
};

// Both mirror outputs of a unit, operation by operation.
__device__ __forceinline__ void bias_acc(BiasAcc& a, BiasAcc& b, f2 th, f2 tl, f2 gH, f2 gL, f2 kH,
                                         f2 kL, f2 c, f2 d) {
    const f2 s = fma2(th, gH, c), t = fma2(th, kH, d);
    const f2 y = sub2(c, s), z = sub2(d, t);
    f2 p = fma2(th, gH, y), q = fma2(th, kH, z);
    p = fma2(th, gL, p);
    q = fma2(th, kL, q);
    p = fma2(tl, gH, p);
    q = fma2(tl, kH, q);
    a.i0 += (unsigned)s;
    a.i1 += (unsigned)(s >> 32);
    b.i0 += (unsigned)t;
    b.i1 += (unsigned)(t >> 32);
    a.lo = add2(a.lo, p);
    b.lo = add2(b.lo, q);
}

// sum += the accumulator's value after n points under bias c; clears it.
__device__ __forceinline__ void bias_fold(BiasAcc& a, f2 c, unsigned n, ulonglong2& sum) {
    const unsigned c0 = (unsigned)c, c1 = (unsigned)(c >> 32);
    const int d0 = (int)(a.i0 - n * c0), d1 = (int)(a.i1 - n * c1);
    // (s - c) / u summed: |d| < 2^31 as two exact floats, high 20 and low 12 bits
    f2 dh = (f2)(0x4B400000u + (unsigned)(d0 >> 12)) | (f2)(0x4B400000u + (unsigned)(d1 >> 12)) << 32;
    f2 dl = (f2)(0x4B000000u | (d0 & 4095)) | (f2)(0x4B000000u | (d1 & 4095)) << 32;
    dh = sub2(dh, pk(12582912.f, 12582912.f));
    dl = sub2(dl, pk(8388608.f, 8388608.f));
    const f2 p = c & 0x7F8000007F800000ull;   // 2^k = 2^23 u
    const f2 A = prod2(prod2(dh, pk(0x1p-11f, 0x1p-11f)), p);
    const f2 B = prod2(prod2(dl, pk(0x1p-23f, 0x1p-23f)), p);
    const f2 vh = add2(A, B);
    const f2 vl = sub2(B, sub2(vh, A));       // |A| >= |B| or A = 0
    const f2 S = sum.x;
    const f2 t = add2(S, vh);                 // TwoSum(S, vh)
    const f2 z = sub2(t, S);
    const f2 e = add2(sub2(S, sub2(t, z)), sub2(vh, z));
    const f2 l = add2(add2(sum.y, e), add2(vl, a.lo));
    const f2 hi = add2(t, l);                 // renormalise
    sum.x = hi;
    sum.y = sub2(l, sub2(hi, t));
    a.i0 = a.i1 = 0u;
    a.lo = 0ull;
}

// Copy bytes (4, 8 or 16) global -> shared, the last `bytes - n` of them zeros.
template <int BYTES>
__device__ __forceinline__ void cp_n(void* dst, const void* src, int n) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n));
    else if (BYTES == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(src), "r"(n));
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(n));
}

// The two forms of the accumulators, for the kernel below: mirror outputs
// [x pair][i][j] of H^XYZ and H^XZY, Y = ty + 8 i, Z = tx + 8 j.
template <bool BIAS>
struct DfAcc {
    // float pairs of -H, updated by TwoSum
    f2 h1[2][2][2], l1[2][2][2], h2[2][2][2], l2[2][2][2];
};
template <>
struct DfAcc<true> {
    BiasAcc h1[2][2][2], h2[2][2][2];
    f2 sg[2][2][2], cb[2][2][2], db[2][2][2];   // biases of t's products, of t G^YZ and of t G^ZY
};

// Grid: block of DX rows X (fastest, so that the blocks running together share
// the G tiles of one (Y, Z) pair in L2), pair of mirror tiles.
// BIAS: bounds ME, MF: [chunk][x pair][P]; MG: [chunk][P][P].  EVEN: P is even, rows of G start on 16-byte boundaries and are
// copied two columns at a time.
// A packed FMA of three distinct register pairs measures 3.3 cycles of a
// scheduler on GB300 and a packed addition 2.3 (peak: 2): the operations here
// are bound by register reads, 138 per unit of two X and two mirror outputs
// against 208 in the TwoSum form, so what comes besides them counts.  The copy
// addresses advance by constants, which is why a thread copies a two-column
// piece of one row of every G tile and one element of E and of F per grid
// point.  P = 400, 400 rows X, 1200 grid points: 46.3 ms (with one bias for both
// mirror outputs, which measures the smaller of H^XYZ and H^XZY by the larger's
// bound, 44.3; 32-wide tiles and one block of 256 threads per SM: 58.5; their
// TwoSum form 68.7), and 0.37 for k_bias_check; TwoSum form, P = 100, 300 points:
// 0.41 (0.60).
// uneven (may be null for the TwoSum form): a block runs where its tile's word
// asks for its form.
template <bool BIAS, bool EVEN>
__global__ void __launch_bounds__(DTH, 2)
    k_triangle_df(double* H, const float4* E4, const float4* F4, const float2* G2,
                  const uint2* ME, const uint2* MF, const unsigned* MG, const int* uneven, int P,
                  int nX, int nI) {
    grid_wait();
    if (BIAS ? uneven[blockIdx.x] != 0 : uneven && uneven[blockIdx.x] == 0) return;
    extern __shared__ __align__(16) unsigned char df_raw[];
    DfSmem<BIAS>& sm = *reinterpret_cast<DfSmem<BIAS>*>(df_raw);
    const int nb = (P + DT - 1) / DT;
    const int nxb = (nX + DX - 1) / DX, xb = (int)(blockIdx.x % (unsigned)nxb);
    int pidx = (int)(blockIdx.x / (unsigned)nxb), Yb = 0;
    while (pidx >= nb - Yb) {
        pidx -= nb - Yb;
        ++Yb;
    }
    const int Zb = Yb + pidx;
    const int Y0 = Yb * DT, Z0 = Zb * DT, X0 = xb * DX;
    const int nXp = (nX + 1) / 2, xp0 = xb * DP;
    const bool diag = Yb == Zb;
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3 & 7, xg = tid >> 6 << 1;
    const long long PP = (long long)P * P, XP = (long long)nXp * P;

    // Copies of this thread per grid point: columns 2 gc, 2 gc + 1 of row gr of
    // both G tiles, and one column of one row of E and of F.
    const int gr = tid >> 3, gc = tid & 7;
    const char *g1p, *g2p, *ep, *fp;
    int g1n, g2n, en;         // bytes inside the array
    {
        const int c1 = Z0 + 2 * gc, c2 = Y0 + 2 * gc;
        g1n = Y0 + gr < P ? 8 * max(0, min(2, P - c1)) : 0;
        g2n = Z0 + gr < P ? 8 * max(0, min(2, P - c2)) : 0;
        g1p = reinterpret_cast<const char*>(G2 + (g1n ? (long long)(Y0 + gr) * P + c1 : 0));
        g2p = reinterpret_cast<const char*>(G2 + (g2n ? (long long)(Z0 + gr) * P + c2 : 0));
    }
    // Z side (or Y), X pair cx, column c
    const int cz = tid >> 6, cx = tid >> 4 & 3, c = tid & 15;
    const char *mp = nullptr, *np = nullptr;      // the bounds of the same elements, per chunk
    {
        const int col = (cz ? Z0 : Y0) + c;
        const bool ok = xp0 + cx < nXp && col < P;
        const long long at = ok ? (long long)(xp0 + cx) * P + col : 0;
        en = ok ? 16 : 0;
        ep = reinterpret_cast<const char*>(E4 + at);
        fp = reinterpret_cast<const char*>(F4 + at);
        if (BIAS) {
            mp = reinterpret_cast<const char*>(ME + at);
            np = reinterpret_cast<const char*>(MF + at);
        }
    }
    const int gsw = 2 * (gc ^ swz(gr));
    auto load = [&](int k, int b) {
        const int I0 = k * BS;
        auto& st = sm.st[b];
#pragma unroll
        for (int s = 0; s < BS; ++s) {
            const bool in = I0 + s < nI;        // else the grid point's values are zeros
            const int n1 = in ? g1n : 0, n2 = in ? g2n : 0, n = in ? en : 0;
            const char* p1 = n1 ? g1p + s * PP * 8 : reinterpret_cast<const char*>(G2);
            const char* p2 = n2 ? g2p + s * PP * 8 : reinterpret_cast<const char*>(G2);
            if (EVEN) {
                cp_n<16>(&st.g1[s][gr][gsw], p1, n1);
                cp_n<16>(&st.g2[s][gr][gsw], p2, n2);
            } else {
                cp_n<8>(&st.g1[s][gr][gsw], p1, min(n1, 8));
                cp_n<8>(&st.g1[s][gr][gsw + 1], n1 > 8 ? p1 + 8 : p1, max(n1 - 8, 0));
                cp_n<8>(&st.g2[s][gr][gsw], p2, min(n2, 8));
                cp_n<8>(&st.g2[s][gr][gsw + 1], n2 > 8 ? p2 + 8 : p2, max(n2 - 8, 0));
            }
            cp_n<16>(cz ? &st.ez[s][cx][c] : &st.ey[s][cx][c],
                     n ? ep + s * XP * 16 : reinterpret_cast<const char*>(E4), n);
            cp_n<16>(cz ? &st.fz[s][cx][c] : &st.fy[s][cx][c],
                     n ? fp + s * XP * 16 : reinterpret_cast<const char*>(F4), n);
        }
        if constexpr (BIAS) {
            // the chunk's bounds with its first stage
            if (I0 % BC == 0) {
                auto& mx = sm.mx[(I0 / BC) & 1];
                cp_n<8>(cz ? &mx.ez[cx][c] : &mx.ey[cx][c], mp, en / 2);
                cp_n<8>(cz ? &mx.fz[cx][c] : &mx.fy[cx][c], np, en / 2);
                mp += XP * 8;
                np += XP * 8;
                const unsigned* m = MG + I0 / BC * PP +
                                 (g1n ? (long long)(Y0 + gr) * P + Z0 + 2 * gc : 0);
                cp_n<4>(&mx.g1[gr][2 * gc], m, min(g1n / 2, 4));
                cp_n<4>(&mx.g1[gr][2 * gc + 1], g1n > 8 ? m + 1 : m, max(g1n / 2 - 4, 0));
                m = MG + I0 / BC * PP + (g2n ? (long long)(Z0 + gr) * P + Y0 + 2 * gc : 0);
                cp_n<4>(&mx.g2[gr][2 * gc], m, min(g2n / 2, 4));
                cp_n<4>(&mx.g2[gr][2 * gc + 1], g2n > 8 ? m + 1 : m, max(g2n / 2 - 4, 0));
            }
        }
        g1p += BS * PP * 8;
        g2p += BS * PP * 8;
        ep += BS * XP * 16;
        fp += BS * XP * 16;
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    DfAcc<BIAS> A;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if constexpr (BIAS) {
                    A.h1[a][i][j] = BiasAcc{0u, 0u, 0ull};
                    A.h2[a][i][j] = BiasAcc{0u, 0u, 0ull};
                    A.sg[a][i][j] = A.cb[a][i][j] = A.db[a][i][j] = 0ull;
                    sm.sum[(a * 4 + i * 2 + j) * 2][tid] = make_ulonglong2(0ull, 0ull);
                    sm.sum[(a * 4 + i * 2 + j) * 2 + 1][tid] = make_ulonglong2(0ull, 0ull);
                } else {
                    A.h1[a][i][j] = A.l1[a][i][j] = A.h2[a][i][j] = A.l2[a][i][j] = 0ull;
                }
            }
    auto fold = [&](unsigned n) {
        if constexpr (BIAS) {
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int u = (a * 4 + i * 2 + j) * 2;
                        bias_fold(A.h1[a][i][j], A.cb[a][i][j], n, sm.sum[u][tid]);
                        bias_fold(A.h2[a][i][j], A.db[a][i][j], n, sm.sum[u + 1][tid]);
                    }
        }
    };
    const int nsteps = (nI + BS - 1) / BS;
#pragma unroll
    for (int k = 0; k < BST - 1; ++k) {
        if (k < nsteps) load(k, k);
        else asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    int inchunk = 0;   // grid points summed under the present biases
    int b = 0;         // stage of step k
    for (int k = 0; k < nsteps; ++k) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(BST - 2) : "memory");
        __syncthreads();   // stage k is there, stage k - 1 is free
        if (k + BST - 1 < nsteps) load(k + BST - 1, b == 0 ? BST - 1 : b - 1);
        else asm volatile("cp.async.commit_group;\n" ::: "memory");
        if constexpr (BIAS) {
            if (k * BS % BC == 0) {
                if (k > 0) fold((unsigned)inchunk);
                inchunk = 0;
                const auto& mx = sm.mx[(k * BS / BC) & 1];
#pragma unroll
                for (int a = 0; a < 2; ++a)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            const f2 ey = bound2(mx.ey[xg + a][ty + 8 * i]);
                            const f2 fy = bound2(mx.fy[xg + a][ty + 8 * i]);
                            const f2 ez = bound2(mx.ez[xg + a][tx + 8 * j]);
                            const f2 fz = bound2(mx.fz[xg + a][tx + 8 * j]);
                            const float g1 = bf_lo(mx.g1[ty + 8 * i][tx + 8 * j]);
                            const float g2 = bf_lo(mx.g2[tx + 8 * j][ty + 8 * i]);
                            const f2 p1 = prod2(ey, fz), p2 = prod2(ez, fy), p = add2(p1, p2);
                            A.sg[a][i][j] = bias_of(max2(p1, p2));
                            A.cb[a][i][j] = bias_of(prod2(p, pk(g1, g1)));
                            A.db[a][i][j] = bias_of(prod2(p, pk(g2, g2)));
                        }
            }
        }
        const auto& cur = sm.st[b];
#pragma unroll
        for (int st = 0; st < BS; ++st) {
            // G^(Y_i, Z_j) and G^(Z_j, Y_i), the same value in both lanes
            f2 g1h[2][2], g1l[2][2], g2h[2][2], g2l[2][2];
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float2 u =
                        cur.g1[st][ty + 8 * i][2 * ((tx / 2 + 4 * j) ^ swz(ty)) + (tx & 1)];
                    const float2 v =
                        cur.g2[st][tx + 8 * j][2 * ((ty / 2 + 4 * i) ^ swz(tx)) + (ty & 1)];
                    g1h[i][j] = pk(u.x, u.x);
                    g1l[i][j] = pk(u.y, u.y);
                    g2h[i][j] = pk(v.x, v.x);
                    g2l[i][j] = pk(v.y, v.y);
                }
#pragma unroll
            for (int xp = 0; xp < 2; ++xp) {
                // {h(x), h(x+1)} and {l(x), l(x+1)} as two 64-bit lanes
                ulonglong2 ey[2], fy[2], ez[2], fz[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    ey[i] = reinterpret_cast<const ulonglong2&>(cur.ey[st][xg + xp][ty + 8 * i]);
                    fy[i] = reinterpret_cast<const ulonglong2&>(cur.fy[st][xg + xp][ty + 8 * i]);
                    ez[i] = reinterpret_cast<const ulonglong2&>(cur.ez[st][xg + xp][tx + 8 * i]);
                    fz[i] = reinterpret_cast<const ulonglong2&>(cur.fz[st][xg + xp][tx + 8 * i]);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if constexpr (BIAS) {
                        f2 th[2], tl[2];
                        bias_dot2(ey[i], fy[i], ez, fz, A.sg[xp][i], th, tl);
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            bias_acc(A.h1[xp][i][j], A.h2[xp][i][j], th[j], tl[j], g1h[i][j],
                                     g1l[i][j], g2h[i][j], g2l[i][j], A.cb[xp][i][j], A.db[xp][i][j]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            f2 th, tl;
                            df_dot2(ey[i].x, ey[i].y, fz[j].x, fz[j].y, ez[j].x, ez[j].y, fy[i].x,
                                    fy[i].y, th, tl);
                            const f2 thn = neg2(th);
                            df_acc(A.h1[xp][i][j], A.l1[xp][i][j], th, tl, thn, g1h[i][j],
                                   g1l[i][j]);
                            df_acc(A.h2[xp][i][j], A.l2[xp][i][j], th, tl, thn, g2h[i][j],
                                   g2l[i][j]);
                        }
                    }
                }
            }
        }
        inchunk += BS;
        b = b + 1 == BST ? 0 : b + 1;
    }
    if (nsteps > 0) fold((unsigned)inchunk);
    // On a diagonal pair both accumulators cover the same tile and count
    // every (Y, Z) twice.
    const double scale = (diag ? 0.5 : 1.0) * (BIAS ? 1.0 : -1.0);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
        if (m == 1 && diag) __syncthreads();   // mirror targets overlap other threads' first targets
#pragma unroll
        for (int xp = 0; xp < 2; ++xp)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int Y = Y0 + ty + 8 * i, Z = Z0 + tx + 8 * j;
                    if (Y >= P || Z >= P) continue;
                    float a0, a1, b0, b1;
                    if constexpr (BIAS) {
                        const ulonglong2 v = sm.sum[(xp * 4 + i * 2 + j) * 2 + m][tid];
                        upk(v.x, a0, a1);
                        upk(v.y, b0, b1);
                    } else {
                        upk(m == 0 ? A.h1[xp][i][j] : A.h2[xp][i][j], a0, a1);
                        upk(m == 0 ? A.l1[xp][i][j] : A.l2[xp][i][j], b0, b1);
                    }
                    const int x = X0 + 2 * (xg + xp);
                    const long long at = m == 0 ? (long long)Y * P + Z : (long long)Z * P + Y;
                    if (x < nX) H[x * PP + at] += scale * ((double)a0 + (double)b0);
                    if (x + 1 < nX) H[(x + 1) * PP + at] += scale * ((double)a1 + (double)b1);
                }
    }
}

// ---------------------------------------------------------------------------
// Which tiles the sums with bounds are accurate enough for.  With b_c the bounds
// of an output's chunks, the rms error of the bounded sum is close to 2^-46.5
// sqrt(16 sum_c b_c^2), the TwoSum form's between 2^-47 and 2^-43.5 of W = sum_I
// (|E^XY F^XZ| + |E^XZ F^XY|) |G^YZ|.  A lower bound of W follows from each factor by
// itself: the sum of n terms is at least n times their geometric mean, which is
// the product of the factors' geometric means.  With those of a chunk, a tile is
// even if
//   sqrt(16 max_c b_c sum_c b_c) <= kEven sum_c n_c (<E^XY><F^XZ> + <E^XZ><F^XY>) <G^YZ>
// (max b sum b >= sum b^2 keeps squares out of float32's range), that is, if the
// rms error is at most 2^-43.2 W.  The left side over the right one's sum is 4.1
// to 6.5 on Gaussian operands at 512 grid points, 2.9 to 3.5 at 1200; 10 is where the
// bounded form begins to be less accurate than TwoSum (by 0.4 bits, for entries
// spread over a factor of 2, 512 points); a spread over 2^-4 .. 1 gives 70 and
// more, a decay of exp(-I / 8) 260.  Sums outside 2^-100 .. 2^120 are refused as well
// (the biases end at 1.5 2^126); all-zero outputs are not.
// A block looks at 256 outputs of 32 X and one (Y, Z) tile and both mirrors, with
// X pair q = Y + Z mod 16, so that every element of E, F and G of the tile enters
// one of them: the ratio of bound to mean is the product of the factors', each at
// least 1, and an uneven element shows in any output.  (All 4096 outputs took
// 5.9 ms at the size above.)
constexpr float kEven = 10.f;
constexpr int CX = 32;                      // X per block

__global__ void __launch_bounds__(256)
    k_bias_check(const uint2* ME, const uint2* MF, const unsigned* MG, int P, int nX, int nI,
                 int* uneven) {
    grid_wait();
    const int nb = (P + DT - 1) / DT, nxb = (nX + DX - 1) / DX, nsx = (nX + CX - 1) / CX;
    const int sx = (int)(blockIdx.x % (unsigned)nsx);
    const int pair = (int)(blockIdx.x / (unsigned)nsx);
    int pidx = pair, Yb = 0;
    while (pidx >= nb - Yb) {
        pidx -= nb - Yb;
        ++Yb;
    }
    const int y = threadIdx.x & 15, q = threadIdx.x >> 4;
    const int Y = Yb * DT + y, Z = (Yb + pidx) * DT + ((q - y) & 15);
    const int nXp = (nX + 1) / 2, xp = sx * (CX / 2) + q;
    const long long PP = (long long)P * P, XP = (long long)nXp * P;
    bool good = true;
    if (Y < P && Z < P && xp < nXp) {
        const uint2 *ey = ME + (long long)xp * P + Y, *ez = ME + (long long)xp * P + Z;
        const uint2 *fy = MF + (long long)xp * P + Y, *fz = MF + (long long)xp * P + Z;
        const unsigned *g1 = MG + (long long)Y * P + Z, *g2 = MG + (long long)Z * P + Y;
        float sb[2][2] = {}, mb[2][2] = {}, w[2][2] = {};   // [mirror][lane]
        const int nch = (nI + BC - 1) / BC;
#pragma unroll 4
        for (int c = 0; c < nch; ++c) {
            const uint2 a = ey[c * XP], b = ez[c * XP], d = fy[c * XP], e = fz[c * XP];
            const unsigned g[2] = {g1[c * PP], g2[c * PP]};
            const float n = (float)min(BC, nI - c * BC);
            const float tb[2] = {fmaf(bf_lo(d.x), bf_lo(b.x), bf_lo(a.x) * bf_lo(e.x)),
                                 fmaf(bf_hi(d.x), bf_hi(b.x), bf_hi(a.x) * bf_hi(e.x))};
            const float tw[2] = {fmaf(bf_lo(d.y), bf_lo(b.y), bf_lo(a.y) * bf_lo(e.y)),
                                 fmaf(bf_hi(d.y), bf_hi(b.y), bf_hi(a.y) * bf_hi(e.y))};
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    const float v = tb[l] * bf_lo(g[m]);
                    sb[m][l] += v;
                    mb[m][l] = fmaxf(mb[m][l], v);
                    w[m][l] = fmaf(tw[l], n * bf_hi(g[m]), w[m][l]);
                }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                const float v = w[m][l] * (kEven / 4.f);
                const bool in = mb[m][l] > 0x1p-100f && mb[m][l] < 0x1p120f;
                good = good && (mb[m][l] == 0.f || (in && mb[m][l] / v * (sb[m][l] / v) <= 1.f));
            }
    }
    const int all = __syncthreads_and(good);
    if (threadIdx.x < CX / DX && sx * (CX / DX) + (int)threadIdx.x < nxb)
        uneven[(long long)pair * nxb + sx * (CX / DX) + threadIdx.x] = all ? 0 : 1;
}

template <bool BIAS, bool EVEN>
cudaError_t launch_df(double* H, const float4* E4, const float4* F4, const float2* G2,
                      const uint2* ME, const uint2* MF, const unsigned* MG, const int* uneven, int P,
                      int nX, int nI, cudaStream_t s) {
    const int smem = (int)sizeof(DfSmem<BIAS>);
    const cudaError_t e = smem_optin((const void*)k_triangle_df<BIAS, EVEN>, smem);
    if (e != cudaSuccess) return e;
    const long long grid = triangle_df_tiles(P, nX);
    if (grid > INT32_MAX) return cudaErrorInvalidValue;
    launch_chained(k_triangle_df<BIAS, EVEN>, (unsigned)grid, DTH, smem, s, H, E4, F4, G2, ME, MF,
                   MG, uneven, P, nX, nI);
    count_launches(1);
    return cudaGetLastError();
}

// Largest value (rounded up) and geometric mean (rounded down, from the sum of n
// binary logarithms) in bf16; a zero makes the mean zero.
__device__ __forceinline__ unsigned bf_up(float v) {
    return (__float_as_uint(v) + 0xFFFFu) >> 16;
}
__device__ __forceinline__ unsigned bf_mean(float logs, int n) {
    return __float_as_uint(exp2f(logs / (float)n)) >> 16;
}

// M[chunk][Y][Z] = {largest, mean} |G_h^YZ| of the chunk's grid points (grid y: chunks).
__global__ void __launch_bounds__(256) k_chunk_max(const float2* G2, int nI, int P, unsigned* M) {
    grid_wait();
    const int ch = blockIdx.y, lo = ch * BC, n = min(nI - lo, BC);
    const long long PP = (long long)P * P;
    for (long long e = blockIdx.x * 256LL + threadIdx.x; e < PP; e += gridDim.x * 256LL) {
        const float2* g = G2 + lo * PP + e;
        float m = 0.f, s = 0.f;
#pragma unroll 4
        for (int I = 0; I < n; ++I) {
            const float v = fabsf(g[I * PP].x);
            m = fmaxf(m, v);
            s += __log2f(v);
        }
        M[ch * PP + e] = bf_up(m) | bf_mean(s, n) << 16;
    }
}

// {h, l} = {fl32(d), fl32(d - fl32(d))}.  The float64 form takes four
// float64-pipe operations (1/64 of the float32 rate on GB300: it kept the
// split kernels' float64 pipe 88 % busy), so for 2^-60 <= |d| < 2^60 the
// split is done on the IEEE-754 fields with integer operations: h rounds the
// 53-bit significand to 24 bits (nearest, ties to even); the signed
// remainder, below 2^29 units of 2^(e - 1075), is rounded to float32 and
// given its exponent.  Bit-identical to the float64 form (checked on the host
// over 2e7 values, ties and carries included).  Other values (zero among
// them) take the float64 form out of line, so that the common path carries
// no predicated float64 operations.
__device__ __noinline__ void split1_f64(double d, float& h, float& l) {
    h = __double2float_rn(d);
    l = __double2float_rn(d - (double)h);   // d - h is exact in float64
}

__device__ __forceinline__ bool split1_int(double d, float& h, float& l) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e < 1023 - 60 || e >= 1023 + 60) return false;
    const unsigned long long m = (b & 0xfffffffffffffULL) | (1ULL << 52);
    unsigned long long q = m >> 29;
    const unsigned long long rem = m & ((1ULL << 29) - 1);
    if (rem > (1ULL << 28) || (rem == (1ULL << 28) && (q & 1ULL))) ++q;
    const long long rs = (long long)m - (long long)(q << 29);   // |rs| <= 2^28
    int eh = e;
    if (q >> 24) {
        q >>= 1;
        ++eh;
    }
    const unsigned sgn = (unsigned)(b >> 63) << 31;
    h = __uint_as_float(sgn | ((unsigned)(eh - 1023 + 127) << 23) | (unsigned)(q & 0x7fffffULL));
    unsigned lb = __float_as_uint(__int2float_rn((int)rs));
    if (rs != 0) lb += (unsigned)(e - 1075) << 23;
    l = rs != 0 ? __uint_as_float(lb ^ sgn) : 0.f;
    return true;
}

__device__ __forceinline__ void split1(double d, float& h, float& l) {
    if (!split1_int(d, h, l)) split1_f64(d, h, l);
}

// One block per output row (I, q) at a time, threads along the P columns
// (no 64-bit division per element).  With M, a block takes the rows of one q
// for the BC grid points of a chunk and also writes the largest |h| and the
// geometric mean of every column, M[chunk][q][P].
__global__ void k_split_pairs(const double* E, int nI, int nX, int P, float4* out, uint2* M) {
    grid_wait();
    const int nXp = (nX + 1) / 2, per = M ? BC : 1;
    const long long rows = (long long)((nI + per - 1) / per) * nXp;
    for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
        const long long ch = row / nXp;
        const int q = (int)(row - ch * nXp), x = 2 * q;
        const int lo = (int)ch * per, hi = min(nI, lo + per);
        const bool two = x + 1 < nX;
        for (int c = threadIdx.x; c < P; c += blockDim.x) {
            float m0 = 0.f, m1 = 0.f, s0 = 0.f, s1 = 0.f;
            for (int I = lo; I < hi; ++I) {
                const double* e0 = E + ((long long)I * nX + x) * P;
                const double d0 = e0[c];
                const double d1 = two ? e0[P + c] : 0.0;
                float h0, l0, h1, l1;
                split1(d0, h0, l0);
                split1(d1, h1, l1);
                out[((long long)I * nXp + q) * P + c] = make_float4(h0, h1, l0, l1);
                m0 = fmaxf(m0, fabsf(h0));
                m1 = fmaxf(m1, fabsf(h1));
                s0 += __log2f(fabsf(h0));
                s1 += __log2f(fabsf(h1));
            }
            if (M)
                M[row * P + c] = make_uint2(bf_up(m0) | bf_up(m1) << 16,
                                            bf_mean(s0, hi - lo) | bf_mean(s1, hi - lo) << 16);
        }
    }
}

// in and out may be the same buffer: element i's float64 value is replaced
// by its float pair in the same eight bytes.
__global__ void k_split_df(const double* in, long long n, float2* out) {
    grid_wait();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        float h, l;
        split1(in[i], h, l);
        out[i] = make_float2(h, l);
    }
}

unsigned grid_for(long long n) {
    return (unsigned)std::max<long long>(1, std::min<long long>((n + 255) / 256, 152LL * 16));
}

}  // namespace

cudaError_t split_df_pairs(const double* E, int nI, int nX, int P, float4* out, uint2* bounds,
                           cudaStream_t s) {
    if (nI <= 0 || nX <= 0 || P <= 0) return cudaSuccess;
    const long long rows = (long long)(bounds ? cdiv(nI, BC) : nI) * ((nX + 1) / 2);
    launch_chained(k_split_pairs, (unsigned)std::min<long long>(rows, 152LL * 16), 128, 0, s, E, nI,
                   nX, P, out, bounds);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t chunk_max(const float2* G2, int nI, int P, unsigned* M, cudaStream_t s) {
    if (nI <= 0 || P <= 0) return cudaSuccess;
    const unsigned nb = (unsigned)std::min<long long>(((long long)P * P + 255) / 256, 152LL * 8);
    launch_chained(k_chunk_max, dim3(nb, cdiv(nI, BC)), 256, 0, s, G2, nI, P, M);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t split_df(const double* in, long long n, float2* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    launch_chained(k_split_df, grid_for(n), 256, 0, s, in, n, out);
    count_launches(1);
    return cudaGetLastError();
}

long long triangle_df_tiles(int P, int nX) {
    const long long nb = cdiv(P, DT);
    return cdiv(nX, DX) * (nb * (nb + 1) / 2);
}

cudaError_t triangle_df(double* H, const float4* E4, const float4* F4, const float2* G2,
                        const uint2* ME, const uint2* MF, const unsigned* MG, int* uneven, int P,
                        int nX, int nI, cudaStream_t s) {
    if (nX <= 0 || nI <= 0) return cudaSuccess;
    const bool bounds = ME && MF && MG && uneven && nI >= kBiasMinPoints;
    if (bounds) {
        const long long nb = cdiv(P, DT), grid = cdiv(nX, CX) * (nb * (nb + 1) / 2);
        if (grid > INT32_MAX) return cudaErrorInvalidValue;
        launch_chained(k_bias_check, (unsigned)grid, 256, 0, s, ME, MF, MG, P, nX, nI, uneven);
        count_launches(1);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess)
            e = P % 2 ? launch_df<true, false>(H, E4, F4, G2, ME, MF, MG, uneven, P, nX, nI, s)
                      : launch_df<true, true>(H, E4, F4, G2, ME, MF, MG, uneven, P, nX, nI, s);
        if (e != cudaSuccess) return e;
    }
    const int* rest = bounds ? uneven : nullptr;
    return P % 2 ? launch_df<false, false>(H, E4, F4, G2, ME, MF, MG, rest, P, nX, nI, s)
                 : launch_df<false, true>(H, E4, F4, G2, ME, MF, MG, rest, P, nX, nI, s);
}

}  // namespace thc
