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
#ifdef THC_DF_SUBNEG
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(0ull), "l"(a));
    return d;
#else
    return a ^ 0x8000000080000000ull;
#endif
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
// (k_split_pairs and k_pair_max write them), for every (X, Y, Z) of its own;
// after BC points the integer and float32 sums are added to a float pair in
// shared memory.  Accuracy: an error u per term relative to the chunk's
// bound instead of relative to the running sum, so it does not grow with the
// number of grid points as the TwoSum form's does: on Gaussian operands, rms
// over the sum of |terms|, 2^-46.1 / -46.6 / -47.1 for 300 / 600 / 1200 points
// against 2^-46.7 / -46.2 / -45.7.  Hence the rule kBiasMinPoints: below it
// the other kernel is the more accurate one (and the step is short).
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
        float2 ey[DP][DT], ez[DP][DT], fy[DP][DT], fz[DP][DT];   // [x pair][.]
        float g[DT][DT];
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
                                         f2 kL, f2 c) {
    const f2 s = fma2(th, gH, c), t = fma2(th, kH, c);
    const f2 y = sub2(c, s), z = sub2(c, t);
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
    f2 sg[2][2][2], cb[2][2][2];   // biases of t's products and of t G
};

// Grid: block of DX rows X (fastest, so that the blocks running together share
// the G tiles of one (Y, Z) pair in L2), pair of mirror tiles.
// BIAS: bounds ME, MF: [chunk][x pair][P] (lanes x, x + 1); MG: [chunk][P][P],
// symmetric.  EVEN: P is even, rows of G start on 16-byte boundaries and are
// copied two columns at a time.
// A packed FMA of three distinct register pairs measures 3.3 cycles of a
// scheduler on GB300 and a packed addition 2.3 (peak: 2): the operations here
// are bound by register reads, 138 per unit of two X and two mirror outputs
// against 208 in the TwoSum form, so what comes besides them counts.  The copy
// addresses advance by constants, which is why a thread copies a two-column
// piece of one row of every G tile and one element of E and of F per grid
// point.  P = 400, 400 rows X, 1200 grid points: 44.3 ms (32-wide tiles and one
// block of 256 threads per SM: 58.5; their TwoSum form 68.7); P = 200, 200 X,
// 600 points: 3.19 ms (4.93); TwoSum form, P = 100, 300 points: 0.41 (0.60).
template <bool BIAS, bool EVEN>
__global__ void __launch_bounds__(DTH, 2)
    k_triangle_df(double* H, const float4* E4, const float4* F4, const float2* G2,
                  const float2* ME, const float2* MF, const float* MG, int P, int nX, int nI) {
    grid_wait();
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
                const float* m = MG + I0 / BC * PP +
                                 (g1n ? (long long)(Y0 + gr) * P + Z0 + 2 * gc : 0);
                cp_n<4>(&mx.g[gr][2 * gc], m, min(g1n / 2, 4));
                cp_n<4>(&mx.g[gr][2 * gc + 1], g1n > 8 ? m + 1 : m, max(g1n / 2 - 4, 0));
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
                    A.sg[a][i][j] = A.cb[a][i][j] = 0ull;
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
                        bias_fold(A.h2[a][i][j], A.cb[a][i][j], n, sm.sum[u + 1][tid]);
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
                            const f2 ey = reinterpret_cast<const f2&>(mx.ey[xg + a][ty + 8 * i]);
                            const f2 fy = reinterpret_cast<const f2&>(mx.fy[xg + a][ty + 8 * i]);
                            const f2 ez = reinterpret_cast<const f2&>(mx.ez[xg + a][tx + 8 * j]);
                            const f2 fz = reinterpret_cast<const f2&>(mx.fz[xg + a][tx + 8 * j]);
                            const float g = mx.g[ty + 8 * i][tx + 8 * j];
                            const f2 p1 = prod2(ey, fz), p2 = prod2(ez, fy);
                            A.sg[a][i][j] = bias_of(max2(p1, p2));
                            A.cb[a][i][j] = bias_of(prod2(add2(p1, p2), pk(g, g)));
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
                                     g1l[i][j], g2h[i][j], g2l[i][j], A.cb[xp][i][j]);
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

template <bool BIAS, bool EVEN>
cudaError_t launch_df(double* H, const float4* E4, const float4* F4, const float2* G2,
                      const float2* ME, const float2* MF, const float* MG, int P, int nX, int nI,
                      cudaStream_t s) {
    const int smem = (int)sizeof(DfSmem<BIAS>);
    const cudaError_t e = smem_optin((const void*)k_triangle_df<BIAS, EVEN>, smem);
    if (e != cudaSuccess) return e;
    const long long nb = cdiv(P, DT), grid = cdiv(nX, DX) * (nb * (nb + 1) / 2);
    if (grid > INT32_MAX) return cudaErrorInvalidValue;
    launch_chained(k_triangle_df<BIAS, EVEN>, (unsigned)grid, DTH, smem, s, H, E4, F4, G2, ME, MF,
                   MG, P, nX, nI);
    count_launches(1);
    return cudaGetLastError();
}

// M[chunk][Y][Z] = max over the chunk's grid points of |G_h^YZ| and |G_h^ZY|.
// Block: one 32 x 32 tile and its mirror (grid x: tile pairs, y: chunks).
__global__ void __launch_bounds__(256) k_pair_max(const float2* G2, int nI, int P, float* M) {
    grid_wait();
    __shared__ float t1[32][33], t2[32][33];
    const int nb = (P + 31) / 32;
    int pidx = blockIdx.x, Yb = 0;
    while (pidx >= nb - Yb) {
        pidx -= nb - Yb;
        ++Yb;
    }
    const int Y0 = Yb * 32, Z0 = (Yb + pidx) * 32, ch = blockIdx.y;
    const int c = threadIdx.x & 31, r0 = threadIdx.x >> 5;
    const long long PP = (long long)P * P;
    const int lo = ch * BC, hi = min(nI, lo + BC);
    for (int r = r0; r < 32; r += 8) {
        float a = 0.f, b = 0.f;
        const bool ok1 = Y0 + r < P && Z0 + c < P, ok2 = Z0 + r < P && Y0 + c < P;
        for (int I = lo; I < hi; ++I) {
            if (ok1) a = fmaxf(a, fabsf(G2[I * PP + (long long)(Y0 + r) * P + Z0 + c].x));
            if (ok2) b = fmaxf(b, fabsf(G2[I * PP + (long long)(Z0 + r) * P + Y0 + c].x));
        }
        t1[r][c] = a;
        t2[r][c] = b;
    }
    __syncthreads();
    for (int r = r0; r < 32; r += 8) {
        if (Y0 + r < P && Z0 + c < P)
            M[ch * PP + (long long)(Y0 + r) * P + Z0 + c] = fmaxf(t1[r][c], t2[c][r]);
        if (Z0 + r < P && Y0 + c < P)
            M[ch * PP + (long long)(Z0 + r) * P + Y0 + c] = fmaxf(t2[r][c], t1[c][r]);
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
// for the BC grid points of a chunk and also writes the largest |h| of every
// column, M[chunk][q][P].
__global__ void k_split_pairs(const double* E, int nI, int nX, int P, float4* out, float2* M) {
    grid_wait();
    const int nXp = (nX + 1) / 2, per = M ? BC : 1;
    const long long rows = (long long)((nI + per - 1) / per) * nXp;
    for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
        const long long ch = row / nXp;
        const int q = (int)(row - ch * nXp), x = 2 * q;
        const int lo = (int)ch * per, hi = min(nI, lo + per);
        const bool two = x + 1 < nX;
        for (int c = threadIdx.x; c < P; c += blockDim.x) {
            float m0 = 0.f, m1 = 0.f;
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
            }
            if (M) M[row * P + c] = make_float2(m0, m1);
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

cudaError_t split_df_pairs(const double* E, int nI, int nX, int P, float4* out, float2* bounds,
                           cudaStream_t s) {
    if (nI <= 0 || nX <= 0 || P <= 0) return cudaSuccess;
    const long long rows = (long long)(bounds ? cdiv(nI, BC) : nI) * ((nX + 1) / 2);
    launch_chained(k_split_pairs, (unsigned)std::min<long long>(rows, 152LL * 16), 128, 0, s, E, nI,
                   nX, P, out, bounds);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t pair_max(const float2* G2, int nI, int P, float* M, cudaStream_t s) {
    if (nI <= 0 || P <= 0) return cudaSuccess;
    const unsigned nb = cdiv(P, 32);
    launch_chained(k_pair_max, dim3(nb * (nb + 1) / 2, cdiv(nI, BC)), 256, 0, s, G2, nI, P, M);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t split_df(const double* in, long long n, float2* out, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    launch_chained(k_split_df, grid_for(n), 256, 0, s, in, n, out);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t triangle_df(double* H, const float4* E4, const float4* F4, const float2* G2,
                        const float2* ME, const float2* MF, const float* MG, int P, int nX, int nI,
                        cudaStream_t s) {
    if (nX <= 0 || nI <= 0) return cudaSuccess;
    if (ME && MF && MG)
        return P % 2 ? launch_df<true, false>(H, E4, F4, G2, ME, MF, MG, P, nX, nI, s)
                     : launch_df<true, true>(H, E4, F4, G2, ME, MF, MG, P, nX, nI, s);
    return P % 2 ? launch_df<false, false>(H, E4, F4, G2, ME, MF, MG, P, nX, nI, s)
                 : launch_df<false, true>(H, E4, F4, G2, ME, MF, MG, P, nX, nI, s);
}

}  // namespace thc
