// Shared-memory FFT over lines of vectors of NC components, for any even
// 7-smooth length with the radix plan known only at run time.
//
// A thread owns one butterfly of one line and carries it for NC components
// (three or one); with three, a pass's index arithmetic and twiddles are paid once
// for three transforms, and the 3x3 tensor product finds the components of a
// wave number in one thread's registers; with one, three times the threads
// share the work (FP64 passes other than the tensor product).
// Element e of line l and component c lives at s[c plane + place(e) B + l];
// the passes are in place (every thread reads its butterfly, the CTA
// synchronises, every thread writes).
//
// Self-sorting Stockham passes: butterfly b of a pass of radix R and span Ns
// (the product of the earlier radices) reads elements b + q L/R, multiplies
// input q by W_{Ns R}^(q k), k = b mod Ns, and writes output q to
// (b - k) R + k + q Ns.  The first pass has no twiddles, and the last pass's
// outputs lie at b + q L/R again: a forward transform can hand its outputs to
// the inverse's first pass, run with the radices in reverse order, in
// registers.  The plan's first radix is even, so that the zero-padded upper
// half of a forward's input, and the dropped half of an inverse's output, are
// the registers q >= R/2 of that pass.
//
// Twiddled radix-2 steps are folded into multiply-adds (LineTwiddle), in FP64 six
// for both outputs: 3 instructions per point and level against 3.5 for radix-8
// passes that multiply first.  FP64 instructions are what an FP64
// pass spends its time on (one warp instruction per 19 cycles and SM; 64
// cycles for a single warp of a quarter SM, dependent or not), so FP64 plans
// take radix 4, many threads and, against a radix-2 pass left over, radix 8;
// FP32 passes are bound by the shared-memory exchanges and take radix 8.
#pragma once

#include "common.cuh"

namespace mm {

constexpr int kLineMaxPass = 12;
// entries of the concatenated tables W_L^m; behind them, in FP64, the same twiddles
// as LineTwiddle takes them
constexpr int kTwRt = 173884;
// |Im W_L^m| > |Re W_L^m| (8 m mod 4 L between L and 3 L)
__host__ __device__ __forceinline__ constexpr bool line_turn(int m, int L) {
    const int q = 8 * m - (2 * m >= L ? 4 * L : 0);
    return q > L && q < 3 * L;
}
constexpr int kLineIdle = 1 << 20;       // butterfly number of a thread without a line: past every pass's count

struct LinePlan {
    int L, np;
    int tw;                            // offset of W_L^m in the table
    int rmin;                          // smallest radix: L / rmin butterflies in the widest pass
    short R[kLineMaxPass];             // forward order; the inverse runs them backwards
    short Ns[kLineMaxPass];            // forward spans
    short Nsi[kLineMaxPass];           // spans of the inverse's passes, in its order
    unsigned mg[kLineMaxPass], mgi[kLineMaxPass];   // ceil(2^32 / span)
};

// The factors of L, as few as radices up to rmax (and 3, 5, 7) allow and among
// those the largest smallest one, largest first: from radix number `at` on,
// appended to cur[0..n).
struct LineFactors {
    int n = 0, f[kLineMaxPass] = {};
};
constexpr void line_factors(int L, int rmax, int at, LineFactors cur, LineFactors& best) {
    constexpr int radix[7] = {8, 7, 6, 5, 4, 3, 2};
    if (L == 1) {
        if (best.n == 0 || cur.n < best.n || (cur.n == best.n && cur.f[cur.n - 1] > best.f[best.n - 1])) best = cur;
        return;
    }
    if (cur.n == kLineMaxPass || (best.n && cur.n >= best.n)) return;
    for (int i = at; i < 7; ++i) {
        const int r = radix[i];
        if (L % r || (r > rmax && r % 2 == 0)) continue;
        LineFactors next = cur;
        next.f[next.n++] = r;
        line_factors(L / r, rmax, i, next, best);
    }
}

// The plan of an even length (np = 0: not one of the engine's): an even radix
// first, the largest of the others last.
constexpr LinePlan line_plan(int L, int rmax) {
    LinePlan p{};
    p.L = L;
    LineFactors f;
    line_factors(L, rmax, 0, LineFactors(), f);
    if (f.n == 0) return p;
    p.np = f.n;
    p.rmin = f.f[f.n - 1];
    int first = 0;
    while (f.f[first] % 2) ++first;
    p.R[0] = (short)f.f[first];
    for (int i = 0, at = f.n - 1; i < f.n; ++i)
        if (i != first) p.R[at--] = (short)f.f[i];
    for (int i = 0, a = 1, b = 1; i < p.np; ++i) {
        p.Ns[i] = (short)a;
        p.Nsi[i] = (short)b;
        p.mg[i] = (unsigned)(((1ull << 32) + a - 1) / a);
        p.mgi[i] = (unsigned)(((1ull << 32) + b - 1) / b);
        a *= p.R[i];
        b *= p.R[p.np - 1 - i];
    }
    return p;
}
// threads of a CTA at most.  FP32 passes wait on memory: three CTAs of 256
// threads per SM (85 registers); the 512-thread variant takes the lines with
// more butterflies.
constexpr int kLineThreads = 512, kLineThreads32 = 256;
// plan of an FP32 compiled length
template <typename T> __host__ __device__ constexpr LinePlan line_ct(int L) { return line_plan(L, 8); }
// FP64 z lines whose three components fit a CTA side by side take a thread per
// butterfly and component (32x32x4: 9.5 -> 6.6 us, 128x128x32: 416 -> 382 us; in
// FP32 the extra exchange costs more than the threads bring: 32 grids of
// 256x256x1 105 against 68 us).  M: butterflies of the widest pass.
template <typename T> __host__ __device__ constexpr bool line_split(int M) { return sizeof(T) == 8 && M <= 128; }
// their columns per CTA (log2): a sector of each row at least, and three warps
__host__ __device__ constexpr int line_split_lb(int M) {
    int lb = 1;
    while (lb < 5 && ((3 * M) << lb) < 96) ++lb;
    return lb;
}
// columns per CTA (log2) of a compiled length otherwise: a sector of each row at least, and two warps
template <typename T> __host__ __device__ constexpr int line_ct_lb(int L) {
    const LinePlan p = line_ct<T>(L);
    int lb = sizeof(T) == 4 ? 2 : 1;
    while (lb < 5 && ((L / p.rmin) << lb) < 64) ++lb;
    while (lb > 0 && ((L / p.rmin) << lb) > 512) --lb;
    return lb;
}

// b mod Ns for b < 4096 with mg = ceil(2^32 / Ns): b mg / 2^32 is exact for b Ns < 2^32
// (mg = 0: Ns is a constant)
__device__ __forceinline__ int line_mod(int b, int Ns, unsigned mg) {
    return mg == 0 ? b % Ns : Ns == 1 ? 0 : b - (int)__umulhi((unsigned)b, mg) * Ns;
}

// One slot of padding every 2^SH elements spreads the strided writes of the
// first passes over the banks: every eight where several lines lie side by side
// (a warp reads eight elements of four lines), every sixteen where one line
// does (a half warp reads sixteen elements).
template <int SH> __host__ __device__ __forceinline__ int line_place(int e) { return e + (e >> SH); }
__host__ __device__ __forceinline__ constexpr int line_len(int L) { return L + (L >> 3) + 1; }

// Whether a CTA holds an FP64 line of L points with every plan the launches may
// choose (radices up to 2, 4 or 8), alone for the y and x passes and with its three
// components for the z pass: the lengths whose launches have nothing else to turn
// to.  (The one other reason to refuse, more than 65535 grids, is 16 times the
// largest batch.)
constexpr bool line_holds_fp64(int L) {
    for (int rmax = 2; rmax <= 8; rmax *= 2) {
        const LinePlan p = line_plan(L, rmax);
        if (p.np < (rmax < 8 ? 2 : 1) || L / p.rmin > kLineThreads) return false;
    }
    return 3 * 2 * sizeof(double) * line_len(L) <= 160 * 1024;
}

// -v or v; FP64 on the integer side (FP64 instructions are what an FP64 pass is made of)
__device__ __forceinline__ float line_flip(float v, bool neg) { return neg ? -v : v; }
__device__ __forceinline__ double line_flip(double v, bool neg) {
    return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000 : 0), __double2loint(v));
}

// Twiddles of the folded butterflies and x = a + w b, y = a - w b, neither formed
// from the other: y = 2 a - x would carry the rounding of a large x into a small
// y, as the spectrum of a nearly uniform magnetisation has them side by side.
//
// FP32 takes w as it is, eight multiply-adds.
template <typename T, int DIR> struct LineTwiddle {
    float2 w;
    __device__ __forceinline__ LineTwiddle(const float2* tw, int m, int) : w(__ldg(tw + m)) {
        if (DIR > 0) w.y = -w.y;
    }
    __device__ __forceinline__ void bf2(float2& a, float2& b) const { bf2(a, b, w); }
    __device__ __forceinline__ void bf2i(float2& a, float2& b) const { bf2(a, b, mul_i<DIR>(w)); }
    static __device__ __forceinline__ void bf2(float2& a, float2& b, float2 w) {
        const float2 x = make_float2(fma(w.x, b.x, fma(-w.y, b.y, a.x)), fma(w.x, b.y, fma(w.y, b.x, a.y)));
        b = make_float2(fma(-w.x, b.x, fma(w.y, b.y, a.x)), fma(-w.x, b.y, fma(-w.y, b.x, a.y)));
        a = x;
    }
};
// FP64, whose instructions bound the pass, takes w = c (1 + i t), |t| <= 1, after
// a quarter turn where |Im w| > |Re w| (Linzer and Feig 1993): w b costs two
// multiply-adds up to the factor c, which the two sums take in, six in all.  The
// turn costs selections on the integer side, which the twiddle's index decides:
// kept with the twiddle they would wait for its load (32x32x4: 1342 against 1304 us
// for ten RK4 steps).
template <int DIR> struct LineTwiddle<double, DIR> {
    double c, t;
    bool turn;
    __device__ __forceinline__ LineTwiddle(const double2* tw, int m, int L) : turn(line_turn(m, L)) {
        const double2 e = __ldg(tw + kTwRt + m);
        c = e.x;
        t = e.y;
    }
    __device__ __forceinline__ void bf2(double2& a, double2& b) const { bf2(a, b, turn, false); }
    __device__ __forceinline__ void bf2i(double2& a, double2& b) const { bf2(a, b, !turn, !turn); }
    // u = b, or -DIR i b (quarter), or DIR i b (quarter and back)
    __device__ __forceinline__ void bf2(double2& a, double2& b, bool quarter, bool back) const {
        const double ux = quarter ? b.y : b.x, uy = quarter ? b.x : b.y;
        const bool nx = quarter && (DIR < 0) != back, ny = quarter && (DIR > 0) != back;
        const double px = line_flip(ux, nx), py = line_flip(uy, ny);
        const double vx = fma(DIR < 0 ? -t : t, py, px), vy = fma(DIR < 0 ? t : -t, px, py);
        b = make_double2(fma(-c, vx, a.x), fma(-c, vy, a.y));
        a = make_double2(fma(c, vx, a.x), fma(c, vy, a.y));
    }
};

// DFT of R values, no twiddles; HALF: the upper half of the inputs is zero
template <int DIR, int R, bool HALF, typename C> __device__ __forceinline__ void line_dft(C (&x)[R]) {
    if constexpr (R == 2) {
        if constexpr (HALF) x[1] = x[0]; else dft2<DIR>(x[0], x[1]);
    } else if constexpr (R == 3) {
        dft3<DIR>(x[0], x[1], x[2]);
    } else if constexpr (R == 4) {
        if constexpr (HALF) {
            const C a = x[0], b = x[1], ib = mul_i<DIR>(b);
            x[0] = cadd(a, b); x[2] = csub(a, b); x[1] = cadd(a, ib); x[3] = csub(a, ib);
        } else {
            dft4<DIR>(x[0], x[1], x[2], x[3]);
        }
    } else if constexpr (R == 5) {
        dft5<DIR>(x[0], x[1], x[2], x[3], x[4]);
    } else if constexpr (R == 6) {
        if constexpr (HALF) x[3] = x[4] = x[5] = mk<C>(0, 0);
        dft6<DIR>(x);
    } else if constexpr (R == 7) {
        dft7<DIR>(x);
    } else if constexpr (R == 12) {
        if constexpr (HALF) {
#pragma unroll
            for (int q = 6; q < 12; ++q) x[q] = mk<C>(0, 0);
        }
        dft12<DIR>(x);
    } else if constexpr (R == 16) {
        dft16<DIR, HALF>(x);
    } else {
        static_assert(R == 8, "no such radix");
        if constexpr (HALF) dft8_half<DIR>(x); else dft8<DIR>(x);
    }
}

// one butterfly of NC components: twiddles (none for span 1), then the DFT
template <typename T, int DIR, int R, int NC>
__device__ __forceinline__ void line_butterfly(typename Cplx<T>::type (&x)[NC][R], const typename Cplx<T>::type* tw,
                                               int k, int step, int L) {
    using C = typename Cplx<T>::type;
    using Tw = LineTwiddle<T, DIR>;
    auto W = [&](int m) {
        C w = __ldg(tw + m);
        if (DIR > 0) w.y = -w.y;
        return w;
    };
    if constexpr (R == 2) {
        const Tw w(tw, k * step, L);
#pragma unroll
        for (int c = 0; c < NC; ++c) w.bf2(x[c][0], x[c][1]);
    } else if constexpr (R == 4) {
        const Tw w1(tw, k * step, L), w2(tw, 2 * k * step, L);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            C* a = x[c];
            w2.bf2(a[0], a[2]);           // t0, t1
            w2.bf2(a[1], a[3]);           // t2, t3
            w1.bf2(a[0], a[1]);           // X0, X2
            w1.bf2i(a[2], a[3]);          // X1, X3
            const C x1 = a[2];
            a[2] = a[1]; a[1] = x1;
        }
    } else if constexpr (R == 8) {
        // W_8 w1 = W_L^(k step + L/8)
        const Tw w1(tw, k * step, L), w2(tw, 2 * k * step, L), w4(tw, 4 * k * step, L), u(tw, k * step + L / 8, L);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            C* a = x[c];
            w4.bf2(a[0], a[4]); w4.bf2(a[2], a[6]);
            w2.bf2(a[0], a[2]); w2.bf2i(a[4], a[6]);     // E0 E2 | E1 E3 in a0 a2 a4 a6
            w4.bf2(a[1], a[5]); w4.bf2(a[3], a[7]);
            w2.bf2(a[1], a[3]); w2.bf2i(a[5], a[7]);     // O0 O2 | O1 O3 in a1 a3 a5 a7
            w1.bf2(a[0], a[1]);             // X0, X4
            u.bf2(a[4], a[5]);              // X1, X5
            w1.bf2i(a[2], a[3]);            // X2, X6
            u.bf2i(a[6], a[7]);             // X3, X7
            const C x4 = a[1], x1 = a[4], x6 = a[3], x3 = a[6];
            a[1] = x1; a[3] = x3; a[4] = x4; a[6] = x6;
        }
    } else {
#pragma unroll
        for (int q = 1; q < R; ++q) {
            const C w = W(q * k * step);
#pragma unroll
            for (int c = 0; c < NC; ++c) x[c][q] = cmul(x[c][q], w);
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) line_dft<DIR, R, false>(x[c]);
    }
}

template <int SH, typename C, int R, int NC>
__device__ __forceinline__ void line_load(C (&x)[NC][R], const C* s, int plane, int lb, int b, int M) {
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const C* p = s + (line_place<SH>(b + q * M) << lb);
#pragma unroll
        for (int c = 0; c < NC; ++c) x[c][q] = p[c * plane];
    }
}
template <int SH, typename C, int R, int NC>
__device__ __forceinline__ void line_store(const C (&x)[NC][R], C* s, int plane, int lb, int b, int k, int Ns) {
#pragma unroll
    for (int q = 0; q < R; ++q) {
        C* p = s + (line_place<SH>((b - k) * R + k + q * Ns) << lb);
#pragma unroll
        for (int c = 0; c < NC; ++c) p[c * plane] = x[c][q];
    }
}

// a pass between two others, in place; s is the thread's line.  Every thread of
// the CTA calls it.
template <typename T, int DIR, int R, int NC, int SH>
__device__ __forceinline__ void line_mid(typename Cplx<T>::type* s, int plane, int lb, int b, int L, int Ns,
                                         unsigned mg, const typename Cplx<T>::type* tw) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    // threads without a butterfly compute the first one and store nothing: values
    // set under a condition would stay live around the loop over passes and spill
    const bool on = b < M;
    if (!on) b = 0;
    C x[NC][R];
    const int k = line_mod(b, Ns, mg);
    line_load<SH>(x, s, plane, lb, b, M);
    line_butterfly<T, DIR>(x, tw, k, L / (Ns * R), L);
    __syncthreads();
    if (on) line_store<SH>(x, s, plane, lb, b, k, Ns);
    __syncthreads();
}

// a first pass in place: no twiddles, any input
template <typename T, int DIR, int R, int NC, int SH>
__device__ __forceinline__ void line_start(typename Cplx<T>::type* s, int plane, int lb, int b, int L) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    const bool on = b < M;
    if (!on) b = 0;
    C x[NC][R];
    line_load<SH>(x, s, plane, lb, b, M);
#pragma unroll
    for (int c = 0; c < NC; ++c) line_dft<DIR, R, false>(x[c]);
    __syncthreads();
    if (on) line_store<SH>(x, s, plane, lb, b, 0, 1);
    __syncthreads();
}

// Whether a warp has no butterfly in a pass of radix R (IDLE kernels: FP64 plans of
// unequal radices).  Plans of one radix 2 and odd ones have 2.5 to 3.5 times as
// many threads as their odd passes have butterflies, and in FP64 idle threads'
// instructions take the pipe from the others: with them an RK4 stage of 64x32x245
// (2 5 7 7) took 3307 us, without 1640.  FP32, bound by its exchanges, does without
// the vote, and so do plans of equal radices (32x32x4 with the vote in its kernels:
// 1342 against 1304 us).  Every warp is whole.
template <bool IDLE> __device__ __forceinline__ bool line_warp_idle(const LinePlan& pl, int R, int b) {
    return IDLE && !__any_sync(0xffffffffu, b * R < pl.L);
}
// the two barriers of a pass in place, for a warp that leaves it out
__device__ __forceinline__ void line_pass_over() {
    asm volatile("bar.sync 0;\n\tbar.sync 0;" ::: "memory");
}

// CALL with R_ = the radix (Wv: plans with a 6 or an 8 come here too)
#define MM_LINE_RADIX(Wv, Rv, CALL)                                           \
    switch (Rv) {                                                         \
        case 2: { constexpr int R_ = 2; CALL; } break;                     \
        case 3: { constexpr int R_ = 3; CALL; } break;                     \
        case 4: { constexpr int R_ = 4; CALL; } break;                     \
        case 5: { constexpr int R_ = 5; CALL; } break;                     \
        case 7: { constexpr int R_ = 7; CALL; } break;                     \
        case 6: { constexpr int R_ = (Wv) ? 6 : 2; CALL; } break; \
        default: { constexpr int R_ = (Wv) ? 8 : 2; CALL; } break; \
    }
#define MM_LINE_RADIX_EVEN(Wv, Rv, CALL)                                      \
    switch (Rv) {                                                         \
        case 2: { constexpr int R_ = 2; CALL; } break;                     \
        case 4: { constexpr int R_ = 4; CALL; } break;                     \
        case 6: { constexpr int R_ = (Wv) ? 6 : 2; CALL; } break; \
        default: { constexpr int R_ = (Wv) ? 8 : 2; CALL; } break; \
    }

template <typename T, int DIR, int NC, int SH, bool WIDE, bool IDLE>
__device__ __forceinline__ void line_mid_any(typename Cplx<T>::type* s, int plane, int lb, int b, const LinePlan& pl,
                                             int i, const typename Cplx<T>::type* tw) {
    const int R = DIR < 0 ? pl.R[i] : pl.R[pl.np - 1 - i];
    const int Ns = DIR < 0 ? pl.Ns[i] : pl.Nsi[i];
    const unsigned mg = DIR < 0 ? pl.mg[i] : pl.mgi[i];
    if (line_warp_idle<IDLE>(pl, R, b)) return line_pass_over();
    MM_LINE_RADIX(WIDE, R, (line_mid<T, DIR, R_, NC, SH>(s, plane, lb, b, pl.L, Ns, mg, tw)));
}

// passes I .. END-1 of a compiled length
template <typename T, int DIR, int NC, int SH, int LC, int I, int END>
__device__ __forceinline__ void line_mids_ct(typename Cplx<T>::type* s, int plane, int lb, int b,
                                             const typename Cplx<T>::type* tw) {
    if constexpr (I < END) {
        constexpr LinePlan P = line_ct<T>(LC);
        constexpr int R = DIR < 0 ? P.R[I] : P.R[P.np - 1 - I], Ns = DIR < 0 ? P.Ns[I] : P.Nsi[I];
        line_mid<T, DIR, R, NC, SH>(s, plane, lb, b, LC, Ns, 0, tw);
        line_mids_ct<T, DIR, NC, SH, LC, I + 1, END>(s, plane, lb, b, tw);
    }
}

}  // namespace mm
