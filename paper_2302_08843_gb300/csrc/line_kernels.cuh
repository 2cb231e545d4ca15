// Kernels of the line engine.  Each is written for a plan known at run time
// (LC = 0) and for a compiled length LC (FP32): the plan is then a constant and
// the index arithmetic, more than half of the instructions otherwise, folds into
// addresses.  tw: the table W_L^m of the line's length.
//
// x passes: x-forward (r2c) of Ms m, or of a Runge-Kutta
// combination formed on the way; x-inverse (c2r) of the demag spectrum; and the
// fused x-inverse + local terms + LLG + Runge-Kutta combination + x-forward of
// the next stage input (FP32).
//
// A line is two real rows a + i b.  With NC = 3 they are two neighbouring rows
// of y of one plane, for all three components; with NC = 1 two consecutive rows
// of the 3 ny nz rows of a grid, whatever their component.  Rows never pair
// across grids of a batch.  One line after another in shared memory
// (line l, component c at (l NC + c) len), threads of a line side by side.
#pragma once

#include "demag.h"
#include "fft_pair.cuh"
#include "line_engine.cuh"
#include "tma.cuh"

namespace mm {

template <typename T, int MAXT> constexpr int line_blocks() { return sizeof(T) == 4 && MAXT == kLineThreads32 ? 3 : 1; }


// the rows a CTA's line stands for: first row of each component and their distance
struct LineRows {
    long ra;         // row index of a's first component within the grid
    int z, y;        // NC = 3: plane and first row of y
    bool on, two;    // a line of this grid; b exists
};
template <int NC> __device__ __forceinline__ LineRows line_rows(const DemagDims& d, int q) {
    LineRows r;
    if (NC == 3) {
        const int ppz = (d.ny + 1) >> 1;
        r.z = q / ppz;
        r.y = 2 * (q - r.z * ppz);
        r.on = r.z < d.nz;
        r.two = r.y + 1 < d.ny;
        r.ra = (long)r.z * d.ny + r.y;
    } else {
        const long rows = 3L * d.ny * d.nz;
        r.ra = 2L * q;
        r.on = r.ra < rows;
        r.two = r.ra + 1 < rows;
        r.z = r.y = 0;
    }
    if (!r.on) r.ra = 0;
    if (!r.on) r.two = false;
    return r;
}

// c2r input element e of a line from its two spectrum rows
template <typename T>
__device__ __forceinline__ typename Cplx<T>::type line_c2r(const typename Cplx<T>::type* sa,
                                                           const typename Cplx<T>::type* sb, int e, int L) {
    using C = typename Cplx<T>::type;
    const bool up = 2 * e > L;
    const int k = up ? L - e : e;
    C a = sa[k], b = sb[k];
    if (k == 0 || 2 * k == L) a.y = b.y = 0;      // a real row has real DC and Nyquist
    return up ? mk<C>(a.x + b.y, b.x - a.y) : mk<C>(a.x - b.y, a.y + b.x);
}

// first pass of the x-inverse, straight from the spectrum rows
template <typename T, int R, int NC>
__device__ __forceinline__ void line_x_first(const typename Cplx<T>::type* sa, const typename Cplx<T>::type* sb,
                                             long cs, typename Cplx<T>::type* s, int plane, int b, int L) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    if (b >= M) return;
    C x[NC][R];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int q = 0; q < R; ++q) x[c][q] = line_c2r<T>(sa + c * cs, sb + c * cs, b + q * M, L);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) line_dft<+1, R, false>(x[c]);
    line_store<4>(x, s, plane, 0, b, 0, 1);
}

// last pass of the x-inverse: the kept half back to its natural places
template <typename T, int R, int NC>
__device__ __forceinline__ void line_x_last(typename Cplx<T>::type* s, int plane, int b, int L, int Ns, unsigned mg,
                                            const typename Cplx<T>::type* tw) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    const bool on = b < M;
    if (!on) b = 0;
    C x[NC][R];
    line_load<4>(x, s, plane, 0, b, M);
    line_butterfly<T, +1>(x, tw, line_mod(b, Ns, mg), L / (Ns * R), L);
    __syncthreads();
    if (on) {
#pragma unroll
        for (int q = 0; q < R / 2; ++q)
#pragma unroll
            for (int c = 0; c < NC; ++c) s[c * plane + line_place<4>(b + q * M)] = x[c][q];
    }
    __syncthreads();
}

// first pass of the x-forward, in place, inputs e < nx at their natural places
template <typename T, int R, int NC>
__device__ __forceinline__ void line_f_first(typename Cplx<T>::type* s, int plane, int b, int L, int nx) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    const bool on = b < M;
    if (!on) b = 0;
    C x[NC][R];
#pragma unroll
    for (int q = 0; q < R / 2; ++q) {
        const int e = b + q * M;
#pragma unroll
        for (int c = 0; c < NC; ++c) x[c][q] = e < nx ? s[c * plane + line_place<4>(e)] : mk<C>(0, 0);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) line_dft<-1, R, true>(x[c]);
    __syncthreads();
    if (on) line_store<4>(x, s, plane, 0, b, 0, 1);
    __syncthreads();
}

// inverse of one line in shared memory (the first pass reads global memory); ends synchronised
template <typename T, int NC, int LC, bool IDLE = false>
__device__ __forceinline__ void line_inverse(const typename Cplx<T>::type* sa, const typename Cplx<T>::type* sb,
                                             long cs, typename Cplx<T>::type* s, int plane, int b,
                                             const LinePlan& pl, const typename Cplx<T>::type* tw) {
    if constexpr (LC > 0) {
        constexpr LinePlan P = line_ct<T>(LC);
        constexpr int np = P.np;
        line_x_first<T, P.R[np - 1], NC>(sa, sb, cs, s, plane, b, LC);
        __syncthreads();
        line_mids_ct<T, +1, NC, 4, LC, 1, np - 1>(s, plane, 0, b, tw);
        line_x_last<T, P.R[0], NC>(s, plane, b, LC, P.Nsi[np - 1], 0, tw);
    } else {
        const int np = pl.np, L = pl.L;
        MM_LINE_RADIX(true, pl.R[np - 1], (line_x_first<T, R_, NC>(sa, sb, cs, s, plane, b, L)));
        __syncthreads();
        for (int i = 1; i < np - 1; ++i) line_mid_any<T, +1, NC, 4, true, IDLE>(s, plane, 0, b, pl, i, tw);
        if (line_warp_idle<IDLE>(pl, pl.R[0], b)) return line_pass_over();
        MM_LINE_RADIX_EVEN(true, pl.R[0], (line_x_last<T, R_, NC>(s, plane, b, L, pl.Nsi[np - 1], pl.mgi[np - 1], tw)));
    }
}

// forward of one line in shared memory and the r2c split into the two
// spectrum rows; nt threads per line, this one b; called with the inputs in place and synchronised
template <typename T, int NC, int LC, bool IDLE = false>
__device__ __forceinline__ void line_forward(typename Cplx<T>::type* s, int plane, int b, int nt, int nx,
                                             const LinePlan& pl, const typename Cplx<T>::type* tw,
                                             typename Cplx<T>::type* sa, typename Cplx<T>::type* sb, long cs,
                                             bool on, bool two) {
    using C = typename Cplx<T>::type;
    const int L = LC ? LC : pl.L;
    if constexpr (LC > 0) {
        constexpr LinePlan P = line_ct<T>(LC);
        line_f_first<T, P.R[0], NC>(s, plane, b, LC, nx);
        line_mids_ct<T, -1, NC, 4, LC, 1, P.np>(s, plane, 0, b, tw);
    } else {
        if (line_warp_idle<IDLE>(pl, pl.R[0], b)) line_pass_over();
        else MM_LINE_RADIX_EVEN(true, pl.R[0], (line_f_first<T, R_, NC>(s, plane, b, L, nx)));
        for (int i = 1; i < pl.np; ++i) line_mid_any<T, -1, NC, 4, true, IDLE>(s, plane, 0, b, pl, i, tw);
    }
    if (!on) return;
    const T half = (T)0.5;
    for (int k = b; 2 * k <= L; k += nt) {
        const int pk = line_place<4>(k), pm = line_place<4>(k ? L - k : 0);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const C zk = s[c * plane + pk], zm = s[c * plane + pm];
            sa[c * cs + k] = mk<C>(half * (zk.x + zm.x), half * (zk.y - zm.y));
            if (two) sb[c * cs + k] = mk<C>(half * (zk.y + zm.y), half * (zm.x - zk.x));
        }
    }
}

// what a CTA's thread works on: line l of the CTA, butterfly b of nt
struct LineThread {
    int l, b;
    bool in;       // a thread of one of the CTA's lines (not of the tail of the last warp)
};
__device__ __forceinline__ LineThread line_thread(int nt, int lines) {
    LineThread t;
    t.l = threadIdx.x / nt;
    t.b = threadIdx.x - t.l * nt;
    t.in = t.l < lines;
    // tail threads follow the last line as butterflies past every pass's count
    if (!t.in) { t.l = lines - 1; t.b = kLineIdle; }
    return t;
}

// x-forward of Ms m (comb: of Ms (m + dt ca k), which is also stored in y)
template <typename T> struct LineForward {
    const T* m;
    const T* Ms_cell;
    T Ms;
    const T* k;           // null: m itself
    T* y;
    T ca;                 // dt ca, one grid
    const double* dt_b;   // per grid, times a
    double a;
    const int* mask;      // grids to work on, or null
};

template <typename T, int MAXT, int LC, bool IDLE = false>
__global__ void __launch_bounds__(MAXT)
line_x_forward(DemagDims d, LineForward<T> f, typename Cplx<T>::type* __restrict__ S1,
               const __grid_constant__ LinePlan pl, const typename Cplx<T>::type* __restrict__ tw, int nt, int lines) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    if constexpr (LC > 0) {
        constexpr int kNt = LC / line_ct<T>(LC).rmin;
        nt = kNt;
    }
    const LineThread t = line_thread(nt, lines);
    const int g = blockIdx.y, nx = d.nx, plane = line_len(LC ? LC : pl.L);
    const LineRows r = line_rows<1>(d, blockIdx.x * lines + t.l);
    const long rows = (long)d.ny * d.nz;             // rows of one component
    C* s = reinterpret_cast<C*>(smraw) + (size_t)t.l * plane;
    grid_dep_wait();
    if (f.mask && !f.mask[g]) return;
    const T* Ms_b = static_cast<const T*>(d.Ms_b);
    const T msu = Ms_b ? Ms_b[g] : f.Ms;
    const T ca = f.dt_b ? (T)(f.dt_b[g] * f.a) : f.ca;
    const long off = (long)g * 3 * rows;
    if (r.on && t.in) {
        // kBatch elements of both rows in flight per thread
        constexpr int kBatch = 4;
        for (int x0 = t.b; x0 < nx; x0 += kBatch * nt) {
            C v[kBatch];
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const int x = min(x0 + q * nt, nx - 1);
                const T* m = f.m + (off + r.ra) * nx + x;
                v[q] = mk<C>(__ldcg(m), r.two ? __ldcg(m + nx) : (T)0);
                if (f.k) {
                    const T* k = f.k + (m - f.m);
                    v[q].x += ca * __ldcg(k);
                    if (r.two) v[q].y += ca * __ldcg(k + nx);
                }
            }
#pragma unroll
            for (int q = 0; q < kBatch; ++q) {
                const int x = x0 + q * nt;
                if (x >= nx) break;
                if (f.k) {
                    T* y = f.y + (off + r.ra) * nx + x;
                    y[0] = v[q].x;
                    if (r.two) y[nx] = v[q].y;
                }
                T ma = msu, mb = msu;
                if (f.Ms_cell && !Ms_b) {
                    ma = f.Ms_cell[(r.ra % rows) * nx + x];
                    mb = r.two ? f.Ms_cell[((r.ra + 1) % rows) * nx + x] : (T)0;
                }
                s[line_place<4>(x)] = mk<C>(ma * v[q].x, mb * v[q].y);
            }
        }
    }
    __syncthreads();
    C* sa = S1 + (off + r.ra) * d.KXS;
    line_forward<T, 1, LC, IDLE>(s, plane, t.b, nt, nx, pl, tw, sa, sa + d.KXS, 0, r.on && t.in, r.two);
}

template <typename T, int MAXT, int LC, bool IDLE = false>
__global__ void __launch_bounds__(MAXT)
line_x_inverse(DemagDims d, const typename Cplx<T>::type* __restrict__ S1, T* __restrict__ h,
               const __grid_constant__ LinePlan pl, const typename Cplx<T>::type* __restrict__ tw, int nt, int lines) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    if constexpr (LC > 0) {
        constexpr int kNt = LC / line_ct<T>(LC).rmin;
        nt = kNt;
    }
    const LineThread t = line_thread(nt, lines);
    const int nx = d.nx, plane = line_len(LC ? LC : pl.L);
    const LineRows r = line_rows<1>(d, blockIdx.x * lines + t.l);
    const long rows = (long)d.ny * d.nz, off = (long)blockIdx.y * 3 * rows;
    C* s = reinterpret_cast<C*>(smraw) + (size_t)t.l * plane;
    const C* sa = S1 + (off + r.ra) * d.KXS;
    grid_dep_wait();
    line_inverse<T, 1, LC, IDLE>(sa, r.two ? sa + d.KXS : sa, 0, s, plane, t.b, pl, tw);
    if (!r.on || !t.in) return;
    for (int x = t.b; x < nx; x += nt) {
        const C v = s[line_place<4>(x)];
        T* o = h + (off + r.ra) * nx + x;
        o[0] = v.x;
        if (r.two) o[nx] = v.y;
    }
}


// ---------------------------------------------------------- fused stage ----
__device__ __forceinline__ float line_harm(float a, float b) {
    const float s = a + b;
    return s != 0.f ? 2.f * a * b / s : 0.f;
}
__device__ __forceinline__ float line_thick(float a, float b, float ha, float hb) {
    const float s = ha * b + hb * a;
    return s != 0.f ? (ha + hb) * a * b / s : 0.f;
}
__device__ __forceinline__ float line_davg(float a, float b) {
    const float prod = a * b, s = a + b;
    if (prod >= 0.f) return s != 0.f ? 2.f * prod / s : 0.f;
    return copysignf(sqrtf(sqrtf(-prod) * fabsf(s) * 0.5f), s);
}

// Reductions a thread carries over its cells.
struct LineRed {
    float tq2, tq, en, ed;     // largest |m x h|^2 (uniform Ms) and |m x h| / Ms, error ratio en / ed
    int nf;
    float2 e[5];               // energy sums, sum Ms m.h per term, as high and low parts
};

// Sums of FP32 products kept exact to 48 bits as high and low parts (products
// and sums with their rounding errors: Dekker 1971, Knuth's two-sum): FP64
// instructions run at 1/64 of the FP32 rate here, and a field of 100x65x27 cells
// with its energies took 35.6 us in FP64 sums, 30.8 us so.
__device__ __forceinline__ void line_acc(float2& s, float p, float e) {
    const float t = __fadd_rn(s.x, p), z = __fsub_rn(t, s.x);
    s.y = __fadd_rn(s.y, __fadd_rn(__fadd_rn(__fsub_rn(s.x, __fsub_rn(t, z)), __fsub_rn(p, z)), e));
    s.x = t;
}
__device__ __forceinline__ void line_acc_prod(float2& s, float a, float b) {
    const float p = __fmul_rn(a, b);
    line_acc(s, p, __fmaf_rn(a, b, -p));
}

// One item: the cells (x, ya) and (x, yb) of the line's two rows as the lanes
// of paired FP32 instructions.  ia, ib: their indices in the grid (ib = ia for
// a missing second row); v: the demag field in, Ms next out; rk: the known part
// of the derivatives' sum and of the error (line_known).
template <bool GEN>
__device__ __forceinline__ void line_cells(const StageParams<float>& p, const LineBatch& bt, int g, long off, int x,
                                           int y, int z, bool two, const float2 (&rk)[6], float2 (&v)[3],
                                           LineRed& red) {
    const int nx = p.nx, ny = p.ny, nz = p.nz, N = (int)p.N;
    const int ia = x + nx * (y + ny * z), ib = two ? ia + nx : ia;
    const bool batch = bt.mask != nullptr;
    const float* m = p.m + off;
    auto ld = [&](const float* q) { return make_float2(q[ia], q[ib]); };
    // streams that are read once pass the L1 by, which the twiddles and the stencil share
    auto lds = [&](const float* q) { return make_float2(__ldcg(q + ia), __ldcg(q + ib)); };
    const float2 mx = ld(m), my = ld(m + N), mz = ld(m + 2 * N);
    const float Msu = batch ? bt.Ms[g] : p.Ms, Au = batch ? bt.A[g] : p.A;
    const float2 Ms = GEN && !batch && p.Ms_cell ? ld(p.Ms_cell) : f2s(Msu);
    const bool a_cell = GEN && !batch && p.A_cell;
    const float2 A = a_cell ? ld(p.A_cell) : f2s(Au);
    const int kind = GEN && batch ? bt.kind[g] : 0;
    const bool dmi = GEN && (batch ? kind != 0 : p.dmi != 0);
    const bool d_cell = GEN && !batch && p.D_cell;
    const float Du = GEN && dmi ? (batch ? bt.D[g] : p.D) : 0.f;
    const float2 Dc = d_cell ? ld(p.D_cell) : f2s(Du);
    const float* ev = batch ? bt.dmi_e[kind] : p.dmi_e;
    const float2 zero = f2s(0.f);
    float2 sx = zero, sy = zero, sz = zero, qx = zero, qy = zero, qz = zero;
    // link to cells ja, jb; a missing neighbour (ha, hb false) stands in as the
    // cell itself and adds nothing
    auto link = [&](int ja, int jb, bool ha, bool hb, float id2, const float* e, float si2d, bool thick, float hk,
                    float hn) {
        const float2 a = make_float2(m[ja], m[jb]), b = make_float2(m[N + ja], m[N + jb]),
                     c = make_float2(m[2 * N + ja], m[2 * N + jb]);
        float2 w = f2s(Au * id2);
        if (a_cell) {
            const float2 An = make_float2(p.A_cell[ja], p.A_cell[jb]);
            w = thick ? make_float2(id2 * line_thick(A.x, An.x, hk, hn), id2 * line_thick(A.y, An.y, hk, hn))
                      : make_float2(id2 * line_harm(A.x, An.x), id2 * line_harm(A.y, An.y));
        }
        sx = f2fma(w, f2sub(a, mx), sx);
        sy = f2fma(w, f2sub(b, my), sy);
        sz = f2fma(w, f2sub(c, mz), sz);
        if (GEN && dmi) {
            float2 D = Dc;
            if (d_cell) D = make_float2(line_davg(Dc.x, p.D_cell[ja]), line_davg(Dc.y, p.D_cell[jb]));
            D = f2mul(D, make_float2(ha ? si2d : 0.f, hb ? si2d : 0.f));
            qx = f2fma(D, f2sub(f2mul(f2s(e[1]), c), f2mul(f2s(e[2]), b)), qx);
            qy = f2fma(D, f2sub(f2mul(f2s(e[2]), a), f2mul(f2s(e[0]), c)), qy);
            qz = f2fma(D, f2sub(f2mul(f2s(e[0]), b), f2mul(f2s(e[1]), a)), qz);
        }
    };
    // (no branches along x and y: the loads of all four links go out together)
    {
        const bool xl = x > 0, xr = x < nx - 1, lo = y > 0, hi = two && y + 2 < ny;
        link(ia - xl, ib - xl, xl, xl, p.idx2, ev, -p.i2dx, false, 0.f, 0.f);
        link(ia + xr, ib + xr, xr, xr, p.idx2, ev, p.i2dx, false, 0.f, 0.f);
        link(lo ? ia - nx : ia, ia, lo, two, p.idy2, ev + 3, -p.i2dy, false, 0.f, 0.f);
        link(ib, hi ? ib + nx : ib, two, hi, p.idy2, ev + 3, p.i2dy, false, 0.f, 0.f);
    }
    const int pl = nx * ny;
    if (GEN && p.lay) {
        const float hk = p.lay[z];
        if (z > 0) link(ia - pl, ib - pl, true, true, p.lay[2 * nz + z], ev + 6, -p.i2dz, true, hk, p.lay[z - 1]);
        if (z < nz - 1) link(ia + pl, ib + pl, true, true, p.lay[nz + z], ev + 6, p.i2dz, true, hk, p.lay[z + 1]);
    } else {
        if (z > 0) link(ia - pl, ib - pl, true, true, p.idz2, ev + 6, -p.i2dz, false, 0.f, 0.f);
        if (z < nz - 1) link(ia + pl, ib + pl, true, true, p.idz2, ev + 6, p.i2dz, false, 0.f, 0.f);
    }
    // field
    const float c2 = (float)(2.0 / kMu0);
    float2 cex, on = f2s(1.f);
    if (GEN && !batch && p.Ms_cell) {
        cex = make_float2(Ms.x != 0.f ? c2 * (1.f / Ms.x) : 0.f, Ms.y != 0.f ? c2 * (1.f / Ms.y) : 0.f);
        on = make_float2(Ms.x != 0.f ? 1.f : 0.f, Ms.y != 0.f ? 1.f : 0.f);
    } else if (batch) {
        cex = f2s(Msu != 0.f ? c2 / Msu : 0.f);
        if (Msu == 0.f) on = zero;
    } else {
        cex = f2s(p.cex_u);
        if (GEN && Msu == 0.f) on = zero;
    }
    const float2 hex = f2mul(cex, sx), hey = f2mul(cex, sy), hez = f2mul(cex, sz);
    float2 hax = zero, hay = zero, haz = zero;
    const float2 Ku = GEN && !batch && p.Ku_cell ? ld(p.Ku_cell) : f2s(batch ? 0.f : p.Ku);
    if (Ku.x != 0.f || Ku.y != 0.f) {
        float2 ex = f2s(p.ex), ey = f2s(p.ey), ez = f2s(p.ez);
        if (p.grain) {
            const int g0 = 3 * p.grain[ia], g1 = 3 * p.grain[ib];
            ex = make_float2(p.axis_tab[g0], p.axis_tab[g1]);
            ey = make_float2(p.axis_tab[g0 + 1], p.axis_tab[g1 + 1]);
            ez = make_float2(p.axis_tab[g0 + 2], p.axis_tab[g1 + 2]);
        }
        const float2 ck = GEN && (p.Ms_cell || p.Ku_cell) ? f2mul(Ku, cex) : f2s(p.cani_u);
        const float2 c = f2mul(ck, f2fma(ex, mx, f2fma(ey, my, f2mul(ez, mz))));
        hax = f2mul(c, ex); hay = f2mul(c, ey); haz = f2mul(c, ez);
    }
    const float2 zw = GEN && p.zw ? ld(p.zw) : f2s(1.f);
    const float2 hzx = f2mul(zw, f2s(p.hx0)), hzy = f2mul(zw, f2s(p.hy0)), hzz = f2mul(zw, f2s(p.hz0));
    const float2 hmx = f2mul(cex, qx), hmy = f2mul(cex, qy), hmz = f2mul(cex, qz);
    float2 hx = f2add(f2add(v[0], hex), f2add(hax, hzx)), hy = f2add(f2add(v[1], hey), f2add(hay, hzy)),
           hz = f2add(f2add(v[2], hez), f2add(haz, hzz));
    if (GEN && dmi) { hx = f2add(hx, hmx); hy = f2add(hy, hmy); hz = f2add(hz, hmz); }
    if (GEN) {     // cells without magnetisation carry no field, whatever the sums hold
        if (on.x == 0.f) hx.x = hy.x = hz.x = 0.f;
        if (on.y == 0.f) hx.y = hy.y = hz.y = 0.f;
    }
    // Eq. llg
    float2 cx = f2sub(f2mul(my, hz), f2mul(mz, hy)), cy = f2sub(f2mul(mz, hx), f2mul(mx, hz)),
           cz = f2sub(f2mul(mx, hy), f2mul(my, hx));
    // a missing second row is the first one again, its field included: the
    // reductions see the first row's cells twice
    if (!two) { cx.y = cx.x; cy.y = cy.x; cz.y = cz.x; }
    const float2 dx_ = f2sub(f2mul(my, cz), f2mul(mz, cy)), dy_ = f2sub(f2mul(mz, cx), f2mul(mx, cz)),
                 dz_ = f2sub(f2mul(mx, cy), f2mul(my, cx));
    float2 al = f2s(batch ? bt.alpha[g] : p.alpha), gp = f2s(p.gp_u);
    if (GEN && !batch && p.alpha_cell) al = ld(p.alpha_cell);
    if ((GEN && p.alpha_cell) || batch)
        gp = make_float2((float)(-kGamma) / (1.f + al.x * al.x), (float)(-kGamma) / (1.f + al.y * al.y));
    const float2 pc = f2s(batch ? bt.pc[g] : (p.no_precession ? 0.f : 1.f));
    const float2 kx = f2mul(gp, f2fma(al, dx_, f2mul(pc, cx))), ky = f2mul(gp, f2fma(al, dy_, f2mul(pc, cy))),
                 kz = f2mul(gp, f2fma(al, dz_, f2mul(pc, cz)));
    auto st = [&](float* q, float2 a, float2 b, float2 c) {
        q[ia] = a.x; q[N + ia] = b.x; q[2 * N + ia] = c.x;
        if (two) { q[ib] = a.y; q[N + ib] = b.y; q[2 * N + ib] = c.y; }
    };
    if (p.want_torque || p.want_err || p.want_energy) {
        if (!(isfinite(kx.x) && isfinite(ky.x) && isfinite(kz.x) && isfinite(kx.y) && isfinite(ky.y) && isfinite(kz.y)))
            red.nf = 1;
        const float2 c2v = f2fma(cx, cx, f2fma(cy, cy, f2mul(cz, cz)));
        if (GEN && !batch && p.Ms_cell) {
            if (on.x != 0.f) red.tq = fmaxf(red.tq, sqrtf(c2v.x) / Ms.x);
            if (on.y != 0.f) red.tq = fmaxf(red.tq, sqrtf(c2v.y) / Ms.y);
        } else {
            red.tq2 = fmaxf(red.tq2, fmaxf(c2v.x, c2v.y));
        }
    }
    if (GEN && p.want_energy) {
        auto add = [&](int q, float2 a, float2 b, float2 c) {
#pragma unroll
            for (int lane = 0; lane < 2; ++lane) {
                if (lane && !two) break;
                float2 dot = f2s(0.f);
                line_acc_prod(dot, lane ? mx.y : mx.x, lane ? a.y : a.x);
                line_acc_prod(dot, lane ? my.y : my.x, lane ? b.y : b.x);
                line_acc_prod(dot, lane ? mz.y : mz.x, lane ? c.y : c.x);
                const float ms = lane ? Ms.y : Ms.x, h = __fadd_rn(dot.x, dot.y), l = __fadd_rn(__fsub_rn(dot.x, h), dot.y);
                if (ms == 0.f) continue;
                const float w = __fmul_rn(ms, h);
                line_acc(red.e[q], w, __fadd_rn(__fmaf_rn(ms, h, -w), __fmul_rn(ms, l)));
            }
        };
        add(0, v[0], v[1], v[2]);
        add(1, hex, hey, hez);
        add(2, hax, hay, haz);
        add(3, hzx, hzy, hzz);
        if (dmi) add(4, hmx, hmy, hmz);
    }
    if (p.h_out) st(p.h_out + off, hx, hy, hz);
    if (p.k_out) st(p.k_out + off, kx, ky, kz);
    if (p.acc_out) {
        float2 a = f2mul(f2s(p.acc_bT), kx), b = f2mul(f2s(p.acc_bT), ky), c = f2mul(f2s(p.acc_bT), kz);
        if (p.acc_in) { a = f2add(a, lds(p.acc_in)); b = f2add(b, lds(p.acc_in + N)); c = f2add(c, lds(p.acc_in + 2 * N)); }
        st(p.acc_out, a, b, c);
    }
    if (p.next || p.want_err) {
        // m + dt (sum of all derivatives): one rounding at the size of m
        const float2 dt = f2s(batch ? (float)bt.dt[g] : p.dtT), ck = f2s(p.ckT);
        const float* mn = p.mn + off;
        const float2 m0x = lds(mn), m0y = lds(mn + N), m0z = lds(mn + 2 * N);
        float2 ox = f2fma(dt, f2fma(ck, kx, rk[0]), m0x), oy = f2fma(dt, f2fma(ck, ky, rk[1]), m0y),
               oz = f2fma(dt, f2fma(ck, kz, rk[2]), m0z);
        if (p.want_err) {
            auto worst = [&](float e, float m0, float u) {
                const float n = fabsf(e), sc = p.atolT + p.rtolT * fmaxf(fabsf(m0), fabsf(u));
                if (!isfinite(n)) red.nf = 1;
                if (n * red.ed > red.en * sc) { red.en = n; red.ed = sc; }
            };
            const bool on_next = p.err_on_next;
            const float2 ebk = f2mul(dt, f2s(p.eb_kT));
            const float2 eX = f2fma(ebk, kx, rk[3]), eY = f2fma(ebk, ky, rk[4]), eZ = f2fma(ebk, kz, rk[5]);
            worst(eX.x, m0x.x, on_next ? ox.x : mx.x); worst(eX.y, m0x.y, on_next ? ox.y : mx.y);
            worst(eY.x, m0y.x, on_next ? oy.x : my.x); worst(eY.y, m0y.y, on_next ? oy.y : my.y);
            worst(eZ.x, m0z.x, on_next ? oz.x : mz.x); worst(eZ.y, m0z.y, on_next ? oz.y : mz.y);
        }
        if (p.next) {
            if (p.renorm) {
                const float2 nn = f2fma(ox, ox, f2fma(oy, oy, f2mul(oz, oz)));
                const float2 sc = make_float2(nn.x > 0.f ? 1.f / sqrtf(nn.x) : 1.f, nn.y > 0.f ? 1.f / sqrtf(nn.y) : 1.f);
                ox = f2mul(ox, sc); oy = f2mul(oy, sc); oz = f2mul(oz, sc);
            }
            st(p.next + off, ox, oy, oz);
            v[0] = f2mul(Ms, ox); v[1] = f2mul(Ms, oy); v[2] = f2mul(Ms, oz);
            if (!two) v[0].y = v[1].y = v[2].y = 0.f;
        }
    }
}

// The part of an item's Runge-Kutta combination that does not wait for the
// field: sum_j kc_j kin_j (w[0..2]) and dt sum_j eb_j kin_j (w[3..5]).  The state
// is left to the cell update: added here it would be rounded once more.
template <int NK>
__device__ __forceinline__ void line_known(const StageParams<float>& p, float dtv, long off, int ia, int ib,
                                           float2 (&w)[6]) {
    const int N = (int)p.N;
    float2 k[NK > 0 ? NK : 1][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int q = 0; q < NK; ++q) {
            const float* a = p.kin[q] + off + c * N;
            k[q][c] = make_float2(__ldcg(a + ia), __ldcg(a + ib));
        }
    }
    const float2 dt = f2s(dtv);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float2 n = f2s(0.f), e = f2s(0.f);
#pragma unroll
        for (int q = 0; q < NK; ++q) {
            n = f2fma(f2s(p.kcT[q]), k[q][c], n);
            e = f2fma(f2s(p.ebT[q]), k[q][c], e);
        }
        w[c] = n;
        w[3 + c] = f2mul(dt, e);
    }
}

// threads of a fused CTA at most, and the CTAs per SM asked of the register
// allocator: 64 registers a thread, 128 with every term (GEN).  The passes wait
// on memory and shared memory, so warps count for more than registers (one
// thread for all three components: 80 registers, 19 warps per SM, 95 us on 32
// grids of 256x256x1).
template <int LC> constexpr int line_fused_threads() {
    constexpr int n = LC > 0 ? (3 * (LC / line_ct<float>(LC > 0 ? LC : 16).rmin) + 31) / 32 * 32 : 0;
    return n > 256 ? n : 256;
}
template <bool GEN, int MAXT> constexpr int line_fused_ctas() {
    constexpr int n = (GEN ? 576 : 1024) / MAXT;
    return n > 0 ? n : 1;
}

// A CTA takes `lines` row pairs of one grid, three lines (components) of nt
// threads each: x-inverse in shared memory, the cell updates (an item is one x
// of both rows, all components), and, unless fwd is 0, the x-forward of Ms next
// over the same rows of S1.  It replaces an x-inverse, a stage and an x-forward
// pass, and with them the demag field's and the next input's trips through memory.
template <bool GEN, int MAXT, int LC>
__global__ void __launch_bounds__(MAXT, (line_fused_ctas<GEN, MAXT>()))
line_fused(DemagDims d, float2* __restrict__ S1, const __grid_constant__ StageParams<float> p,
           const __grid_constant__ LineBatch bt, const __grid_constant__ LinePlan pl,
           const float2* __restrict__ tw, int nt, int lines, int park_n, int fwd) {
    using C = float2;
    extern __shared__ __align__(16) unsigned char smraw[];
    if constexpr (LC > 0) {
        constexpr int kNt = LC / line_ct<float>(LC).rmin;
        nt = kNt;
    }
    const LineThread t = line_thread(nt, 3 * lines);
    const int pair = t.l / 3, c = t.l - 3 * pair;
    const int g = blockIdx.y, nx = d.nx, plane = line_len(LC ? LC : pl.L);
    const LineRows r = line_rows<3>(d, blockIdx.x * lines + pair);
    const long rows = (long)d.ny * d.nz, off = (long)g * 3 * rows;
    C* sp = reinterpret_cast<C*>(smraw) + (size_t)pair * 3 * plane;     // the pair's three lines
    C* s = sp + c * plane;
    C* sa = S1 + (off + c * rows + r.ra) * d.KXS;
    C* sb = r.two ? sa + d.KXS : sa;
    grid_dep_wait();
    if (bt.mask && !bt.mask[g]) return;
    // The Runge-Kutta combination of the derivatives that are there, summed
    // while the registers are free and all its loads can be in flight, and
    // parked in shared memory for this thread's cell updates: [next][err][3][nx]
    const bool next = p.next != nullptr, err = p.want_err != 0;
    float2* park = reinterpret_cast<float2*>(smraw) + (size_t)lines * 3 * plane + (size_t)pair * park_n * nx;
    if (r.on && t.in && (next || err)) {
        const float dtv = bt.mask ? (float)bt.dt[g] : p.dtT;
#pragma unroll 1
        for (int x = c * nt + t.b; x < nx; x += 3 * nt) {
            const int ia = x + nx * (int)r.ra, ib = r.two ? ia + nx : ia;
            float2 w[6];
            switch (p.nk) {
                case 0: line_known<0>(p, dtv, off * nx, ia, ib, w); break;
                case 1: line_known<1>(p, dtv, off * nx, ia, ib, w); break;
                case 2: line_known<2>(p, dtv, off * nx, ia, ib, w); break;
                case 3: line_known<3>(p, dtv, off * nx, ia, ib, w); break;
                case 4: line_known<4>(p, dtv, off * nx, ia, ib, w); break;
                case 5: line_known<5>(p, dtv, off * nx, ia, ib, w); break;
                default: line_known<6>(p, dtv, off * nx, ia, ib, w); break;
            }
            float2* o = park + x;
            if (next) { o[0] = w[0]; o[nx] = w[1]; o[2 * nx] = w[2]; o += 3 * nx; }
            if (err) { o[0] = w[3]; o[nx] = w[4]; o[2 * nx] = w[5]; }
        }
    }
    line_inverse<float, 1, LC>(sa, sb, 0, s, plane, t.b, pl, tw);
    LineRed red;
    red.tq2 = red.tq = red.en = 0.f;
    red.ed = 1.f;
    red.nf = 0;
    for (int q = 0; q < 5; ++q) red.e[q] = f2s(0.f);
    if (r.on && t.in) {
#pragma unroll 1
        for (int x = c * nt + t.b; x < nx; x += 3 * nt) {
            C* w = sp + line_place<4>(x);
            float2 v[3] = {w[0], w[plane], w[2 * plane]};
            float2 rk[6];
            const float2* o = park + x;
            if (next) { rk[0] = o[0]; rk[1] = o[nx]; rk[2] = o[2 * nx]; o += 3 * nx; }
            if (err) { rk[3] = o[0]; rk[4] = o[nx]; rk[5] = o[2 * nx]; }
            line_cells<GEN>(p, bt, g, off * nx, x, r.y, r.z, r.two, rk, v, red);
            w[0] = v[0]; w[plane] = v[1]; w[2 * plane] = v[2];
        }
    }
    double* part = bt.mask ? bt.partials : p.partials;
    if (part) {
        // block maxima, and sums of the energies, in a fixed order
        __shared__ float rt[MAXT / 32][4];
        __shared__ int rn[MAXT / 32];
        __shared__ double re[MAXT / 32][5];
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
        double en[5] = {0, 0, 0, 0, 0};
        if (GEN && p.want_energy) {
            const double f = -0.5 * kMu0 * (p.lvol ? p.lvol[min(r.z, d.nz - 1)] : p.V);
#pragma unroll
            for (int q = 0; q < 5; ++q) en[q] = (q == 3 ? 2.0 : 1.0) * f * ((double)red.e[q].x + (double)red.e[q].y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float n2 = __shfl_down_sync(0xffffffffu, red.en, o), d2 = __shfl_down_sync(0xffffffffu, red.ed, o);
            if (n2 * red.ed > red.en * d2) { red.en = n2; red.ed = d2; }
            red.tq2 = fmaxf(red.tq2, __shfl_down_sync(0xffffffffu, red.tq2, o));
            red.tq = fmaxf(red.tq, __shfl_down_sync(0xffffffffu, red.tq, o));
            if (GEN && p.want_energy) {
#pragma unroll
                for (int q = 0; q < 5; ++q) en[q] += __shfl_down_sync(0xffffffffu, en[q], o);
            }
        }
        const int nf = __any_sync(0xffffffffu, red.nf);
        if (lane == 0) {
            rt[w][0] = red.tq2; rt[w][1] = red.tq; rt[w][2] = red.en; rt[w][3] = red.ed;
            rn[w] = nf;
            for (int q = 0; q < 5; ++q) re[w][q] = en[q];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            float t2 = rt[0][0], tq = rt[0][1], n = rt[0][2], e = rt[0][3];
            int f = rn[0];
            for (int q = 1; q < nw; ++q) {
                t2 = fmaxf(t2, rt[q][0]);
                tq = fmaxf(tq, rt[q][1]);
                if (rt[q][2] * e > n * rt[q][3]) { n = rt[q][2]; e = rt[q][3]; }
                f |= rn[q];
            }
            const float ms = bt.mask ? bt.Ms[g] : p.Ms;
            if (ms != 0.f && !(GEN && !bt.mask && p.Ms_cell)) tq = sqrtf(t2) / ms;
            if (bt.mask) {
                double* o = part + ((long)g * gridDim.x + blockIdx.x) * 3;
                o[0] = tq; o[1] = n / e; o[2] = f;
            } else {
                double* o = part + (long)blockIdx.x * kNPart;
                o[R_TORQUE] = tq; o[R_ERR] = n / e; o[R_NONFINITE] = f;
                const int slot[5] = {R_EDEM, R_EEX, R_EANI, R_EZEE, R_EDMI};
                for (int q = 0; q < 5; ++q) {
                    double sum = re[0][q];
                    for (int k = 1; k < nw; ++k) sum += re[k][q];
                    o[slot[q]] = sum;
                }
            }
        }
    }
    if (!fwd) return;
    __syncthreads();
    line_forward<float, 1, LC>(s, plane, t.b, nt, nx, pl, tw, sa, sb, 0, r.on && t.in, r.two);
}

// ---------------------------------------------------- y passes, z pass ----
// A CTA takes 2^lb columns, one thread per butterfly of a column.

// first pass of a transform along a strided line: elements b + q M straight
// from global memory (at g[e es + c cs]; e < n, the rest zero)
template <typename T, int DIR, int R, bool HALF, int NC>
__device__ __forceinline__ void line_first(const typename Cplx<T>::type* g, long es, long cs, int n,
                                           typename Cplx<T>::type* s, int plane, int lb, int b, int L) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    if (b >= M) return;
    C x[NC][R];
#pragma unroll
    for (int q = 0; q < (HALF ? R / 2 : R); ++q) {
        const int e = b + q * M;
        const bool in = !HALF || e < n;
#pragma unroll
        for (int c = 0; c < NC; ++c) x[c][q] = in ? __ldcg(g + c * cs + e * es) : mk<C>(0, 0);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) line_dft<DIR, R, HALF>(x[c]);
    line_store<3>(x, s, plane, lb, b, 0, 1);
}

// last pass: outputs b + q M to global memory; HALF: only e < n
template <typename T, int DIR, int R, bool HALF, int NC>
__device__ __forceinline__ void line_last(const typename Cplx<T>::type* s, int plane, int lb, int b, int L, int Ns,
                                          unsigned mg, const typename Cplx<T>::type* tw,
                                          typename Cplx<T>::type* g, long es, long cs, int n, bool valid) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    if (b >= M) return;
    C x[NC][R];
    line_load<3>(x, s, plane, lb, b, M);
    line_butterfly<T, DIR>(x, tw, line_mod(b, Ns, mg), L / (Ns * R), L);
#pragma unroll
    for (int q = 0; q < (HALF ? R / 2 : R); ++q) {
        const int e = b + q * M;
        if (valid && (!HALF || e < n)) {
#pragma unroll
            for (int c = 0; c < NC; ++c) g[c * cs + e * es] = x[c][q];
        }
    }
}

// h^ = T M^ of one wave number; t: the octant's xx, xy, xz, yy, yz, zz; ny, nz:
// whether the odd components along y and along z change sign here
template <typename T, typename C>
__device__ __forceinline__ void line_mul(const T (&t)[6], bool ny, bool nz, C& x, C& y, C& z) {
    const T txy = line_flip(t[1], ny), txz = line_flip(t[2], nz), tyz = line_flip(t[4], ny != nz);
    const C mx = x, my = y, mz = z;
    x = mk<C>(t[0] * mx.x + txy * my.x + txz * mz.x, t[0] * mx.y + txy * my.y + txz * mz.y);
    y = mk<C>(txy * mx.x + t[3] * my.x + tyz * mz.x, txy * mx.y + t[3] * my.y + tyz * mz.y);
    z = mk<C>(txz * mx.x + tyz * my.x + t[5] * mz.x, txz * mx.y + tyz * my.y + t[5] * mz.y);
}

// h^ = T M^ at the R wave numbers b + q M of one column; tp points at the
// column's folded ky row, tz between kz planes, tc between components
template <typename T, int R>
__device__ __forceinline__ void line_tensor(typename Cplx<T>::type (&x)[3][R], const T* __restrict__ tp, long tz, long tc,
                                            int b, int M, int L, bool sy, int swap) {
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int kz = b + q * M;
        const bool sz = 2 * kz > L;
        const T* g = tp + (sz ? L - kz : kz) * tz;
        const T t[6] = {g[0], g[tc], g[2 * tc], g[3 * tc], g[4 * tc], g[5 * tc]};
        line_mul(t, swap ? sz : sy, swap ? sy : sz, x[0][q], x[1][q], x[2][q]);
    }
}

// the forward's last pass, the tensor product and the inverse's first pass
template <typename T, int R>
__device__ __forceinline__ void line_product(typename Cplx<T>::type* s, int plane, int lb, int b, int L, int Ns,
                                             unsigned mg, const typename Cplx<T>::type* tw, const T* tp, long tz, long tc,
                                             bool sy, int swap) {
    using C = typename Cplx<T>::type;
    const int M = L / R;
    const bool on = b < M;
    if (!on) b = 0;
    C x[3][R];
    line_load<3>(x, s, plane, lb, b, M);
    line_butterfly<T, -1>(x, tw, line_mod(b, Ns, mg), L / (Ns * R), L);
    line_tensor<T, R>(x, tp, tz, tc, b, M, L, sy, swap);
#pragma unroll
    for (int c = 0; c < 3; ++c) line_dft<+1, R, false>(x[c]);
    __syncthreads();
    if (on) line_store<3>(x, s, plane, lb, b, 0, 1);
    __syncthreads();
}

// the whole column in one thread's registers (L = R)
template <typename T, int R>
__device__ __forceinline__ void line_product_one(typename Cplx<T>::type* g, long es, long cs, int n, const T* tp,
                                                 long tz, long tc, bool sy, int swap) {
    using C = typename Cplx<T>::type;
    constexpr int H = R == 1 ? 1 : R / 2;
    C x[3][R];
#pragma unroll
    for (int q = 0; q < H; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) x[c][q] = q < n ? g[c * cs + q * es] : mk<C>(0, 0);
    if constexpr (R > 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) line_dft<-1, R, true>(x[c]);
    }
    line_tensor<T, R>(x, tp, tz, tc, 0, 1, R, sy, swap);
    if constexpr (R > 1) {
#pragma unroll
        for (int c = 0; c < 3; ++c) line_dft<+1, R, false>(x[c]);
    }
#pragma unroll
    for (int q = 0; q < H; ++q)
        if (q < n) {
#pragma unroll
            for (int c = 0; c < 3; ++c) g[c * cs + q * es] = x[c][q];
        }
}

// z pass: per (kx, ky) column z-forward (z < nz, the rest zero), h^ = T M^ with
// the octant-folded real tensor (sign flips of the odd components from the
// parity of ky and kz, or of the transformed axis on 2-D grids), z-inverse,
// keep z < nz; in place.  Columns are numbered kx-fastest over (ky, kx <= Px/2);
// blockIdx.y is the grid of a batch.
// (The tensor slice copied to shared memory during the forward passes measured
// slower, 90 against 80 us on 32 grids of 256x256x1: fewer CTAs per SM.)
// FORM: kConvOne, a column in one thread's registers; kConvThree, a thread per
// butterfly of all three components; kConvSplit, a thread per butterfly and
// component, the product then taken wave number by wave number by all of them;
// kConvSplitWide, that with radices 6 and 8 too, whose registers cost the plans
// without them 1 to 3 % (film of 512x128x1: 47.5 -> 49.0 us).
enum { kConvOne, kConvThree, kConvSplit, kConvSplitWide };
template <typename T, int FORM, int MAXT, int LC, bool IDLE = false>
__global__ void __launch_bounds__(MAXT, FORM >= kConvSplit ? (MAXT <= 384 ? 2 : 1) : FORM == kConvOne ? 2 : LC > 0 && MAXT == kLineThreads32 ? 2 : line_blocks<T, MAXT>())
line_conv(DemagDims d, typename Cplx<T>::type* __restrict__ S2, const T* __restrict__ tens,
          const __grid_constant__ LinePlan pl, const typename Cplx<T>::type* __restrict__ tw, int lb, int ncol) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int L = LC ? LC : pl.L, tid = threadIdx.x;
    int M = L / pl.rmin;
    if constexpr (LC > 0) {
        constexpr int kM = LC / line_ct<T>(LC).rmin;
        constexpr int kLb = line_ct_lb<T>(LC);
        M = kM;
        lb = kLb;
    }
    const int l = tid & ((1 << lb) - 1), u = tid >> lb;
    const int c = FORM >= kConvSplit ? min(u / M, 2) : 0;
    const int b = FORM < kConvSplit ? u : u < 3 * M ? u - c * M : kLineIdle;
    const int col = (blockIdx.x << lb) + l;
    const bool valid = col < ncol;
    const int cc = valid ? col : ncol - 1;      // columns past the end follow the last one and store nothing
    const int ky = cc / d.KX, kx = cc - ky * d.KX;
    const int LY = d.LY, KY2 = LY / 2 + 1;
    const bool up = 2 * ky > LY;
    const long zs = (long)LY * d.KXS, cs = (long)d.nz * zs;
    C* g = S2 + (long)blockIdx.y * 3 * cs + (long)ky * d.KXS + kx;
    const long tz = (long)KY2 * d.KXS, tc = (long)(L / 2 + 1) * tz;
    const T* tp = tens + (long)(up ? LY - ky : ky) * d.KXS + kx;
    if constexpr (FORM >= kConvSplit) {
        // this thread's wave numbers u + 3 M i; their tensor entries (written long
        // before the previous pass) are on their way from the start
        static_assert(LC == 0 && sizeof(T) == 8, "the split form is FP64's");
        constexpr bool kWide = FORM == kConvSplitWide;
        constexpr int KP = kWide ? 3 : 2;               // the smallest radix of a plan is 8, or 4, at most
        T t[KP][6];
#pragma unroll
        for (int i = 0; i < KP; ++i) {
            const int kz = min(u + 3 * M * i, L - 1);
            const T* q = tp + (2 * kz > L ? L - kz : kz) * tz;
#pragma unroll
            for (int j = 0; j < 6; ++j) t[i][j] = __ldg(q + j * tc);
        }
        grid_dep_wait();
        C* s0 = reinterpret_cast<C*>(smraw) + l;
        const int plane = line_len(L) << lb;
        C* s = s0 + c * plane;
        g += c * cs;
        auto product = [&]() {
#pragma unroll
            for (int i = 0; i < KP; ++i) {
                const int kz = u + 3 * M * i;
                if (u < 3 * M && kz < L) {
                    C* q = s0 + (line_place<3>(kz) << lb);
                    const bool sz = 2 * kz > L;
                    C x = q[0], y = q[plane], z = q[2 * plane];
                    line_mul(t[i], d.yz_swap ? sz : up, d.yz_swap ? up : sz, x, y, z);
                    q[0] = x; q[plane] = y; q[2 * plane] = z;
                }
            }
            __syncthreads();
        };
        const int np = pl.np;
        MM_LINE_RADIX_EVEN(kWide, pl.R[0], (line_first<T, -1, R_, true, 1>(g, zs, 0, d.nz, s, 0, lb, b, L)));
        __syncthreads();
        for (int i = 1; i < np; ++i) line_mid_any<T, -1, 1, 3, kWide, IDLE>(s, 0, lb, b, pl, i, tw);
        product();
        if (line_warp_idle<IDLE>(pl, pl.R[np - 1], b)) line_pass_over();
        else MM_LINE_RADIX(kWide, pl.R[np - 1], (line_start<T, +1, R_, 1, 3>(s, 0, lb, b, L)));
        for (int i = 1; i < np - 1; ++i) line_mid_any<T, +1, 1, 3, kWide, IDLE>(s, 0, lb, b, pl, i, tw);
        MM_LINE_RADIX_EVEN(kWide, pl.R[0], (line_last<T, +1, R_, true, 1>(s, 0, lb, b, L, pl.Nsi[np - 1], pl.mgi[np - 1],
                                                                      tw, g, zs, 0, d.nz, valid)));
        return;
    }
    grid_dep_wait();
    if (d.early) grid_dep_launch();
    if constexpr (FORM == kConvOne) {
        if (!valid) return;
        switch (L) {
            case 1: line_product_one<T, 1>(g, zs, cs, d.nz, tp, tz, tc, up, d.yz_swap); break;
            case 2: line_product_one<T, 2>(g, zs, cs, d.nz, tp, tz, tc, up, d.yz_swap); break;
            case 4: line_product_one<T, 4>(g, zs, cs, d.nz, tp, tz, tc, up, d.yz_swap); break;
            case 6: line_product_one<T, sizeof(T) == 4 ? 6 : 1>(g, zs, cs, d.nz, tp, tz, tc, up, d.yz_swap); break;
            case 8: line_product_one<T, sizeof(T) == 4 ? 8 : 1>(g, zs, cs, d.nz, tp, tz, tc, up, d.yz_swap); break;
            case 12: line_product_one<T, sizeof(T) == 4 ? 12 : 1>(g, zs, cs, d.nz, tp, tz, tc, up, d.yz_swap); break;
            default: line_product_one<T, sizeof(T) == 4 ? 16 : 1>(g, zs, cs, d.nz, tp, tz, tc, up, d.yz_swap); break;
        }
    } else {
        C* s = reinterpret_cast<C*>(smraw) + l;
        const int plane = line_len(L) << lb;
        if constexpr (LC > 0) {
            constexpr LinePlan P = line_ct<T>(LC);
            constexpr int np = P.np;
            line_first<T, -1, P.R[0], true, 3>(g, zs, cs, d.nz, s, plane, lb, b, L);
            __syncthreads();
            line_mids_ct<T, -1, 3, 3, LC, 1, np - 1>(s, plane, lb, b, tw);
            line_product<T, P.R[np - 1]>(s, plane, lb, b, L, P.Ns[np - 1], 0, tw, tp, tz, tc, up, d.yz_swap);
            line_mids_ct<T, +1, 3, 3, LC, 1, np - 1>(s, plane, lb, b, tw);
            line_last<T, +1, P.R[0], true, 3>(s, plane, lb, b, L, P.Nsi[np - 1], 0, tw, g, zs, cs, d.nz, valid);
        } else {
            MM_LINE_RADIX_EVEN(true, pl.R[0], (line_first<T, -1, R_, true, 3>(g, zs, cs, d.nz, s, plane, lb, b, L)));
            __syncthreads();
            const int np = pl.np;
            for (int i = 1; i < np - 1; ++i) line_mid_any<T, -1, 3, 3, true, IDLE>(s, plane, lb, b, pl, i, tw);
            if (line_warp_idle<IDLE>(pl, pl.R[np - 1], b)) line_pass_over();
            else MM_LINE_RADIX(true, pl.R[np - 1], (line_product<T, R_>(s, plane, lb, b, L, pl.Ns[np - 1], pl.mg[np - 1], tw, tp,
                                                                tz, tc, up, d.yz_swap)));
            for (int i = 1; i < np - 1; ++i) line_mid_any<T, +1, 3, 3, true, IDLE>(s, plane, lb, b, pl, i, tw);
            MM_LINE_RADIX_EVEN(true, pl.R[0], (line_last<T, +1, R_, true, 3>(s, plane, lb, b, L, pl.Nsi[np - 1],
                                                                          pl.mgi[np - 1], tw, g, zs, cs, d.nz, valid)));
        }
    }
}

// y passes.  DIR = -1: S1 (ny rows) -> S2 (Py rows), forward, zero upper half;
// DIR = +1: S2 -> S1, keep y < ny.  Columns kx-fastest over component and z,
// kx <= Px/2, a thread per butterfly of one component (three per thread: 11.3 and
// 9.6 against 8.7 and 8.8 us on 140-point lines of 100x65x27).
template <typename T, int DIR, int MAXT, bool IDLE = false>
__global__ void __launch_bounds__(MAXT)
line_y(DemagDims d, const typename Cplx<T>::type* __restrict__ in, typename Cplx<T>::type* __restrict__ out,
       const __grid_constant__ LinePlan pl, const typename Cplx<T>::type* __restrict__ tw, int lb, int ncol) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int L = pl.L, np = pl.np, tid = threadIdx.x;
    const int l = tid & ((1 << lb) - 1), b = tid >> lb;
    const int col = (blockIdx.x << lb) + l;
    const bool valid = col < ncol;
    const int cc = valid ? col : ncol - 1;
    const int cz = cc / d.KX, kx = cc - cz * d.KX;
    const int rin = DIR < 0 ? d.ny : L, rout = DIR < 0 ? L : d.ny;
    const long plane = (long)blockIdx.y * 3 * d.nz + cz;
    const C* gi = in + plane * rin * d.KXS + kx;
    C* go = out + plane * rout * d.KXS + kx;
    grid_dep_wait();
    C* s = reinterpret_cast<C*>(smraw) + l;
    if constexpr (DIR < 0) {
        MM_LINE_RADIX_EVEN(true, pl.R[0], (line_first<T, -1, R_, true, 1>(gi, d.KXS, 0, d.ny, s, 0, lb, b, L)));
    } else {
        MM_LINE_RADIX(true, pl.R[np - 1], (line_first<T, +1, R_, false, 1>(gi, d.KXS, 0, L, s, 0, lb, b, L)));
    }
    __syncthreads();
    for (int i = 1; i < np - 1; ++i) line_mid_any<T, DIR, 1, 3, true, IDLE>(s, 0, lb, b, pl, i, tw);
    if constexpr (DIR < 0) {
        MM_LINE_RADIX(true, pl.R[np - 1], (line_last<T, -1, R_, false, 1>(s, 0, lb, b, L, pl.Ns[np - 1], pl.mg[np - 1], tw, go,
                                                                       d.KXS, 0, L, valid)));
    } else {
        MM_LINE_RADIX_EVEN(true, pl.R[0], (line_last<T, +1, R_, true, 1>(s, 0, lb, b, L, pl.Nsi[np - 1], pl.mgi[np - 1], tw, go,
                                                                      d.KXS, 0, d.ny, valid)));
    }
}

// kernels of the compiled lengths, by kind: null for a length without them
enum LineKind { kLineFused, kLineFusedGen, kLineXFwd, kLineXInv, kLineConv };
const void* line_ct_kernel0(LineKind kind, int L);      // 16 .. 128
const void* line_ct_kernel1(LineKind kind, int L);      // 256 .. 1024
const void* line_ct_kernel2(LineKind kind, int L);      // 96 .. 224
const void* line_ct_kernel3(LineKind kind, int L);      // 384 .. 896

template <int LC> const void* line_ct_pick(LineKind kind) {
    constexpr LinePlan P = line_ct<float>(LC);
    constexpr int M = LC / P.rmin, FT = line_fused_threads<LC>(), YT = (M << line_ct_lb<float>(LC)) <= 256 ? 256 : 512;
    switch (kind) {
        case kLineFused: return (const void*)line_fused<false, FT, LC>;
        case kLineFusedGen: return (const void*)line_fused<true, FT, LC>;
        case kLineXFwd: return (const void*)line_x_forward<float, 256, LC>;
        case kLineXInv: return (const void*)line_x_inverse<float, 256, LC>;
        default:
            // z lines of up to 16 points stay in one thread's registers
            if constexpr (LC <= 16) return nullptr;
            else return (const void*)line_conv<float, kConvThree, YT, LC>;
    }
}

}  // namespace mm
