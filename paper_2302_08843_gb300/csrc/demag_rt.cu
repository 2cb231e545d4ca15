// Demag FFT passes for every 7-smooth padded length 2^a 3^b 5^c 7^d (even,
// <= 4096) that has no compiled engine: the same five passes as
// demag_passes.cu (x-forward r2c, y-forward, z-forward + 3x3 tensor multiply
// + z-inverse, y-inverse, x-inverse c2r; Sec. 4.4), with the line length and
// its radix plan known only at run time.
//
// Engine: a self-sorting Stockham FFT over a batch of lines held in shared
// memory (element e of line l at s[e NLc + l]), all threads of the CTA
// sharing the butterflies of every pass: a pass of radix R and span Ns reads
// butterfly b's inputs at b + q L/R, multiplies input q by W_{Ns R}^(q k)
// (k = b mod Ns), transforms them and writes output q to
// (b - k) R + k + q Ns, ping-ponging between two buffers.  Plan: every radix 7,
// then 5, then 3, then radix-4 passes and at most one radix-2 pass.
// Twiddles W_L^m (m < L) come from one double-precision table per length,
// all lengths concatenated (g_twrt64 / g_twrt32), built on the host with the
// octant-exact evaluation of the other tables and uploaded once per device.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <utility>
#include <vector>

#include "demag.h"
#include "line_kernels.cuh"
#include "tensor_host.h"
#include "tma.cuh"

namespace mm {

namespace {

constexpr int kRtMaxPass = 16;
constexpr int kRtThreads = 256;
constexpr int kRtMaxLines = 16;

struct RtPlan {
    int L;
    int np;
    int R[kRtMaxPass];
    int tw;          // offset of this length's table W_L^m in g_twrt
};

// every padded length the library uses above 1 (even, 7-smooth; 4096 beyond
// kMaxRtFft), their twiddle offsets and the table size
struct RtTable {
    std::vector<int> lengths;
    std::vector<int> offsets;
    int total = 0;
};

const RtTable& rt_table() {
    static RtTable t;
    static std::once_flag once;
    std::call_once(once, [] {
        for (int L = 2; L <= kMaxFft; L += 2)
            if (fft_extent(L / 2) == L) {
                t.lengths.push_back(L);
                t.offsets.push_back(t.total);
                t.total += L;
            }
    });
    return t;
}

// offset of W_L^m in the table, -1 for a length that is not in it
int rt_offset(int L) {
    const RtTable& t = rt_table();
    const auto it = std::lower_bound(t.lengths.begin(), t.lengths.end(), L);
    return it == t.lengths.end() || *it != L ? -1 : t.offsets[it - t.lengths.begin()];
}

// the engine's plan of a length; one: a single pass of radix L
LinePlan host_plan(int L, int rmax, bool one) {
    LinePlan p{};
    if (one) {
        p.L = L;
        p.np = 1;
        p.rmin = p.R[0] = (short)L;
        p.Ns[0] = p.Nsi[0] = 1;
        return p;
    }
    p = line_plan(L, rmax);
    p.tw = rt_offset(L);
    if (p.tw < 0) p.np = 0;
    return p;
}

}  // namespace

// the concatenated twiddle tables (kTwRt, a compile-time bound, is checked against
// the host table at upload)
static __device__ double2 g_twrt64[2 * kTwRt];
static __device__ float2 g_twrt32[kTwRt];

// device addresses of the tables, per device (set by the upload)
constexpr int kMaxDevices = 128;
static const double2* g_tab64[kMaxDevices];
static const float2* g_tab32[kMaxDevices];
template <typename T> const typename Cplx<T>::type* line_table(const LinePlan& pl) {
    int dev = 0;
    cudaGetDevice(&dev);
    if constexpr (sizeof(T) == 4) return g_tab32[dev] + pl.tw;
    else return g_tab64[dev] + pl.tw;
}

template <typename T> struct TwRt;
template <> struct TwRt<float> {
    static __device__ __forceinline__ float2 get(int m) { return __ldg(&g_twrt32[m]); }
};
template <> struct TwRt<double> {
    static __device__ __forceinline__ double2 get(int m) { return __ldg(&g_twrt64[m]); }
};

bool fft_rt_length(int L) {
    if (L < 2 || L > kMaxRtFft || (L & 1)) return false;
    if (is_pow2(L)) return false;
    static const int compiled[12] = {96, 100, 112, 192, 200, 224, 384, 400, 448, 768, 800, 896};
    for (int c : compiled)
        if (c == L) return false;
    int v = L;
    for (int p : {2, 3, 5, 7})
        while (v % p == 0) v /= p;
    return v == 1;
}

static RtPlan make_plan(int L) {
    RtPlan pl{};
    pl.L = L;
    int v = L;
    for (int r : {7, 5, 3})
        while (v % r == 0) {
            pl.R[pl.np++] = r;
            v /= r;
        }
    while (v % 4 == 0) {
        pl.R[pl.np++] = 4;
        v /= 4;
    }
    if (v == 2) pl.R[pl.np++] = 2;
    const RtTable& t = rt_table();
    pl.tw = -1;
    for (size_t i = 0; i < t.lengths.size(); ++i)
        if (t.lengths[i] == L) pl.tw = t.offsets[i];
    return pl;
}

cudaError_t upload_twiddles_rt() {
    const RtTable& t = rt_table();
    if (t.total != kTwRt) return cudaErrorInvalidValue;
    static std::vector<double2> h64;
    static std::vector<float2> h32;
    if (h64.empty()) {
        h64.resize(2 * kTwRt);
        h32.resize(kTwRt);
        for (size_t i = 0; i < t.lengths.size(); ++i) {
            const int L = t.lengths[i];
            for (int m = 0; m < L; ++m) {
                double c, sn;
                twiddle_entry(L, m, &c, &sn);
                h64[t.offsets[i] + m] = make_double2(c, sn);
                h64[kTwRt + t.offsets[i] + m] = line_turn(m, L) ? make_double2(sn, -c / sn) : make_double2(c, sn / c);
                h32[t.offsets[i] + m] = make_float2((float)c, (float)sn);
            }
        }
    }
    cudaError_t e = cudaMemcpyToSymbol(g_twrt64, h64.data(), sizeof(double2) * 2 * kTwRt);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_twrt32, h32.data(), sizeof(float2) * kTwRt);
    int dev = 0;
    void *p64 = nullptr, *p32 = nullptr;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess && (dev < 0 || dev >= kMaxDevices)) e = cudaErrorInvalidDevice;
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&p64, g_twrt64);
    if (e == cudaSuccess) e = cudaGetSymbolAddress(&p32, g_twrt32);
    if (e == cudaSuccess) {
        g_tab64[dev] = static_cast<const double2*>(p64);
        g_tab32[dev] = static_cast<const float2*>(p32);
    }
    return e;
}

// One radix-R Stockham pass of span Ns over NLc lines of length L.
template <typename T, int DIR, int R>
__device__ __forceinline__ void rt_pass(const typename Cplx<T>::type* __restrict__ src,
                                        typename Cplx<T>::type* __restrict__ dst, int NLc, int L, int Ns, int tw) {
    using C = typename Cplx<T>::type;
    const int M = L / R, step = L / (Ns * R);
    for (int idx = threadIdx.x; idx < M * NLc; idx += blockDim.x) {
        const int l = idx % NLc, b = idx / NLc;
        const int k = b % Ns;
        C x[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            C v = src[(b + q * M) * NLc + l];
            if (q > 0 && k > 0) {
                C w = TwRt<T>::get(tw + q * k * step);
                if (DIR > 0) w.y = -w.y;
                v = cmul(v, w);
            }
            x[q] = v;
        }
        if constexpr (R == 2) dft2<DIR>(x[0], x[1]);
        else if constexpr (R == 3) dft3<DIR>(x[0], x[1], x[2]);
        else if constexpr (R == 4) dft4<DIR>(x[0], x[1], x[2], x[3]);
        else if constexpr (R == 5) dft5<DIR>(x[0], x[1], x[2], x[3], x[4]);
        else dft7<DIR>(x);
        const int base = (b - k) * R + k;
#pragma unroll
        for (int q = 0; q < R; ++q) dst[(base + q * Ns) * NLc + l] = x[q];
    }
}

// One Stockham transform of NLc lines of length pl.L in shared memory (src,
// with dst as the other buffer of the ping-pong); returns the buffer holding
// the result.  Every thread of the CTA must call it.  DIR = -1 forward,
// +1 inverse (unnormalised).
template <typename T, int DIR>
__device__ typename Cplx<T>::type* rt_fft(typename Cplx<T>::type* src, typename Cplx<T>::type* dst, int NLc,
                                         const RtPlan& pl) {
    using C = typename Cplx<T>::type;
    int Ns = 1;
    for (int p = 0; p < pl.np; ++p) {
        const int R = pl.R[p];
        switch (R) {
            case 2: rt_pass<T, DIR, 2>(src, dst, NLc, pl.L, Ns, pl.tw); break;
            case 3: rt_pass<T, DIR, 3>(src, dst, NLc, pl.L, Ns, pl.tw); break;
            case 4: rt_pass<T, DIR, 4>(src, dst, NLc, pl.L, Ns, pl.tw); break;
            case 5: rt_pass<T, DIR, 5>(src, dst, NLc, pl.L, Ns, pl.tw); break;
            default: rt_pass<T, DIR, 7>(src, dst, NLc, pl.L, Ns, pl.tw); break;
        }
        __syncthreads();
        C* t = src;
        src = dst;
        dst = t;
        Ns *= R;
    }
    return src;
}

// ------------------------------------------------------------- x passes ----
// Two real rows per complex line, paired within one grid of a batch as in the
// compiled x passes (an odd row count leaves the last row with a zero partner).
__device__ __forceinline__ void rt_pair(const DemagDims& d, int NLc, long* ra_s, long* rb_s) {
    if (threadIdx.x < NLc) {
        const long R = 3L * d.ny * d.nz, ppg = (R + 1) / 2;
        const long q = (long)blockIdx.x * NLc + threadIdx.x;
        const long b = q / ppg, lp = q - b * ppg;
        const bool ok = b < d.nb;
        ra_s[threadIdx.x] = ok ? b * R + 2 * lp : -1;
        rb_s[threadIdx.x] = ok && 2 * lp + 1 < R ? b * R + 2 * lp + 1 : -1;
    }
}

template <typename T>
__global__ void __launch_bounds__(kRtThreads)
rt_x_forward(DemagDims d, const T* __restrict__ m, const T* __restrict__ Ms_cell, T Ms_const,
             typename Cplx<T>::type* __restrict__ S1, RtPlan pl, int NLc) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int L = pl.L;
    C* a = reinterpret_cast<C*>(smraw);
    C* b = a + (size_t)L * NLc;
    __shared__ long ra_s[kRtMaxLines], rb_s[kRtMaxLines];
    rt_pair(d, NLc, ra_s, rb_s);
    __syncthreads();
    const long plane = (long)d.ny * d.nz;
    const T* Ms_b = static_cast<const T*>(d.Ms_b);
    for (int idx = threadIdx.x; idx < L * NLc; idx += blockDim.x) {
        const int l = idx % NLc, x = idx / NLc;
        const long ra = ra_s[l], rb = rb_s[l];
        T va = 0, vb = 0;
        if (x < d.nx) {
            if (ra >= 0) {
                const T ms = Ms_b ? Ms_b[ra / (3 * plane)] : (Ms_cell ? Ms_cell[(ra % plane) * d.nx + x] : Ms_const);
                va = m[ra * d.nx + x] * ms;
            }
            if (rb >= 0) {
                const T ms = Ms_b ? Ms_b[rb / (3 * plane)] : (Ms_cell ? Ms_cell[(rb % plane) * d.nx + x] : Ms_const);
                vb = m[rb * d.nx + x] * ms;
            }
        }
        a[x * NLc + l] = mk<C>(va, vb);
    }
    __syncthreads();
    const C* z = rt_fft<T, -1>(a, b, NLc, pl);
    const int KX = L / 2 + 1;
    const T half = (T)0.5;
    for (int idx = threadIdx.x; idx < KX * NLc; idx += blockDim.x) {
        const int l = idx % NLc, k = idx / NLc;
        const long ra = ra_s[l], rb = rb_s[l];
        const C zk = z[k * NLc + l];
        const C zm = z[(k == 0 ? 0 : L - k) * NLc + l];
        if (ra >= 0) S1[ra * d.KXS + k] = mk<C>(half * (zk.x + zm.x), half * (zk.y - zm.y));
        if (rb >= 0) S1[rb * d.KXS + k] = mk<C>(half * (zk.y + zm.y), half * (zm.x - zk.x));
    }
}

template <typename T>
__global__ void __launch_bounds__(kRtThreads)
rt_x_inverse(DemagDims d, const typename Cplx<T>::type* __restrict__ S1, T* __restrict__ h, RtPlan pl, int NLc) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int L = pl.L;
    C* a = reinterpret_cast<C*>(smraw);
    C* b = a + (size_t)L * NLc;
    __shared__ long ra_s[kRtMaxLines], rb_s[kRtMaxLines];
    rt_pair(d, NLc, ra_s, rb_s);
    __syncthreads();
    const int KX = L / 2 + 1;
    for (int idx = threadIdx.x; idx < KX * NLc; idx += blockDim.x) {
        const int l = idx % NLc, k = idx / NLc;
        const long ra = ra_s[l], rb = rb_s[l];
        C A = mk<C>(0, 0), Bv = mk<C>(0, 0);
        if (ra >= 0) A = S1[ra * d.KXS + k];
        if (rb >= 0) Bv = S1[rb * d.KXS + k];
        if (k == 0 || 2 * k == L) { A.y = 0; Bv.y = 0; }   // a real row has real DC and Nyquist
        a[k * NLc + l] = mk<C>(A.x - Bv.y, A.y + Bv.x);
        if (k > 0 && 2 * k < L) a[(L - k) * NLc + l] = mk<C>(A.x + Bv.y, Bv.x - A.y);
    }
    __syncthreads();
    const C* z = rt_fft<T, +1>(a, b, NLc, pl);
    for (int idx = threadIdx.x; idx < d.nx * NLc; idx += blockDim.x) {
        const int l = idx % NLc, x = idx / NLc;
        const long ra = ra_s[l], rb = rb_s[l];
        const C v = z[x * NLc + l];
        if (ra >= 0) h[ra * d.nx + x] = v.x;
        if (rb >= 0) h[rb * d.nx + x] = v.y;
    }
}

// --------------------------------- y and z passes of the longest lines ----
// (those whose widest pass has more butterflies than a CTA threads)
// DIR = -1: S1 (ny rows) -> S2 (Py rows), forward.  DIR = +1: S2 -> S1, keep y < ny.
// A CTA takes B kx columns of one (grid, component, z) plane.
template <typename T, int DIR>
__global__ void __launch_bounds__(kRtThreads)
rt_y_pass(DemagDims d, const typename Cplx<T>::type* __restrict__ in, typename Cplx<T>::type* __restrict__ out,
          RtPlan pl, int B) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int L = pl.L;
    C* a = reinterpret_cast<C*>(smraw);
    C* b = a + (size_t)L * B;
    const int kx0 = blockIdx.x * B;
    const long cz = blockIdx.y;
    const int rows_in = DIR < 0 ? d.ny : L;
    const int rows_out = DIR < 0 ? L : d.ny;
    const C* src = in + (cz * rows_in) * d.KXS;
    C* dst = out + (cz * rows_out) * d.KXS;
    for (int idx = threadIdx.x; idx < L * B; idx += blockDim.x) {
        const int l = idx % B, e = idx / B;
        const int kx = kx0 + l;
        a[e * B + l] = (e < rows_in && kx < d.KX) ? src[(long)e * d.KXS + kx] : mk<C>(0, 0);
    }
    __syncthreads();
    const C* z = rt_fft<T, DIR>(a, b, B, pl);
    for (int idx = threadIdx.x; idx < rows_out * B; idx += blockDim.x) {
        const int l = idx % B, e = idx / B;
        const int kx = kx0 + l;
        if (kx < d.KX) dst[(long)e * d.KXS + kx] = z[e * B + l];
    }
}

// -------------------------------------------------------------- z pass ----
// Per (kx, ky) column: z-forward of the three components, h^ = T M^ with the
// octant-folded real tensor (sign flips of the odd components from the
// parity of ky and kz, or of the transformed axis on 2-D grids), z-inverse,
// keep z < nz; in place in S2.  A CTA takes B kx columns of one ky; blockIdx.z
// is the grid of a batch.
template <typename T>
__global__ void __launch_bounds__(kRtThreads)
rt_z_conv(DemagDims d, typename Cplx<T>::type* __restrict__ S2, const T* __restrict__ tens, RtPlan pl, int B) {
    using C = typename Cplx<T>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int LZ = pl.L;
    C* buf[4];
    buf[0] = reinterpret_cast<C*>(smraw);
    for (int q = 1; q < 4; ++q) buf[q] = buf[q - 1] + (size_t)LZ * B;
    const int LY = d.LY;
    const int KY2 = LY / 2 + 1;
    const int p = blockIdx.y >> 1, side = blockIdx.y & 1;
    if (!(p < KY2 && (side == 0 || (p > 0 && 2 * p < LY)))) return;      // uniform over the CTA
    const int ky = side ? LY - p : p;
    const int kx0 = blockIdx.x * B;
    const long cstride = (long)d.nz * LY * d.KXS;
    const long zs = (long)LY * d.KXS;
    C* col = S2 + (long)blockIdx.z * 3 * cstride + (long)ky * d.KXS + kx0;
    C* area[3] = {buf[0], buf[1], buf[2]};
    C* scratch = buf[3];
    for (int c = 0; c < 3; ++c)
        for (int idx = threadIdx.x; idx < LZ * B; idx += blockDim.x) {
            const int l = idx % B, z = idx / B;
            area[c][z * B + l] = (z < d.nz && kx0 + l < d.KX) ? col[c * cstride + z * zs + l] : mk<C>(0, 0);
        }
    __syncthreads();
    for (int c = 0; c < 3; ++c) {
        C* r = rt_fft<T, -1>(area[c], scratch, B, pl);
        if (r != area[c]) { scratch = area[c]; area[c] = r; }
    }
    const int KZ2 = LZ / 2 + 1;
    const long tcomp = (long)KZ2 * KY2 * d.KXS;
    const T sy = side ? (T)-1 : (T)1;
    for (int idx = threadIdx.x; idx < LZ * B; idx += blockDim.x) {
        const int l = idx % B, kz = idx / B;
        const int kx = kx0 + l;
        if (kx >= d.KX) continue;
        const int kzf = (2 * kz <= LZ) ? kz : LZ - kz;
        const T sz = (2 * kz <= LZ) ? (T)1 : (T)-1;
        const T* tp = tens + ((long)kzf * KY2 + p) * d.KXS + kx;
        const T txx = __ldg(tp);
        const T txy = (d.yz_swap ? sz : sy) * __ldg(tp + tcomp);
        const T txz = (d.yz_swap ? sy : sz) * __ldg(tp + 2 * tcomp);
        const T tyy = __ldg(tp + 3 * tcomp);
        const T tyz = sy * sz * __ldg(tp + 4 * tcomp);
        const T tzz = __ldg(tp + 5 * tcomp);
        const int o = kz * B + l;
        const C mx = area[0][o], my = area[1][o], mz = area[2][o];
        area[0][o] = mk<C>(txx * mx.x + txy * my.x + txz * mz.x, txx * mx.y + txy * my.y + txz * mz.y);
        area[1][o] = mk<C>(txy * mx.x + tyy * my.x + tyz * mz.x, txy * mx.y + tyy * my.y + tyz * mz.y);
        area[2][o] = mk<C>(txz * mx.x + tyz * my.x + tzz * mz.x, txz * mx.y + tyz * my.y + tzz * mz.y);
    }
    __syncthreads();
    for (int c = 0; c < 3; ++c) {
        C* r = rt_fft<T, +1>(area[c], scratch, B, pl);
        if (r != area[c]) { scratch = area[c]; area[c] = r; }
    }
    for (int c = 0; c < 3; ++c)
        for (int idx = threadIdx.x; idx < d.nz * B; idx += blockDim.x) {
            const int l = idx % B, z = idx / B;
            if (kx0 + l < d.KX) col[c * cstride + z * zs + l] = area[c][z * B + l];
        }
}

// ------------------------------------------------------------- launchers ----
// The limit belongs to a kernel and a device, not to a launch, and one kernel
// serves lines of many lengths: it is raised once, to all that a CTA may have.
// Set to each launch's own size, a thread with a shorter line would take it from
// under another's longer one between that thread's two calls.  (Requests that
// stay clear of the 48 KB every kernel may use, a little static shared memory
// included, need nothing.)  A limit that could not be raised shows as the
// launch's own error.
void allow_shared(const void* kernel, size_t bytes) {
    if (bytes <= 40 * 1024) return;
    struct Raised { const void* kernel; int device; };
    constexpr size_t kSlots = 2048;             // open addressing; when full, kernels are raised anew each time
    static Raised raised[kSlots];
    static std::mutex lock;
    int dev = 0, most = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    const size_t h = ((reinterpret_cast<uintptr_t>(kernel) >> 4) * 0x9E3779B97F4A7C15ull >> 40) + dev;
    std::lock_guard<std::mutex> guard(lock);
    Raised* slot = nullptr;
    for (size_t q = 0; q < 64 && !slot; ++q) {
        Raised& r = raised[(h + q) % kSlots];
        if (r.kernel == kernel && r.device == dev) return;
        if (!r.kernel) slot = &r;
    }
    cudaFuncAttributes a;
    if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess ||
        cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)a.sharedSizeBytes) !=
            cudaSuccess)
        return;
    if (slot) *slot = Raised{kernel, dev};
}

namespace {
template <typename K> void rt_smem(K kernel, size_t bytes) {
    allow_shared(reinterpret_cast<const void*>(kernel), bytes);
}
constexpr size_t kRtSmem = 200 * 1024;
// lines (or columns) per CTA: up to `cap`, as many as two (or four) buffers of L complex values allow
int rt_lines(int L, size_t csz, int nbuf, int cap) {
    int n = cap;
    while (n > 1 && (size_t)nbuf * L * n * csz > kRtSmem) --n;
    return n;
}
}  // namespace

template <typename T>
void launch_rt_x_fwd(const DemagDims& d, const T* m, const T* Ms_cell, T Ms, typename Cplx<T>::type* S1,
                     cudaStream_t st) {
    LineXIn<T> in;
    in.m = m; in.Ms_cell = Ms_cell; in.Ms = Ms;
    if (!d.classic && launch_line_x_fwd<T>(d, in, S1, st)) return;
    using C = typename Cplx<T>::type;
    const RtPlan pl = make_plan(d.LX);
    const int NL = rt_lines(d.LX, sizeof(C), 2, kRtMaxLines);
    const size_t sm = 2 * (size_t)d.LX * NL * sizeof(C);
    const long pairs = (long)d.nb * ((3L * d.ny * d.nz + 1) / 2);
    auto k = rt_x_forward<T>;
    rt_smem(k, sm);
    k<<<(unsigned)((pairs + NL - 1) / NL), kRtThreads, sm, st>>>(d, m, Ms_cell, Ms, S1, pl, NL);
}

template <typename T>
void launch_rt_x_inv(const DemagDims& d, const typename Cplx<T>::type* S1, T* h, cudaStream_t st) {
    if (!d.classic && launch_line_x_inv<T>(d, S1, h, st)) return;
    using C = typename Cplx<T>::type;
    const RtPlan pl = make_plan(d.LX);
    const int NL = rt_lines(d.LX, sizeof(C), 2, kRtMaxLines);
    const size_t sm = 2 * (size_t)d.LX * NL * sizeof(C);
    const long pairs = (long)d.nb * ((3L * d.ny * d.nz + 1) / 2);
    auto k = rt_x_inverse<T>;
    rt_smem(k, sm);
    k<<<(unsigned)((pairs + NL - 1) / NL), kRtThreads, sm, st>>>(d, S1, h, pl, NL);
}

// ---- line-engine launches ----
namespace {

// A launch of the line engine: 2^lb columns per CTA and the plan.
struct LineShape {
    LinePlan pl;
    int lb, threads;
    size_t smem;
    long ctas;
};

// The plan of a line, of which a launch has `lines`.  Radices are bounded by 8
// (FP32, which shared-memory exchanges bound) or 4 (FP64, whose instructions
// bound it: small radices cost no more of them and put more warps on them; the x
// lines of 128x128x32 took 84 and 80 us with radix 4, 124 and 105 with 8).  An
// FP64 length whose radix-4 plan keeps a radix-2 pass takes radices up to 8
// instead: the wide first pass would idle half its threads in every other
// (128x128x64's 128-point z lines 1351 -> 923 us, 256x256x64's 512-point lines
// 1490 -> 1010 and 1486 -> 1056 along y, 988 -> 649 and 953 -> 631 along x).  An
// FP64 grid that would leave quarter SMs idle takes radix 2; the grids of a batch
// do not count, so that a grid's rounding does not depend on the others.
bool line_few(int L, long lines) {
    return L > 2 && lines * (L / 4) < kSms * 128L;
}
template <typename T> LinePlan line_radices(int L, long lines, bool one) {
    if (sizeof(T) == 4) return host_plan(L, 8, one);
    if (line_few(L, lines)) return host_plan(L, 2, one);
    const LinePlan p = host_plan(L, 4, one);
    if (one || p.rmin != 2) return p;
    const LinePlan wide = host_plan(L, 8, one);
    return wide.np > 1 ? wide : p;          // 6 and 8 points keep two passes
}

// As many columns per CTA (at least one 32-byte sector of each row) as leave two
// CTAs for every SM.
template <typename T> bool line_shape(int L, long ncol, int nb, int nc, bool conv, LineShape* o) {
    constexpr int full = 128 / (2 * sizeof(T)), sector = 32 / (2 * sizeof(T));
    // FP32 z lines of up to 16 points stay in one thread's registers
    const bool one = conv && (L <= 2 || L == 4 || (sizeof(T) == 4 && (L == 6 || L == 8 || L == 12 || L == 16)));
    o->pl = line_radices<T>(L, ncol, one);
    const int M = L / o->pl.rmin;
    if (o->pl.np < 1 || o->pl.np > kLineMaxPass) return false;
    int lb = 0;
    while ((1 << lb) < full) ++lb;
    const size_t column = 2 * sizeof(T) * nc * line_len(L);
    auto fits = [&](int q) { return ((long)M << q) <= kLineThreads && column << q <= 160 * 1024; };
    while (lb > 0 && (!fits(lb) || (M << lb) > 256)) --lb;
    while (lb > 0 && (2 << lb) > 2 * sector && (M << lb) > 32 && ((ncol + (1 << lb) - 1) >> lb) * nb < 2 * kSms) --lb;
    if (!fits(lb)) return false;
    // short lines: whole warps
    while ((M << lb) < 32 || ((M << lb) < 64 && ((ncol + (2 << lb) - 1) >> (lb + 1)) * nb >= 4 * kSms)) ++lb;
    o->lb = lb;
    o->threads = (int)((((long)M << lb) + 31) / 32 * 32);
    o->smem = o->pl.np == 1 ? 0 : column << lb;
    o->ctas = (ncol + (1 << lb) - 1) >> lb;
    return true;
}

// Launched with programmatic stream serialisation, so that a kernel's set-up
// overlaps the end of the previous one; none but line_conv before a short y pass
// (DemagDims::early) triggers the next one earlier.  CTAs
// placed while the previous grid still runs crowd on the SMs that finish first:
// with a trigger at the start of launches of at most 304 CTAs an RK4 step of
// 512x128x1 in FP32 took 92 us instead of 59, 300x128x1 74 instead of 54, four FP64
// Dormand-Prince steps of the film 3080 us instead of 2831.
template <typename... KArgs, typename... Args>
void line_launch(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args&&... args) {
    allow_shared(reinterpret_cast<const void*>(kernel), smem);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// FP64 plans whose passes have unequal numbers of butterflies (line_warp_idle);
// lines: of all grids, as no result depends on it.
// Where few lines leave the pipe idle anyway the vote pays from a third of the
// threads without work on: an RK4 step of 16x16x49 (98 points, 52 % busy) 367 ->
// 219 us, five of a 20x45x4 stack (40 and 90 points, 85 and 68 %) 979 -> 992.
template <typename T> bool line_idle(const LinePlan& pl, long lines) {
    if (sizeof(T) == 4) return false;
    double busy = 0;
    for (int i = 0; i < pl.np; ++i) busy += (double)pl.rmin / pl.R[i] / pl.np;
    return busy < (line_few(pl.L, lines) ? 0.65 : 0.999);
}

// the kernel of a compiled length in place of the run-time one, if there is one
template <typename... KArgs> bool line_ct_use(LineKind kind, int L, void (**kernel)(KArgs...)) {
    const void* k = line_ct_kernel0(kind, L);
    if (!k) k = line_ct_kernel1(kind, L);
    if (!k) k = line_ct_kernel2(kind, L);
    if (!k) k = line_ct_kernel3(kind, L);
    if (!k) return false;
    *kernel = reinterpret_cast<void (*)(KArgs...)>(const_cast<void*>(k));
    return true;
}

}  // namespace

namespace {

// A launch of the x passes: nt threads for each of a CTA's lines.
struct LineXShape {
    LinePlan pl;
    int nt, lines, threads;
    bool ct;             // a compiled length's kernel holds that many threads
    size_t smem;
    long ctas;
};

// As many lines per CTA (up to 256 threads) as leave two CTAs for every SM
// (nb = 1 for the fused stage: its block partials must not depend on a batch's
// other grids); never more CTAs than max_ctas for each grid.  nc: lines of a row
// pair (3: the fused stage's components).  FP64 radices as in line_shape.
template <typename T> bool line_x_shape(int L, long pairs, int nb, int nc, long max_ctas, LineXShape* o) {
    o->pl = line_radices<T>(L, pairs, false);
    if (o->pl.np < 2) return false;
    o->nt = L / o->pl.rmin;
    const int per = nc * o->nt, most = nc == 3 ? 1024 : kLineThreads;
    // (the fused stage parks up to 6 float2 values for each x of a row pair besides)
    const size_t one = 2 * sizeof(T) * nc * line_len(L) + (nc == 3 ? 6 * sizeof(float2) * (L / 2) : 0);
    if (per > most || one > 200 * 1024) return false;
    long lines = per >= 256 ? 1 : 256 / per;
    while (lines > 1 && (lines * (long)one > 100 * 1024 || (pairs + lines - 1) / lines * nb < 2 * kSms)) --lines;
    while ((pairs + lines - 1) / lines > max_ctas) ++lines;
    if (lines * per > most || lines * (long)one > 200 * 1024) return false;
    o->lines = (int)lines;
    o->threads = (int)((lines * per + 31) / 32 * 32);
    o->ct = o->threads <= (nc == 1 || per <= 256 ? 256 : (per + 31) / 32 * 32);
    o->smem = lines * 2 * sizeof(T) * nc * line_len(L);
    o->ctas = (pairs + lines - 1) / lines;
    return true;
}
constexpr long kAnyCtas = 1L << 40;

long line_x_pairs(const DemagDims& d) { return (3L * d.ny * d.nz + 1) / 2; }
long line_fused_pairs(const DemagDims& d) { return (long)d.nz * ((d.ny + 1) / 2); }

}  // namespace

template <typename T>
bool launch_line_x_fwd(const DemagDims& d, const LineXIn<T>& in, typename Cplx<T>::type* S1, cudaStream_t st) {
    LineXShape o;
    if (d.nb > 65535 || !line_x_shape<T>(d.LX, line_x_pairs(d), d.nb, 1, kAnyCtas, &o)) return false;
    LineForward<T> f{in.m, in.Ms_cell, in.Ms, in.k, in.y, in.ca, in.dt_b, in.a, in.mask};
    auto k = o.threads <= 256 ? line_x_forward<T, 256, 0> : line_x_forward<T, kLineThreads, 0>;
    if constexpr (sizeof(T) == 8) {
        if (line_idle<T>(o.pl, line_x_pairs(d) * d.nb))
            k = o.threads <= 256 ? line_x_forward<T, 256, 0, true> : line_x_forward<T, kLineThreads, 0, true>;
    } else {
        if (o.ct) line_ct_use(kLineXFwd, d.LX, &k);
    }
    line_launch(k, dim3((unsigned)o.ctas, d.nb), o.threads, o.smem, st, d, f, S1, o.pl, line_table<T>(o.pl), o.nt, o.lines);
    return true;
}

template <typename T>
bool launch_line_x_inv(const DemagDims& d, const typename Cplx<T>::type* S1, T* h, cudaStream_t st) {
    LineXShape o;
    if (d.nb > 65535 || !line_x_shape<T>(d.LX, line_x_pairs(d), d.nb, 1, kAnyCtas, &o)) return false;
    auto k = o.threads <= 256 ? line_x_inverse<T, 256, 0> : line_x_inverse<T, kLineThreads, 0>;
    if constexpr (sizeof(T) == 8) {
        if (line_idle<T>(o.pl, line_x_pairs(d) * d.nb))
            k = o.threads <= 256 ? line_x_inverse<T, 256, 0, true> : line_x_inverse<T, kLineThreads, 0, true>;
    } else {
        if (o.ct) line_ct_use(kLineXInv, d.LX, &k);
    }
    line_launch(k, dim3((unsigned)o.ctas, d.nb), o.threads, o.smem, st, d, S1, h, o.pl, line_table<T>(o.pl), o.nt, o.lines);
    return true;
}

// The fused stage indexes the three components of a grid in 32 bits (in 64, five
// RK4 steps of a 20x45x4 stack of layers took 461 us instead of 441): 716 million
// cells and more take the separate passes, whose stage kernel has 64.
static bool line_fused_fits(const DemagDims& d) { return 3L * d.nx * d.ny * d.nz < 1L << 31; }

int line_fused_blocks(const DemagDims& d, long max_ctas) {
    LineXShape o;
    if (!line_fused_fits(d)) return 0;
    if (d.nb > 65535 || !line_x_shape<float>(d.LX, line_fused_pairs(d), 1, 3, max_ctas, &o)) return 0;
    return (int)o.ctas;
}

bool launch_line_fused(const DemagDims& d, float2* S1, const StageParams<float>& p, const LineBatch* bt, bool gen,
                       bool fwd, long max_ctas, cudaStream_t st) {
    LineXShape o;
    if (!line_fused_fits(d) || d.nb > 65535 || !line_x_shape<float>(d.LX, line_fused_pairs(d), 1, 3, max_ctas, &o))
        return false;
    LineBatch b{};
    if (bt) b = *bt;
    auto k = gen ? (o.threads <= 256 ? line_fused<true, 256, 0> : line_fused<true, 1024, 0>)
                 : (o.threads <= 256 ? line_fused<false, 256, 0> : line_fused<false, 1024, 0>);
    if (o.ct) line_ct_use(gen ? kLineFusedGen : kLineFused, d.LX, &k);
    // parked float2 values per x of a row pair (line_fused)
    const int park = (p.next ? 3 : 0) + (p.want_err ? 3 : 0);
    const size_t smem = o.smem + (size_t)o.lines * park * d.nx * sizeof(float2);
    line_launch(k, dim3((unsigned)o.ctas, d.nb), o.threads, smem, st, d, S1, p, b, o.pl, line_table<float>(o.pl), o.nt,
                o.lines, park, (int)fwd);
    return true;
}

// the column shape a compiled length's kernel is built for
static void line_ct_shape(int L, long ncol, LineShape* o) {
    o->lb = line_ct_lb<float>(L);
    const int M = L / o->pl.rmin;
    o->threads = ((M << o->lb) + 31) / 32 * 32;
    o->smem = (size_t)3 * line_len(L) * (sizeof(float2) << o->lb);
    o->ctas = (ncol + (1 << o->lb) - 1) >> o->lb;
}

template <typename T, int DIR>
bool launch_line_y(const DemagDims& d, const typename Cplx<T>::type* in, typename Cplx<T>::type* out,
                   cudaStream_t st) {
    LineShape o;
    const long ncol = 3L * d.KX * d.nz;
    if (d.nb > 65535 || !line_shape<T>(d.LY, ncol, d.nb, 1, false, &o) || o.pl.np < 2) return false;
    auto k = o.threads <= 256 ? line_y<T, DIR, 256> : line_y<T, DIR, kLineThreads>;
    if constexpr (sizeof(T) == 8) {
        if (line_idle<T>(o.pl, ncol * d.nb)) k = o.threads <= 256 ? line_y<T, DIR, 256, true> : line_y<T, DIR, kLineThreads, true>;
    }
    line_launch(k, dim3((unsigned)o.ctas, d.nb), o.threads, o.smem, st, d, in, out, o.pl, line_table<T>(o.pl), o.lb,
                (int)ncol);
    return true;
}

template <typename T>
bool launch_line_conv(const DemagDims& d, typename Cplx<T>::type* S2, const T* tens, cudaStream_t st) {
    LineShape o;
    const long ncol = (long)d.KX * d.LY;
    if (d.nb > 65535 || !line_shape<T>(d.LZ, ncol, d.nb, 3, true, &o)) return false;
    constexpr int kSmall = sizeof(T) == 4 ? kLineThreads32 : kLineThreads;
    const int M = o.pl.np ? d.LZ / o.pl.rmin : 0;
    const bool split = o.pl.np > 1 && line_split<T>(M);
    if (split) {
        o.lb = line_split_lb(M);
        o.threads = (((3 * M) << o.lb) + 31) / 32 * 32;
        o.smem = (size_t)3 * line_len(d.LZ) * (2 * sizeof(T) << o.lb);
        o.ctas = (ncol + (1 << o.lb) - 1) >> o.lb;
    }
    auto k = o.pl.np == 1 ? line_conv<T, kConvOne, 256, 0>
             : o.threads > kSmall ? line_conv<T, kConvThree, kLineThreads, 0> : line_conv<T, kConvThree, kSmall, 0>;
    if constexpr (sizeof(T) == 4) {
        if (o.pl.np > 1 && line_ct_use(kLineConv, d.LZ, &k)) line_ct_shape(d.LZ, ncol, &o);
    } else if (o.pl.np > 1) {
        const bool wide = std::any_of(o.pl.R, o.pl.R + o.pl.np, [](int r) { return r == 6 || r == 8; });
        const bool idle = line_idle<T>(o.pl, ncol * d.nb);
        // components lie side by side in a CTA's threads, and whole warps are idle only
        // where there are many of them (an RK4 step of 128x128x25: 4880 -> 4150 us)
        while (split && idle && ((6 * M) << o.lb) <= 384 && (ncol >> (o.lb + 1)) >= 8 * kSms) {
            ++o.lb;
            o.threads = (((3 * M) << o.lb) + 31) / 32 * 32;
            o.smem *= 2;
            o.ctas = (ncol + (1 << o.lb) - 1) >> o.lb;
        }
        const bool small = o.threads <= 384;
        if (!split) {
            if (idle) k = line_conv<T, kConvThree, kLineThreads, 0, true>;
        } else if (idle) {
            if (wide) k = small ? line_conv<T, kConvSplitWide, 384, 0, true> : line_conv<T, kConvSplitWide, 768, 0, true>;
            else k = small ? line_conv<T, kConvSplit, 384, 0, true> : line_conv<T, kConvSplit, 768, 0, true>;
        } else {
            if (wide) k = small ? line_conv<T, kConvSplitWide, 384, 0> : line_conv<T, kConvSplitWide, 768, 0>;
            else k = small ? line_conv<T, kConvSplit, 384, 0> : line_conv<T, kConvSplit, 768, 0>;
        }
    }
    const dim3 grid((unsigned)o.ctas, d.nb);
    line_launch(k, grid, o.threads, o.smem, st, d, S2, tens, o.pl, line_table<T>(o.pl), o.lb, (int)ncol);
    return true;
}

template <typename T, int DIR>
void launch_rt_y(const DemagDims& d, const typename Cplx<T>::type* in, typename Cplx<T>::type* out,
                 cudaStream_t st) {
    if (!d.classic && launch_line_y<T, DIR>(d, in, out, st)) return;
    using C = typename Cplx<T>::type;
    const RtPlan pl = make_plan(d.LY);
    const int B = rt_lines(d.LY, sizeof(C), 2, (int)(128 / sizeof(C)));
    const size_t sm = 2 * (size_t)d.LY * B * sizeof(C);
    dim3 grid((d.KX + B - 1) / B, (unsigned)(d.nb * 3 * d.nz));
    auto k = rt_y_pass<T, DIR>;
    rt_smem(k, sm);
    k<<<grid, kRtThreads, sm, st>>>(d, in, out, pl, B);
}

template <typename T>
void launch_rt_z(const DemagDims& d, typename Cplx<T>::type* S2, const T* tens, cudaStream_t st) {
    if (!d.classic && launch_line_conv<T>(d, S2, tens, st)) return;
    using C = typename Cplx<T>::type;
    const RtPlan pl = make_plan(d.LZ);
    const int B = rt_lines(d.LZ, sizeof(C), 4, (int)(128 / sizeof(C)));
    const size_t sm = 4 * (size_t)d.LZ * B * sizeof(C);
    dim3 grid((d.KX + B - 1) / B, 2 * (d.LY / 2 + 1), d.nb);
    auto k = rt_z_conv<T>;
    rt_smem(k, sm);
    k<<<grid, kRtThreads, sm, st>>>(d, S2, tens, pl, B);
}

template void launch_rt_x_fwd<float>(const DemagDims&, const float*, const float*, float, float2*, cudaStream_t);
template void launch_rt_x_fwd<double>(const DemagDims&, const double*, const double*, double, double2*,
                                      cudaStream_t);
template void launch_rt_x_inv<float>(const DemagDims&, const float2*, float*, cudaStream_t);
template void launch_rt_x_inv<double>(const DemagDims&, const double2*, double*, cudaStream_t);
template bool launch_line_y<float, -1>(const DemagDims&, const float2*, float2*, cudaStream_t);
template bool launch_line_y<float, +1>(const DemagDims&, const float2*, float2*, cudaStream_t);
template bool launch_line_y<double, -1>(const DemagDims&, const double2*, double2*, cudaStream_t);
template bool launch_line_y<double, +1>(const DemagDims&, const double2*, double2*, cudaStream_t);
template bool launch_line_conv<float>(const DemagDims&, float2*, const float*, cudaStream_t);
template bool launch_line_conv<double>(const DemagDims&, double2*, const double*, cudaStream_t);

template void launch_rt_y<float, -1>(const DemagDims&, const float2*, float2*, cudaStream_t);
template void launch_rt_y<float, +1>(const DemagDims&, const float2*, float2*, cudaStream_t);
template void launch_rt_y<double, -1>(const DemagDims&, const double2*, double2*, cudaStream_t);
template void launch_rt_y<double, +1>(const DemagDims&, const double2*, double2*, cudaStream_t);
template void launch_rt_z<float>(const DemagDims&, float2*, const float*, cudaStream_t);
template void launch_rt_z<double>(const DemagDims&, double2*, const double*, cudaStream_t);

template bool launch_line_x_fwd<float>(const DemagDims&, const LineXIn<float>&, float2*, cudaStream_t);
template bool launch_line_x_fwd<double>(const DemagDims&, const LineXIn<double>&, double2*, cudaStream_t);
template bool launch_line_x_inv<float>(const DemagDims&, const float2*, float*, cudaStream_t);
template bool launch_line_x_inv<double>(const DemagDims&, const double2*, double*, cudaStream_t);

}  // namespace mm
