// Coarse solve K x2 = t (Sec. 2.3.3, eq. block_matrix_inversion): dense K^-1 GEMV forms for
// small coarse systems, the nested-dissection multifrontal solve, and the CSR residual of
// the refinement step.
#include "ddh_fixed.cuh"
#include "ddh_kcommon.cuh"
#include <type_traits>
#include <utility>

namespace ddh {

// ------------------------------------------------------------------ split matrices (ddh_fixed.cuh)
// row a[j cs], j < n, to d[j cs], its exponent to ex, by one warp
__device__ __forceinline__ void fix_row(const double2* a, const FxMat& d, int64_t cs, int n, int* ex) {
    const int lane = threadIdx.x & 31;
    unsigned m = 0;
    for (int j = lane; j < n; j += 32) m = max(m, fx_mag(a[j * cs]));
    const int ef = fx_exp(__reduce_max_sync(0xffffffffu, m));
    for (int j = lane; j < n; j += 32) fx_put(d, j * cs, a[j * cs], ef);
    if (lane == 0) *ex = ef;
}
// K^-1, packed: one exponent per row and tile of kGemvTile columns
constexpr int kGemvThreads = 512, kGemvTile = 736;
__global__ void k_fix_dense(const double2* __restrict__ A, int n, longlong2* __restrict__ d, int* __restrict__ ex) {
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const int nt = (n + kGemvTile - 1) / kGemvTile;
    if (row >= n) return;
    for (int t = 0; t < nt; ++t) {
        const int64_t at = (int64_t)row * n + t * kGemvTile;
        const int w = min(kGemvTile, n - t * kGemvTile);
        unsigned m = 0;
        for (int j = lane; j < w; j += 32) m = max(m, fx_mag(A[at + j]));
        const int ef = fx_exp(__reduce_max_sync(0xffffffffu, m));
        for (int j = lane; j < w; j += 32) d[at + j] = make_longlong2(fx_pack(A[at + j].x, ef), fx_pack(A[at + j].y, ef));
        if (lane == 0) ex[(int64_t)row * nt + t] = ef;
    }
}
// the two matrices of one nested-dissection front per CTA (layouts: NDDev)
__global__ void k_fix_fronts(NDDev d) {
    const int node = blockIdx.x, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nF = d.nF[node], nB = d.nB[node], n = nF + nB;
    const int64_t go = d.g_off[node], mo = d.m_off[node];
    const bool gs = nF <= kNDShortRow, ms = n <= kNDShortRow;
    for (int r = warp; r < nB; r += nw) {
        const int64_t at = go + (gs ? r : (int64_t)r * nF);
        fix_row((const double2*)d.G + at, d.gfx.at(at), gs ? nB : 1, nF, d.gexp + d.u_off[node] + r);
    }
    for (int r = warp; r < nF; r += nw) {
        const int64_t at = mo + (ms ? r : (int64_t)r * n);
        fix_row((const double2*)d.M + at, d.mfx.at(at), ms ? nF : 1, n, d.mexp + d.f0[node] + r);
    }
}

// ------------------------------------------------------------------ dense K^-1
// y = K^-1 x for the complex64 copy (the mixed-precision inner solves with coarse_fp32) and RB right-hand sides,
// one warp per row; vectors and accumulation FP64, which bounds it.  n = 1921, one right-hand side: 57 us; two
// warps per row or two rows per warp measured the same within 3 %.
template <int RB>
__global__ void k_gemv(const float2* __restrict__ A, int n, const double2* __restrict__ x, double2* __restrict__ y, int r0,
                       const int* __restrict__ done) {
    if (done && *done) return;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= n) return;
    const float2* a = A + (int64_t)warp * n;
    const double2* xr = x + (int64_t)r0 * n;
    double sx[RB], sy[RB];
#pragma unroll
    for (int q = 0; q < RB; ++q) { sx[q] = 0; sy[q] = 0; }
    int j = lane;
    if (RB == 1) {
        // one right-hand side: four loads in flight per lane, two accumulator chains
        double tx = 0, ty = 0;
        for (; j + 96 < n; j += 128) {
            const float2 a0 = a[j], a1 = a[j + 32], a2 = a[j + 64], a3 = a[j + 96];
            const double2 x0 = xr[j], x1 = xr[j + 32], x2 = xr[j + 64], x3 = xr[j + 96];
            sx[0] = fma((double)a0.x, x0.x, fma(-(double)a0.y, x0.y, sx[0]));
            sy[0] = fma((double)a0.x, x0.y, fma((double)a0.y, x0.x, sy[0]));
            tx = fma((double)a1.x, x1.x, fma(-(double)a1.y, x1.y, tx));
            ty = fma((double)a1.x, x1.y, fma((double)a1.y, x1.x, ty));
            sx[0] = fma((double)a2.x, x2.x, fma(-(double)a2.y, x2.y, sx[0]));
            sy[0] = fma((double)a2.x, x2.y, fma((double)a2.y, x2.x, sy[0]));
            tx = fma((double)a3.x, x3.x, fma(-(double)a3.y, x3.y, tx));
            ty = fma((double)a3.x, x3.y, fma((double)a3.y, x3.x, ty));
        }
        sx[0] += tx;
        sy[0] += ty;
    }
    for (; j < n; j += 32) {
        const float2 av = a[j];
        const double ax = (double)av.x, ay = (double)av.y;
#pragma unroll
        for (int q = 0; q < RB; ++q) {
            const double2 xv = xr[(int64_t)q * n + j];
            sx[q] = fma(ax, xv.x, fma(-ay, xv.y, sx[q]));
            sy[q] = fma(ax, xv.y, fma(ay, xv.x, sy[q]));
        }
    }
#pragma unroll
    for (int q = 0; q < RB; ++q) {
        for (int o = 16; o > 0; o >>= 1) {
            sx[q] += __shfl_xor_sync(0xffffffffu, sx[q], o);
            sy[q] += __shfl_xor_sync(0xffffffffu, sy[q], o);
        }
    }
    if (lane < RB) {
        double vx = 0, vy = 0;
#pragma unroll
        for (int q = 0; q < RB; ++q) if (q == lane) { vx = sx[q]; vy = sy[q]; }
        y[(int64_t)(r0 + lane) * n + warp] = make_double2(vx, vy);
    }
}

__host__ __device__ constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v / 2); }

// Warp sum of V values per lane by a transposing butterfly: each of the first log2(V) rounds
// halves the values a lane carries (it keeps one half, sends the other half to its partner and
// adds what it receives); the remaining rounds are a plain butterfly on the one value left.
// V - 1 + 5 - log2(V) adds per lane instead of 5 V.  On return every lane holds the full sum of
// value index lane >> (5 - log2(V)).
template <class T, int V>
__device__ __forceinline__ T warp_sum_transpose(T (&v)[V]) {
    static_assert(V >= 1 && V <= 32 && (V & (V - 1)) == 0, "V must be a power of two <= 32");
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = V / 2, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T send = up ? v[i] : v[i + h];
            const T keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = 16 >> ilog2(V); o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// ------------------------------------------------------------------ coarse solve
// Nested-dissection solve of K x = t, one launch per tree level (see NDDev).  A CTA of 128
// threads takes rows of one node's matrix for a block of RB right-hand sides after staging
// the node's input vector in shared memory ([RB][stride], odd stride against bank
// conflicts).  Long rows: up to 4 rows per item, one warp per row, lanes across the row.
// Short rows (column-major matrix): up to 16 rows per item, 32/S rows per warp at a time with S lanes
// (column slices) each, and all right-hand sides of the block in a lane, so that an entry of the matrix
// is loaded once; small items spread a level over all SMs.
// Arithmetic follows the factor's storage type MT: the FP64-accurate products of ddh_fixed.cuh for the
// complex128 factor, FP32 for its complex64 copy (vectors stay complex128 in global memory and are
// converted when they are staged).
template <class MT> constexpr bool kNDFixed = std::is_same<MT, double2>::value;
// bytes of a staged entry, and of len of them (rounded up to keep what follows aligned)
template <class MT> constexpr int kNDEntry = kNDFixed<MT> ? 32 : 8;
template <class MT> __host__ __device__ constexpr size_t nd_bytes(size_t len) { return (kNDEntry<MT> * len + 15) & ~(size_t)15; }
// the longest vector that is staged in limbs; the rows of a front with a longer one are summed in FP64 from
// global memory
constexpr int kNDFixedRows = 6144;
// RB staged vectors at stride: limbs and fractions, or complex64
template <class MT, int RB>
struct NDStaged {
    int4* i;
    float4* f;
    float2* v;
    __device__ __forceinline__ NDStaged(char* sm, int stride)
        : i(reinterpret_cast<int4*>(sm)), f(reinterpret_cast<float4*>(i + RB * stride)), v(reinterpret_cast<float2*>(sm)) {}
};

// Sum of V values per lane over each group of G consecutive lanes (xor offsets G/2, ..., 1, in
// that order for every value, so the result does not depend on V), transposing while a lane
// carries more than one value.  Afterwards, with g = lane & (G - 1): if V >= G, v[i] (i < V/G) is
// the sum of value index (g << log2(V/G)) | i; else v[0] is the sum of value g >> log2(G/V).
template <class T, int V, int G>
__device__ __forceinline__ void group_sum_transpose(T (&v)[V]) {
    static_assert(V >= 1 && (V & (V - 1)) == 0 && G >= 1 && G <= 32 && (G & (G - 1)) == 0, "powers of two");
    if (G == 1) return;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = V / 2, o = G / 2; h >= 1 && o >= 1; h >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T send = up ? v[i] : v[i + h];
            const T keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int o = (G / 2) >> ilog2(V); o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}

// y = K^-1 x with the products of ddh_fixed.cuh.  A CTA of 16 warps owns `rpc` rows (one CTA per SM), one warp
// per row.  It stages x in shared memory as limbs, G tiles of kGemvTile columns at a time (each tile of a
// row and of a vector has its own exponent, so a right-hand side's result does not depend on RB), and adds
// the tiles up in FP64.  K^-1 is packed: in the 24 bytes of the split form it does not stay in L2 between the
// iterations of a solve (n = 1921, one right-hand side: 1.95 ms a solve instead of 1.77 ms).  n = 1921: 25 us for one
// right-hand side (35 us in FP64), 138 us for eight; n = 2961: 59 and 301 us.
template <int RB>
__global__ void __launch_bounds__(kGemvThreads) k_gemv_fx(const double2* __restrict__ A, const longlong2* __restrict__ Ap,
                                                         const int* __restrict__ aex, int n,
                                                         const double2* __restrict__ x, double2* __restrict__ y,
                                                         int r0, int nr, int rpc, const int* __restrict__ done) {
    if (done && *done) return;
    extern __shared__ __align__(16) char gv_raw[];
    constexpr int nw = kGemvThreads / 32, G = 8 / RB, stride = G * kGemvTile + 1;
    __shared__ unsigned wmax[nw][8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int4* xs = reinterpret_cast<int4*>(gv_raw);                                             // [RB][stride]
    float4* xf = reinterpret_cast<float4*>(xs + RB * stride);
    double* acc = reinterpret_cast<double*>(xf + RB * stride);                              // [rpc][2 RB]
    const int row0 = blockIdx.x * rpc, rows = min(rpc, n - row0), nt = (n + kGemvTile - 1) / kGemvTile;
    for (int g0 = 0; g0 < n; g0 += G * kGemvTile) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {                      // (tile, vector)
            const int q = k % RB, c0 = g0 + k / RB * kGemvTile, w = min(kGemvTile, n - c0);
            const double2* xq = x + (int64_t)(r0 + q) * n + c0;
            double2* d = reinterpret_cast<double2*>(xs) + q * stride + k / RB * kGemvTile;
            unsigned m = 0;
#pragma unroll
            for (int u = 0; u < 2; ++u) {                  // kGemvTile <= 2 kGemvThreads
                const int i = threadIdx.x + u * kGemvThreads;
                if (i < w) {
                    const double2 v = q < nr ? xq[i] : make_double2(0.0, 0.0);
                    d[i] = v;
                    m = max(m, fx_mag(v));
                }
            }
            m = __reduce_max_sync(0xffffffffu, m);
            if (lane == 0) wmax[warp][k] = m;
        }
        __syncthreads();
        int ex[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int at = k % RB * stride + k / RB * kGemvTile, w = min(kGemvTile, n - (g0 + k / RB * kGemvTile));
            unsigned m = 0;
#pragma unroll
            for (int i = 0; i < nw; ++i) m = max(m, wmax[i][k]);
            ex[k] = fx_exp(m);
            for (int i = threadIdx.x; i < w; i += kGemvThreads) {
                const FxVec v = fx_vec(reinterpret_cast<double2*>(xs)[at + i], ex[k]);
                xs[at + i] = v.i;
                xf[at + i] = v.f;
            }
        }
        __syncthreads();
        for (int k = warp; k < rows; k += nw) {
            constexpr int sh = 5 - ilog2(2 * RB);
            const int q = lane >> sh;                      // component q & 1 of right-hand side q >> 1
            const bool mine = (lane & ((1 << sh) - 1)) == 0 && (q >> 1) < nr;
            double* d = acc + k * 2 * RB + q;
            double t = g0 && mine ? *d : 0.0;
#pragma unroll 1
            for (int tl = 0; tl < G; ++tl) {
                const int c0 = g0 + tl * kGemvTile, w = min(kGemvTile, n - c0);
                if (w <= 0) break;
                const double2* a = A + (int64_t)(row0 + k) * n + c0;
                const int ea = aex[(int64_t)(row0 + k) * nt + c0 / kGemvTile], o = tl * kGemvTile;
                FxSum s[RB];
#pragma unroll
                for (int i = 0; i < RB; ++i) fx_clear(s[i]);
                constexpr int U = RB == 1 ? 6 : (RB == 2 ? 4 : 2);     // loads issued ahead of their use
                longlong2 av[U];
                const longlong2* ap = Ap + (int64_t)(row0 + k) * n + c0;
#pragma unroll
                for (int u = 0; u < U; ++u) av[u] = lane + 32 * u < w ? __ldg(ap + lane + 32 * u) : make_longlong2(0, 0);
                for (int j = lane; j < w; j += 32 * U) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        int4 ai;
                        float2 af;
                        fx_unpack(av[u], ai, af);
                        const FxEntry v = fx_entry(ai, af);
                        const int jj = o + min(j + 32 * u, w - 1), jn = j + 32 * (U + u);
                        av[u] = jn < w ? __ldg(ap + jn) : make_longlong2(0, 0);
#pragma unroll
                        for (int b = 0; b < RB; ++b) fx_mac(s[b], v, xs[b * stride + jj], xf[b * stride + jj]);
                    }
                }
                long long h[2 * RB], l[2 * RB];
#pragma unroll
                for (int i = 0; i < 2 * RB; ++i) {
                    h[i] = l[i] = 0;
                    fx_flush(s[i >> 1], i & 1, h[i], l[i]);
                }
                const long long hs = warp_sum_transpose<long long, 2 * RB>(h), ls = warp_sum_transpose<long long, 2 * RB>(l);
                int e = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) e = i == tl * RB + (q >> 1) ? ex[i] : e;
                double v = 0;
                const bool bad = (q >> 1) < nr && !fx_value(hs, ls, ea, e, v, kFxSmallPacked);
                if (__any_sync(0xffffffffu, bad)) {
#pragma unroll 1
                    for (int b = 0; b < nr; ++b) {
                        const bool this_b = bad && (q >> 1) == b;
                        if (!__any_sync(0xffffffffu, this_b)) continue;
                        const double2* xq = x + (int64_t)(r0 + b) * n + c0;
                        int eb = 0;
#pragma unroll
                        for (int i = 0; i < 8; ++i) eb = i == tl * RB + b ? ex[i] : eb;
                        double2 r;
                        const int4* xi = xs + b * stride + o;
                        const unsigned keep = fx_again(32, this_b ? 1u << (q & 1) : 0, w, ea, eb, [=](int j) { return a[j]; },
                                                       [=](int j) { const longlong2 u = ap[j]; return make_int2((int)(u.x >> 37), (int)(u.y >> 37)); },
                                                       [=](int j) { return xi[j]; }, [=](int j) { return xq[j]; }, r, kFxSmallPacked);
                        if (this_b && !(keep >> (q & 1) & 1)) v = q & 1 ? r.y : r.x;
                    }
                }
                t += v;
            }
            if (mine) {
                if (g0 + G * kGemvTile < n) *d = t;
                else reinterpret_cast<double*>(y + (int64_t)(r0 + (q >> 1)) * n + row0 + k)[q & 1] = t;
            }
        }
        __syncthreads();                     // the next group overwrites xs
    }
}

// Loads of vectors written during the same launch by other CTAs (the one-launch schedule) go
// through L2 (ld.global.cg): another SM's L1 may hold a stale copy of the line.
template <bool CG>
__device__ __forceinline__ double2 ldv(const double2* p) { return CG ? __ldcg(p) : *p; }
// the children's amounts at offsets a and b of u (-1: none)
template <bool CG>
__device__ __forceinline__ double2 nd_pull(const double2* u, int64_t base, int64_t a, int64_t b) {
    double2 s = make_double2(0.0, 0.0);
    if (a >= 0) { const double2 v = ldv<CG>(u + base + a); s.x += v.x; s.y += v.y; }
    if (b >= 0) { const double2 v = ldv<CG>(u + base + b); s.x += v.x; s.y += v.y; }
    return s;
}
__device__ __forceinline__ void cfma(float& ax, float& ay, float2 a, float2 v) {
    ax = fma(a.x, v.x, fma(-a.y, v.y, ax));
    ay = fma(a.x, v.y, fma(a.y, v.x, ay));
}

// Threads that work on one node: the whole CTA, or (WARP) one warp of it, with its own shared memory.
template <bool WARP>
struct NDGroup {
    __device__ __forceinline__ static int t() { return WARP ? threadIdx.x & 31 : threadIdx.x; }
    __device__ __forceinline__ static int n() { return WARP ? 32 : blockDim.x; }
    __device__ __forceinline__ static int warp() { return WARP ? 0 : threadIdx.x >> 5; }
    __device__ __forceinline__ static int warps() { return WARP ? 1 : blockDim.x >> 5; }
    __device__ __forceinline__ static void sync() { if (WARP) __syncwarp(); else __syncthreads(); }
};
constexpr int kNDThreads = 128;          // level launches: four warps (long rows: a row each)
constexpr int kNDWarps = 8;              // bottom launches, and the most warps of a CTA
// shared memory beside the staged vectors: exponents, and the warps' maxima while they are found
struct NDShared {
    int ex[4];
    unsigned wmax[kNDWarps][4];
};

// Stages RB vectors of length n (odd stride) in shared memory: load(i, v) gives entry i of all of them
// as complex128, so that their index lookups are shared and RB loads are in flight per thread.
// Fixed point: each vector's exponent is that of its largest entry (2047, i.e. FP64 for all results, where
// it is too long to be staged).
template <class MT, int RB, bool WARP, class F>
__device__ __forceinline__ void nd_stage(const F& load, int n, int stride, char* sm, int* ex, NDShared* sh) {
    using G = NDGroup<WARP>;
    const NDStaged<MT, RB> st(sm, stride);
    if constexpr (kNDFixed<MT>) {
        double2* s = reinterpret_cast<double2*>(sm);
        const bool fit = n <= kNDFixedRows;
        unsigned m[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) m[r] = 0;
#pragma unroll 2
        for (int i = G::t(); i < n; i += G::n()) {
            double2 v[RB];
            load(i, v);
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                if (fit) s[r * stride + i] = v[r];
                m[r] = max(m[r], fx_mag(v[r]));
            }
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) m[r] = __reduce_max_sync(0xffffffffu, m[r]);
        if constexpr (!WARP) {
            if ((threadIdx.x & 31) == 0)
#pragma unroll
                for (int r = 0; r < RB; ++r) sh->wmax[threadIdx.x >> 5][r] = m[r];
            __syncthreads();
            for (int k = 0; k < G::warps(); ++k)
#pragma unroll
                for (int r = 0; r < RB; ++r) m[r] = max(m[r], sh->wmax[k][r]);
        }
        if (G::t() == 0)
#pragma unroll
            for (int r = 0; r < RB; ++r) ex[r] = fit ? fx_exp(m[r]) : 0x7ff;
        if (fit)
            for (int i = G::t(); i < n; i += G::n())
#pragma unroll
                for (int r = 0; r < RB; ++r) {
                    const FxVec w = fx_vec(s[r * stride + i], fx_exp(m[r]));
                    st.i[r * stride + i] = w.i;
                    st.f[r * stride + i] = w.f;
                }
    } else {
        for (int i = G::t(); i < n; i += G::n()) {
            double2 v[RB];
            load(i, v);
#pragma unroll
            for (int r = 0; r < RB; ++r) st.v[r * stride + i] = make_float2((float)v[r].x, (float)v[r].y);
        }
    }
    G::sync();
}

// One lane's terms a[j cs] x[j], j = j0, j0 + dj, ... < n, for RB vectors (staged): v[2r + c] is component c of
// vector r (fixed point: with low[]).  kNDAhead loads of A are in flight; pre holds
// the first ones when they were issued before the vectors were staged.
constexpr int kNDAhead = 4;
template <class MT> using NDSum = typename std::conditional<kNDFixed<MT>, long long, float>::type;
// the matrix that the sums read, and an entry of it in registers
struct NDSplit {
    int4 i;
    float2 f;
};
template <class MT> using NDMat = typename std::conditional<kNDFixed<MT>, FxMat, const MT*>::type;
template <class MT> using NDItem = typename std::conditional<kNDFixed<MT>, NDSplit, MT>::type;
template <class MT>
__device__ __forceinline__ void nd_ahead(const NDMat<MT>& a, int64_t cs, int j0, int dj, int n, bool ok,
                                         NDItem<MT> (&pre)[kNDAhead]) {
#pragma unroll
    for (int k = 0; k < kNDAhead; ++k) {
        const int j = j0 + k * dj;
        pre[k] = NDItem<MT>{};
        if (ok && j < n) {
            if constexpr (kNDFixed<MT>) pre[k] = {__ldg(a.i + j * cs), __ldg(a.f + j * cs)};
            else pre[k] = __ldg(a + j * cs);
        }
    }
}
template <class MT, int RB>
__device__ __forceinline__ void nd_dot(const NDMat<MT>& a, int64_t cs, int j0, int dj, int n, bool ok,
                                       NDItem<MT> (&pre)[kNDAhead], int stride, const NDStaged<MT, RB>& st, NDSum<MT> (&v)[2 * RB],
                                       long long (&low)[2 * RB]) {
#pragma unroll
    for (int i = 0; i < 2 * RB; ++i) { v[i] = 0; low[i] = 0; }
    FxSum s[RB];
    if constexpr (kNDFixed<MT>)
#pragma unroll
        for (int r = 0; r < RB; ++r) fx_clear(s[r]);
    auto flush = [&] {
        if constexpr (kNDFixed<MT>)
#pragma unroll
            for (int i = 0; i < 2 * RB; ++i) fx_flush(s[i >> 1], i & 1, v[i], low[i]);
#pragma unroll
        for (int r = 0; r < RB; ++r) fx_clear(s[r]);
    };
    for (int j = j0, c = 0; j < n; j += kNDAhead * dj) {
        NDItem<MT> nxt[kNDAhead];
        nd_ahead<MT>(a, cs, j + kNDAhead * dj, dj, n, ok, nxt);
#pragma unroll
        for (int k = 0; k < kNDAhead; ++k) {
            const int jj = min(j + k * dj, n - 1);         // past the end the entry of A is zero
            if constexpr (kNDFixed<MT>) {
                const FxEntry e = fx_entry(pre[k].i, pre[k].f);
#pragma unroll
                for (int r = 0; r < RB; ++r) fx_mac(s[r], e, st.i[r * stride + jj], st.f[r * stride + jj]);
            } else {
#pragma unroll
                for (int r = 0; r < RB; ++r) cfma(v[2 * r], v[2 * r + 1], pre[k], st.v[r * stride + jj]);
            }
            pre[k] = nxt[k];
        }
        if constexpr (kNDFixed<MT>)
            if ((c += kNDAhead) > kFxChain - kNDAhead) {
                c = 0;
                flush();
            }
    }
    if constexpr (kNDFixed<MT>) flush();
}

// Rows of one front's matrix, A x + add, by 32/S rows per warp: lane = (row, column slice of S).  In the
// constructor-like first step (ahead) a lane finds its row and issues its first loads of A; after the
// vectors are staged, run() forms the sums and hands component c (0 real, 1 imaginary) of right-hand
// side r to out(row, r, c, value).  Sums run in an order fixed by the matrix and S alone, so the result
// does not depend on RB.  cs, rs: strides of A along a row and between rows; load: the staged vectors'
// entries, for the results that are formed again in FP64.
template <class MT, int RB, int S>
struct NDRows {
    static constexpr int nv = 2 * RB >= S ? 2 * RB / S : 1, sh = 2 * RB >= S ? 0 : ilog2(S) - ilog2(2 * RB);
    const MT* a;                         // the row
    NDMat<MT> ax;                        // and split
    int64_t cs;
    int row, n, ea;
    bool ok, mine;
    NDItem<MT> pre[kNDAhead];
    __device__ __forceinline__ static int slice() { return threadIdx.x & (S - 1); }
    // value index (component q & 1 of right-hand side q >> 1) of this lane's i-th sum
    __device__ __forceinline__ static int value(int i) { return 2 * RB >= S ? slice() * nv + i : slice() >> sh; }
    __device__ __forceinline__ void ahead(const MT* A, const FxMat& Ax, int64_t rs, int64_t cs_, int n_, const int* aex, int row_,
                                          int end) {
        row = row_ + ((threadIdx.x & 31) / S);
        ok = row < end;
        mine = ok && (slice() & ((1 << sh) - 1)) == 0;
        a = A + (int64_t)(ok ? row : 0) * rs;
        cs = cs_;
        n = n_;
        ea = 0;
        if constexpr (kNDFixed<MT>) {
            ax = Ax.at((int64_t)(ok ? row : 0) * rs);
            if (ok) ea = aex[row];
        } else ax = a;
        nd_ahead<MT>(ax, cs, slice(), S, n, ok, pre);
    }
    template <class L, class F>
    __device__ __forceinline__ void run(int stride, char* sm, const int* ex, int nr, const double (&add)[nv], const L& load,
                                        const F& out) {
        NDSum<MT> v[2 * RB];
        long long low[2 * RB];
        nd_dot<MT, RB>(ax, cs, slice(), S, kNDFixed<MT> && n > kNDFixedRows ? 0 : n, ok, pre, stride,
                       NDStaged<MT, RB>(sm, stride), v, low);
        group_sum_transpose<NDSum<MT>, 2 * RB, S>(v);
        double val[nv];
        if constexpr (kNDFixed<MT>) {
            group_sum_transpose<long long, 2 * RB, S>(low);
            unsigned bad = 0;                              // bit i: value i is to be formed in FP64
#pragma unroll
            for (int i = 0; i < nv; ++i) {
                const int r = value(i) >> 1;
                val[i] = 0;
                if (mine && r < nr && !fx_value(v[i], low[i], ea, ex[r], val[i])) bad |= 1u << i;
            }
            if (__any_sync(0xffffffffu, bad != 0)) again(bad, nr, val, ex, NDStaged<MT, RB>(sm, stride).i, stride, load);
        } else {
#pragma unroll
            for (int i = 0; i < nv; ++i) val[i] = (double)v[i];
        }
        if (!mine) return;
#pragma unroll
        for (int i = 0; i < nv; ++i) {
            const int q = value(i), r = q >> 1;
            if (r < nr) out(row, r, q & 1, add[i] + val[i]);
        }
    }
    template <class L>
    __device__ __forceinline__ void again(unsigned bad, int nr, double (&val)[nv], const int* ex, const int4* xi, int stride,
                                          const L& load) {
#pragma unroll 1
        for (int r = 0; r < nr; ++r) {
            unsigned b = 0;
#pragma unroll
            for (int i = 0; i < nv; ++i)
                if ((bad >> i & 1) && (value(i) >> 1) == r) b |= 1u << (value(i) & 1);
            if (!__any_sync(0xffffffffu, b != 0)) continue;
            double2 d;
            const MT* a_ = a;
            const int4 *ai = ax.i, *xr = xi + r * stride;
            const int64_t cs_ = cs;
            b &= ~fx_again(S, b, n, ea, ex[r], [=](int j) { const MT u = a_[j * cs_]; return make_double2((double)u.x, (double)u.y); },
                           [=](int j) { const int4 u = ai[j * cs_]; return make_int2(u.x, u.z); }, [=](int j) { return xr[j]; },
                           [=](int j) { double2 x[RB]; load(j, x); return x[r]; }, d);
#pragma unroll
            for (int i = 0; i < nv; ++i)
                if ((value(i) >> 1) == r && (b >> (value(i) & 1) & 1) && (bad >> i & 1)) val[i] = value(i) & 1 ? d.y : d.x;
        }
    }
};

// Where rows [row0, row0 + nrows) of a front are worked on: by the warps of a CTA (32/S rows each at a
// time), or (WARP) by one warp alone.
// Forward: stage y_F = t_F - w_F (w = the children's amounts), write y_F when asked, then
// u_N[row] = w_B[row] + (G_N y_F)[row].  Ends without a trailing barrier.
template <class MT, int RB, int S, bool CG, bool WARP>
__device__ __forceinline__ void nd_forward_rows(const NDDev& d, int node, int row0, int nrows, bool write_y,
                                                const double2* __restrict__ t, double2* __restrict__ y,
                                                double2* __restrict__ u, int r0, int nr,
                                                char* nd_sm, int* ex, NDShared* sh) {
    using G = NDGroup<WARP>;
    const int f0 = d.f0[node], nF = d.nF[node], nB = d.nB[node], sF = nF | 1;
    const int64_t nc = d.nc, ul = d.u_len, so = d.s_off[node], uo = d.u_off[node];
    const bool cm = nF <= kNDShortRow;
    const MT* A = (const MT*)d.G + d.g_off[node];
    NDRows<MT, RB, S> R;
    double add[NDRows<MT, RB, S>::nv];
    auto begin = [&](int row) {
        R.ahead(A, d.gfx.at(d.g_off[node]), cm ? 1 : nF, cm ? nB : 1, nF, d.gexp + uo, row, row0 + nrows);
        const int64_t i = so + nF + (R.ok ? R.row : 0);
        const int64_t pa = R.mine ? d.src[2 * i] : -1, pb = R.mine ? d.src[2 * i + 1] : -1;
#pragma unroll
        for (int k = 0; k < R.nv; ++k) {
            const int q = R.value(k), r = q >> 1;
            add[k] = 0;
            if (r >= nr) continue;
            const double* ud = reinterpret_cast<const double*>(u + (r0 + r) * ul) + (q & 1);
            if (pa >= 0) add[k] += CG ? __ldcg(ud + 2 * pa) : ud[2 * pa];
            if (pb >= 0) add[k] += CG ? __ldcg(ud + 2 * pb) : ud[2 * pb];
        }
    };
    constexpr int per = 32 / S;
    int row = row0 + G::warp() * per;
    begin(row);
    const int64_t* src = d.src + 2 * so;
    const auto load = [=](int i, double2 (&v)[RB]) {
        const int64_t a = src[2 * i], b = src[2 * i + 1];
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            v[r] = make_double2(0.0, 0.0);
            if (r >= nr) continue;
            const double2 w = nd_pull<CG>(u, (r0 + r) * ul, a, b);
            v[r] = t[(r0 + r) * nc + f0 + i];
            v[r].x -= w.x; v[r].y -= w.y;
            if (write_y) y[(r0 + r) * nc + f0 + i] = v[r];
        }
    };
    nd_stage<MT, RB, WARP>(load, nF, sF, nd_sm, ex, sh);
    for (; row < row0 + nrows; row += per * G::warps()) {
        if (row != row0 + G::warp() * per) begin(row);
        R.run(sF, nd_sm, ex, nr, add, load, [&](int rw, int r, int c, double v) {
            reinterpret_cast<double*>(u + (r0 + r) * ul + uo + rw)[c] = v;
        });
    }
}

// Backward: x_F[rows] = ([W | -H] [y_F; x_B])[rows].  A node without a boundary has nothing to pass up,
// so it has no forward item when root is set: its y_F = t_F - w_F is formed here.
template <class MT, int RB, int S, bool CG, bool WARP>
__device__ __forceinline__ void nd_backward_rows(const NDDev& d, int node, int row0, int nrows, bool root,
                                                 const double2* __restrict__ t, const double2* __restrict__ u,
                                                 const double2* __restrict__ y, double2* __restrict__ x, int r0,
                                                 int nr, char* nd_sm, int* ex, NDShared* sh) {
    using G = NDGroup<WARP>;
    const int f0 = d.f0[node], nF = d.nF[node], nB = d.nB[node], n = nF + nB, sn = n | 1;
    const int64_t nc = d.nc, ul = d.u_len, so = d.s_off[node];
    const int* bi = d.bidx + d.b_off[node];
    const bool cm = n <= kNDShortRow;
    const MT* A = (const MT*)d.M + d.m_off[node];
    NDRows<MT, RB, S> R;
    double add[NDRows<MT, RB, S>::nv];
#pragma unroll
    for (int k = 0; k < R.nv; ++k) add[k] = 0;
    constexpr int per = 32 / S;
    int row = row0 + G::warp() * per;
    R.ahead(A, d.mfx.at(d.m_off[node]), cm ? 1 : n, cm ? nF : 1, n, d.mexp + f0, row, row0 + nrows);
    const int64_t* src = d.src + 2 * so;
    const auto load = [=](int i, double2 (&v)[RB]) {
        if (root) {
            const int64_t a = src[2 * i], b = src[2 * i + 1];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                v[r] = make_double2(0.0, 0.0);
                if (r >= nr) continue;
                const double2 w = nd_pull<CG>(u, (r0 + r) * ul, a, b);
                v[r] = t[(r0 + r) * nc + f0 + i];
                v[r].x -= w.x; v[r].y -= w.y;
            }
        } else {
            const int pos = i < nF ? f0 + i : bi[i - nF];
            const double2* from = i < nF ? y : x;
#pragma unroll
            for (int r = 0; r < RB; ++r) v[r] = r < nr ? ldv<CG>(from + (r0 + r) * nc + pos) : make_double2(0.0, 0.0);
        }
    };
    nd_stage<MT, RB, WARP>(load, n, sn, nd_sm, ex, sh);
    for (; row < row0 + nrows; row += per * G::warps()) {
        if (row != row0 + G::warp() * per) R.ahead(A, d.mfx.at(d.m_off[node]), cm ? 1 : n, cm ? nF : 1, n, d.mexp + f0, row, row0 + nrows);
        R.run(sn, nd_sm, ex, nr, add, load, [&](int rw, int r, int c, double v) {
            reinterpret_cast<double*>(x + (r0 + r) * nc + f0 + rw)[c] = v;
        });
    }
}

// The column slices of a level item: 32 (one warp per row) for a row-major matrix, 8 for a column-major
// one (long and short rows)
template <class MT, int RB, bool CG = false>
__device__ __forceinline__ void nd_forward_node(const NDDev& d, int node, int row0, int nrows, bool shortm,
                                                bool write_y, const double2* __restrict__ t, double2* __restrict__ y,
                                                double2* __restrict__ u, int r0, int nr,
                                                char* nd_sm, NDShared* sh) {
    if (shortm) nd_forward_rows<MT, RB, 8, CG, false>(d, node, row0, nrows, write_y, t, y, u, r0, nr, nd_sm, sh->ex, sh);
    else nd_forward_rows<MT, RB, 32, CG, false>(d, node, row0, nrows, write_y, t, y, u, r0, nr, nd_sm, sh->ex, sh);
}
template <class MT, int RB, bool CG = false>
__device__ __forceinline__ void nd_backward_node(const NDDev& d, int node, int row0, int nrows, bool shortm, bool root,
                                                 const double2* __restrict__ t, const double2* __restrict__ u,
                                                 const double2* __restrict__ y, double2* __restrict__ x, int r0,
                                                 int nr, char* nd_sm, NDShared* sh) {
    if (shortm) nd_backward_rows<MT, RB, 8, CG, false>(d, node, row0, nrows, root, t, u, y, x, r0, nr, nd_sm, sh->ex, sh);
    else nd_backward_rows<MT, RB, 32, CG, false>(d, node, row0, nrows, root, t, u, y, x, r0, nr, nd_sm, sh->ex, sh);
}

// Programmatic dependent launch between consecutive level launches: a CTA first waits until
// the previous launch in the stream has completed and its writes are visible (a no-op when
// this launch was not made dependent), then lets the next launch be scheduled, so that its
// CTAs are resident when this one ends.  No memory is touched before the wait.
__device__ __forceinline__ void nd_pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// forward level: one item per CTA
template <class MT, int RB>
__global__ void __launch_bounds__(kNDThreads) k_nd_forward(const __grid_constant__ NDDev d, const int4* __restrict__ items,
                                                    const double2* __restrict__ t, double2* __restrict__ y,
                                                    double2* __restrict__ u, int R, const int* __restrict__ done) {
    nd_pdl_enter();
    if (done && *done) return;
    extern __shared__ __align__(16) char nd_raw[];
    __shared__ NDShared sh;
    const int4 it = items[blockIdx.x];
    const int r0 = blockIdx.y * RB, nr = min(RB, R - r0);
    nd_forward_node<MT, RB>(d, it.x, it.y, it.z, it.w != 0, it.y == 0, t, y, u, r0, nr,
                            nd_raw, &sh);
}

// backward level: one item per CTA
template <class MT, int RB>
__global__ void __launch_bounds__(kNDThreads) k_nd_backward(const __grid_constant__ NDDev d, const int4* __restrict__ items, int root,
                                                     const double2* __restrict__ t, const double2* __restrict__ u,
                                                     const double2* __restrict__ y, double2* __restrict__ x, int R,
                                                     const int* __restrict__ done) {
    nd_pdl_enter();
    if (done && *done) return;
    extern __shared__ __align__(16) char nd_raw[];
    __shared__ NDShared sh;
    const int4 it = items[blockIdx.x];
    const int r0 = blockIdx.y * RB, nr = min(RB, R - r0);
    nd_backward_node<MT, RB>(d, it.x, it.y, it.z, it.w != 0, root != 0, t, u, y, x, r0, nr,
                             nd_raw, &sh);
}

// The bottom of the tree in one launch per direction: CTA b owns the subtree below a node of the cut
// level and walks its levels, deepest first (FWD) or last, with a barrier between levels.  Within a
// level each warp takes whole items by itself, so nothing but the level barrier couples the warps: the
// fronts here are small and many, and a launch per level is all latency.  Forward rows are short, and
// there are many of them: a lane per row (S = 1), no sum across lanes.  Backward rows are few and longer:
// 4 rows by 8 slices, or 16 by 2 where a level has rows enough for all warps (item.w: slices).
// 64 x 64 elements, l = 5, 8 right-hand sides: a coarse solve takes 533 us, 715 us with a launch per level.
template <class MT, int RB, bool FWD>
__global__ void __launch_bounds__(32 * kNDWarps) k_nd_bottom(const __grid_constant__ NDDev d, const int4* __restrict__ items,
                                                             const int* __restrict__ ptr, int nlev, int warp_len,
                                                             const double2* __restrict__ t, double2* __restrict__ y,
                                                             double2* __restrict__ x, double2* __restrict__ u, int R,
                                                             const int* __restrict__ done) {
    if (done && *done) return;
    extern __shared__ __align__(16) char nd_raw[];
    __shared__ int ex[kNDWarps][RB];
    const int warp = threadIdx.x >> 5;
    char* sm = nd_raw + nd_bytes<MT>(warp_len) * warp;
    const int r0 = blockIdx.y * RB, nr = min(RB, R - r0);
    const int* p = ptr + (size_t)blockIdx.x * nlev;
    for (int k = 0; k < nlev; ++k) {
        const int lv = FWD ? nlev - 1 - k : k;
        for (int i = p[lv] + warp; i < p[lv + 1]; i += kNDWarps) {
            const int4 it = items[i];
            __syncwarp();
            if (FWD) nd_forward_rows<MT, RB, 1, false, true>(d, it.x, it.y, it.z, it.y == 0, t, y, u, r0, nr, sm, ex[warp], nullptr);
            else if (it.w == 2) nd_backward_rows<MT, RB, 2, false, true>(d, it.x, it.y, it.z, false, t, u, y, x, r0, nr, sm, ex[warp], nullptr);
            else nd_backward_rows<MT, RB, 8, false, true>(d, it.x, it.y, it.z, false, t, u, y, x, r0, nr, sm, ex[warp], nullptr);
        }
        __syncthreads();
    }
}

// ---- the whole solve in one launch (see NDSched): items in dependency-safe ticket order
__device__ __forceinline__ int ld_acquire_gpu(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
// Bounded wait (one thread) until *cnt >= target.  Gives up when another CTA has aborted or
// after about a second, raising the abort flag; returns whether the dependency is met.
__device__ __forceinline__ bool nd_wait(const int* cnt, int target, int* abort_f) {
    if (target <= 0) return true;
    for (int it = 0; it < (1 << 21); ++it) {
        if (ld_acquire_gpu(cnt) >= target) return true;
        if (ld_acquire_gpu(abort_f)) return false;
        if (it > 32) __nanosleep(256);
    }
    atomicExch(abort_f, 1);
    return false;
}

template <class MT, int RB>
__global__ void __launch_bounds__(kNDThreads) k_nd_persistent(const __grid_constant__ NDDev d, NDSched sc, const double2* __restrict__ t,
                                                       double2* y, double2* x, double2* u, int R,
                                                       const int* __restrict__ done, int* err) {
    if (done && *done) return;
    extern __shared__ __align__(16) char nd_raw[];
    __shared__ int s_ticket, s_ok;
    __shared__ NDShared sh;
    const int nrb = (R + RB - 1) / RB;
    const int total = sc.nseq * nrb;
    int* ticket = sc.state;
    int* abort_f = sc.state + 1;
    int* fcnt = sc.state + 2;                       // [nn][nrb] finished forward items
    int* bcnt = fcnt + (size_t)sc.nn * nrb;         // [nn][nrb] finished backward items
    char* sm = nd_raw;
    while (true) {
        if (threadIdx.x == 0) s_ticket = atomicAdd(ticket, 1);
        __syncthreads();
        const int tk = s_ticket;
        if (tk >= total) return;
        const int4 it = sc.seq[tk / nrb];
        const int rb = tk % nrb, node = it.x;
        const bool bwd = (it.w & 2) != 0, shortm = (it.w & 1) != 0;
        if (threadIdx.x == 0) {
            bool ok = true;
            if (!bwd) {
                for (int c = 0; c < 2 && ok; ++c) {
                    const int k = sc.kid[2 * node + c];
                    if (k >= 0) ok = nd_wait(fcnt + (size_t)k * nrb + rb, sc.nfi[k], abort_f);
                }
            } else {
                ok = nd_wait(fcnt + (size_t)node * nrb + rb, sc.nfi[node], abort_f);
                const int a = sc.bdep[node];
                if (ok && a >= 0) ok = nd_wait(bcnt + (size_t)a * nrb + rb, sc.nbi[a], abort_f);
            }
            if (!ok && err) atomicExch(err, 3);
            __threadfence();
            s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) return;
        const int r0 = rb * RB, nr = min(RB, R - r0);
        if (!bwd) nd_forward_node<MT, RB, true>(d, node, it.y, it.z, shortm, it.y == 0, t, y, u, r0, nr, sm, &sh);
        else nd_backward_node<MT, RB, true>(d, node, it.y, it.z, shortm, false, t, u, y, x, r0, nr, sm, &sh);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd((bwd ? bcnt : fcnt) + (size_t)node * nrb + rb, 1);
        }
    }
}

// r = t - K x with K in CSR, one warp per row, lanes across the row's entries, RB right-hand sides per
// pass.  The residual cancels about eight digits of t, so its rounding is what the refined solve, and
// through it a whole FP64 solve, comes out with; here K x is the sum of ddh_fixed.cuh (K scaled by row once,
// x by the largest entry that the row meets) in two FP64 numbers, and t - K x is rounded once.
template <int RB>
__global__ void __launch_bounds__(128) k_csr_residual(const int* __restrict__ ptr, const int* __restrict__ col,
                                                      const double2* __restrict__ val, FxMat vx, const int* __restrict__ vex, int n,
                                                      const double2* __restrict__ x, const double2* __restrict__ t,
                                                      double2* __restrict__ r, int R, const int* __restrict__ done) {
    if (done && *done) return;
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, r0 = blockIdx.y * RB, nr = min(RB, R - r0);
    if (row >= n) return;
    const int a0 = ptr[row], a1 = ptr[row + 1];
    const double2* xr = x + (int64_t)r0 * n;
    int ex[RB];
#pragma unroll
    for (int q = 0; q < RB; ++q) ex[q] = 0;
    for (int a = a0 + lane; a < a1; a += 32) {
        const int c = col[a];
#pragma unroll
        for (int q = 0; q < RB; ++q)
            if (q < nr) ex[q] = max(ex[q], (int)fx_mag(xr[(int64_t)q * n + c]));
    }
#pragma unroll
    for (int q = 0; q < RB; ++q) ex[q] = fx_exp(__reduce_max_sync(0xffffffffu, (unsigned)ex[q]));
    const int ea = vex[row];
    FxSum s[RB];
    long long h[2 * RB], l[2 * RB];
#pragma unroll
    for (int i = 0; i < 2 * RB; ++i) h[i] = l[i] = 0;
#pragma unroll
    for (int q = 0; q < RB; ++q) fx_clear(s[q]);
    auto flush = [&] {
#pragma unroll
        for (int i = 0; i < 2 * RB; ++i) fx_flush(s[i >> 1], i & 1, h[i], l[i]);
#pragma unroll
        for (int q = 0; q < RB; ++q) fx_clear(s[q]);
    };
    for (int a = a0 + lane, c = 0; a < a1; a += 32) {
        const FxEntry v = fx_entry(vx.i[a], vx.f[a]);
        const double2* xc = xr + col[a];
#pragma unroll
        for (int q = 0; q < RB; ++q)
            if (q < nr) {
                const FxVec w = fx_vec(xc[(int64_t)q * n], ex[q]);
                fx_mac(s[q], v, w.i, w.f);
            }
        if (++c == kFxChain) {
            c = 0;
            flush();
        }
    }
    flush();
    const long long hs = warp_sum_transpose<long long, 2 * RB>(h), ls = warp_sum_transpose<long long, 2 * RB>(l);
    constexpr int sh = 5 - ilog2(2 * RB);
    const int k = lane >> sh, q = k >> 1;                  // component k & 1 of right-hand side q
    int e = 0;
#pragma unroll
    for (int i = 0; i < RB; ++i) e = i == q ? ex[i] : e;
    double hi = 0, lo = 0;
    const bool bad = q < nr && !fx_value2(hs, ls, ea, e, hi, lo);
    if (__any_sync(0xffffffffu, bad)) {
#pragma unroll 1
        for (int b = 0; b < nr; ++b) {
            const bool this_b = bad && q == b;
            if (!__any_sync(0xffffffffu, this_b)) continue;
            int eb = 0;
#pragma unroll
            for (int i = 0; i < RB; ++i) eb = i == b ? ex[i] : eb;
            const double2* v0 = val + a0;
            const int4* i0 = vx.i + a0;
            const auto xb = [=](int j) { return xr[(int64_t)b * n + col[a0 + j]]; };
            double2 d;
            const unsigned keep = fx_again(32, this_b ? 1u << (k & 1) : 0, a1 - a0, ea, eb, [=](int j) { return v0[j]; },
                                           [=](int j) { const int4 u = i0[j]; return make_int2(u.x, u.z); },
                                           [=](int j) { return fx_vec(xb(j), eb).i; }, xb, d);
            if (this_b && !(keep >> (k & 1) & 1)) { hi = k & 1 ? d.y : d.x; lo = 0; }
        }
    }
    if ((lane & ((1 << sh) - 1)) == 0 && q < nr) {
        const int64_t at = (int64_t)(r0 + q) * n + row;
        reinterpret_cast<double*>(r + at)[k & 1] = ((k & 1 ? t[at].y : t[at].x) - hi) - lo;
    }
}
// splits the rows of K; one warp per row
__global__ void k_fix_csr(const int* __restrict__ ptr, const double2* __restrict__ val, FxMat vx, int* __restrict__ ex, int n) {
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (row < n) fix_row(val + ptr[row], vx.at(ptr[row]), 1, ptr[row + 1] - ptr[row], ex + row);
}

// ------------------------------------------------------------------ launch wrappers
static constexpr int kNDSmemMax = 200 * 1024;
// bytes of RB staged vectors of up to `rows` entries
template <class MT>
static size_t nd_smem(int rows, int rb) {
    if (kNDFixed<MT>) rows = std::min(rows, kNDFixedRows);
    return std::max<size_t>(16, nd_bytes<MT>((size_t)(rows | 1) * rb));
}
int nd_rhs_block(int smem_rows, int R) {
    int rb = 4;
    while (rb > 1 && (rb >= 2 * R || nd_smem<double2>(smem_rows, rb) > (size_t)kNDSmemMax)) rb >>= 1;
    return rb;
}
template <class MT, int RB>
static void nd_attr() {
    raise_smem_limit(k_nd_forward<MT, RB>, kNDSmemMax);
    raise_smem_limit(k_nd_backward<MT, RB>, kNDSmemMax);
    raise_smem_limit(k_nd_bottom<MT, RB, true>, kNDSmemMax);
    raise_smem_limit(k_nd_bottom<MT, RB, false>, kNDSmemMax);
    raise_smem_limit(k_nd_persistent<MT, RB>, kNDSmemMax);
}
void nd_set_smem_limits() {
    nd_attr<double2, 1>(); nd_attr<double2, 2>(); nd_attr<double2, 4>();
    nd_attr<float2, 1>(); nd_attr<float2, 2>(); nd_attr<float2, 4>();
}
// launch with (pdl) or without the programmatic-stream-serialization attribute
template <typename... Exp, typename... Act>
static void nd_launch(void (*k)(Exp...), dim3 g, size_t sm, cudaStream_t st, bool pdl, Act&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = g;
    cfg.blockDim = dim3(kNDThreads);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    cudaLaunchKernelEx(&cfg, k, std::forward<Act>(args)...);
}
template <class MT, int RB>
static void nd_fwd_t(const NDDev& d, const int4* items, int nitems, int smem_rows, const double2* t, double2* y,
                     double2* u, int R, const int* done, cudaStream_t st, bool pdl) {
    const size_t sm = nd_smem<MT>(smem_rows, RB);
    nd_launch(k_nd_forward<MT, RB>, dim3(nitems, (R + RB - 1) / RB), sm, st, pdl, d, items, t, y, u, R, done);
}
template <class MT, int RB>
static void nd_bwd_t(const NDDev& d, const int4* items, int nitems, int smem_rows, int root, const double2* t,
                     const double2* u, const double2* y, double2* x, int R, const int* done, cudaStream_t st, bool pdl) {
    const size_t sm = nd_smem<MT>(smem_rows, RB);
    nd_launch(k_nd_backward<MT, RB>, dim3(nitems, (R + RB - 1) / RB), sm, st, pdl, d, items, root, t, u, y, x, R, done);
}
void launch_nd_forward(const NDDev& d, bool f32, const int4* items, int nitems, int smem_rows, const double2* t,
                       double2* y, double2* u, int R, const int* done, cudaStream_t st, int rb_want, bool pdl) {
    if (nitems <= 0) return;
    const int rb_max = nd_rhs_block(smem_rows, R);
    const int rb = rb_want > 0 && rb_want <= rb_max ? rb_want : rb_max;
#define ND_F(RBV)                                                                             \
    if (f32) nd_fwd_t<float2, RBV>(d, items, nitems, smem_rows, t, y, u, R, done, st, pdl);   \
    else nd_fwd_t<double2, RBV>(d, items, nitems, smem_rows, t, y, u, R, done, st, pdl);
    switch (rb) {
        case 4: ND_F(4) break;
        case 2: ND_F(2) break;
        default: ND_F(1)
    }
#undef ND_F
}
void launch_nd_backward(const NDDev& d, bool f32, const int4* items, int nitems, int smem_rows, int root,
                        const double2* t, const double2* u, const double2* y, double2* x, int R, const int* done,
                        cudaStream_t st, int rb_want, bool pdl) {
    if (nitems <= 0) return;
    const int rb_max = nd_rhs_block(smem_rows, R);
    const int rb = rb_want > 0 && rb_want <= rb_max ? rb_want : rb_max;
#define ND_B(RBV)                                                                          \
    if (f32) nd_bwd_t<float2, RBV>(d, items, nitems, smem_rows, root, t, u, y, x, R, done, st, pdl);   \
    else nd_bwd_t<double2, RBV>(d, items, nitems, smem_rows, root, t, u, y, x, R, done, st, pdl);
    switch (rb) {
        case 4: ND_B(4) break;
        case 2: ND_B(2) break;
        default: ND_B(1)
    }
#undef ND_B
}
// right-hand sides per CTA of the bottom launches: all warps' staged vectors fit
int nd_bottom_block(int rows, int R) {
    int rb = 4;
    while (rb > 1 && (rb >= 2 * R || nd_smem<double2>(rows, rb) * kNDWarps > (size_t)kNDSmemMax)) rb >>= 1;
    return nd_smem<double2>(rows, rb) * kNDWarps > (size_t)kNDSmemMax ? 0 : rb;
}
template <class MT, int RB>
static void nd_bottom_t(bool fwd, const NDDev& d, const NDBottom& b, const double2* t, double2* y, double2* x, double2* u,
                        int R, const int* done, cudaStream_t st) {
    const int len = RB * ((fwd ? b.fwd_rows : b.bwd_rows) | 1);
    const size_t sm = nd_bytes<MT>(len) * kNDWarps;
    const dim3 g(b.nsub, (R + RB - 1) / RB);
    if (fwd) k_nd_bottom<MT, RB, true><<<g, 32 * kNDWarps, sm, st>>>(d, b.fitems, b.fptr, b.nlev, len, t, y, x, u, R, done);
    else k_nd_bottom<MT, RB, false><<<g, 32 * kNDWarps, sm, st>>>(d, b.bitems, b.bptr, b.nlev, len, t, y, x, u, R, done);
}
void launch_nd_bottom(bool forward, const NDDev& d, bool f32, const NDBottom& b, const double2* t, double2* y, double2* x,
                      double2* u, int R, const int* done, cudaStream_t st, int rb_want) {
    if (b.nsub <= 0) return;
    const int rb_max = nd_bottom_block(forward ? b.fwd_rows : b.bwd_rows, R);
    const int rb = rb_want > 0 && rb_want <= rb_max ? rb_want : rb_max;
#define ND_S(RBV)                                                               \
    if (f32) nd_bottom_t<float2, RBV>(forward, d, b, t, y, x, u, R, done, st);  \
    else nd_bottom_t<double2, RBV>(forward, d, b, t, y, x, u, R, done, st);
    switch (rb) {
        case 4: ND_S(4) break;
        case 2: ND_S(2) break;
        default: ND_S(1)
    }
#undef ND_S
}
size_t nd_state_ints(const NDSched& s, int R) {
    const int rb = nd_rhs_block(s.smem_rows, R);
    return 2 + 2 * (size_t)s.nn * ((R + rb - 1) / rb);
}
template <class MT, int RB>
static void nd_persist_t(const NDDev& d, const NDSched& s, const double2* t, double2* y, double2* x, double2* u,
                         int R, const int* done, int* err, cudaStream_t st) {
    const size_t sm = nd_smem<MT>(s.smem_rows, RB);
    int dev = 0, nsm = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_nd_persistent<MT, RB>, kNDThreads, sm);
    const int nrb = (R + RB - 1) / RB;
    const int grid = std::max(1, std::min(std::max(1, per) * std::max(1, nsm), s.nseq * nrb));
    cudaMemsetAsync(s.state, 0, sizeof(int) * nd_state_ints(s, R), st);
    k_nd_persistent<MT, RB><<<grid, kNDThreads, sm, st>>>(d, s, t, y, x, u, R, done, err);
}
void launch_nd_persistent(const NDDev& d, const NDSched& s, bool f32, const double2* t, double2* y, double2* x,
                          double2* u, int R, const int* done, int* err, cudaStream_t st) {
    if (s.nseq <= 0) return;
    const int rb = nd_rhs_block(s.smem_rows, R);
#define ND_P(RBV)                                                                   \
    if (f32) nd_persist_t<float2, RBV>(d, s, t, y, x, u, R, done, err, st);         \
    else nd_persist_t<double2, RBV>(d, s, t, y, x, u, R, done, err, st);
    switch (rb) {
        case 4: ND_P(4) break;
        case 2: ND_P(2) break;
        default: ND_P(1)
    }
#undef ND_P
}
void launch_fix_csr(const int* ptr, const double2* val, const FxMat& vx, int* ex, int n, cudaStream_t st) {
    k_fix_csr<<<(n + 3) / 4, 128, 0, st>>>(ptr, val, vx, ex, n);
}
void launch_csr_residual(const int* ptr, const int* col, const double2* v, const FxMat& vx, const int* vex, int n,
                         const double2* x, const double2* t, double2* r, int R, const int* done, cudaStream_t st) {
    const int g = (n + 3) / 4;
    if (R >= 3) k_csr_residual<4><<<dim3(g, (R + 3) / 4), 128, 0, st>>>(ptr, col, v, vx, vex, n, x, t, r, R, done);
    else if (R == 2) k_csr_residual<2><<<dim3(g, 1), 128, 0, st>>>(ptr, col, v, vx, vex, n, x, t, r, R, done);
    else k_csr_residual<1><<<dim3(g, 1), 128, 0, st>>>(ptr, col, v, vx, vex, n, x, t, r, R, done);
}
int gemv_tiles(int n) { return (n + kGemvTile - 1) / kGemvTile; }
void launch_fix_dense(const double2* A, int n, longlong2* Ap, int* ex, cudaStream_t st) {
    k_fix_dense<<<(n + 3) / 4, 128, 0, st>>>(A, n, Ap, ex);
}
void launch_fix_fronts(const NDDev& d, int nodes, cudaStream_t st) {
    if (nodes > 0) k_fix_fronts<<<nodes, 256, 0, st>>>(d);
}
void launch_gemv32(const float2* a, int n, const double2* x, double2* y, int R, const int* done, cudaStream_t st) {
    const dim3 g((n + 3) / 4);
    // right-hand sides in chunks of 8, 4, 2, 1: every FMA issued does useful work
    for (int r0 = 0; r0 < R;) {
        const int left = R - r0;
        const int rb = left >= 8 ? 8 : (left >= 4 ? 4 : (left >= 2 ? 2 : 1));
#define DDH_GEMV(RBV) k_gemv<RBV><<<g, 128, 0, st>>>(a, n, x, y, r0, done);
        switch (rb) { case 8: DDH_GEMV(8) break; case 4: DDH_GEMV(4) break; case 2: DDH_GEMV(2) break; default: DDH_GEMV(1) }
#undef DDH_GEMV
        r0 += rb;
    }
}
// one CTA per SM, but at least four rows per CTA (each CTA stages all of x)
static int gemv_rows(int n, int nsm) { return std::max(4, (n + nsm - 1) / nsm); }
void gemv_set_smem_limits() {
    constexpr int most = 216 * 1024;          // eight staged tiles and the sums of the rows of n = 16384
    raise_smem_limit(k_gemv_fx<1>, most);
    raise_smem_limit(k_gemv_fx<2>, most);
    raise_smem_limit(k_gemv_fx<4>, most);
}
void launch_gemv(const double2* A, const longlong2* Ap, const int* ex, int n, const double2* x, double2* y, int R, const int* done, int nsm,
                 cudaStream_t st) {
    const int rpc = gemv_rows(n, nsm);
    const int g = (n + rpc - 1) / rpc;
    for (int r0 = 0; r0 < R;) {
        const int left = std::min(R - r0, 4);                  // a sum is twelve registers
        const int rb = left >= 3 ? 4 : left;
        const size_t sm = (size_t)rb * ((8 / rb * kGemvTile + 1) * (sizeof(int4) + sizeof(float4)) + (size_t)rpc * 2 * sizeof(double));
#define DDH_GEMV(RBV) k_gemv_fx<RBV><<<g, kGemvThreads, sm, st>>>(A, Ap, ex, n, x, y, r0, left, rpc, done);
        switch (rb) { case 4: DDH_GEMV(4) break; case 2: DDH_GEMV(2) break; default: DDH_GEMV(1) }
#undef DDH_GEMV
        r0 += left;
    }
}

}  // namespace ddh
