// Krylov-loop element passes with the explicit edge operators, the coarse assembly, the
// jump gather C^ x and the Dirichlet preconditioner (Sec. 2.3.3, eqs. complicated_schur_system,
// general_preconditioner, weight_matrix).
#include "ddh_fixed.cuh"
#include "ddh_kcommon.cuh"
#include <type_traits>

namespace ddh {

// ------------------------------------------------------------------ passes with explicit edge operators
// Inside the Krylov loop the element solves only ever map type-1 edge values to type-1 edge
// values and type-2 values (the jump operator touches nothing else), so with
//   Y = [A11^-1 A_1T]_E = S_E^-1 (A_ET - A_EX G A_XT)      (nE x nT, complex symmetric A)
// pass 1 is  x_E = S_E^-1 r_E,  t_T = Y^T r_E   (t_T = A_T1 A11^-1 [r_E; 0])
// pass 2 is  x1_E = x_E - Y u_T                 (x1 = y1 - A11^-1 A12 x2, edge part)
// -- two small dense products per element and right-hand side block instead of the FDM
// chain.  Y is formed at factor time.  The interior never enters the iteration; it is
// rebuilt by the FDM kernels in the recovery.
//
// The FP64 passes form their products on the integer and FP32 pipes (ddh_fixed.cuh) from the split S_E^-1 and
// Y.  S_E^-1 has an exponent per row (DevModel::sinv_ex, by type-1 slot), Y one per column (y_ex, by type-2
// slot), i.e. per output row of pass 1.  Pass 2, which sums over the columns, reads a copy of Y that is
// column-major, so that a warp's load is contiguous over the rows, with an exponent per row (y2_ex, by type-1
// slot).  In FP64 a staged vector is its limbs, its FP32 parts and, for results that are formed again in FP64,
// its entries.  64 x 64 elements, p = 20, 8 right-hand
// sides, pass 2: 0.13 ms, 0.30 ms in FP64.
template <class T> struct EdgeVec {
    cpx<T>* v;
    __device__ __forceinline__ EdgeVec(void* p, int) : v(reinterpret_cast<cpx<T>*>(p)) {}
};
template <> struct EdgeVec<double> {
    int4* i;
    float4* f;
    double2* d;
    __device__ __forceinline__ EdgeVec(void* p, int n)
        : i(reinterpret_cast<int4*>(p)), f(reinterpret_cast<float4*>(i + n)), d(reinterpret_cast<double2*>(f + n)) {}
};
// In FP64 a thread takes at most four of the RB right-hand sides of a CTA (a sum is twelve registers), and a
// CTA of eight has twice the threads.
template <class T, int RB> constexpr int kEdgeParts = std::is_same<T, double>::value && RB == 8 ? 2 : 1;

// Splits S_E^-1 and Y: one CTA per element, one warp per row of S_E^-1 / column of Y, then one per row of Y
__global__ void __launch_bounds__(256) k_fix_edge(DevModel dm, const double2* __restrict__ sinv,
                                                  const double2* __restrict__ Y, EdgeFix f) {
    const int e = blockIdx.x, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    const int nE = dm.nE1[e], nT = dm.nT[e];
    for (int o = warp; o < nE + nT; o += nw) {
        const bool isS = o < nE;
        const int ld = isS ? nE : nT;
        const int64_t at = isS ? dm.sinv_off[e] + o : dm.pq_off[e] + (o - nE);
        const double2* a = (isS ? sinv : Y) + at;
        const FxMat d = (isS ? f.s : f.y).at(at);
        unsigned m = 0;
        for (int j = lane; j < nE; j += 32) m = max(m, fx_mag(a[(int64_t)j * ld]));
        const int ef = fx_exp(__reduce_max_sync(0xffffffffu, m));
        for (int j = lane; j < nE; j += 32) fx_put(d, (int64_t)j * ld, a[(int64_t)j * ld], ef);
        if (lane == 0) *(isS ? f.sex + dm.e1_off[e] + o : f.yex + dm.t_off[e] + o - nE) = ef;
    }
    const double2* a = Y + dm.pq_off[e];
    const FxMat d = f.y2.at(dm.pq_off[e]);
    for (int i = warp; i < nE; i += nw) {
        unsigned m = 0;
        for (int t = lane; t < nT; t += 32) m = max(m, fx_mag(a[(int64_t)i * nT + t]));
        const int ef = fx_exp(__reduce_max_sync(0xffffffffu, m));
        for (int t = lane; t < nT; t += 32) fx_put(d, (int64_t)t * nE + i, a[(int64_t)i * nT + t], ef);
        if (lane == 0) f.y2ex[dm.e1_off[e] + i] = ef;
    }
}

// Stages cnt vectors of length n (stride vs): load(q, i) gives entry i of vector q.  In FP64 one warp per
// vector (n <= 128: four entries per lane), whose exponent goes to ex[q]; vectors cnt to RB - 1 are zero.
template <class T, int RB, class F>
__device__ __forceinline__ void edge_stage(const F& load, int n, int vs, int cnt, const EdgeVec<T>& sm, int* ex) {
    if constexpr (std::is_same<T, double>::value) {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
        for (int q = warp; q < RB; q += nw) {
            double2 v[4];
            unsigned m = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = lane + 32 * k;
                v[k] = make_double2(0.0, 0.0);
                if (i < n && q < cnt) { const cpx<double> c = load(q, i); v[k] = make_double2(c.x, c.y); }
                m = max(m, fx_mag(v[k]));
            }
            const int ef = fx_exp(__reduce_max_sync(0xffffffffu, m));
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (lane + 32 * k < n) {
                    const FxVec w = fx_vec(v[k], ef);
                    sm.i[q * vs + lane + 32 * k] = w.i;
                    sm.f[q * vs + lane + 32 * k] = w.f;
                    sm.d[q * vs + lane + 32 * k] = v[k];
                }
            if (lane == 0) ex[q] = ef;
        }
    } else {
        for (int idx = threadIdx.x; idx < cnt * n; idx += blockDim.x) sm.v[idx / n * vs + idx % n] = load(idx / n, idx % n);
    }
}

// [x_E; t_T] = [S_E^-1; Y^T] r_E for one element and RB right-hand sides: output row o < nE reads
// S_E^-1 (column-major), o >= nE reads Y (row-major nE x nT, i.e. Y^T column-major); tpr (2 or 4)
// threads per output row.  Every output is the same fixed tree (p0 + p2) + (p1 + p3) of the four
// partial sums p_k over the columns j = k (mod 4), each summed in increasing j, whatever tpr: with
// 4 threads a thread holds one p_k, with 2 it holds p_part and p_(part+2).  So the launch shapes
// the autotuner picks do not change the result.
// Output rows [o_lo, o_hi) only (x_E rows are o < nE, t_T rows o >= nE).
template <class T, int RB>
__device__ __forceinline__ void edge_rows_f(const DevModel& dm, const cpx<T>* S, const cpx<T>* Ye, int nE, int nT,
                                          const cpx<T>* rE, int vs, int cnt, int tpr, int r0, int e1o, int to,
                                          cpx<T>* __restrict__ xE_out, cpx<T>* __restrict__ tT_out, int o_lo,
                                          int o_hi) {
    const int no = o_hi;
    for (int base = 0; base < (o_hi - o_lo) * tpr; base += blockDim.x) {
        const int slot = base + threadIdx.x;
        const int o = o_lo + slot / tpr, part = slot % tpr;
        cpx<T> a0[RB], a1[RB];
#pragma unroll
        for (int q = 0; q < RB; ++q) { a0[q] = mk<T>(0, 0); a1[q] = mk<T>(0, 0); }
        if (o < no) {
            const cpx<T>* col0 = o < nE ? S + o : Ye + (o - nE);
            const int ld = o < nE ? nE : nT;
            if (tpr == 4) {
                for (int j = part; j < nE; j += 4) {
                    const cpx<T> s0 = col0[(int64_t)j * ld];
#pragma unroll
                    for (int q = 0; q < RB; ++q)
                        if (q < cnt) fma_c(a0[q], s0, rE[q * vs + j]);
                }
            } else {
                for (int j = part; j < nE; j += 4) {
                    const cpx<T> s0 = col0[(int64_t)j * ld];
#pragma unroll
                    for (int q = 0; q < RB; ++q)
                        if (q < cnt) fma_c(a0[q], s0, rE[q * vs + j]);
                    if (j + 2 < nE) {
                        const cpx<T> s1 = col0[(int64_t)(j + 2) * ld];
#pragma unroll
                        for (int q = 0; q < RB; ++q)
                            if (q < cnt) fma_c(a1[q], s1, rE[q * vs + j + 2]);
                    }
                }
            }
        }
#pragma unroll
        for (int q = 0; q < RB; ++q) {
            cpx<T> v = a0[q] + a1[q];
            if (tpr == 4) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, 2);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, 2);
            }
            v.x += __shfl_xor_sync(0xffffffffu, v.x, 1);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, 1);
            if (part == 0 && o < no && q < cnt) {
                if (o < nE) xE_out[(int64_t)(r0 + q) * dm.nE1_tot + e1o + o] = v;
                else tT_out[(int64_t)(r0 + q) * dm.nT_tot + to + (o - nE)] = v;
            }
        }
    }
}

// The same with the products of ddh_fixed.cuh.  Two or four threads per output row by the row count alone
// (edge_tpr), so that the order of a row's terms does not depend on the launch form.  Integer multiply-adds bound it (22 per SM
// and clock, twelve a term): 64 x 64 elements, p = 20, 8 right-hand sides 0.48 ms, 1.09 ms in FP64; at two
// CTAs of ten warps per SM, 96 registers a thread.
template <class T>
__device__ __forceinline__ int edge_tpr(int rows, int other) {
    return std::is_same<T, double>::value ? (rows <= 64 ? 4 : 2) : other;
}
template <int RB>
__device__ __forceinline__ void edge_rows_fx(const DevModel& dm, const FxMat& S, const FxMat& Ye, const double2* S64,
                                             const double2* Y64, int nE, int nT,
                                             const EdgeVec<double>& rE, const int* ex, int vs, int cnt, int tpr, int r0, int e1o, int to, cpx<double>* __restrict__ xE_out,
                                             cpx<double>* __restrict__ tT_out, int o_lo, int o_hi, int tid, int nt, int q0) {
    for (int base = 0; base < (o_hi - o_lo) * tpr; base += nt) {
        const int slot = base + tid;
        const int o = o_lo + slot / tpr, part = slot % tpr;
        const bool in = o < o_hi;
        const FxMat col0 = !in || o < nE ? S.at(in ? o : 0) : Ye.at(o - nE);
        const int64_t ld = o < nE ? nE : nT;
        const int ea = !in ? 0 : (o < nE ? dm.sinv_ex[e1o + o] : dm.y_ex[to + o - nE]);
        FxSum s[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i) fx_clear(s[i]);
        if (in) {
            // nE <= 124 terms: one chain; the next entry's load is issued ahead
            auto run = [&](auto all) {
                int4 ni = make_int4(0, 0, 0, 0);
                float2 nf = make_float2(0.f, 0.f);
                if (part < nE) { ni = col0.i[part * ld]; nf = col0.f[part * ld]; }
#pragma unroll(RB <= 2 ? 4 : 1)
                for (int j = part; j < nE; j += tpr) {
                    const FxEntry a = fx_entry(ni, nf);
                    if (j + tpr < nE) { ni = col0.i[(j + tpr) * ld]; nf = col0.f[(j + tpr) * ld]; }
#pragma unroll
                    for (int q = 0; q < RB; ++q)
                        if (decltype(all)::value || q0 + q < cnt) fx_mac(s[q], a, rE.i[(q0 + q) * vs + j], rE.f[(q0 + q) * vs + j]);
                }
            };
            // a block that is not full skips what it has not (thirteen right-hand sides: three of sixteen)
            if (RB < 4 || q0 + RB <= cnt) run(std::true_type());
            else run(std::false_type());
        }
#pragma unroll
        for (int q = 0; q < RB; ++q) {
            bool bad = false;
            double v = 0;
            // the lanes of a row share the conversions: component c of vector q goes to lane part = 2 q + c (mod tpr)
            const bool mine = in && q0 + q < cnt && (part & ~1) == ((2 * q) & (tpr - 1));
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                long long h = 0, l = 0;
                fx_flush(s[q], c, h, l);
                if (tpr == 4) {
                    h += __shfl_xor_sync(0xffffffffu, h, 2);
                    l += __shfl_xor_sync(0xffffffffu, l, 2);
                }
                h += __shfl_xor_sync(0xffffffffu, h, 1);
                l += __shfl_xor_sync(0xffffffffu, l, 1);
                if (mine && (part & 1) == c) bad = !fx_value(h, l, ea, ex[q0 + q], v);
            }
            if (__any_sync(0xffffffffu, bad)) {
                double2 d;
                const double2* c64 = !in || o < nE ? S64 + (in ? o : 0) : Y64 + (o - nE);
                const int4 *ci = col0.i, *xi = rE.i + (q0 + q) * vs;
                const double2* xd = rE.d + (q0 + q) * vs;
                const unsigned keep = fx_again(tpr, bad ? 1u << (part & 1) : 0, nE, ea, ex[q0 + q],
                                               [=](int j) { return c64[j * ld]; },
                                               [=](int j) { const int4 u = ci[j * ld]; return make_int2(u.x, u.z); },
                                               [=](int j) { return xi[j]; }, [=](int j) { return xd[j]; }, d);
                if (bad && !(keep >> (part & 1) & 1)) v = part & 1 ? d.y : d.x;
            }
            if (mine) {
                cpx<double>* d = o < nE ? xE_out + (int64_t)(r0 + q0 + q) * dm.nE1_tot + e1o + o
                                        : tT_out + (int64_t)(r0 + q0 + q) * dm.nT_tot + to + (o - nE);
                reinterpret_cast<double*>(d)[part & 1] = v;
            }
        }
    }
}
// S: S_E^-1, staged or not; in FP64 S, Ye point at the complex128 matrices and Sx at the split S_E^-1
template <class T, int RB>
__device__ __forceinline__ void edge_rows(const DevModel& dm, int e, const cpx<T>* S, const FxMat& Sx, const cpx<T>* Ye, int nE,
                                          int nT, const EdgeVec<T>& rE, const int* ex, int vs, int cnt, int tpr,
                                          int r0, int e1o, int to, cpx<T>* __restrict__ xE_out,
                                          cpx<T>* __restrict__ tT_out, int o_lo, int o_hi) {
    if constexpr (std::is_same<T, double>::value) {
        constexpr int parts = kEdgeParts<T, RB>;
        const int nt = blockDim.x / parts, part = threadIdx.x / nt;
        edge_rows_fx<RB / parts>(dm, Sx, dm.y_fx.at(dm.pq_off[e]), reinterpret_cast<const double2*>(S),
                                 reinterpret_cast<const double2*>(Ye), nE, nT, rE, ex, vs, cnt, tpr, r0, e1o, to, xE_out,
                                 tT_out, o_lo, o_hi, threadIdx.x - part * nt, nt, part * (RB / parts));
    } else edge_rows_f<T, RB>(dm, S, Ye, nE, nT, rE.v, vs, cnt, tpr, r0, e1o, to, xE_out, tT_out, o_lo, o_hi);
}

__device__ __forceinline__ void bulk_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint64_t* bar, void* dst, const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// Staging of S_E^-1 by a bulk copy: in FP64 its limbs; the fractions are read where they lie, so that two CTAs fit
// on an SM up to n_E = 72 (n_E = 64, 8 right-hand sides: 220 us, 366 us with both staged and one CTA)
template <class T>
__device__ __forceinline__ void edge_copy(uint64_t* bar, char* dst, const DevModel& dm, const cpx<T>* sinv, int e, int nE) {
    const size_t n = (size_t)nE * nE;
    const int64_t off = dm.sinv_off[e];
    if constexpr (std::is_same<T, double>::value) {
        const uint32_t b0 = (uint32_t)(n * sizeof(int4));
        bulk_expect(bar, b0);
        bulk_copy(bar, dst, dm.sinv_fx.i + off, b0);
    } else {
        const uint32_t b = (uint32_t)(n * sizeof(cpx<T>) + 15) & ~15u;
        bulk_expect(bar, b);
        bulk_copy(bar, dst, sinv + off, b);
    }
}

// entry i of r_E of right-hand side r0 + q
template <class T>
__device__ __forceinline__ auto pass1_load(const DevModel& dm, const double2* z, double zsign, const double2* bt, int r0,
                                           int e1o, int64_t off) {
    return [dp = &dm, z, zsign, bt, r0, e1o, off](int q, int i) {
        const int r = r0 + q;
        cpx<T> v = mk<T>(0, 0);
        const int row = dp->e1_row[e1o + i];
        if (z && row >= 0) v = (T)(zsign * dp->e1_sign[e1o + i]) * ld<T>(z, (int64_t)r * dp->n_dual + row);
        if (bt) v += ld<T>(bt, (int64_t)r * dp->n_local + off + dp->e1_slot[e1o + i]);
        return v;
    };
}
// the staged matrix: S in complex64, Sx in FP64
template <class T>
__device__ __forceinline__ void edge_staged(char* sm, int nE, const cpx<T>*& S, FxMat& Sx) {
    if constexpr (std::is_same<T, double>::value)
        Sx.i = reinterpret_cast<int4*>(sm);
    else S = reinterpret_cast<const cpx<T>*>(sm);
}

template <class T, int RB>
__global__ void __launch_bounds__(kEdgeParts<T, RB> == 2 ? 640 : 256) k_pass1_edge(const __grid_constant__ DevModel dm, const cpx<T>* __restrict__ sinv,
                                                    const cpx<T>* __restrict__ Y, const double2* __restrict__ z,
                                                    double zsign, const double2* __restrict__ bt, int R,
                                                    cpx<T>* __restrict__ xE_out, cpx<T>* __restrict__ tT_out,
                                                    const int* __restrict__ done, int ntask, int stage_off, int vs,
                                                    int rows) {
    if (done && *done) return;
    extern __shared__ __align__(128) char smem[];
    const CtaGroup g;
    const int task = blockIdx.x;
    if (task >= ntask) return;
    const int e = task % dm.E, r0 = (task / dm.E) * RB;
    const int cnt = min(RB, R - r0);
    const int nE = dm.nE1[e], e1o = dm.e1_off[e], nT = dm.nT[e], to = dm.t_off[e];
    const cpx<T>* S = sinv + dm.sinv_off[e];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + stage_off);
    char* S_s = smem + stage_off + 128;
    if (stage_off > 0 && nE > 0 && threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        edge_copy<T>(bar, S_s, dm, sinv, e, nE);
    }
    FxMat Sx = dm.sinv_fx.at(dm.sinv_off[e]);
    const EdgeVec<T> rE(smem, RB * vs);               // [RB][vs]
    __shared__ int ex[RB];
    const int64_t off = dm.off[e];
    const auto load = pass1_load<T>(dm, z, zsign, bt, r0, e1o, off);
    edge_stage<T, RB>(load, nE, vs, cnt, rE, ex);
    g.sync();
    if (stage_off > 0 && nE > 0) {
        if (!bulk_wait_all(bar, dm.err)) return;
        edge_staged<T>(S_s, nE, S, Sx);
    }
    // every vertex and edge slot is type-1 edge or type-2, so nE + nT = 4p <= 128 (p <= 32): four
    // threads per output row when all rows fit the CTA so, else two
    const int tpr = edge_tpr<T>(nE + nT, (nE + nT) * 4 <= (int)blockDim.x ? 4 : 2);
    // rows: 0 all output rows, 1 the x_E rows only, 2 the t_T rows only (no S_E^-1 read)
    const int o_lo = rows == 2 ? nE : 0, o_hi = rows == 1 ? nE : nE + nT;
    edge_rows<T, RB>(dm, e, S, Sx, Y + dm.pq_off[e], nE, nT, rE, ex, vs, cnt, tpr, r0, e1o, to, xE_out, tT_out, o_lo, o_hi);
}

// The same pass as one persistent launch over a degree-sorted work list.  Task t is (element
// items[item0 + t / nrb], right-hand-side block t % nrb): the heaviest elements come first, and
// the blocks of one element are adjacent, so its S_E^-1 is reused from L2.  A CTA walks tasks
// t = blockIdx.x, blockIdx.x + gridDim.x, ...; while it computes one task, the next task's
// S_E^-1 is already being copied into the other of two shared-memory buffers (bulk copy,
// mbarrier per buffer).  tpr_p[p] (2 or 4 threads per output row) is chosen per degree by the
// autotuner; 0 = the default (4 up to 64 output rows, else 2); tpr_force (2 or 4) overrides it.  FP64 always
// takes the default (edge_tpr).
template <class T, int RB>
__global__ void __launch_bounds__(kEdgeParts<T, RB> == 2 ? 640 : 256) k_pass1_edge_p(const __grid_constant__ DevModel dm, const cpx<T>* __restrict__ sinv,
                                                      const cpx<T>* __restrict__ Y, const double2* __restrict__ z,
                                                      double zsign, const double2* __restrict__ bt, int R,
                                                      cpx<T>* __restrict__ xE_out, cpx<T>* __restrict__ tT_out,
                                                      const int* __restrict__ done, const int* __restrict__ items,
                                                      int item0, int nitems, const signed char* __restrict__ tpr_p,
                                                      int tpr_force, int stage_off, int buf_bytes, int vs) {
    if (done && *done) return;
    extern __shared__ __align__(128) char smem[];
    const int nrb = (R + RB - 1) / RB, ntask = nitems * nrb;
    const EdgeVec<T> rE(smem, RB * vs);               // [RB][vs]
    __shared__ int ex[RB];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + stage_off);        // 2 barriers
    __shared__ int s_fail;
    const bool staged = stage_off > 0;
    auto buf = [&](int b) { return smem + stage_off + 128 + (size_t)b * buf_bytes; };
    auto task_elem = [&](int t) { return items[item0 + t / nrb]; };
    // copy of task t's S_E^-1 into buffer b (thread 0); false when there is nothing to copy
    auto issue = [&](int t, int b) {
        const int e = task_elem(t), nE = dm.nE1[e];
        if (nE == 0) return false;
        edge_copy<T>(bar + b, buf(b), dm, sinv, e, nE);
        return true;
    };
    bool pend[2] = {false, false};        // thread 0: copy in flight per buffer
    uint32_t uses[2] = {0, 0};            // completed phases per buffer
    if (threadIdx.x == 0) {
        s_fail = 0;
        if (staged) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar + 1)) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            if (blockIdx.x < ntask) pend[0] = issue(blockIdx.x, 0);
        }
    }
    __syncthreads();
    int k = 0;
    for (int t = blockIdx.x; t < ntask; t += gridDim.x, ++k) {
        const int b = k & 1;
        const int e = task_elem(t), r0 = (t % nrb) * RB;
        const int cnt = min(RB, R - r0);
        const int nE = dm.nE1[e], e1o = dm.e1_off[e], nT = dm.nT[e], to = dm.t_off[e];
        if (staged && threadIdx.x == 0 && t + (int)gridDim.x < ntask) pend[b ^ 1] = issue(t + gridDim.x, b ^ 1);
        const int64_t off = dm.off[e];
        const auto load = pass1_load<T>(dm, z, zsign, bt, r0, e1o, off);
        edge_stage<T, RB>(load, nE, vs, cnt, rE, ex);
        const cpx<T>* S = sinv + dm.sinv_off[e];
        FxMat Sx = dm.sinv_fx.at(dm.sinv_off[e]);
        if (staged && nE > 0) {
            if (threadIdx.x == 0) {
                bool ok = !pend[b];
                for (int it = 0; it < (1 << 22) && !ok; ++it) ok = mbar_try_wait(bar + b, uses[b] & 1);
                if (pend[b]) { pend[b] = false; ++uses[b]; }
                if (!ok) { s_fail = 1; if (dm.err) atomicExch(dm.err, 2); }
            }
            edge_staged<T>(buf(b), nE, S, Sx);
        }
        __syncthreads();
        if (s_fail) break;
        int tpr = tpr_force > 0 ? tpr_force : (tpr_p ? (int)tpr_p[dm.p[e]] : 0);
        if (tpr != 2 && tpr != 4) tpr = nE + nT <= 64 ? 4 : 2;
        tpr = edge_tpr<T>(nE + nT, tpr);
        edge_rows<T, RB>(dm, e, S, Sx, Y + dm.pq_off[e], nE, nT, rE, ex, vs, cnt, tpr, r0, e1o, to, xE_out, tT_out, 0,
                         nE + nT);
        __syncthreads();
    }
    // copies still in flight (after a failure) land before the CTA leaves (bounded waits)
    if (threadIdx.x == 0)
        for (int bb = 0; bb < 2; ++bb)
            if (pend[bb]) {
                bool ok = false;
                for (int it = 0; it < (1 << 22) && !ok; ++it) ok = mbar_try_wait(bar + bb, uses[bb] & 1);
            }
}

template <class T, int RB>
__global__ void __launch_bounds__(128 * kEdgeParts<T, RB>) k_pass2_edge(const __grid_constant__ DevModel dm, const cpx<T>* __restrict__ Y,
                                                    const double2* __restrict__ x2, const cpx<T>* __restrict__ xE_in,
                                                    cpx<T>* __restrict__ xE_out, int R, const int* __restrict__ done,
                                                    int ntask, int vs, int y_off, int y_staged) {
    if (done && *done) return;
    constexpr bool fx = std::is_same<T, double>::value;
    __shared__ int ex[RB];
    extern __shared__ __align__(128) char smem[];
    const CtaGroup g;
    const int task = blockIdx.x;
    if (task >= ntask) return;
    const int e = task % dm.E, r0 = (task / dm.E) * RB;
    const int cnt = min(RB, R - r0);
    const int nE = dm.nE1[e], e1o = dm.e1_off[e], nT = dm.nT[e], to = dm.t_off[e];
    // FP64: the split Y comes into shared memory (in flight while u_T is gathered); a bulk copy starts at a
    // multiple of 16 bytes, so the fractions of an element at an odd offset are read where they lie
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem + y_off);
    char* Y_s = smem + y_off + 128;
    const bool staged = y_staged && nE > 0 && nT > 0;
    FxMat Yx = dm.y2_fx.at(dm.pq_off[e]);
    if constexpr (fx)
        if (staged) {
            const bool even = (dm.pq_off[e] & 1) == 0;
            const uint32_t b0 = nE * nT * (uint32_t)sizeof(int4), b1 = even ? (nE * nT * (uint32_t)sizeof(float2) + 15) & ~15u : 0;
            if (threadIdx.x == 0) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                bulk_expect(bar, b0 + b1);
                bulk_copy(bar, Y_s, Yx.i, b0);
                if (b1) bulk_copy(bar, Y_s + b0, Yx.f, b1);
            }
            Yx.i = reinterpret_cast<int4*>(Y_s);
            if (b1) Yx.f = reinterpret_cast<float2*>(Y_s + b0);
        }
    const EdgeVec<T> uT(smem, RB * vs);
    const auto load = [dp = &dm, x2, to, r0](int q, int i) {
        const int r = r0 + q;
        cpx<T> u = mk<T>(0, 0);
        for (int a = dp->t_ptr[to + i]; a < dp->t_ptr[to + i + 1]; ++a) {
            const double2 xv = x2[(int64_t)r * dp->n_coarse + dp->t_col[a]];
            const T w = (T)dp->t_w[a];
            u.x += w * (T)xv.x;
            u.y += w * (T)xv.y;
        }
        return u;
    };
    edge_stage<T, RB>(load, nT, vs, cnt, uT, ex);
    g.sync();
    if (staged && !bulk_wait_all(bar, dm.err)) return;
    // one thread per row i of Y, all RB right-hand sides at once: each Y entry is read once
    const cpx<T>* Ye = Y + dm.pq_off[e];
    constexpr int parts = kEdgeParts<T, RB>, RT = RB / parts;
    const int nt = blockDim.x / parts, q0 = threadIdx.x / nt * RT;
    for (int i = threadIdx.x % nt; i < nE; i += nt) {
        const cpx<T>* yr = Ye + (int64_t)i * nT;
        cpx<T> a[RT];
        if constexpr (fx) {
            const double2* yd = reinterpret_cast<const double2*>(yr);
            const int ea = dm.y2_ex[e1o + i];
            FxSum s[RT];
#pragma unroll
            for (int q = 0; q < RT; ++q) fx_clear(s[q]);
            // nT <= 128 terms: one chain; the next entry's load is issued ahead
            int4 ni = make_int4(0, 0, 0, 0);
            float2 nf = make_float2(0.f, 0.f);
            if (nT > 0) { ni = Yx.i[i]; nf = Yx.f[i]; }
#pragma unroll(RT <= 2 ? 4 : 2)
            for (int t = 0; t < nT; ++t) {
                const FxEntry y = fx_entry(ni, nf);
                if (t + 1 < nT) { ni = Yx.i[(t + 1) * nE + i]; nf = Yx.f[(t + 1) * nE + i]; }
#pragma unroll
                for (int q = 0; q < RT; ++q) fx_mac(s[q], y, uT.i[(q0 + q) * vs + t], uT.f[(q0 + q) * vs + t]);
            }
#pragma unroll
            for (int q = 0; q < RT; ++q) {
                a[q] = mk<T>(0, 0);
                if (q0 + q >= cnt) continue;
                unsigned bad = 0;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    long long h = 0, l = 0;
                    fx_flush(s[q], c, h, l);
                    if (!fx_value(h, l, ea, ex[q0 + q], c ? a[q].y : a[q].x)) bad |= 1u << c;
                }
                if (bad) {
                    double2 d;
                    const int4 *yi = Yx.i + i, *xi = uT.i + (q0 + q) * vs;
                    const double2* xd = uT.d + (q0 + q) * vs;
                    bad &= ~fx_again(1, bad, nT, ea, ex[q0 + q], [=](int t) { return yd[t]; },
                                     [=](int t) { const int4 u = yi[t * nE]; return make_int2(u.x, u.z); },
                                     [=](int t) { return xi[t]; }, [=](int t) { return xd[t]; }, d);
                    if (bad & 1) a[q].x = d.x;
                    if (bad & 2) a[q].y = d.y;
                }
            }
        } else {
#pragma unroll
            for (int q = 0; q < RT; ++q) a[q] = mk<T>(0, 0);
            for (int t = 0; t < nT; ++t) {
                const cpx<T> y = yr[t];
#pragma unroll
                for (int q = 0; q < RT; ++q)
                    if (q < cnt) fma_c(a[q], y, uT.v[q * vs + t]);
            }
        }
#pragma unroll
        for (int q = 0; q < RT; ++q)
            if (q0 + q < cnt) {
                const int64_t gi = (int64_t)(r0 + q0 + q) * dm.nE1_tot + e1o + i;
                xE_out[gi] = xE_in[gi] - a[q];
            }
    }
}

// ------------------------------------------------------------------ coarse assembly
// t[g] = bsign * (Z2^T b_T)[g] + zsign * (C2^T z)[g] - (Z2^T tT)[g]   (FP64 output)
template <class T>
__global__ void k_coarse_assemble(DevModel dm, const cpx<T>* __restrict__ tT, const double2* __restrict__ bt,
                                  const double2* __restrict__ z, double zsign, double2* __restrict__ tout,
                                  int R, const int* __restrict__ done) {
    if (done && *done) return;
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (g >= dm.n_coarse) return;
    double2 acc = make_double2(0, 0);
    for (int a = dm.g_ptr[g]; a < dm.g_ptr[g + 1]; ++a) {
        const int ts = dm.g_tslot[a];
        const double w = dm.g_w[a];
        const cpx<T> v = tT[(int64_t)r * dm.nT_tot + ts];
        acc.x -= w * (double)v.x;
        acc.y -= w * (double)v.y;
        if (bt) {
            const int e = dm.t_elem[ts];
            const double2 b = bt[(int64_t)r * dm.n_local + dm.off[e] + dm.t_slot[ts]];
            acc.x += w * b.x;
            acc.y += w * b.y;
        }
    }
    if (z)
        for (int a = dm.c2t_ptr[g]; a < dm.c2t_ptr[g + 1]; ++a) {
            const double w = zsign * dm.c2t_w[a];
            const double2 v = z[(int64_t)r * dm.n_dual + dm.c2t_row[a]];
            acc.x += w * v.x;
            acc.y += w * v.y;
        }
    tout[(int64_t)r * dm.n_coarse + g] = acc;
}

// ------------------------------------------------------------------ jump gather (C^ x)
// w[row] = x1_E[c] - x1_E[f] + sum_k C2[row][k] x2[k] (c absent on hanging rows, f on the
// single-sided rows of a Dirichlet side)
template <class T>
__global__ void k_jump_gather(DevModel dm, const cpx<T>* __restrict__ xE, const double2* __restrict__ x2,
                              double2* __restrict__ w, const int* __restrict__ done) {
    if (done && *done) return;
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (row >= dm.n_dual) return;
    double sx = 0, sy = 0;
    const int c = dm.row_c[row], f = dm.row_f[row];
    if (c >= 0) { const cpx<T> v = xE[(int64_t)r * dm.nE1_tot + c]; sx += (double)v.x; sy += (double)v.y; }
    if (f >= 0) { const cpx<T> v = xE[(int64_t)r * dm.nE1_tot + f]; sx -= (double)v.x; sy -= (double)v.y; }
    for (int a = dm.c2_ptr[row]; a < dm.c2_ptr[row + 1]; ++a) {
        const double2 v = x2[(int64_t)r * dm.n_coarse + dm.c2_col[a]];
        sx += dm.c2_w[a] * v.x;
        sy += dm.c2_w[a] * v.y;
    }
    w[(int64_t)r * dm.n_dual + row] = make_double2(sx, sy);
}

// ------------------------------------------------------------------ preconditioner
// y = D^-1 x, D = C1_E C1_E^T + C2 C2^T: 1/2 on conforming rows, dense blocks on hanging edges;
// in the Poisson mode D = C1 W C1^T (diagonal, one weight per row)
__global__ void k_dinv(DevModel dm, const double2* __restrict__ x, double2* __restrict__ y,
                       const int* __restrict__ done) {
    if (done && *done) return;
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (row >= dm.n_dual) return;
    const int64_t ro = (int64_t)r * dm.n_dual;
    if (dm.row_dinv) {
        const double2 v = x[ro + row];
        const double w = dm.row_dinv[row];
        y[ro + row] = make_double2(w * v.x, w * v.y);
        return;
    }
    const int hb = dm.row_hb[row];
    if (hb < 0) {
        const double2 v = x[ro + row];
        y[ro + row] = make_double2(0.5 * v.x, 0.5 * v.y);
        return;
    }
    const int r0 = dm.hb_row0[hb], nr = dm.hb_n[hb];
    const double* Di = dm.hb_Dinv + dm.hb_off[hb] + (int64_t)(row - r0) * nr;
    double sx = 0, sy = 0;
    for (int j = 0; j < nr; ++j) {
        const double2 v = x[ro + r0 + j];
        sx += Di[j] * v.x;
        sy += Di[j] * v.y;
    }
    y[ro + row] = make_double2(sx, sy);
}

// out_E = S^Lap[E1][E1] (C1^T v) per element (stiffness Schur complement, shared per degree);
// one CTA per (element, block of RB RHS), each S^Lap entry read once per CTA.
// out_E = S x for the restricted stiffness Schur complement S (n_E x n_E, symmetric, read from
// global memory column by column: coalesced across output rows, shared by the elements of a
// degree pattern and L1/L2-resident); tpr adjacent threads share an output row.  FP64: the products of
// ddh_fixed.cuh, exponents pre_ex by row (an application as below 0.28 ms, 0.52 ms in FP64).  At
// most 80 registers a thread: 24 warps per SM instead of 16 (230 -> 228 us here, 73.9 -> 67.7 us at 40 x 40, p = 12).
template <class T, int RB>
__device__ __forceinline__ void pre_apply(const DevModel& dm, int e, int nE, int cnt, const EdgeVec<T>& in, const int* ex,
                                          cpx<T>* __restrict__ out, int64_t ostride,
                                          const double* __restrict__ wout = nullptr) {
    const int tpr = nE <= 32 ? 4 : (nE <= 64 ? 2 : 1);
    const int chunk = (nE + tpr - 1) / tpr;
    const double* S = dm.pre_all + dm.pre_off[e];
    const FxRealMat Sx = dm.pre_fx.at(dm.pre_off[e]);
    constexpr int parts = kEdgeParts<T, RB>, RT = RB / parts;
    const int nt = blockDim.x / parts, q0 = threadIdx.x / nt * RT;
    for (int base = 0; base < nE * tpr; base += nt) {
        const int slot = base + threadIdx.x % nt;
        const int i = slot / tpr, part = slot % tpr;
        const int j1 = i < nE ? min(nE, (part + 1) * chunk) : 0;
        if constexpr (std::is_same<T, double>::value) {
            const int ea = i < nE ? dm.pre_ex[dm.pre_ex_off[e] + i] : 0;
            FxSum s[RT];
#pragma unroll
            for (int k = 0; k < RT; ++k) fx_clear(s[k]);
            // nE <= 124 terms: one chain, loads of the next entries ahead (few right-hand sides: eight, the
            // latency bounds it; 16 x 16 elements, p = 16, one right-hand side)
            constexpr int ahead = RT <= 2 ? 8 : 2;
            int2 ni[ahead];
            float nf[ahead];
            auto fetch = [&](int k, int j) {
                ni[k] = j < j1 ? __ldg(Sx.i + j * nE + i) : make_int2(0, 0);
                nf[k] = j < j1 ? __ldg(Sx.f + j * nE + i) : 0.f;
            };
            const int j0 = part * chunk;
#pragma unroll
            for (int k = 0; k < ahead; ++k) fetch(k, j0 + k);
            for (int jb = j0; jb < j1; jb += ahead)
#pragma unroll
                for (int k = 0; k < ahead; ++k) {
                    const int j = min(jb + k, nE - 1);     // past the end the entry of S is zero
                    const FxReal a = fx_real(ni[k].x, ni[k].y, nf[k]);
                    fetch(k, jb + k + ahead);
#pragma unroll
                    for (int q = 0; q < RT; ++q) fx_mac(s[q], a, in.i[(q0 + q) * nE + j], in.f[(q0 + q) * nE + j]);
                }
#pragma unroll
            for (int q = 0; q < RT; ++q) {
                unsigned bad = 0;
                cpx<double> v = mk<double>(0, 0);
                const bool mine = part == 0 && i < nE && q0 + q < cnt;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    long long h = 0, l = 0;
                    fx_flush(s[q], c, h, l);
                    for (int o = 1; o < tpr; o <<= 1) {
                        h += __shfl_xor_sync(0xffffffffu, h, o);
                        l += __shfl_xor_sync(0xffffffffu, l, o);
                    }
                    if (mine && !fx_value(h, l, ea, ex[q0 + q], c ? v.y : v.x)) bad |= 1u << c;
                }
                if (tpr > 1 ? __any_sync(0xffffffffu, bad != 0) : bad != 0) {
                    double2 d;
                    const double* S64 = S + i;
                    const int2* Si = Sx.i + i;
                    const int4* xi = in.i + (q0 + q) * nE;
                    const double2* xd = in.d + (q0 + q) * nE;
                    bad &= ~fx_again(tpr, bad, nE, ea, ex[q0 + q], [=](int j) { return make_double2(S64[j * nE], 0.0); },
                                     [=](int j) { return make_int2(Si[j * nE].x, 0); }, [=](int j) { return xi[j]; },
                                     [=](int j) { return xd[j]; }, d);
                    if (bad & 1) v.x = d.x;
                    if (bad & 2) v.y = d.y;
                }
                if (mine) out[(int64_t)(q0 + q) * ostride + i] = wout ? wout[i] * v : v;
            }
        } else {
            cpx<T> acc[RB];
#pragma unroll
            for (int q = 0; q < RB; ++q) acc[q] = mk<T>(0, 0);
            for (int j = part * chunk; j < j1; ++j) {
                const T sv = (T)__ldg(S + (int64_t)j * nE + i);
#pragma unroll
                for (int q = 0; q < RB; ++q)
                    if (q < cnt) fma_r(acc[q], sv, in.v[q * nE + j]);
            }
#pragma unroll
            for (int q = 0; q < RB; ++q) {
                for (int o = 1; o < tpr; o <<= 1) {
                    acc[q].x += __shfl_xor_sync(0xffffffffu, acc[q].x, o);
                    acc[q].y += __shfl_xor_sync(0xffffffffu, acc[q].y, o);
                }
                if (part == 0 && i < nE && q < cnt) out[(int64_t)q * ostride + i] = wout ? (T)wout[i] * acc[q] : acc[q];
            }
        }
    }
}
// splits the restricted S^Lap, one warp per row (grid: pattern, 8 warps per CTA)
__global__ void k_fix_pre(const double* __restrict__ S, const int64_t* __restrict__ off, const int* __restrict__ len,
                          const int64_t* __restrict__ eoff, FxRealMat fx, int* __restrict__ ex) {
    const int k = blockIdx.x, nE = len[k], warp = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    for (int i = warp; i < nE; i += nw) {
        const double* a = S + off[k] + i;                  // row i = column i (symmetric)
        unsigned m = 0;
        for (int j = lane; j < nE; j += 32) m = max(m, fx_mag(a[(int64_t)j * nE]));
        const int ef = fx_exp(__reduce_max_sync(0xffffffffu, m));
        for (int j = lane; j < nE; j += 32) fx_put(fx, off[k] + i + (int64_t)j * nE, a[(int64_t)j * nE], ef);
        if (lane == 0) ex[eoff[k] + i] = ef;
    }
}

template <class T, int RB>
__global__ void __launch_bounds__(128 * kEdgeParts<T, RB>, std::is_same<T, double>::value && RB >= 4 ? 6 / kEdgeParts<T, RB> : 1) k_pre_elem(const __grid_constant__ DevModel dm, const double2* __restrict__ v, cpx<T>* __restrict__ outE,
                                                  int R, const int* __restrict__ done, int with_d) {
    if (done && *done) return;
    extern __shared__ __align__(128) char smem[];
    __shared__ int ex[RB];
    const int e = blockIdx.x, r0 = blockIdx.y * RB;
    const int cnt = min(RB, R - r0);
    const int nE = dm.nE1[e], e1o = dm.e1_off[e];
    const EdgeVec<T> in(smem, RB * nE);                           // [RB][nE]
    const auto load = [dp = &dm, v, e1o, r0, with_d](int q, int i) {
        const int row = dp->e1_row[e1o + i];
        cpx<T> val = mk<T>(0, 0);
        if (row >= 0) {
            const double w = dp->e1_win ? dp->e1_sign[e1o + i] * dp->e1_win[e1o + i] : dp->e1_sign[e1o + i];
            double2 x = v[(int64_t)(r0 + q) * dp->n_dual + row];
            if (with_d) {
                const double dd = dp->row_dinv ? dp->row_dinv[row] : 0.5;
                x = make_double2(dd * x.x, dd * x.y);
            }
            val = (T)w * mk<T>((T)x.x, (T)x.y);
        }
        return val;
    };
    edge_stage<T, RB>(load, nE, nE, cnt, in, ex);
    __syncthreads();
    // Poisson mode: out = (rho_e w) .* (S^Lap (w .* C1^T v)), the diagonally scaled W^T A W
    pre_apply<T, RB>(dm, e, nE, cnt, in, ex, outE + (int64_t)r0 * dm.nE1_tot + e1o, dm.nE1_tot,
                     dm.e1_wout ? dm.e1_wout + e1o : nullptr);
}

// Conforming meshes (no hanging rows: D = 2 I, no C2 K C2^T term), fused with the Krylov
// fetch: v = V[r][j] read directly (j = ctl[0]), D^-1 = 1/2 applied in the gather.
template <class T, int RB>
__global__ void __launch_bounds__(128 * kEdgeParts<T, RB>, std::is_same<T, double>::value && RB >= 4 ? 6 / kEdgeParts<T, RB> : 1) k_pre_elem_kry(const __grid_constant__ DevModel dm, const __grid_constant__ KrylovDev K, cpx<T>* __restrict__ outE, int R) {
    if (K.ctl[1]) return;
    const int jj = K.ctl[0];
    extern __shared__ __align__(128) char smem[];
    __shared__ int ex[RB];
    const int e = blockIdx.x, r0 = blockIdx.y * RB;
    const int cnt = min(RB, R - r0);
    const int nE = dm.nE1[e], e1o = dm.e1_off[e];
    const EdgeVec<T> in(smem, RB * nE);
    const auto load = [dp = &dm, kp = &K, e1o, r0, jj](int q, int i) {
        const int row = dp->e1_row[e1o + i];
        cpx<T> val = mk<T>(0, 0);
        if (row >= 0) {
            const int64_t at = ((int64_t)(r0 + q) * (kp->m + 1) + jj) * kp->nd + row;
            if (kp->Vf) {
                const float2 x = kp->Vf[at];
                val = (T)(0.5 * dp->e1_sign[e1o + i]) * mk<T>((T)x.x, (T)x.y);
            } else {
                val = (T)(0.5 * dp->e1_sign[e1o + i]) * ld<T>(kp->V, at);
            }
        }
        return val;
    };
    edge_stage<T, RB>(load, nE, nE, cnt, in, ex);
    __syncthreads();
    pre_apply<T, RB>(dm, e, nE, cnt, in, ex, outE + (int64_t)r0 * dm.nE1_tot + e1o, dm.nE1_tot);
}

// z = D^-1 (outE[c] - outE[f]) with D = 2 I, written to zw and to the Krylov store Zb[r][j]
template <class T>
__global__ void k_pre_rows_kry(DevModel dm, KrylovDev K, const cpx<T>* __restrict__ outE) {
    if (K.ctl[1]) return;
    const int jj = K.ctl[0];
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (row >= dm.n_dual) return;
    double sx = 0, sy = 0;
    const int c = dm.row_c[row], f = dm.row_f[row];
    if (c >= 0) { const cpx<T> a = outE[(int64_t)r * dm.nE1_tot + c]; sx += (double)a.x; sy += (double)a.y; }
    if (f >= 0) { const cpx<T> a = outE[(int64_t)r * dm.nE1_tot + f]; sx -= (double)a.x; sy -= (double)a.y; }
    const double2 z = make_double2(0.5 * sx, 0.5 * sy);
    K.zw[(int64_t)r * K.nd + row] = z;
    K.Zb[((int64_t)r * K.m + jj) * K.nd + row] = z;
}

// m[row] = outE[c] - outE[f] + (C2 K^Lap C2^T v)[row]
template <class T>
__global__ void k_pre_rows(DevModel dm, const cpx<T>* __restrict__ outE, const double2* __restrict__ v,
                           double2* __restrict__ m, int with_d, const int* __restrict__ done) {
    if (done && *done) return;
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (row >= dm.n_dual) return;
    double sx = 0, sy = 0;
    const int c = dm.row_c[row], f = dm.row_f[row];
    if (c >= 0) { const cpx<T> a = outE[(int64_t)r * dm.nE1_tot + c]; sx += (double)a.x; sy += (double)a.y; }
    if (f >= 0) { const cpx<T> a = outE[(int64_t)r * dm.nE1_tot + f]; sx -= (double)a.x; sy -= (double)a.y; }
    if (with_d) {
        const double dd = dm.row_dinv ? dm.row_dinv[row] : 0.5;
        sx *= dd;
        sy *= dd;
    } else
        for (int a = dm.mh_ptr[row]; a < dm.mh_ptr[row + 1]; ++a) {
            const double2 vv = v[(int64_t)r * dm.n_dual + dm.mh_col[a]];
            sx += dm.mh_val[a] * vv.x;
            sy += dm.mh_val[a] * vv.y;
        }
    m[(int64_t)r * dm.n_dual + row] = make_double2(sx, sy);
}

// ------------------------------------------------------------------ launch wrappers
// shared memory of the persistent edge pass: r_E block, then (when two fit) two staging buffers
// for S_E^-1 behind two mbarriers; returns the staging offset (0 = read S_E^-1 from global)
template <class T>
static int edge_p_layout(int rb, int maxE1, int* buf_bytes, size_t* total) {
    const size_t base = edge_vec_bytes<T>(rb, maxE1);
    const size_t one = edge_mat_bytes<T>(maxE1);
    const bool fit = maxE1 > 0 && base + 128 + 2 * one <= 200 * 1024;
    *buf_bytes = (int)one;
    *total = fit ? base + 128 + 2 * one : base;
    return fit ? (int)base : 0;
}
template <class T, int RB>
static void edge_p_t(const DevModel& dm, const cpx<T>* S, const cpx<T>* Yp, const double2* z, double zsign,
                     const double2* bt, void* xE, void* tT, int R, const int* done, const EdgeSched& es, int item0,
                     int nitems, int tpr_force, cudaStream_t st) {
    int buf = 0;
    size_t sm = 0;
    const int so = edge_p_layout<T>(RB, dm.maxE1, &buf, &sm);
    const int vs = std::max(1, dm.maxE1);
    const int ntask = nitems * ((R + RB - 1) / RB);
    int dev = 0, nsm = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pass1_edge_p<T, RB>, 256 * kEdgeParts<T, RB>, sm);
    const int grid = std::max(1, std::min(ntask, std::max(1, per) * std::max(1, nsm)));
    k_pass1_edge_p<T, RB><<<grid, 256 * kEdgeParts<T, RB>, sm, st>>>(dm, S, Yp, z, zsign, bt, R, (cpx<T>*)xE, (cpx<T>*)tT, done, es.items,
                                                 item0, nitems, es.tpr_p, tpr_force, so, buf, vs);
}
int edge_cta_threads(int maxNo) { return maxNo > 64 ? std::min(256, (2 * maxNo + 31) / 32 * 32) : 256; }

template <class T>
void launch_pass1_edge(const DevModel& dm, const void* sinv, const void* Y, const double2* z, double zsign,
                       const double2* bt, void* xE, void* tT, int R, const int* done, cudaStream_t st,
                       const EdgeSched* es, int item0, int nitems, int tpr_force, int rows) {
    const int rb = rhs_block(R);
    const cpx<T>* S = (const cpx<T>*)sinv;
    const cpx<T>* Yp = (const cpx<T>*)Y;
    if (es && es->items && rows == 0) {
        if (nitems < 0) nitems = dm.E;
        switch (rb) {
            case 8: edge_p_t<T, 8>(dm, S, Yp, z, zsign, bt, xE, tT, R, done, *es, item0, nitems, tpr_force, st); break;
            case 4: edge_p_t<T, 4>(dm, S, Yp, z, zsign, bt, xE, tT, R, done, *es, item0, nitems, tpr_force, st); break;
            case 2: edge_p_t<T, 2>(dm, S, Yp, z, zsign, bt, xE, tT, R, done, *es, item0, nitems, tpr_force, st); break;
            default: edge_p_t<T, 1>(dm, S, Yp, z, zsign, bt, xE, tT, R, done, *es, item0, nitems, tpr_force, st);
        }
        return;
    }
    // the t_T rows alone read no S_E^-1: no staging
    const bool stage = rows != 2 && !(es && !es->stage);
    const int so = stage ? edge_stage_off<T>(rb, dm.maxE1) : 0;
    const int ntask = dm.E * ((R + rb - 1) / rb);
    const size_t sm = stage ? edge_smem_total<T>(rb, dm.maxE1) : edge_vec_bytes<T>(rb, dm.maxE1);
    const int vs = std::max(1, dm.maxE1);
    // CTA size: two threads per output row of the widest element when that is more than 64
    // rows (rounded up to whole warps), else 256; the CTA takes the rows in one pass and fewer
    // threads idle (80 rows at p = 20, l = 5: 160 threads instead of 256 with 96 idle)
    const int nt = es && es->cta_threads > 0 ? es->cta_threads : edge_cta_threads(dm.maxNo);
    switch (rb) {
        case 8: k_pass1_edge<T, 8><<<ntask, nt * kEdgeParts<T, 8>, sm, st>>>(dm, S, Yp, z, zsign, bt, R, (cpx<T>*)xE, (cpx<T>*)tT, done, ntask, so, vs, rows); break;
        case 4: k_pass1_edge<T, 4><<<ntask, nt, sm, st>>>(dm, S, Yp, z, zsign, bt, R, (cpx<T>*)xE, (cpx<T>*)tT, done, ntask, so, vs, rows); break;
        case 2: k_pass1_edge<T, 2><<<ntask, nt, sm, st>>>(dm, S, Yp, z, zsign, bt, R, (cpx<T>*)xE, (cpx<T>*)tT, done, ntask, so, vs, rows); break;
        default: k_pass1_edge<T, 1><<<ntask, nt, sm, st>>>(dm, S, Yp, z, zsign, bt, R, (cpx<T>*)xE, (cpx<T>*)tT, done, ntask, so, vs, rows);
    }
}
template <class T>
void launch_pass2_edge(const DevModel& dm, const void* Y, const double2* x2, const void* xE_in, void* xE_out, int R,
                       const int* done, cudaStream_t st) {
    const int rb = rhs_block(R);
    const int ntask = dm.E * ((R + rb - 1) / rb);
    const cpx<T>* Yp = (const cpx<T>*)Y;
    const cpx<T>* xi = (const cpx<T>*)xE_in;
    cpx<T>* xo = (cpx<T>*)xE_out;
    // one thread per edge row: 64-thread CTAs when every element has at most 64 (more CTAs
    // resident per SM to hide the gather latency)
    const int nt = dm.maxE1 <= 64 ? 64 : 128;
    // FP64: room for the largest Y (nE + nT <= 4 p = 128, so at most 64 x 64 entries)
    const int vs = std::max(1, dm.maxT), yo = (int)edge_vec_bytes<T>(rb, vs);
    const int ys = std::is_same<T, double>::value && dm.maxY > 0 && dm.maxY <= 64 * 64;
    const size_t sm = yo + (ys ? 128 + dm.maxY * kEdgeMatBytes<T> + 16 : 0);
    switch (rb) {
        case 8: k_pass2_edge<T, 8><<<ntask, nt * kEdgeParts<T, 8>, sm, st>>>(dm, Yp, x2, xi, xo, R, done, ntask, vs, yo, ys); break;
        case 4: k_pass2_edge<T, 4><<<ntask, nt, sm, st>>>(dm, Yp, x2, xi, xo, R, done, ntask, vs, yo, ys); break;
        case 2: k_pass2_edge<T, 2><<<ntask, nt, sm, st>>>(dm, Yp, x2, xi, xo, R, done, ntask, vs, yo, ys); break;
        default: k_pass2_edge<T, 1><<<ntask, nt, sm, st>>>(dm, Yp, x2, xi, xo, R, done, ntask, vs, yo, ys);
    }
}
template void launch_pass1_edge<double>(const DevModel&, const void*, const void*, const double2*, double, const double2*, void*, void*, int, const int*, cudaStream_t, const EdgeSched*, int, int, int, int);
template void launch_pass1_edge<float>(const DevModel&, const void*, const void*, const double2*, double, const double2*, void*, void*, int, const int*, cudaStream_t, const EdgeSched*, int, int, int, int);
template void launch_pass2_edge<double>(const DevModel&, const void*, const double2*, const void*, void*, int, const int*, cudaStream_t);
template void launch_pass2_edge<float>(const DevModel&, const void*, const double2*, const void*, void*, int, const int*, cudaStream_t);
template <class T>
void launch_coarse_assemble(const DevModel& dm, const void* tT, const double2* bt, const double2* z, double zsign,
                            double2* t, int R, const int* done, cudaStream_t st) {
    k_coarse_assemble<T><<<dim3((dm.n_coarse + 127) / 128, R), 128, 0, st>>>(dm, (const cpx<T>*)tT, bt, z, zsign, t, R, done);
}
template <class T>
void launch_jump_gather(const DevModel& dm, const void* xE, const double2* x2, double2* w, int R, const int* done,
                        cudaStream_t st) {
    k_jump_gather<T><<<dim3((dm.n_dual + 127) / 128, R), 128, 0, st>>>(dm, (const cpx<T>*)xE, x2, w, done);
}
template <class T>
int launch_pre(const DevModel& dm, const double2* v, double2* vd, void* outE, double2* m, double2* z,
               int R, const int* done, cudaStream_t st) {
    const dim3 gr((dm.n_dual + 127) / 128, R);
    // without hanging rows D is diagonal and there is no C2 K C2^T: D^-1 goes into the two kernels (64 x 64
    // elements, p = 20, 8 right-hand sides: 275 us for an application, 12 us less than with launches of their own)
    const int with_d = dm.n_hb == 0;
    if (!with_d) k_dinv<<<gr, 128, 0, st>>>(dm, v, vd, done);
    const double2* in = with_d ? v : vd;
    const int rb = rhs_block(R);
    const dim3 g(dm.E, (R + rb - 1) / rb);
    const size_t sm = kEdgeVecBytes<T> * (size_t)rb * dm.maxE1 + 16;
    switch (rb) {
        case 8: k_pre_elem<T, 8><<<g, 128 * kEdgeParts<T, 8>, sm, st>>>(dm, in, (cpx<T>*)outE, R, done, with_d); break;
        case 4: k_pre_elem<T, 4><<<g, 128, sm, st>>>(dm, in, (cpx<T>*)outE, R, done, with_d); break;
        case 2: k_pre_elem<T, 2><<<g, 128, sm, st>>>(dm, in, (cpx<T>*)outE, R, done, with_d); break;
        default: k_pre_elem<T, 1><<<g, 128, sm, st>>>(dm, in, (cpx<T>*)outE, R, done, with_d);
    }
    k_pre_rows<T><<<gr, 128, 0, st>>>(dm, (const cpx<T>*)outE, in, with_d ? z : m, with_d, done);
    if (!with_d) k_dinv<<<gr, 128, 0, st>>>(dm, m, z, done);
    return with_d ? 2 : 4;
}

template void launch_coarse_assemble<double>(const DevModel&, const void*, const double2*, const double2*, double, double2*, int, const int*, cudaStream_t);
template void launch_coarse_assemble<float>(const DevModel&, const void*, const double2*, const double2*, double, double2*, int, const int*, cudaStream_t);
template void launch_jump_gather<double>(const DevModel&, const void*, const double2*, double2*, int, const int*, cudaStream_t);
template void launch_jump_gather<float>(const DevModel&, const void*, const double2*, double2*, int, const int*, cudaStream_t);
template int launch_pre<double>(const DevModel&, const double2*, double2*, void*, double2*, double2*, int, const int*, cudaStream_t);
template int launch_pre<float>(const DevModel&, const double2*, double2*, void*, double2*, double2*, int, const int*, cudaStream_t);
void launch_fix_edge(const DevModel& dm, const void* sinv, const void* Y, const EdgeFix& f, cudaStream_t st) {
    k_fix_edge<<<dm.E, 256, 0, st>>>(dm, (const double2*)sinv, (const double2*)Y, f);
}
void launch_fix_pre(const double* S, int npat, const int64_t* off, const int* len, const int64_t* eoff,
                    const FxRealMat& fx, int* ex, cudaStream_t st) {
    if (npat > 0) k_fix_pre<<<npat, 256, 0, st>>>(S, off, len, eoff, fx, ex);
}
void launch_dinv(const DevModel& dm, const double2* x, double2* y, int R, const int* done, cudaStream_t st) {
    k_dinv<<<dim3((dm.n_dual + 127) / 128, R), 128, 0, st>>>(dm, x, y, done);
}
template <class T>
void launch_pre_krylov(const DevModel& dm, const KrylovDev& K, void* outE, int R, cudaStream_t st) {
    const int rb = rhs_block(R);
    const dim3 g(dm.E, (R + rb - 1) / rb);
    const size_t sm = kEdgeVecBytes<T> * (size_t)rb * dm.maxE1 + 16;
    switch (rb) {
        case 8: k_pre_elem_kry<T, 8><<<g, 128 * kEdgeParts<T, 8>, sm, st>>>(dm, K, (cpx<T>*)outE, R); break;
        case 4: k_pre_elem_kry<T, 4><<<g, 128, sm, st>>>(dm, K, (cpx<T>*)outE, R); break;
        case 2: k_pre_elem_kry<T, 2><<<g, 128, sm, st>>>(dm, K, (cpx<T>*)outE, R); break;
        default: k_pre_elem_kry<T, 1><<<g, 128, sm, st>>>(dm, K, (cpx<T>*)outE, R);
    }
    k_pre_rows_kry<T><<<dim3((dm.n_dual + 127) / 128, R), 128, 0, st>>>(dm, K, (const cpx<T>*)outE);
}
template void launch_pre_krylov<double>(const DevModel&, const KrylovDev&, void*, int, cudaStream_t);
template void launch_pre_krylov<float>(const DevModel&, const KrylovDev&, void*, int, cudaStream_t);


template <class T, int RB>
static void set_edge_pass_limits(int maxE1) {
    raise_smem_limit(k_pass1_edge<T, RB>, (int)edge_smem_total<T>(RB, maxE1));
    // the whole unified L1/shared array as shared memory: the staged S_E^-1 limits residency
    cudaFuncSetAttribute(k_pass1_edge<T, RB>, cudaFuncAttributePreferredSharedMemoryCarveout,
                         (int)cudaSharedmemCarveoutMaxShared);
    if (std::is_same<T, double>::value)
        raise_smem_limit(k_pass2_edge<T, RB>, (int)edge_vec_bytes<T>(RB, 128) + 128 + 64 * 64 * kEdgeMatBytes<T> + 16);
    int buf = 0;
    size_t tot = 0;
    edge_p_layout<T>(RB, maxE1, &buf, &tot);
    raise_smem_limit(k_pass1_edge_p<T, RB>, (int)tot);
}
void set_edge_limits(int pmax, int maxE1) {
    (void)pmax;
    set_edge_pass_limits<double, 1>(maxE1); set_edge_pass_limits<double, 2>(maxE1);
    set_edge_pass_limits<double, 4>(maxE1); set_edge_pass_limits<double, 8>(maxE1);
    set_edge_pass_limits<float, 1>(maxE1); set_edge_pass_limits<float, 2>(maxE1);
    set_edge_pass_limits<float, 4>(maxE1); set_edge_pass_limits<float, 8>(maxE1);
    const int pre64 = kEdgeVecBytes<double> * 8 * maxE1 + 16, pre32 = kEdgeVecBytes<float> * 8 * maxE1 + 16;
    raise_smem_limit(k_pre_elem<double, 1>, pre64);
    raise_smem_limit(k_pre_elem<double, 2>, pre64);
    raise_smem_limit(k_pre_elem<double, 4>, pre64);
    raise_smem_limit(k_pre_elem<double, 8>, pre64);
    raise_smem_limit(k_pre_elem<float, 1>, pre32);
    raise_smem_limit(k_pre_elem<float, 2>, pre32);
    raise_smem_limit(k_pre_elem<float, 4>, pre32);
    raise_smem_limit(k_pre_elem<float, 8>, pre32);
    raise_smem_limit(k_pre_elem_kry<double, 1>, pre64);
    raise_smem_limit(k_pre_elem_kry<double, 2>, pre64);
    raise_smem_limit(k_pre_elem_kry<double, 4>, pre64);
    raise_smem_limit(k_pre_elem_kry<double, 8>, pre64);
    raise_smem_limit(k_pre_elem_kry<float, 1>, pre32);
    raise_smem_limit(k_pre_elem_kry<float, 2>, pre32);
    raise_smem_limit(k_pre_elem_kry<float, 4>, pre32);
    raise_smem_limit(k_pre_elem_kry<float, 8>, pre32);
}

}  // namespace ddh
