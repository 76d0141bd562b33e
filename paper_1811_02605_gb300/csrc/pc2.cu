// PC2 (Sec. 2.2): PCG with a block-Jacobi preconditioner that uses a zero-fill incomplete LU
// factorisation (ILU(0)) in each block. The blocks are the periodic phi lines (i, j) of each
// component: the r and theta couplings are left out of the preconditioner, so every line is an
// independent block (nr nt of them per component) instead of one block per MPI rank as in the
// paper. For a periodic tridiagonal block zero fill changes only the diagonal:
//     dt_0 = m,  dt_k = m - w^2 / dt_{k-1},  dt_{np-1} -= w^2 / dt_0,
// m the diagonal on the line and -w its phi coupling, and P = (dt + L) dt^-1 (dt + U).
//
// The solve runs on the Jacobi-scaled system A~ = S M S (S = diag(M)^-1/2, unit diagonal, the
// PC1 path's tables and stencil kernels), whose ILU(0) is S ILU(0)(M) S: the same iterates as PCG
// with PC2 on M, in exact arithmetic. On a line of A~: m = 1 and w = the scaled phi coefficient.
//
// z = P^-1 r is a forward and a backward substitution along each line, both first-order linear
// recurrences u_k = a_k u_{k-1} + b_k, which the lanes of a line evaluate as an affine scan: each
// lane composes the maps of its segment, a shuffle scan composes
// the segments, and each lane replays its segment from the value entering it. The multipliers
// (a_k = w / dt_k) do not depend on the component, so their segment products and the scan's
// per-step multipliers are formed once per line and reused by the three components; per
// component only the additive parts are scanned. The periodic wrap enters as u_0 in the last
// forward step and as z_{np-1} in the first backward one, both known before the replays.
//
// FP64 solves use the line kernel in double; the mixed-precision inner solves use it in float
// (vectors, factor and scans in FP32; each lane's dot partials over one line, at most 3 np / 32
// products, are formed in FP32 and summed over lines in FP64),
// with the FP64 outer residual of the reliable-update scheme followed by one preconditioner pass
// that recomputes z and <r, z> for the replaced residual.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "mhd_internal.cuh"
#include "reduce.cuh"

namespace mhd {

namespace {

constexpr unsigned kFull = 0xffffffffu;

enum { kIter = 0, kInit = 1, kReliable = 2 };

// launch shape of the line kernel: lanes and elements per lane of a line (0: the generic kernel), warps per CTA,
// dynamic shared memory, CTAs
struct LineShape {
    int lanes, seg, warps, blocks;
    size_t smem;
};

struct Pc2Work {
    double* idt;      // [N] 1 / dt of the scaled lines (FP64)
    float* idt32;     // [N] the same in FP32
    float* z32;       // [3N] z~ of the FP32 iteration (the p double buffer keeps both halves for p~)
    LineShape shape[2];   // of the line kernel, [0] FP64, [1] FP32
};

// 1 / dt along every phi line of A~ (one thread per line); a non-positive pivot flags a breakdown
__global__ void k_pc2_factor(Dims d, OpTab<double> t, double* __restrict__ idt, float* __restrict__ idt32,
                             PcgScalars* sc) {
    const int nl = d.nr * d.nt;
    for (int ij = blockIdx.x * blockDim.x + threadIdx.x; ij < nl; ij += gridDim.x * blockDim.x) {
        const double w = t.ap[ij];
        const double w2 = w * w;
        const long long base = (long long)ij * d.np;
        double dt = 1.0;
        bool bad = false;
        idt[base] = 1.0;
        idt32[base] = 1.0f;
        for (int k = 1; k < d.np; k++) {
            dt = 1.0 - w2 / dt;
            if (k == d.np - 1) dt -= w2;
            bad = bad || !(dt > 0.0);
            const double id = 1.0 / dt;
            idt[base + k] = id;
            idt32[base + k] = (float)id;
        }
        if (bad) sc->done = 4;
    }
}

// Shared memory per warp: 1/dt, w/dt and a work line, each np + ceil(np / S) elements (one pad
// after each lane segment of S = ceil(np / 32) elements; element k sits at k + k / S).
__host__ __device__ inline int padded_len(int np) {
    const int S = (np + 31) / 32;
    return np + (np + S - 1) / S;
}

// end of a line kernel: <r~, z~> and ||r||^2 over the grid; the last CTA does the scalar recurrence of its mode
template <typename T, int MODE>
__device__ __forceinline__ void line_finish(double a_rz, double a_rr, PcgScalars* sc, double* __restrict__ partials,
                                            int restart) {
    double val[2] = {a_rz, a_rr}, out[2];
    if (reduce_last<2>(val, partials, &sc->count, out) && threadIdx.x == 0) {
        const double rz = out[0], rr = out[1];
        if (MODE == kReliable) {
            const bool keep = !restart && sc->rho_prev > 0.0 && rz <= 4.0 * sc->rho;
            sc->beta = keep ? rz / sc->rho_prev : 0.0;
            sc->rho = rz;
            sc->rr = rr;
            if (!isfinite(rz) || !isfinite(rr)) {
                sc->done = 3;
                sc->outer_done = 3;
            } else if (!(rz > 0.0)) {
                sc->done = 4;
            }
            return;
        }
        if (MODE == kInit) {
            sc->beta = 0.0;
        } else {
            sc->iter += 1;
            sc->total_iter += 1;
            sc->beta = rz / sc->rho;
            sc->rho_prev = sc->rho;
            sc->ax = sc->alpha;   // x~ += alpha p~ is left to the next p update
        }
        sc->rho = rz;
        sc->rr = rr;
        if (!isfinite(rz) || !isfinite(rr)) sc->done = 3;
        else if (sc->bb == 0.0 || sqrt(rr) <= sc->tol * sqrt(sc->bb)) sc->done = 1;
        else if (sc->iter >= sc->max_iter) sc->done = 2;
        else if (!(rz > 0.0)) sc->done = 4;
    }
}

// One warp per phi line of the scaled system.
//   kIter:     r~ -= alpha q~; z~ = P~^-1 r~; <r~, z~> and
//              ||r||^2 = sum dg r~^2; last CTA: beta = rho_new / rho, stop test, iteration count.
//              alpha is handed on in sc->ax, and the p update of the next iteration (or the kernel
//              that takes x~ over when the solve stops here) adds alpha p~ to x~.
//   kInit:     z~ = P~^-1 r~, p~ = z~; last CTA: rho, beta = 0, stop test (after the FP64 set-up).
//   kReliable: z~ = P~^-1 r~ for the replaced residual; last CTA: rho = <r~, z~>, and the
//              recurrence continues (beta = rho / rho_prev) while rho stays within 4x of the
//              recursive one, else restarts (beta = 0); the stop flags are the outer kernel's.
// This is the form for lines longer than the register kernel (k_pc2_seg) takes: the segments are in shared memory.
template <typename T, int MODE>
__global__ void __launch_bounds__(kThreads) k_pc2_line(Dims d, int nc, OpTab<T> t, const double* __restrict__ dgv,
                                                       const T* __restrict__ idt,
                                                       T* __restrict__ p, T* __restrict__ r,
                                                       const T* __restrict__ q, T* __restrict__ z,
                                                       PcgScalars* sc, double* __restrict__ partials, int restart) {
    if (sc->done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* smem = reinterpret_cast<T*>(smem_raw);
    const int warps = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int np = d.np;
    const int S = (np + 31) >> 5;
    const int P = padded_len(np);
    T* ib = smem + (size_t)warp * 3 * P;   // 1 / dt_k
    T* gb = ib + P;                        // w / dt_k
    T* ub = gb + P;                        // work line
    const T al = (MODE == kIter) ? (T)sc->alpha : T(0);
    const T zero = T(0);
    const int k0 = lane * S;
    const int s0 = lane * (S + 1);         // element k0 + t of this lane's segment sits at s0 + t
    // element k0 + t is in the line / is its first / is its last element
#define IN_LINE(tt) (k0 + (tt) < np)
#define FIRST(tt) ((tt) == 0 && lane == 0)
#define LAST(tt) (k0 + (tt) == np - 1)
    double a_rz = 0.0, a_rr = 0.0;   // per-line partials (in T) are added here in FP64
    const int nl = d.nr * d.nt;
    for (int line = blockIdx.x * warps + warp; line < nl; line += gridDim.x * warps) {
        const T w = t.ap[line];
        const long long base = (long long)line * np;
        for (int k = lane; k < np; k += 32) {
            const T id = idt[base + k];
            ib[k + k / S] = id;
            gb[k + k / S] = w * id;
        }
        __syncwarp();
        // component-independent multipliers: forward a_k (a_0 = 0), backward c_k (c_{np-1} = 0)
        T A = T(1), Cm = T(1);
#pragma unroll
        for (int tt = 0; tt < S; tt++) {
            if (IN_LINE(tt)) {
                const T g = gb[s0 + tt];
                A *= FIRST(tt) ? zero : g;
                Cm *= LAST(tt) ? zero : g;
            }
        }
        T As[5], Cs[5];
#pragma unroll
        for (int st = 0; st < 5; st++) {
            const int o = 1 << st;
            const T Ao = __shfl_up_sync(kFull, A, o), Co = __shfl_down_sync(kFull, Cm, o);
            As[st] = A;
            Cs[st] = Cm;
            if (lane >= o) A *= Ao;
            if (lane + o < 32) Cm *= Co;
        }
        T line_rz = zero, line_rr = zero;
#pragma unroll 1
        for (int c = 0; c < nc; c++) {
            const long long off = c * d.N + base;
            for (int k = lane; k < np; k += 32) {
                T rv = r[off + k];
                if (MODE == kIter) {
                    rv = fma(-al, q[off + k], rv);
                    r[off + k] = rv;
                }
                ub[k + k / S] = rv;
            }
            __syncwarp();
            // forward: u_0 = r_0 / dt_0; u_k = (r_k + w u_{k-1}) / dt_k; the last also + w u_0 / dt
            const T u0 = ub[0] * ib[0];
            __syncwarp();
            T B = zero;
#pragma unroll
            for (int tt = 0; tt < S; tt++) {
                if (IN_LINE(tt)) {
                    const int sx = s0 + tt;
                    T bk = ub[sx] * ib[sx];
                    if (LAST(tt)) bk = fma(gb[sx], u0, bk);
                    ub[sx] = bk;
                    B = fma(FIRST(tt) ? zero : gb[sx], B, bk);
                }
            }
#pragma unroll
            for (int st = 0; st < 5; st++) {
                const int o = 1 << st;
                const T Bo = __shfl_up_sync(kFull, B, o);
                if (lane >= o) B = fma(As[st], Bo, B);
            }
            T u = __shfl_up_sync(kFull, B, 1);
            if (lane == 0) u = zero;
#pragma unroll
            for (int tt = 0; tt < S; tt++) {
                if (IN_LINE(tt)) {
                    const int sx = s0 + tt;
                    u = fma(FIRST(tt) ? zero : gb[sx], u, ub[sx]);
                    ub[sx] = u;
                }
            }
            __syncwarp();
            // backward: z_{np-1} = u_{np-1}; z_k = u_k + w z_{k+1} / dt_k; the first also + w z_{np-1} / dt_0
            const T zl = ub[(np - 1) + (np - 1) / S];
            __syncwarp();
            T E = zero;
#pragma unroll
            for (int tt = S - 1; tt >= 0; tt--) {
                if (IN_LINE(tt)) {
                    const int sx = s0 + tt;
                    T e = ub[sx];
                    if (FIRST(tt)) e = fma(gb[sx], zl, e);
                    ub[sx] = e;
                    E = fma(LAST(tt) ? zero : gb[sx], E, e);
                }
            }
#pragma unroll
            for (int st = 0; st < 5; st++) {
                const int o = 1 << st;
                const T Eo = __shfl_down_sync(kFull, E, o);
                if (lane + o < 32) E = fma(Cs[st], Eo, E);
            }
            T zz = __shfl_down_sync(kFull, E, 1);
            if (lane == 31) zz = zero;
#pragma unroll
            for (int tt = S - 1; tt >= 0; tt--) {
                if (IN_LINE(tt)) {
                    const int sx = s0 + tt;
                    zz = fma(LAST(tt) ? zero : gb[sx], zz, ub[sx]);
                    ub[sx] = zz;
                }
            }
            __syncwarp();
            for (int k = lane; k < np; k += 32) {
                const T zv = ub[k + k / S];
                const T rv = r[off + k];
                z[off + k] = zv;
                if (MODE == kInit) p[off + k] = zv;
                line_rz = fma(rv, zv, line_rz);
                line_rr = fma(rv, rv, line_rr);
            }
            __syncwarp();
        }
        a_rz += (double)line_rz;
        a_rr = fma(dgv[line], (double)line_rr, a_rr);
    }
#undef IN_LINE
#undef FIRST
#undef LAST
    line_finish<T, MODE>(a_rz, a_rr, sc, partials, restart);
}

constexpr int kSegMax = 24;   // most elements of a lane in the register kernel

__device__ __forceinline__ void copy_async(void* dst, const void* src, int bytes16) {
    const unsigned int d = (unsigned int)__cvta_generic_to_shared(dst);
    if (bytes16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// V consecutive elements as one access (8 or 16 bytes, aligned to their size)
template <typename T, int V>
struct alignas(V * sizeof(T)) Pack {
    T v[V];
};
template <typename T, int V>
__device__ __forceinline__ Pack<T, V> load(const T* p) {
    return *reinterpret_cast<const Pack<T, V>*>(p);
}
template <typename T, int V>
__device__ __forceinline__ void store(T* p, const Pack<T, V>& a) {
    *reinterpret_cast<Pack<T, V>*>(p) = a;
}
// f(integral_constant i) for the same i in [LO, HI) in all lanes, by bisection (registers cannot be indexed)
template <int HI, int LO = 0, typename F>
__device__ __forceinline__ void one_of(int i, F f) {
    if constexpr (HI - LO == 1) f(std::integral_constant<int, LO>());
    else if (i < (LO + HI) / 2) one_of<(LO + HI) / 2, LO>(i, f);
    else one_of<HI, (LO + HI) / 2>(i, f);
}
// distance of two segments in shared memory: an odd number of 16-byte units, so that 16-byte accesses by segment
// meet no bank conflicts
template <typename T, int S>
constexpr int kSegDist = (S * sizeof(T)) % 32 == 0 ? S + 16 / (int)sizeof(T) : S;

// The same line solve with each lane's segment in registers. L lanes hold a line in segments of S elements (the last
// ones shorter or empty, their missing elements zero), so a warp takes 32 / L consecutive lines, which are contiguous
// in memory: loads and stores are coalesced, and one exchange through shared memory in either direction brings an
// element to its lane and back, 16 bytes at a time. 1 / dt and the multipliers stay in registers for the
// components. What a warp reads next is copied ahead (cp.async) while it solves: the registers allow 12 (FP64) to 20
// warps per SM, too few to hide the loads' latency otherwise (96x96x192, FP64: 176 us a call without the copies, with
// them 121).
// In FP64 the floor is the FP64 instructions, each taking a scheduler's pipe 64 cycles: five
// per element for the two recurrences (scale, compose and replay forwards, the same backwards), three for r~ and
// the sums, and per line and lane two for the multipliers and four per scan step. Short scans and long segments are
// the cheap ones, so L is the least that 16 elements a lane allow. In FP32 the floor is HBM; L is 32, which keeps the
// FP32 partial sums short. x~ += alpha p~ is left to the next p update, which reads p~ anyway.
// us per call, 3 components, the shared-memory form / this: FP64 64x64x128 65 / 43, 96x96x192 166 / 114; FP32
// 256x256x512 334 / 295 (at 6.8 TB/s: 257).
template <typename T, int S, int MODE>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? (S > 16 ? 2 : 3) : (S > 16 ? 4 : 5))
    k_pc2_seg(Dims d, int nc, int lanes, OpTab<T> t, const double* __restrict__ dgv, const T* __restrict__ idt,
              T* __restrict__ p, T* __restrict__ r, const T* __restrict__ q, T* __restrict__ z, PcgScalars* sc,
              double* __restrict__ partials, int restart) {
    if (sc->done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int L = sizeof(T) == 4 ? 32 : lanes;
    const int warps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int np = d.np, nl = d.nr * d.nt, lpw = 32 / L;
    constexpr int D = kSegDist<T, S>, W = 16 / (int)sizeof(T);
    T* const sr = reinterpret_cast<T*>(smem_raw) + (size_t)warp * 32 * (3 * S + D);   // r~, q~ and 1 / dt copied ahead
    T* const sq = sr + 32 * S;
    T* const si = sq + 32 * S;
    T* const wb = si + 32 * S;                                                        // r~, then z~, by segments
    const T al = (MODE == kIter) ? (T)sc->alpha : T(0);
    const T zero = T(0);
    const int ln = lane / L, gl = lane - ln * L;
    T* const seg = wb + lane * D;
    const int lastl = (np - 1) / S, lastt = (np - 1) - lastl * S;
    // element e of the warp's lines -> its place by segments (quotient exact for e < 32 kSegMax)
    const unsigned int m_np = (1u << 20) / np + 1;
    auto place = [&](unsigned int e) {
        const unsigned int line = sizeof(T) == 4 ? 0u : (e * m_np) >> 20, k = e - line * np;
        return line * (L * D) + k + k / S * (D - S);
    };
    // f(e, place of e) for the lane's packs of V elements; where a pass of the warp over 32 V elements is a whole
    // number of segments of one line, the places follow from the first
    auto packs = [&](auto width, int l0, int E, auto f) {
        constexpr int V = decltype(width)::value, n = S / V;
        if constexpr (sizeof(T) == 4 && (32 * V) % S == 0) {
            const int e0 = V * l0, p0 = (int)place(e0);
#pragma unroll
            for (int m = 0; m < n; m++)
                if (e0 + 32 * V * m < E) f(e0 + 32 * V * m, p0 + m * (32 * V / S) * D);
        } else {
#pragma unroll 2
            for (int e = V * l0; e < E; e += 32 * V) f(e, (int)place(e));
        }
    };
    const int step = gridDim.x * warps * lpw;
    // rows of np elements start on 16 bytes, except in FP32 when np is not a multiple of 4 (np is even)
    const int b16 = (np * (int)sizeof(T)) % 16 == 0, per = (b16 ? 16 : 8) / (int)sizeof(T);
    auto fetch = [&](int l0, int c) {
        const int E = min(lpw, nl - l0) * np;
        const long long base = (long long)l0 * np, off = c * d.N + base;
        for (int e = per * lane; e < E; e += 32 * per) {
            copy_async(sr + e, r + off + e, b16);
            if (MODE == kIter) copy_async(sq + e, q + off + e, b16);
            if (c == 0) copy_async(si + e, idt + base + e, b16);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // Elements past a line's end are zeros here and stay so: with g = 0 and 1 / dt = 0 there, whatever is formed from
    // them is 0 (unless the system holds a NaN or an infinity, which ends the solve).
    for (int e = lane; e < 32 * D; e += 32) wb[e] = zero;
    double a_rz = 0.0, a_rr = 0.0;   // per-line partials (in T) are added here in FP64
    int line0 = (blockIdx.x * warps + warp) * lpw;
    if (line0 < nl) fetch(line0, 0);
    for (; line0 < nl; line0 += step) {
        const int E = min(lpw, nl - line0) * np;
        const bool valid = line0 + ln < nl;
        const T w = valid ? t.ap[line0 + ln] : zero;
        const long long base = (long long)line0 * np;
        T g[S], id[S], b[S];
        T A = T(1);
        // scan multipliers, forwards and backwards (a wrong product in the lane at an end of the line is never used)
        T As[5], Cs[5];
        T line_rz = zero, line_rr = zero;
#pragma unroll 1
        for (int c = 0; c < nc; c++) {
            const long long off = c * d.N + base;
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            // (a value the compiler cannot see through: the places of all elements, formed once for the three
            // components, would not fit the registers)
            int l0 = lane;
            asm volatile("" : "+r"(l0));
            if (c == 0) {
                packs(std::integral_constant<int, 2>(), l0, E, [&](int e, int w0) { store<T, 2>(wb + w0, load<T, 2>(si + e)); });
                __syncwarp();
#pragma unroll
                for (int tt = 0; tt < S; tt += W) {
                    const Pack<T, W> v = load<T, W>(seg + tt);
#pragma unroll
                    for (int m = 0; m < W; m++) {
                        id[tt + m] = valid ? v.v[m] : zero;
                        g[tt + m] = w * id[tt + m];
                        A *= g[tt + m];
                    }
                }
                T C = A;
#pragma unroll
                for (int st = 0; st < 5; st++) {
                    const int o = 1 << st;
                    As[st] = A;
                    Cs[st] = C;
                    if (o < L) {
                        const T Ao = __shfl_up_sync(kFull, A, o, L), Co = __shfl_down_sync(kFull, C, o, L);
                        if (gl >= o) A *= Ao;
                        if (gl + o < L) C *= Co;
                    }
                }
                __syncwarp();
            }
            T* const rc = r + off;
            auto update = [&](auto width) {
                constexpr int V = decltype(width)::value;
                packs(width, l0, E, [&](int e, int w0) {
                    Pack<T, V> rv = load<T, V>(sr + e);
                    if (MODE == kIter) {
                        const Pack<T, V> qv = load<T, V>(sq + e);
#pragma unroll
                        for (int m = 0; m < V; m++) rv.v[m] = fma(-al, qv.v[m], rv.v[m]);
                        store<T, V>(rc + e, rv);
                    }
                    store<T, V>(wb + w0, rv);
                });
            };
            if (b16) update(std::integral_constant<int, W>());
            else update(std::integral_constant<int, 2>());
            __syncwarp();
            if (c + 1 < nc) fetch(line0, c + 1);
            else if (line0 + step < nl) fetch(line0 + step, 0);
            // forward: u_0 = r_0 / dt_0; u_k = (r_k + w u_{k-1}) / dt_k; the last also + w u_0 / dt
            T B = zero;
#pragma unroll
            for (int tt = 0; tt < S; tt += W) {
                const Pack<T, W> v = load<T, W>(seg + tt);
#pragma unroll
                for (int m = 0; m < W; m++) b[tt + m] = v.v[m] * id[tt + m];
            }
            const T u0 = __shfl_sync(kFull, b[0], 0, L);
#pragma unroll
            for (int tt = 0; tt < S; tt++) {
                B = tt == 0 ? b[0] : fma(g[tt], B, b[tt]);
            }
#pragma unroll
            for (int st = 0; st < 5; st++) {
                const int o = 1 << st;
                if (o < L) {
                    const T Bo = __shfl_up_sync(kFull, B, o, L);
                    if (gl >= o) B = fma(As[st], Bo, B);
                }
            }
            T u = __shfl_up_sync(kFull, B, 1, L);
            if (gl == 0) u = zero;
#pragma unroll
            for (int tt = 0; tt < S; tt++) {
                u = fma(g[tt], u, b[tt]);
                b[tt] = u;
            }
            // (nothing follows the last element, so its wrap term is added to it alone)
            T ul = zero;
            one_of<S>(lastt, [&](auto at) {
                constexpr int tt = decltype(at)::value;
                if (gl == lastl) b[tt] = fma(g[tt], u0, b[tt]);
                ul = b[tt];
            });
            // backward: z_{np-1} = u_{np-1}; z_k = u_k + w z_{k+1} / dt_k; the first also + w z_{np-1} / dt_0
            const T zl = __shfl_sync(kFull, ul, lastl, L);
            if (gl == 0) b[0] = fma(g[0], zl, b[0]);
            T En = b[S - 1];
#pragma unroll
            for (int tt = S - 2; tt >= 0; tt--) En = fma(g[tt], En, b[tt]);
#pragma unroll
            for (int st = 0; st < 5; st++) {
                const int o = 1 << st;
                if (o < L) {
                    const T Eo = __shfl_down_sync(kFull, En, o, L);
                    if (gl + o < L) En = fma(Cs[st], Eo, En);
                }
            }
            T zz = __shfl_down_sync(kFull, En, 1, L);
            if (gl == L - 1) zz = zero;
#pragma unroll
            for (int tt = S - W; tt >= 0; tt -= W) {
                const Pack<T, W> rv = load<T, W>(seg + tt);
                Pack<T, W> zv;
#pragma unroll
                for (int m = W - 1; m >= 0; m--) {
                    zz = fma(g[tt + m], zz, b[tt + m]);
                    zv.v[m] = zz;
                    line_rz = fma(rv.v[m], zz, line_rz);
                    line_rr = fma(rv.v[m], rv.v[m], line_rr);
                }
                store<T, W>(seg + tt, zv);
            }
            __syncwarp();
            T* const zc = z + off;
            auto hand_out = [&](auto width) {
                constexpr int V = decltype(width)::value;
                packs(width, l0, E, [&](int e, int w0) {
                    const Pack<T, V> zv = load<T, V>(wb + w0);
                    store<T, V>(zc + e, zv);
                    if (MODE == kInit) store<T, V>(p + off + e, zv);
                });
            };
            if (b16) hand_out(std::integral_constant<int, W>());
            else hand_out(std::integral_constant<int, 2>());
            __syncwarp();
        }
        if (valid) {
            a_rz += (double)line_rz;
            a_rr = fma(dgv[line0 + ln], (double)line_rr, a_rr);
        }
    }
    line_finish<T, MODE>(a_rz, a_rr, sc, partials, restart);
}

template <typename T>
size_t line_smem(const Dims& d, int warps) {
    return (size_t)warps * 3 * padded_len(d.np) * sizeof(T);
}

// the kernel of a mode for a segment length
template <typename T, int MODE>
auto seg_kernel(int seg) {
    switch (seg) {
        case 4: return k_pc2_seg<T, 4, MODE>;
        case 8: return k_pc2_seg<T, 8, MODE>;
        case 12: return k_pc2_seg<T, 12, MODE>;
        case 16: return k_pc2_seg<T, 16, MODE>;
        case 20: return k_pc2_seg<T, 20, MODE>;
        default: return k_pc2_seg<T, kSegMax, MODE>;
    }
}

template <typename T, int MODE>
cudaError_t set_smem(const LineShape& s) {
    return s.seg ? cudaFuncSetAttribute(seg_kernel<T, MODE>(s.seg), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s.smem)
                 : cudaFuncSetAttribute(k_pc2_line<T, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s.smem);
}

// Lines of up to 32 kSegMax elements take the register kernel, longer ones the generic kernel (up to 8 warps per
// CTA within 200 KB).
template <typename T>
mhd_status_t line_shape(mhd_grid_s* g, LineShape* s) {
    const int np = g->d.np, nl = g->d.nr * g->d.nt;
    int per_cta = 0;   // lines a CTA takes at once
    if (np <= 32 * kSegMax) {
        s->lanes = sizeof(T) == 4 ? 32 : (np <= 128 ? 8 : np <= 256 ? 16 : 32);
        s->seg = ((np + s->lanes - 1) / s->lanes + 3) & ~3;
        s->warps = 4;
        s->smem = (size_t)s->warps * 32 * (4 * s->seg + 16 / sizeof(T)) * sizeof(T);   // at most (kSegDist)
        per_cta = s->warps * (32 / s->lanes);
    } else {
        s->lanes = s->seg = 0;
        s->warps = 8;
        while (s->warps > 1 && line_smem<T>(g->d, s->warps) > 200 * 1024) s->warps >>= 1;
        s->smem = line_smem<T>(g->d, s->warps);
        if (s->smem > 200 * 1024) return set_error(g, MHD_ERR_ARG, "PC2: np too large for the line kernel");
        per_cta = s->warps;
    }
    constexpr int kFirst = sizeof(T) == 8 ? kInit : kReliable;   // the mode that starts or renews a recurrence
    if (set_smem<T, kIter>(*s) != cudaSuccess || set_smem<T, kFirst>(*s) != cudaSuccess)
        return check_cuda(g, "PC2: shared memory attribute");
    int per_sm = 0;
    if (s->seg) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, seg_kernel<T, kIter>(s->seg), 32 * s->warps, s->smem);
    else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pc2_line<T, kIter>, 32 * s->warps, s->smem);
    if (per_sm < 1) per_sm = 1;
    s->blocks = std::min(std::min(g->num_sms * per_sm, (nl + per_cta - 1) / per_cta), kMaxBlocks);
    return MHD_OK;
}

mhd_status_t pc2_workspace(mhd_grid_s* g, Pc2Work** out) {
    if (g->pc2_mem) {
        *out = reinterpret_cast<Pc2Work*>(g->pc2_mem);
        return MHD_OK;
    }
    auto* w = new Pc2Work{};
    const size_t N = (size_t)g->d.N;
    if (cudaMalloc(&w->idt, sizeof(double) * N) != cudaSuccess ||
        cudaMalloc(&w->idt32, sizeof(float) * N) != cudaSuccess ||
        cudaMalloc(&w->z32, sizeof(float) * 3 * N) != cudaSuccess) {
        if (w->idt) cudaFree(w->idt);
        if (w->idt32) cudaFree(w->idt32);
        delete w;
        cudaGetLastError();
        return set_error(g, MHD_ERR_OOM, "PC2: workspace allocation failed");
    }
    mhd_status_t st = line_shape<double>(g, &w->shape[0]);
    if (st == MHD_OK) st = line_shape<float>(g, &w->shape[1]);
    if (st == MHD_OK && cudaMemsetAsync(w->z32, 0, sizeof(float) * 3 * N, g->stream) != cudaSuccess)
        st = check_cuda(g, "PC2: workspace clear");
    if (st != MHD_OK) {
        cudaFree(w->idt);
        cudaFree(w->idt32);
        cudaFree(w->z32);
        delete w;
        return st;
    }
    g->pc2_mem = w;
    *out = w;
    return MHD_OK;
}

template <typename T, int MODE>
void launch_line(mhd_grid_s* g, cudaStream_t st, int nc, int restart = 0) {
    const auto* w = reinterpret_cast<const Pc2Work*>(g->pc2_mem);
    const Dims d = g->d;
    const LineShape& s = w->shape[sizeof(T) == 8 ? 0 : 1];
    T *p, *r, *q;
    const T* idt;
    OpTab<T> t;
    if constexpr (sizeof(T) == 8) {
        p = g->p64; r = g->r64; q = g->q64; idt = w->idt; t = g->t64;
    } else {
        p = g->p32; r = g->r32; q = g->q32; idt = w->idt32; t = g->t32;
    }
    // z~: FP64 in the second half of the p double buffer, FP32 in the workspace
    T* z;
    if constexpr (sizeof(T) == 8) z = p + 3 * (size_t)d.N;
    else z = w->z32;
    if (s.seg)
        seg_kernel<T, MODE>(s.seg)<<<s.blocks, 32 * s.warps, s.smem, st>>>(d, nc, s.lanes, t, g->tu.dg, idt, p, r, q, z,
                                                                          g->sc, g->partials, restart);
    else
        k_pc2_line<T, MODE><<<s.blocks, 32 * s.warps, s.smem, st>>>(d, nc, t, g->tu.dg, idt, p, r, q, z, g->sc, g->partials,
                                                                    restart);
}

}  // namespace

void pc2_free(mhd_grid_s* g) {
    if (!g->pc2_mem) return;
    auto* w = reinterpret_cast<Pc2Work*>(g->pc2_mem);
    cudaFree(w->idt);
    cudaFree(w->idt32);
    cudaFree(w->z32);
    delete w;
    g->pc2_mem = nullptr;
}

float* pc2_z32(mhd_grid_s* g) { return reinterpret_cast<Pc2Work*>(g->pc2_mem)->z32; }

// factorise the lines of A~ for the current tables (FP64 and FP32 copies)
mhd_status_t pc2_factor(mhd_grid_s* g) {
    Pc2Work* w = nullptr;
    mhd_status_t st = pc2_workspace(g, &w);
    if (st != MHD_OK) return st;
    const int nl = g->d.nr * g->d.nt;
    k_pc2_factor<<<(nl + kThreads - 1) / kThreads, kThreads, 0, g->stream>>>(g->d, g->t64, w->idt, w->idt32, g->sc);
    return check_cuda(g, "PC2 factorisation");
}

// FP64: after the scaled set-up (x~, r~, rr, bb, done) form z~ = P~^-1 r~, p~ = z~, rho
void pc2_init64(mhd_grid_s* g, int nc) { launch_line<double, kInit>(g, g->stream, nc); }

// FP32 inner solves: after the outer residual replaced r~32, recompute z~32 and rho and decide
// between continuing the recurrence and restarting it
void pc2_reliable32(mhd_grid_s* g, int nc, int restart) { launch_line<float, kReliable>(g, g->stream, nc, restart); }

// the line kernel of one iteration (x / r update, z = P^-1 r, dots)
void pc2_enqueue_line(mhd_grid_s* g, cudaStream_t st, int nc, bool fp32) {
    if (fp32) launch_line<float, kIter>(g, st, nc);
    else launch_line<double, kIter>(g, st, nc);
}

// PC2 workspace, allocated ahead of the first PC2 solve
mhd_status_t pc2_reserve(mhd_grid_s* g) {
    Pc2Work* w = nullptr;
    return pc2_workspace(g, &w);
}

}  // namespace mhd
