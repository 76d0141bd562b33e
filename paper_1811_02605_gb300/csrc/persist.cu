// Point-Jacobi PCG of one system as ONE cooperative launch: every iteration of a solve (FP64) or of
// an inner solve (FP32) runs inside the kernel, with one CTA per SM.
//
// Why: below about a million cells an iteration's kernels are shorter than the launches and the
// last-block reductions between them (32x32x64, FP64: 3.7 us of FP64 instructions in a 20.0 us
// iteration of three kernels). Here the CTAs stay resident, each owns the same cells throughout, and
// the vectors that only their owner touches (x~, r~, q~ and its share of p~) stay in shared memory;
// only p~ is also written to global memory, where the neighbouring CTAs read it.
//
// The stacked vector is cut into groups of V phi-neighbours (16 bytes) in component-major order, CTA b
// owns groups [b C, (b + 1) C) and a thread the groups b C + t + m blockDim. An iteration is the
// Hestenes-Stiefel one of pcg.cu, same expressions and rounding:
//   p = r + beta p                               | exchange 1: p visible to the neighbours
//   q = A~ p, <p, q>                             | exchange 2: sum of <p, q>, alpha
//   r -= alpha q, <r, r>, sum dg r^2             | exchange 3: sums, beta, stop test; x += alpha p
//                                                | before it (FP32) or meanwhile (FP64)
//
// Exchange 1 waits for the CTAs whose groups a chunk's stencil reads, one flag each. Exchanges 2 and 3
// go through CTA 0: each CTA posts its partial sums in its own slot, a warp of CTA 0 reads the slots,
// adds them in slot order, forms the scalars and posts them for all. (All CTAs reading all slots took
// 3.4 us an exchange, an atomic counter with the sums read afterwards 2.6 us, this 2.0 us.) A value
// travels as two 64-bit words, each half value, half tag, so that a word with the awaited tag carries
// its half of the value whatever the order of arrival; no fence is needed for it. Reuse is safe without a
// second buffer: a slot is written again only after an exchange that follows its reading.
// Results are deterministic: the order of every sum is fixed by the partition.
//
// FP64 runs at half a lane per cycle and scheduler on this part: an FP64 operation of every thread costs 64
// cycles a warp, as much as 64 FP32 operations (a dependent addition takes 56 cycles, a division 576). So
// scalars are formed by one warp, two sums share one shuffle tree, and FP32 partials are summed in
// compensated FP32. 512 threads a CTA: 64x64x128 FP64 took 48.5 us an iteration with 256, 43.9 with 384,
// 42.7 with 512, 43.3 with 768.
//
// Every wait is bounded (polls and a %globaltimer budget): a CTA that gives up sets an error word
// that the others see, all return, and the solve reports MHD_ERR_TIMEOUT.
#include <algorithm>
#include <cstdlib>

#include "mhd_internal.cuh"

namespace mhd {

namespace {

constexpr int kPT = 768;                  // most threads per CTA (85 registers each)
constexpr int kPMaxCta = 160;             // capacity of the slots
constexpr size_t kPSmemMax = 220 * 1024;  // dynamic shared memory a CTA may use
constexpr int kPCoef = 6;                 // per row: -ar low, -ar high, -at low, -at high, -ap, unused

constexpr int kPCopies = 8;               // copies of what CTA 0 posts, to spread its readers

struct PersistBuf {
    unsigned int flag[kPMaxCta][8];        // exchange 1, 32 bytes apart
    ulonglong2 slot[3][kPMaxCta];          // <p, q>; <r, r>; sum dg r^2
    ulonglong2 post[2][kPCopies][2];       // alpha; beta (32 bytes apart)
    int err;
};

template <typename T, int V>
struct Vec;
template <>
struct Vec<double, 2> { using type = double2; };
template <>
struct Vec<float, 4> { using type = float4; };
template <>
struct Vec<float, 2> { using type = float2; };

template <typename T, int V>
__device__ __forceinline__ void get(const typename Vec<T, V>::type* p, T (&o)[V]) {
    const auto t = *p;
    o[0] = t.x;
    o[1] = t.y;
    if constexpr (V == 4) {
        o[2] = t.z;
        o[3] = t.w;
    }
}
template <typename T, int V>
__device__ __forceinline__ void put(typename Vec<T, V>::type* p, const T (&o)[V]) {
    typename Vec<T, V>::type t;
    t.x = o[0];
    t.y = o[1];
    if constexpr (V == 4) {
        t.z = o[2];
        t.w = o[3];
    }
    *p = t;
}

// running sum of one thread: plain in FP64, Neumaier-compensated in FP32
template <typename T>
struct Sum;
template <>
struct Sum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ double get() const { return s; }
};
template <>
struct Sum<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x;
        c += (fabsf(s) >= fabsf(x)) ? ((s - t) + x) : ((x - t) + s);
        s = t;
    }
    __device__ __forceinline__ double get() const { return (double)s + (double)c; }
};

__device__ __forceinline__ unsigned long long now() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void slot_store(ulonglong2* s, double v, unsigned int tag) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const unsigned long long lo = (b << 32) | tag, hi = (b & 0xffffffff00000000ull) | tag;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(s), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ void slot_read(const ulonglong2* s, unsigned long long& lo, unsigned long long& hi) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(s) : "memory");
}
__device__ __forceinline__ double slot_value(unsigned long long lo, unsigned long long hi) {
    return __longlong_as_double((long long)((lo >> 32) | (hi & 0xffffffff00000000ull)));
}
// (an FP64 comparison would run on the FP64 pipe)
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ unsigned int flag_load(const unsigned int* f) {
    unsigned int v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
    return v;
}

// one poll round done by a whole warp: true when it has to give up
struct Patience {
    unsigned int polls = 0;
    unsigned long long t0 = 0;
    __device__ __forceinline__ bool spent(PersistBuf* buf, unsigned long long budget_ns) {
        if ((++polls & 255u) != 0u) return false;
        const unsigned long long t = now();
        if (t0 == 0) t0 = t;
        const bool stop = *(volatile int*)&buf->err || polls > (1u << 28) || t - t0 > budget_ns;
        if (!__any_sync(0xffffffffu, stop)) return false;
        if ((threadIdx.x & 31) == 0) atomicExch(&buf->err, 1);
        return true;
    }
};

struct PersistShared {
    double part[2][kPT / 32];   // per-warp partials (FP64)
    float2 part32[kPT / 32];    // per-warp partials of a compensated FP32 sum
    double alpha, beta;
    int state;
};

__device__ __forceinline__ void warp_partial(const Sum<double>& a, PersistShared& sh) {
    double v = a.s;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh.part[0][threadIdx.x >> 5] = v;
}
__device__ __forceinline__ void warp_partial(const Sum<float>& a, PersistShared& sh) {
    float s = a.s, c = a.c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float s2 = __shfl_xor_sync(0xffffffffu, s, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
        const float t = s + s2, b = t - s;   // two-sum: t + e = s + s2 exactly
        c = (c + c2) + ((s - (t - b)) + (s2 - b));
        s = t;
    }
    if ((threadIdx.x & 31) == 0) sh.part32[threadIdx.x >> 5] = make_float2(s, c);
}
// two FP64 sums over the lanes in one tree: lanes 0-15 end with the sum of a, lanes 16-31 of b
__device__ __forceinline__ double lane_sum2(double a, double b) {
    const bool up = (threadIdx.x & 16) != 0;
    double v = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double lane_sum(double s, int width) {
    for (int o = width / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// CTA 0's side of exchanges 2 (K = 1) and 3 (K = 2), run by a warp: sums of all slots in every lane.
// `expect`: slots waited for, one per CTA (one more under fault injection)
template <int K>
__device__ __forceinline__ bool gather(double (&v)[2], PersistBuf* buf, int first, unsigned int tag, int expect,
                                       unsigned long long budget_ns) {
    const int lane = threadIdx.x & 31;
    constexpr int Q = kPMaxCta / 32;
    double got[K][Q];
    Patience wait;
    for (;;) {
        // all loads of a round are issued before any is looked at (a lane without a slot reads the last)
        unsigned long long lo[K][Q], hi[K][Q];
#pragma unroll
        for (int q = 0; q < Q; q++)
#pragma unroll
            for (int k = 0; k < K; k++) slot_read(&buf->slot[first + k][min(32 * q + lane, expect - 1)], lo[k][q], hi[k][q]);
        bool all = true;
#pragma unroll
        for (int q = 0; q < Q; q++)
#pragma unroll
            for (int k = 0; k < K; k++) {
                all = (unsigned int)lo[k][q] == tag && (unsigned int)hi[k][q] == tag && all;
                got[k][q] = 32 * q + lane < (int)gridDim.x ? slot_value(lo[k][q], hi[k][q]) : 0.0;
            }
        if (__all_sync(0xffffffffu, all)) break;
        if (wait.spent(buf, budget_ns)) return false;
    }
    double s[K];
#pragma unroll
    for (int k = 0; k < K; k++) {
        s[k] = got[k][0];
#pragma unroll
        for (int q = 1; q < Q; q++)
            if (32 * q < (int)gridDim.x) s[k] += got[k][q];
    }
    if constexpr (K == 1) {
        v[0] = lane_sum(s[0], 32);
    } else {
        const double u = lane_sum2(s[0], s[1]);
        v[0] = __shfl_sync(0xffffffffu, u, 0);
        v[1] = __shfl_sync(0xffffffffu, u, 16);
    }
    return true;
}

// the other CTAs' side: what CTA 0 posted (value and state)
__device__ __forceinline__ int await_post(double& v, PersistBuf* buf, int which, unsigned int tag,
                                          unsigned long long budget_ns) {
    Patience wait;
    for (;;) {
        unsigned long long lo, hi;
        slot_read(buf->post[which][blockIdx.x % kPCopies], lo, hi);
        if (((unsigned int)lo & ~7u) == tag && (unsigned int)hi == (unsigned int)lo) {
            v = slot_value(lo, hi);
            return (int)((unsigned int)lo & 7u);
        }
        if (wait.spent(buf, budget_ns)) return 6;
    }
}

// SM: x~, r~, q~ and the own p~ in shared memory; otherwise in their global arrays
template <typename T, int V, bool SM>
__global__ void __launch_bounds__(kPT, 1) k_persist(Dims d, unsigned int groups, unsigned int chunk, T* __restrict__ xg,
                                                    T* __restrict__ rg, T* pbuf, T* __restrict__ qg, OpTab<T> t,
                                                    const double* __restrict__ dg, PcgScalars* sc, PersistBuf* buf,
                                                    int expect, unsigned long long budget_ns) {
    using VT = typename Vec<T, V>::type;
    constexpr bool kLateX = sizeof(T) == 8;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ PersistShared sh;
    if (sc->done) return;
    const unsigned int npv = d.np / V, plane = (unsigned int)d.nt * npv, rows_c = (unsigned int)(d.nr * d.nt);
    const unsigned int g0 = blockIdx.x * chunk, g1 = min(g0 + chunk, groups);
    const unsigned int n = g1 > g0 ? g1 - g0 : 0u;
    // FP32: the half of the p double buffer that holds the current p (FP64: par is 0)
    VT* const pg = reinterpret_cast<VT*>(pbuf + (long long)sc->par * 3 * d.N);
    VT* const xgv = reinterpret_cast<VT*>(xg) + g0;
    VT* const rgv = reinterpret_cast<VT*>(rg) + g0;
    // shared memory: [x r q p] of the chunk (SM), then the coefficient rows of the chunk
    VT* const xs = SM ? reinterpret_cast<VT*>(dyn) : xgv;
    VT* const rs = SM ? xs + chunk : rgv;
    VT* const qs = SM ? rs + chunk : reinterpret_cast<VT*>(qg) + g0;
    VT* const ps = SM ? qs + chunk : pg + g0;
    const unsigned int row0 = g0 / npv;
    const unsigned int nrows = n ? (g1 - 1) / npv - row0 + 1 : 0u;
    double* const dgs = reinterpret_cast<double*>(reinterpret_cast<VT*>(dyn) + (SM ? 4 * (size_t)chunk : 0));
    T* const co = reinterpret_cast<T*>(dgs + nrows);
    for (unsigned int q = threadIdx.x; q < nrows; q += blockDim.x) {
        const unsigned int ij = (row0 + q) % rows_c;
        const unsigned int i = ij / d.nt, j = ij - i * d.nt;
        T* c = co + kPCoef * q;
        c[0] = -t.ar[i * d.nt + j];
        c[1] = -t.ar[(i + 1) * d.nt + j];
        c[2] = -t.at[i * (d.nt + 1) + j];
        c[3] = -t.at[i * (d.nt + 1) + j + 1];
        c[4] = -t.ap[ij];
        dgs[q] = dg[ij];
    }
    if (SM)
        for (unsigned int l = threadIdx.x; l < n; l += blockDim.x) {
            xs[l] = xgv[l];
            rs[l] = rgv[l];
            ps[l] = pg[g0 + l];
        }
    // the CTAs that own what this chunk's stencil reads: three ranges of groups, shifted down by a
    // plane, up by a plane, and the chunk with a row on either side
    auto owner = [&](long long g) { return (int)(min(max(g, 0ll), (long long)groups - 1) / chunk); };
    const int dep[6] = {owner((long long)g0 - plane), owner((long long)g1 - 1 - plane), owner((long long)g0 + plane),
                        owner((long long)g1 - 1 + plane), owner((long long)g0 - npv), owner((long long)g1 - 1 + npv)};
    // warp 0 keeps the scalars (CTA 0's the sums too); the other warps read them from shared memory
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    const bool lead = threadIdx.x < 32, master = blockIdx.x == 0;
    double rho = sc->rho, rho_prev = sc->rho_prev, rr = sc->rr, pq = sc->pq;
    const double bound = sc->tol * sqrt(sc->bb), near = bound * bound * (1.0 + 1e-12);
    const int max_iter = sc->max_iter, total0 = sc->total_iter - sc->iter;
    int iter = sc->iter;
    unsigned int tag = 0;
    if (threadIdx.x == 0) {
        sh.alpha = 0.0;
        sh.beta = sc->beta;
        sh.state = 0;
    }
    __syncthreads();
    for (;;) {
        tag += 8;   // the low 3 bits carry a state
        const T be = (T)sh.beta;
#pragma unroll 4
        for (unsigned int l = threadIdx.x; l < n; l += blockDim.x) {
            T a[V], b[V];
            get<T, V>(rs + l, a);
            get<T, V>(ps + l, b);
#pragma unroll
            for (int e = 0; e < V; e++) b[e] = fma(be, b[e], a[e]);
            if (SM) put<T, V>(ps + l, b);
            put<T, V>(pg + g0 + l, b);
        }
        __syncthreads();
        if (lead) {
            // exchange 1: release the own p, wait for the neighbours' flags, acquire theirs
            __threadfence();
            if (lane == 0) *(volatile unsigned int*)buf->flag[blockIdx.x] = tag;
            bool ok = true;
            if (n) {
                Patience wait;
                for (;;) {
                    bool all = true;
#pragma unroll
                    for (int q = 0; q < 3; q++)
                        for (int c = dep[2 * q] + lane; c <= dep[2 * q + 1]; c += 32)
                            all = flag_load(buf->flag[c]) == tag && all;
                    if (__all_sync(0xffffffffu, all)) break;
                    if (wait.spent(buf, budget_ns)) { ok = false; break; }
                }
            }
            __threadfence();
            if (!ok && lane == 0) sh.state = 6;
        }
        __syncthreads();
        if (sh.state) break;
        Sum<T> acc;
#pragma unroll 2
        for (unsigned int l = threadIdx.x; l < n; l += blockDim.x) {
            const unsigned int g = g0 + l, row = g / npv, kv = g - row * npv;
            const unsigned int ij = row % rows_c, i = ij / d.nt, j = ij - i * d.nt;
            const T* c = co + kPCoef * (row - row0);
            // own groups from shared memory, the others from the global copy; at a wall the cell
            // itself, with a coefficient that is exactly 0
            auto at = [&](unsigned int gn) -> const VT* {
                if (!SM) return pg + gn;
                const unsigned int ln = gn - g0;
                return ln < n ? ps + ln : pg + gn;
            };
            const VT *pim = at(i > 0 ? g - plane : g), *pip = at(i + 1 < (unsigned)d.nr ? g + plane : g);
            const VT *pjm = at(j > 0 ? g - npv : g), *pjp = at(j + 1 < (unsigned)d.nt ? g + npv : g);
            const VT *pkm = at(kv > 0 ? g - 1 : g + npv - 1), *pkp = at(kv + 1 < npv ? g + 1 : g + 1 - npv);
            T v[V], a[V], b[V], e0[V], e1[V], o[V];
            get<T, V>(pim, a);
            get<T, V>(pip, b);
            get<T, V>(pjm, e0);
            get<T, V>(pjp, e1);
            const T left0 = reinterpret_cast<const T*>(pkm)[V - 1], right1 = reinterpret_cast<const T*>(pkp)[0];
            get<T, V>(ps + l, v);
            const T cim = c[0], cip = c[1], cjm = c[2], cjp = c[3], cp = c[4];
#pragma unroll
            for (int e = 0; e < V; e++) {
                const T left = (e == 0) ? left0 : v[e - 1];
                const T right = (e == V - 1) ? right1 : v[e + 1];
                o[e] = fma(cp, left + right, v[e]);
                o[e] = fma(cim, a[e], o[e]);
                o[e] = fma(cip, b[e], o[e]);
                o[e] = fma(cjm, e0[e], o[e]);
                o[e] = fma(cjp, e1[e], o[e]);
                if constexpr (sizeof(T) == 8) acc.s = fma(v[e], o[e], acc.s);
                else acc.add(v[e] * o[e]);
            }
            put<T, V>(qs + l, o);
        }
        warp_partial(acc, sh);
        __syncthreads();
        if (lead) {
            // exchange 2
            double v[2] = {0.0, 0.0}, al64 = 0.0;
            if (lane < nw) {
                if constexpr (sizeof(T) == 8) v[0] = sh.part[0][lane];
                else v[0] = (double)sh.part32[lane].x + (double)sh.part32[lane].y;
            }
            v[0] = lane_sum(v[0], 32);
            if (lane == 0) slot_store(&buf->slot[0][blockIdx.x], v[0], tag);
            int state;
            if (master) {
                state = gather<1>(v, buf, 0, tag, expect, budget_ns) ? 0 : 6;
                pq = v[0];
                if (!state && !finite_bits(pq)) state = 3;
                if (!state && !(pq > 0.0)) state = 4;
                al64 = rho / pq;
                if (state != 6 && lane < kPCopies) slot_store(buf->post[0][lane], al64, tag | state);
            } else {
                state = await_post(al64, buf, 0, tag, budget_ns);
            }
            if (lane == 0) {
                sh.state = state;
                sh.alpha = al64;
            }
        }
        __syncthreads();
        if (sh.state) break;
        const T al = (T)sh.alpha;
        auto add_x = [&](unsigned int l) {
            T xv[V], pv[V];
            get<T, V>(xs + l, xv);
            get<T, V>(ps + l, pv);
#pragma unroll
            for (int e = 0; e < V; e++) xv[e] = fma(al, pv[e], xv[e]);
            put<T, V>(xs + l, xv);
        };
        Sum<T> a_rho;
        Sum<double> a_rr;
#pragma unroll 2
        for (unsigned int l = threadIdx.x; l < n; l += blockDim.x) {
            T rv[V], qv[V];
            get<T, V>(rs + l, rv);
            get<T, V>(qs + l, qv);
            if constexpr (!kLateX) add_x(l);
            T cell = T(0);
#pragma unroll
            for (int e = 0; e < V; e++) {
                rv[e] = fma(-al, qv[e], rv[e]);
                cell = fma(rv[e], rv[e], cell);
            }
            put<T, V>(rs + l, rv);
            a_rho.add(cell);
            a_rr.s = fma(dgs[(g0 + l) / npv - row0], (double)cell, a_rr.s);
        }
        if constexpr (sizeof(T) == 8) {
            const double u = lane_sum2(a_rho.s, a_rr.s);
            if ((lane & 15) == 0) sh.part[lane >> 4][threadIdx.x >> 5] = u;
        } else {
            warp_partial(a_rho, sh);
            const double u = lane_sum(a_rr.s, 32);
            if (lane == 0) sh.part[1][threadIdx.x >> 5] = u;
        }
        __syncthreads();
        if (lead) {
            // exchange 3
            double v[2] = {0.0, 0.0}, be64 = 0.0;
            if (lane < nw) {
                if constexpr (sizeof(T) == 8) v[0] = sh.part[0][lane];
                else v[0] = (double)sh.part32[lane].x + (double)sh.part32[lane].y;
                v[1] = sh.part[1][lane];
            }
            const double u = lane_sum2(v[0], v[1]);
            if ((lane & 15) == 0) slot_store(&buf->slot[1 + (lane >> 4)][blockIdx.x], u, tag);
            int state;
            iter++;
            if (master) {
                state = gather<2>(v, buf, 1, tag, expect, budget_ns) ? 0 : 6;
                rho_prev = rho;
                rho = v[0];
                rr = v[1];
                be64 = rho / rho_prev;
                if (!state && (!finite_bits(rr) || !finite_bits(rho))) state = 3;
                // the stop test sqrt(rr) <= tol sqrt(bb); the square root only where it can decide
                if (!state && rr <= near && sqrt(rr) <= bound) state = 1;
                if (!state && iter >= max_iter) state = 2;
                if (state != 6 && lane < kPCopies) slot_store(buf->post[1][lane], be64, tag | state);
            } else {
                state = await_post(be64, buf, 1, tag, budget_ns);
            }
            if (lane == 0) {
                sh.state = state;
                sh.beta = be64;
            }
        } else if (kLateX && (threadIdx.x & 96)) {
            // meanwhile x += alpha p, by the warps that share no scheduler with the first one, whose FP64 sums
            // would queue behind theirs (warps are dealt to the four schedulers in turn). us per iteration:
            // 32x32x64 13.5 -> 13.1, 48x48x96 23.5 -> 22.7, 61x47x118 30.7 -> 29.8; in FP32 it gave nothing.
            const unsigned int w = threadIdx.x >> 5, helpers = nw - (nw + 3) / 4, at = w - 1 - w / 4;
#pragma unroll 4
            for (unsigned int l = 32 * at + lane; l < n; l += 32 * helpers) add_x(l);
        }
        __syncthreads();
        if (sh.state) break;
    }
    if (SM)
        for (unsigned int l = threadIdx.x; l < n; l += blockDim.x) xgv[l] = xs[l];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->iter = iter;
        sc->total_iter = total0 + iter;
        sc->rho_prev = rho_prev;
        sc->rho = rho;
        sc->beta = sh.beta;
        sc->rr = rr;
        sc->pq = pq;
        sc->alpha = sh.alpha;
        sc->ax = 0.0;   // x is complete
        sc->done = sh.state;
    }
}

template <typename T, int V>
constexpr size_t smem_bytes(unsigned int chunk, unsigned int rows, bool sm) {
    return (sm ? 4 * (size_t)chunk * sizeof(typename Vec<T, V>::type) : 0) + rows * (sizeof(double) + kPCoef * sizeof(T));
}

struct Shape {
    unsigned int groups, chunk, rows;
    int threads;
};

Shape shape_of(const mhd_grid_s* g, int nc, int V, bool sm) {
    Shape s;
    s.groups = (unsigned int)(nc * g->d.N / V);
    const unsigned int nb = g->num_sms;
    s.chunk = ((s.groups + nb - 1) / nb + 3u) & ~3u;   // 64-byte multiples
    s.rows = s.chunk / (g->d.np / V) + 2;
    const unsigned int most = sm ? 512 : kPT;
    const unsigned int m = (s.chunk + most - 1) / most;
    s.threads = std::max<int>((((s.chunk + m - 1) / m + 31) / 32) * 32, 128);
    return s;
}

// refused: the launch needs more SMs than this context may use (a green context, a partition); nothing has run
template <typename T, int V, bool SM>
mhd_status_t launch(mhd_grid_s* g, const Shape& s, T* x, T* r, T* p, T* q, const OpTab<T>& t, bool* refused) {
    const size_t bytes = smem_bytes<T, V>(s.chunk, s.rows, SM);
    if (cudaFuncSetAttribute(k_persist<T, V, SM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPSmemMax) != cudaSuccess)
        return check_cuda(g, "persistent PCG: shared memory");
    PersistBuf* buf = reinterpret_cast<PersistBuf*>(g->persist_buf);
    int expect = g->num_sms;
    unsigned long long budget = 20ull * 1000 * 1000 * 1000;
    // Fault injection for tests (no GPU fault): wait for one arrival that never comes, for so long
    if (const char* f = std::getenv("MHD_FAULT_BARRIER_MS")) {
        const long ms = std::strtol(f, nullptr, 10);
        if (ms > 0) {
            expect++;
            budget = (unsigned long long)ms * 1000 * 1000;
        }
    }
    cudaMemsetAsync(buf, 0, sizeof(PersistBuf), g->stream);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g->num_sms);
    cfg.blockDim = dim3(s.threads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = g->stream;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeCooperative;
    a[0].val.cooperative = 1;
    cfg.attrs = a;
    cfg.numAttrs = 1;
    // (the environment variable stands in for the refusal in tests, on the host)
    const cudaError_t e = std::getenv("MHD_FAULT_COOP_LAUNCH")
                              ? cudaErrorCooperativeLaunchTooLarge
                              : cudaLaunchKernelEx(&cfg, k_persist<T, V, SM>, g->d, s.groups, s.chunk, x, r, p, q, t,
                                                   (const double*)g->tu.dg, g->sc, buf, expect, budget);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        *refused = true;
        return MHD_OK;
    }
    return check_cuda(g, "persistent PCG launch");
}

}  // namespace

size_t persist_buf_bytes() { return sizeof(PersistBuf); }

// 1: the chunks fit shared memory; 2: only with the vectors in global memory; 0: not available
int persist_mode(const mhd_grid_s* g, bool fp32, int nc) {
    if (g->num_sms + 1 > kPMaxCta) return 0;
    const int V = fp32 ? (g->d.np % 4 == 0 ? 4 : 2) : 2;
    const Shape s = shape_of(g, nc, V, true);
    const size_t item = fp32 ? 4 * V : 8 * V, coef = s.rows * (8 + (size_t)kPCoef * (fp32 ? 4 : 8));
    if (4 * (size_t)s.chunk * item + coef <= kPSmemMax) return 1;
    return coef <= kPSmemMax ? 2 : 0;
}

// the iterations of a solve (FP64) or of an inner solve (FP32), after its set-up kernel; done, the
// counts and the final scalars are in g->sc, x~ complete. refused: the kernel cannot run here and has not touched
// anything; the caller takes another form
mhd_status_t persist_iterate(mhd_grid_s* g, bool fp32, int nc, bool* refused) {
    const int mode = persist_mode(g, fp32, nc);
    *refused = !mode;
    if (!mode) return MHD_OK;
    const int slot = prof_begin(g, g->stream, fp32 ? MHD_KERNEL_PERSIST32 : MHD_KERNEL_PERSIST64);
    mhd_status_t st;
    if (!fp32) {
        const Shape s = shape_of(g, nc, 2, mode == 1);
        st = mode == 1 ? launch<double, 2, true>(g, s, g->x64, g->r64, g->p64, g->q64, g->t64, refused)
                       : launch<double, 2, false>(g, s, g->x64, g->r64, g->p64, g->q64, g->t64, refused);
    } else if (g->d.np % 4 == 0) {
        const Shape s = shape_of(g, nc, 4, mode == 1);
        st = mode == 1 ? launch<float, 4, true>(g, s, g->x32, g->r32, g->p32, g->q32, g->t32, refused)
                       : launch<float, 4, false>(g, s, g->x32, g->r32, g->p32, g->q32, g->t32, refused);
    } else {
        const Shape s = shape_of(g, nc, 2, mode == 1);
        st = mode == 1 ? launch<float, 2, true>(g, s, g->x32, g->r32, g->p32, g->q32, g->t32, refused)
                       : launch<float, 2, false>(g, s, g->x32, g->r32, g->p32, g->q32, g->t32, refused);
    }
    prof_end(g, g->stream, slot);
    return st;
}

}  // namespace mhd
