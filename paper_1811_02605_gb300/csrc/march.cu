// FP32 single-reduction CG iteration of the mixed-precision inner solve as ONE plane-marching kernel.
//
// The iteration is the single-reduction pair of pcg.cu (k_cgr32 + k_cgu32), whose residual kernel reads
// r~ a second time only because A~ r~ needs the neighbours' new r~. Here a CTA carries its tile two
// cells further than what it writes, so the neighbours' new r~ are its own recomputed values (the same
// expressions in the same order, hence the same bits as their owner's) and the whole iteration is one pass:
//   p = r + beta p_old, q = A~ p, r' = r - alpha q, x += alpha p + ax p_old (every second iteration),
//   gamma = <r', r'>, w = <r', q>, delta = <r', A~ r'>, sum dg r'^2 -> the next alpha, beta, stop test.
// It moves r and p in, r' and p out, and half of x in and out: 5 vector passes (60 B per cell) instead of 6.
//
// What bounded the pair was not those bytes: every value went to its thread seven times, mostly through
// L2 (13 TB/s of L2 reads for 2.7 to 5 TB/s of HBM traffic). A CTA here owns a column of one component, up to 20
// theta rows by 14 groups of four phi cells, and marches along r. A thread owns three adjacent rows of one
// group: its r neighbours and part of its theta neighbours are its registers, the phi neighbours come by
// shuffles within half a warp (16 lanes, 14 groups and a halo group on either side), and only the outer two of its
// rows go through shared memory. What it reads from memory is copied a plane ahead (cp.async) into a slot of
// its own, so no barrier orders it. The halo (24 x 16) / (20 x 14) is read from L2; neighbouring columns
// march in step, so HBM sees it once.
//
// us per iteration, the pair / this: 128x128x256 86.6 / 62.7, 192x192x384 247 / 162, 256x256x512 542 / 376 (5
// passes at 6.8 TB/s are 296). What bounds it now is the latency of the steps (3 CTAs of 128 threads per SM
// at 152 registers; issue slots half used, 5.3 TB/s of HBM by the 60 B a cell). Other shapes at 192x192x384: one row a thread 242
// (bound by instructions and shared-memory wavefronts), 2 rows 164 to 175, 4 rows 167 to 187, 5 rows 217.
//
// The sums are FP32 over the thread's 12 cells of a plane (<r', q>: 24 of two) and compensated beyond; the weights dg of the stop norm
// have 48 bits and each product's rounding is kept, as FP64 at this rate would take longer than all the rest (with
// dg and the products rounded to FP32 an iteration at 256x256x512 took 0.9% less).
//
// One block barrier a plane: in step n a thread writes p of plane n and r' of plane n-1 to shared memory and
// reads the neighbours' p of plane n-1 and r' of plane n-2, written in the step before.
#include <algorithm>

#include "mhd_internal.cuh"
#include "reduce.cuh"

namespace mhd {

namespace {

constexpr int kRT = 3;               // theta rows of a thread
constexpr int kTR = 8;               // thread rows of a CTA
constexpr int kLanes = 16;           // lanes of a row: half a warp
constexpr int kMT = kTR * kLanes;    // 128 threads
constexpr int kCtas = 3;             // CTAs per SM
constexpr int kRows = kTR * kRT;
constexpr int kTJ = kRows - 4;       // most theta rows a CTA writes
constexpr int kTG = kLanes - 2;      // most groups of four phi cells a CTA writes in a row

struct Smem {
    float4 in[2][3][kRT][kMT];               // r, p_old, x of the thread's own groups, two planes
    float4 p[2][kTR][2][kLanes];             // first and last row's p of each thread row, two planes
    float4 r[2][kTR][2][kLanes];             // the same of r'
    float4 co[4][kRows][2];                  // coefficients of four planes, by row
};

__device__ __forceinline__ void copy16(void* dst, const void* src, bool ok) {
    const unsigned int d = (unsigned int)__cvta_generic_to_shared(dst);
    const int bytes = ok ? 16 : 0;   // 0: the destination is filled with zeros
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ float4 fma4(float a, float4 b, float4 c) {
    return make_float4(fmaf(a, b.x, c.x), fmaf(a, b.y, c.y), fmaf(a, b.z, c.z), fmaf(a, b.w, c.w));
}

// o = u - sum c_nb u_nb at the four cells of a group (scaled operator, unit diagonal)
__device__ __forceinline__ float4 stencil4(float4 u, float left, float right, float4 im, float4 ip, float4 jm, float4 jp,
                                           float4 c0, float cp) {
    float4 o;
    o.x = fmaf(-cp, left + u.y, u.x);
    o.y = fmaf(-cp, u.x + u.z, u.y);
    o.z = fmaf(-cp, u.y + u.w, u.z);
    o.w = fmaf(-cp, u.z + right, u.w);
    o = fma4(-c0.x, im, o);
    o = fma4(-c0.y, ip, o);
    o = fma4(-c0.z, jm, o);
    return fma4(-c0.w, jp, o);
}

// compensated FP32 sum (two-sum)
struct Sum2 {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {
        const float t = s + x, b = t - s;
        c += (s - (t - b)) + (x - b);
        s = t;
    }
    // of a product g (hi + lo): its rounding and the low part go to the correction
    __device__ __forceinline__ void add_product(float g, float hi, float lo) {
        const float x = g * hi, t = s + x, b = t - s;
        c += fmaf(g, lo, fmaf(g, hi, -x)) + ((s - (t - b)) + (x - b));
        s = t;
    }
    __device__ __forceinline__ double get() const { return (double)s + (double)c; }
};

struct Tiling {
    int tj, tg;              // theta rows and phi groups a CTA writes
    int njt, nkt, cols;      // columns: components x njt x nkt
    int full;                // columns marched over all planes by one unit
    int slabs;               // the others are cut into this many units
    int units;
};

__global__ void __launch_bounds__(kMT, kCtas) k_march32(Dims d, Tiling T, float* __restrict__ x, float* __restrict__ ra,
                                                    float* __restrict__ rb, float* __restrict__ pbuf,
                                                    const float4* __restrict__ tab, PcgScalars* sc,
                                                    double* __restrict__ partials) {
    if (sc->done) return;
    extern __shared__ __align__(16) unsigned char dyn[];
    Smem& S = *reinterpret_cast<Smem*>(dyn);
    const int par = sc->par;
    const float* __restrict__ rin = par ? rb : ra;
    float* __restrict__ rout = par ? ra : rb;
    const float* __restrict__ pin = pbuf + (long long)par * 3 * d.N;
    float* __restrict__ pout = pbuf + (long long)(1 - par) * 3 * d.N;
    float beta = (float)sc->beta, al = (float)sc->alpha, axp = (float)sc->ax;
    int pair = (sc->ax != 0.0);
    // keep the converted scalars in registers (left alone, the compiler converts them again in every step, on the
    // FP64 pipe)
    asm volatile("" : "+f"(beta), "+f"(al), "+f"(axp), "+r"(pair));
    const int tid = threadIdx.x, tr = tid / kLanes, lane = tid % kLanes;   // lane 0 is the halo group
    const int npg = d.np / 4, plane = d.nt * d.np;
    float4* const in = &S.in[0][0][0][tid];
    Sum2 s_g, s_w, s_d, s_rr;
    for (int u = blockIdx.x; u < T.units; u += gridDim.x) {
        // unit -> column and planes [i0, i1)
        int col = u, i0 = 0, i1 = d.nr;
        if (u >= T.full) {
            const int rest = T.cols - T.full, v = u - T.full, sl = v / rest, len = (d.nr + T.slabs - 1) / T.slabs;
            col = T.full + v - sl * rest;
            i0 = sl * len;
            i1 = min(i0 + len, d.nr);
        }
        const int kt = col % T.nkt, jt = (col / T.nkt) % T.njt, comp = col / (T.nkt * T.njt);
        const int j0 = jt * T.tj, g0 = kt * T.tg;
        const int rows = min(T.tj, d.nt - j0), groups = min(T.tg, npg - g0);
        const int jb = j0 - 2 + tr * kRT;   // theta row of the thread's first row (tile row 0 is j0 - 2)
        int g = g0 - 1 + lane;              // phi group, periodic
        g = g < 0 ? g + npg : (g >= npg ? g - npg : g);
        const bool lane_in = lane < groups + 2, lane_out = lane >= 1 && lane <= groups;
        // per row: inside the tile and the grid (read), written by this CTA
        bool rd[kRT], wr[kRT];
#pragma unroll
        for (int a = 0; a < kRT; a++) {
            const int row = tr * kRT + a, j = jb + a;
            rd[a] = lane_in && row < rows + 4 && j >= 0 && j < d.nt;
            wr[a] = rd[a] && lane_out && row >= 2 && row < rows + 2;
        }
        const long long cell = (long long)comp * d.N + (long long)jb * d.np + 4 * (lane_in ? g : 0);
        const int steps = i1 - i0 + 4;      // step n forms p of plane i0 - 2 + n
        auto fetch = [&](int n, int slot) {
            if (n < steps) {
                const int s = i0 - 2 + n;
                const bool in_r = (unsigned)s < (unsigned)d.nr, xs = pair && n >= 2 && n < steps - 2;
                const long long o = cell + (long long)s * plane;
#pragma unroll
                for (int a = 0; a < kRT; a++) {
                    const bool ok = rd[a] && in_r;
                    const long long oa = ok ? o + a * d.np : 0;
                    copy16(in + ((slot * 3 + 0) * kRT + a) * kMT, rin + oa, ok);
                    copy16(in + ((slot * 3 + 1) * kRT + a) * kMT, pin + oa, ok);
                    if (xs && wr[a]) copy16(in + ((slot * 3 + 2) * kRT + a) * kMT, x + oa, true);
                }
                // a row of the coefficient table, clamped outside the grid (what is formed there meets
                // coefficients that are exactly 0)
                if (tid < 2 * kRows) {
                    const int jc = min(max(j0 - 2 + tid / 2, 0), d.nt - 1), sc_ = min(max(s, 0), d.nr - 1);
                    copy16(&S.co[n & 3][0][0] + tid, tab + 2 * (sc_ * d.nt + jc) + (tid & 1), true);
                }
            }
            copy_commit();
        };
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        // before step n: p of planes n-1 and n-2, r of n-1, r' of n-2 and n-3
        float4 p1[kRT], p2[kRT], rk[kRT], r2[kRT], r3[kRT];
#pragma unroll
        for (int a = 0; a < kRT; a++) p1[a] = p2[a] = rk[a] = r2[a] = r3[a] = z4;
        const int tu = tr > 0 ? tr - 1 : 0, td = tr < kTR - 1 ? tr + 1 : tr;   // thread rows above and below
        fetch(0, 0);
        for (int n0 = 0; n0 < steps; n0 += 2) {
            float pw = 0.f;   // plain over the thread's 24 cells of two planes, then compensated
#pragma unroll
            for (int t = 0; t < 2; t++) {
                float pg = 0.f, pd = 0.f;   // over the 12 of one
                const int n = n0 + t;
                fetch(n + 1, t ^ 1);
                copy_wait<1>();
                const int b0 = t, b1 = t ^ 1;
                const long long o = cell + (long long)(i0 - 2 + n) * plane;
                const bool wp = n >= 2 && n < steps - 2, wr1 = n >= 3 && n < steps - 1, wd = n >= 4 && n < steps;
                float4 p0[kRT];
#pragma unroll
                for (int a = 0; a < kRT; a++) {
                    const float4 rv = in[((t * 3 + 0) * kRT + a) * kMT], pv = in[((t * 3 + 1) * kRT + a) * kMT];
                    p0[a] = fma4(beta, pv, rv);
                    if (wp && wr[a]) {
                        *reinterpret_cast<float4*>(pout + o + a * d.np) = p0[a];
                        if (pair)
                            *reinterpret_cast<float4*>(x + o + a * d.np) =
                                fma4(al, p0[a], fma4(axp, pv, in[((t * 3 + 2) * kRT + a) * kMT]));
                    }
                }
                S.p[b0][tr][0][lane] = p0[0];
                S.p[b0][tr][1][lane] = p0[kRT - 1];
                // q and r' of plane n - 1 (of use from n = 2 on)
                float4 r1[kRT];
                {
                    const float4 above = S.p[b1][tu][1][lane], below = S.p[b1][td][0][lane];
#pragma unroll
                    for (int a = 0; a < kRT; a++) {
                        const float4 c0 = S.co[(n + 3) & 3][tr * kRT + a][0];
                        const float4 c1 = S.co[(n + 3) & 3][tr * kRT + a][1];
                        const float left = __shfl_up_sync(0xffffffffu, p1[a].w, 1, kLanes);
                        const float right = __shfl_down_sync(0xffffffffu, p1[a].x, 1, kLanes);
                        const float4 q = stencil4(p1[a], left, right, p2[a], p0[a], a > 0 ? p1[a > 0 ? a - 1 : 0] : above,
                                                  a < kRT - 1 ? p1[a < kRT - 1 ? a + 1 : a] : below, c0, c1.x);
                        // the residual at hand is plane n - 1's: it is overwritten by the next one below
                        r1[a] = fma4(-al, q, rk[a]);
                        if (wr1 && wr[a]) {
                            *reinterpret_cast<float4*>(rout + (o - plane) + a * d.np) = r1[a];
                            const float gg = fmaf(r1[a].x, r1[a].x, fmaf(r1[a].y, r1[a].y, fmaf(r1[a].z, r1[a].z, r1[a].w * r1[a].w)));
                            pg += gg;
                            // the stop norm's weight has 48 bits: the product is exact but for the low part's rounding
                            s_rr.add_product(gg, c1.y, c1.z);
                            pw = fmaf(r1[a].x, q.x, fmaf(r1[a].y, q.y, fmaf(r1[a].z, q.z, fmaf(r1[a].w, q.w, pw))));
                        }
                    }
                }
                S.r[b1][tr][0][lane] = r1[0];
                S.r[b1][tr][1][lane] = r1[kRT - 1];
                // A~ r' of plane n - 2
                {
                    const float4 above = S.r[b0][tu][1][lane], below = S.r[b0][td][0][lane];
#pragma unroll
                    for (int a = 0; a < kRT; a++) {
                        const float4 c0 = S.co[(n + 2) & 3][tr * kRT + a][0];
                        const float cp = S.co[(n + 2) & 3][tr * kRT + a][1].x;
                        const float left = __shfl_up_sync(0xffffffffu, r2[a].w, 1, kLanes);
                        const float right = __shfl_down_sync(0xffffffffu, r2[a].x, 1, kLanes);
                        const float4 q = stencil4(r2[a], left, right, r3[a], r1[a], a > 0 ? r2[a > 0 ? a - 1 : 0] : above,
                                                  a < kRT - 1 ? r2[a < kRT - 1 ? a + 1 : a] : below, c0, cp);
                        if (wd && wr[a])
                            pd = fmaf(r2[a].x, q.x, fmaf(r2[a].y, q.y, fmaf(r2[a].z, q.z, fmaf(r2[a].w, q.w, pd))));
                    }
                }
#pragma unroll
                for (int a = 0; a < kRT; a++) {
                    p2[a] = p1[a];
                    p1[a] = p0[a];
                    r3[a] = r2[a];
                    r2[a] = r1[a];
                    rk[a] = in[((t * 3 + 0) * kRT + a) * kMT];
                }
                s_g.add(pg);
                s_d.add(pd);
                __syncthreads();
            }
            s_w.add(pw);
        }
    }
    copy_wait<0>();
    double val[4] = {s_g.get(), s_w.get(), s_d.get(), s_rr.get()}, out[4];
    if (reduce_last<4>(val, partials, &sc->count, out) && threadIdx.x == 0) {
        const double gam = out[0], del = out[2], rr = ldexp(out[3], __float_as_int(tab[1].w));
        sc->wp = out[1];
        sc->par = 1 - par;
        sc->ax = pair ? 0.0 : sc->alpha;   // pending: alpha p, p in the new current half
        sc->iter += 1;
        sc->total_iter += 1;
        single_reduction_finish(sc, gam, del, rr);
    }
}

// Tile sizes and units. The cost of a choice is what the slowest CTA marches: rounds of units times a unit's
// planes and 6 more (halo and pipeline fill). Considered: the smallest tile counts that fit and up to three
// more, all columns cut into slabs, or as many rounds of whole columns as fill every CTA and the rest in slabs.
// A row of a tile is an even number of groups, so that rows start on 32-byte sectors (256x256x512: 13 groups
// 415 us an iteration, 12 groups 368 us, 11 groups 443 us, 10 groups 398 us); multiples of 64 bytes win a tie.
Tiling tiling(const mhd_grid_s* g, int nc) {
    const int npg = g->d.np / 4, nt = g->d.nt, nr = g->d.nr, ctas = kCtas * g->num_sms;
    Tiling best{};
    long long best_cost = -1;
    const int nj0 = (nt + kTJ - 1) / kTJ, nk0 = (npg + kTG - 1) / kTG;
    for (int nk = nk0; nk <= nk0 + 3; nk++)
        for (int nj = nj0; nj <= nj0 + 3; nj++) {
            Tiling T;
            T.tg = std::min(kTG, ((npg + nk - 1) / nk + 1) & ~1);
            T.tj = (nt + nj - 1) / nj;
            T.nkt = (npg + T.tg - 1) / T.tg;
            T.njt = (nt + T.tj - 1) / T.tj;
            T.cols = nc * T.njt * T.nkt;
            auto consider = [&](int full, int slabs) {
                const int rest = T.cols - full, len = (nr + slabs - 1) / slabs;
                slabs = (nr + len - 1) / len;
                const long long rounds = ((long long)rest * slabs + ctas - 1) / ctas;
                const long long cost = 2 * ((full / ctas) * (long long)(nr + 6) + rounds * (len + 6)) + (T.tg % 4 != 0);
                if (best_cost < 0 || cost < best_cost) {
                    best_cost = cost;
                    best = T;
                    best.full = full;
                    best.slabs = slabs;
                    best.units = full + rest * slabs;
                }
            };
            const int full = T.cols / ctas * ctas;
            for (int s = 1; s <= nr && s <= 64; s++) {
                consider(0, s);
                if (full && full < T.cols) consider(full, s);
            }
        }
    return best;
}

}  // namespace

bool march32_ok(const mhd_grid_s* g) { return g->d.np % 4 == 0; }

void enqueue_march32(mhd_grid_s* g, cudaStream_t st, int nc) {
    const Tiling T = tiling(g, nc);
    cudaFuncSetAttribute(k_march32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
    const int slot = prof_begin(g, st, MHD_KERNEL_MARCH32);
    k_march32<<<std::min(T.units, kCtas * g->num_sms), kMT, sizeof(Smem), st>>>(
        g->d, T, g->x32, g->r32, g->q32, g->p32, reinterpret_cast<const float4*>(g->row32), g->sc, g->partials);
    prof_end(g, st, slot);
}

}  // namespace mhd
