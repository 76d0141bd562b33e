// Explicit parts of the zero-beta step (Eq. 1; Sec. 2.2 explicit predictor-corrector
// upwinding), all FP64, a warp or a part of one per row of output elements:
//   - step coefficients: dt from the flow CFL, C_w, the semi-implicit coefficient (Sec. 2.1)
//   - J = curl_h B on edges (Stokes on the dual faces around each edge)
//   - momentum force b = rho V dt (-(v.grad)v + J x B / rho)
//   - E = -v x B + eta J at cell centres, averaged to edges; B <- B - dt curl_h E (Stokes)
// Pole and boundary rules:
//   - B_theta at a cell centre in the two polar rings is the mean of the non-polar face and of
//     the pole value along the cell's meridian (first phi harmonic of the face ring next to the
//     pole, divided by cos(dth)).
//   - The polar radial edge carries one value: the cap circulation of B_phi for J, the ring
//     mean of the polar cells for E.
//   - The polar phi edges have zero length; their J is 0 and left out of the centre average.
//   - Ghost tangential B beyond r0 and r1 equals the first interior value, at mirrored radii.
//   - Advection: Dirichlet mirror ghost (-u) at r0, zero gradient at r1, no flux from the pole.
//   - Tangential E is 0 on r0 (line-tied); on r1 it is the mean of the two interior cells.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <utility>

#include "mhd_internal.cuh"
#include "reduce.cuh"

namespace mhd {

namespace {


// FP64 runs at 2 multiply-adds per clock and SM on this part (64 cycles a warp instruction and scheduler), so
// these kernels are bound by their count of FP64 instructions; integer work, loads and address arithmetic are
// free beside it. Hence: a row (i, j) of np elements, or a part of it, to a group of lanes, so that whatever depends on the row alone is
// formed once a row; the means are kept as plain sums (B_c doubled, J_c and the edge E by powers of two, which
// scale exactly) and the factor goes into a row constant; signs and maxima are integer tests; the upwind
// difference is |u_d| / h (u - u_upwind), one form for both signs. Coefficients, force, induction with
// resistivity and diagnostics of a 256x256x512 grid: 21.3 -> 13.0 ms, at about 190 FP64 instructions a cell and 82 to
// 89% of the pipe.

// How rows of np elements are dealt to lanes: `lanes` of a warp (a power of two) take a row, or one of its `parts` of
// len elements each.
struct RowMap {
    int lanes, parts, len;
    // WHOLE: a warp takes whole rows, known at compile time (k_current takes 8 registers less then, so a CTA per SM
    // more: 740 us at 256x256x512, else 790)
    template <bool WHOLE>
    __host__ __device__ RowMap fixed(int np) const {
        return WHOLE ? RowMap{32, 1, np} : *this;
    }
};

// a thread's place: rows (or parts of rows) w, w + stride, ...; lane is its lane within the row
struct Lanes {
    unsigned int first, stride, mask;
    int lane, n;
    __device__ __forceinline__ explicit Lanes(const RowMap& M) : n(M.lanes) {
        const unsigned int sh = 31 - __clz(M.lanes);
        first = (blockIdx.x * kThreads + threadIdx.x) >> sh;
        stride = (gridDim.x * kThreads) >> sh;
        lane = threadIdx.x & (M.lanes - 1);
        mask = (0xffffffffu >> (32 - M.lanes)) << (threadIdx.x & 31 & ~(M.lanes - 1));
    }
    // sum over the row's lanes, in all of them
    __device__ __forceinline__ double sum(double s) const {
        for (int o = n / 2; o > 0; o >>= 1) s += __shfl_xor_sync(mask, s, o);
        return s;
    }
};
// item -> row and the elements [lo, hi) of it, lo the lane's first
struct Part {
    unsigned int row;
    int part, lo, hi;
    __device__ __forceinline__ Part(const RowMap& M, const Lanes& L, unsigned int item, int np) {
        row = item / (unsigned int)M.parts;
        part = (int)(item - row * (unsigned int)M.parts);
        lo = part * M.len + L.lane;
        hi = min(part * M.len + M.len, np);
    }
};
// x > 0 (true also for a NaN with a clear sign, which makes every use of the result a NaN)
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }
// m = max(m, |x|) on the bits of non-negative doubles; a NaN is ignored, as by fmax
__device__ __forceinline__ void max_abs(long long& m, double x) {
    const long long b = __double_as_longlong(x) & 0x7fffffffffffffffll;
    if (b > m && b <= 0x7ff0000000000000ll) m = b;
}

// a row (i, j) of cells: the addresses of the faces around it, and the polar rule
struct FaceRow {
    const double *r0, *r1, *t0, *t1, *p0;
    const double* h;   // polar rings: the two harmonic sums of the B_theta ring beside it
    const double* pcs;
    double pole_f;
    int np;
    __device__ __forceinline__ FaceRow(const Dims& d, const Geo& G, const double* __restrict__ bh, const double* br,
                                       const double* bt, const double* bp, int i, int j)
        : r0(br + ix(d, i, j, 0)), r1(br + ix(d, i + 1, j, 0)), t0(bt + ixt(d, i, j, 0)), t1(bt + ixt(d, i, j + 1, 0)),
          p0(bp + ix(d, i, j, 0)), h(j == 0 ? bh + 2 * i : (j == d.nt - 1 ? bh + 2 * (d.nr + i) : nullptr)), pcs(G.pcs),
          pole_f(G.pole_f), np(d.np) {
        if (j == 0) t0 = t1;        // the non-polar face on either side
        else if (j == d.nt - 1) t1 = t0;
    }
    // twice the cell-centred B: sums of opposite faces; in the polar rings (POLAR) B_theta is the non-polar face and
    // the pole value (first phi harmonic of the ring, see polar_btc)
    template <bool POLAR>
    __device__ __forceinline__ void twice(int k, int kp, double (&o)[3]) const {
        o[0] = r0[k] + r1[k];
        if constexpr (POLAR) o[1] = t0[k] + (h[0] * pcs[k] + h[1] * pcs[np + k]) * pole_f;
        else o[1] = t0[k] + t1[k];
        o[2] = p0[k] + p0[kp];
    }
    // f(polar) with polar a compile-time truth value: a loop over the row of its own for the polar rings (the pole
    // value as a choice within one loop takes its turns of the FP64 pipe in every row)
    template <typename F>
    __device__ __forceinline__ void over(F f) const {
        if (h) f(std::true_type());
        else f(std::false_type());
    }
};

// four times J at the cells of a row, from the edge arrays (polar phi edges left out)
struct EdgeRow {
    const double *r0, *r1, *t0, *t1, *p00, *p01, *p10, *p11;
    __device__ __forceinline__ EdgeRow(const Dims& d, const double* jr, const double* jt, const double* jp, int i, int j)
        : r0(jr + ixt(d, i, j, 0)), r1(jr + ixt(d, i, j + 1, 0)), t0(jt + ix(d, i, j, 0)), t1(jt + ix(d, i + 1, j, 0)) {
        const int lo = j == 0 ? 1 : j, hi = j == d.nt - 1 ? d.nt - 1 : j + 1;
        p00 = jp + ixt(d, i, lo, 0);
        p01 = jp + ixt(d, i, hi, 0);
        p10 = jp + ixt(d, i + 1, lo, 0);
        p11 = jp + ixt(d, i + 1, hi, 0);
    }
    __device__ __forceinline__ void four(int k, int kp, double (&o)[3]) const {
        o[0] = (r0[k] + r0[kp]) + (r1[k] + r1[kp]);
        o[1] = (t0[k] + t0[kp]) + (t1[k] + t1[kp]);
        o[2] = (p00[k] + p01[k]) + (p10[k] + p11[k]);
    }
};

// velocity u = v + f * dlt; DLT false: u = v (a test of the pointer at run time would leave the multiply-adds in
// place, switched off but taking their turn of the FP64 pipe: force 69 FP64 instructions a cell instead of 54)
template <bool DLT>
struct Vel {
    const double *vr, *vt, *vp, *dl;
    double f;
    long long N;
    __device__ __forceinline__ void at(long long c, double (&u)[3]) const {
        u[0] = vr[c];
        u[1] = vt[c];
        u[2] = vp[c];
        if constexpr (DLT) {
            u[0] += f * dl[c];
            u[1] += f * dl[N + c];
            u[2] += f * dl[2 * N + c];
        }
    }
};

// Lanes and parts of rows of np elements, and the CTAs of a kernel over them: as many as are resident at once.
// Parts: where rows are so few that they would not fill the resident warps, a row is cut, down to 4 passes of its
// lanes. Lanes: 32 while a row is many passes long (smaller groups at np = 512 took 15 to 50% longer: their accesses are spread
// over more rows); below that the number with the least estimated time, which is the items that the busiest
// SM gets, a CTA's worth at a time, times the passes of an item, with a factor for the spread. Times in us, coefficients + force +
// induction without and with resistivity + diagnostics, with 32 lanes and one part for every row / by this rule:
// 256x256x8 1332 / 477, 300x200x34 2293 / 1306, 100x100x48 530 / 423, 16x16x4096 2010 / 806, 4x4x8192 3433 / 301.
struct RowLaunch {
    RowMap m;
    int blocks;
};
RowLaunch row_launch(const mhd_grid_s* g, long long rows, int resident) {
    const int np = g->d.np;
    const long long room = (long long)g->num_sms * resident * kThreads;
    auto map = [&](int lanes) {
        RowMap m{lanes, 1, 0};
        m.parts = (int)std::max<long long>(1, std::min<long long>(np / (4 * lanes), (room + rows * lanes - 1) / (rows * lanes)));
        const int len = (np + m.parts - 1) / m.parts;
        m.len = (len + lanes - 1) / lanes * lanes;
        m.parts = (np + m.len - 1) / m.len;
        return m;
    };
    auto cost = [&](const RowMap& m, double spread) {
        const long long ctas = (rows * m.parts * m.lanes + kThreads - 1) / kThreads;
        return (double)((ctas + g->num_sms - 1) / g->num_sms) * (m.len / m.lanes + 0.2) * spread;
    };
    RowLaunch r{map(32), 0};
    if (np < 256) {
        double least = cost(r.m, 1.0);
        for (const auto& [lanes, spread] : {std::pair(16, 1.15), std::pair(8, 1.15), std::pair(4, 1.2), std::pair(2, 1.4)}) {
            const RowMap m = map(lanes);
            const double c = cost(m, spread);
            if (c < least) {
                least = c;
                r.m = m;
            }
        }
    }
    r.blocks = grid_blocks(g, rows * r.m.parts * r.m.lanes, resident);
    return r;
}
// launch a row kernel: W where warps take whole rows, P otherwise
template <auto W, auto P, typename... Args>
void launch_rows(const mhd_grid_s* g, cudaStream_t st, long long rows, int max_blocks, Args... args) {
    RowLaunch r = row_launch(g, rows, resident_per_sm<W>());
    if (r.m.lanes == 32 && r.m.parts == 1) {
        W<<<std::min(r.blocks, max_blocks), kThreads, 0, st>>>(g->d, r.m, args...);
        return;
    }
    r = row_launch(g, rows, resident_per_sm<P>());
    P<<<std::min(r.blocks, max_blocks), kThreads, 0, st>>>(g->d, r.m, args...);
}

}  // namespace

// ------------------------------------------------------------------------------------------
// step coefficients
// ------------------------------------------------------------------------------------------
// Every term of a row has the same factors, and rounding is monotone, so the row's largest |v|^2 and |B|^2 give
// the largest products bit for bit.
template <bool WHOLE>
__global__ void __launch_bounds__(kThreads) k_coeffs(Dims d, RowMap map, Geo G, Vel<false> v, const double* __restrict__ bh,
                                                     const double* __restrict__ br,
                                                     const double* __restrict__ bt,
                                                     const double* __restrict__ bp, double nu, double cfl,
                                                     double dt_fixed, double dt_max, double asi_fixed,
                                                     StepScalars* ss, double* __restrict__ partials) {
    double mkv = 0.0, mka = 0.0;
    const unsigned int rows = (unsigned int)(d.nr * d.nt);
    const RowMap M = map.fixed<WHOLE>(d.np);
    const Lanes L(M);
    for (unsigned int it = L.first; it < rows * M.parts; it += L.stride) {
        const Part S(M, L, it, d.np);
        const unsigned int ij = S.row;
        const int i = (int)(ij / d.nt), j = (int)(ij - (unsigned int)i * d.nt);
        const FaceRow F(d, G, bh, br, bt, bp, i, j);
        long long mv = 0, mb = 0;
        F.over([&](auto polar) {
#pragma unroll 4
            for (int k = S.lo; k < S.hi; k += L.n) {
                double u[3], B[3];
                v.at((long long)ij * d.np + k, u);
                F.twice<decltype(polar)::value>(k, kp1(d, k), B);
                max_abs(mv, u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
                max_abs(mb, B[0] * B[0] + B[1] * B[1] + B[2] * B[2]);
            }
        });
        const double kt2 = G.kt2[ij];
        mkv = fmax(mkv, kt2 * __longlong_as_double(mv));
        mka = fmax(mka, kt2 * (0.25 * __longlong_as_double(mb)) / G.rho[i]);
    }
    double val[2] = {mkv, mka}, out[2];
    if (reduce_last<2, OpMax>(val, partials, &ss->count, out) && threadIdx.x == 0) {
        const double kv = sqrt(out[0]), ka = sqrt(out[1]);
        ss->max_kv2 = out[0];
        ss->max_kva2 = out[1];
        ss->max_kt2 = G.max_kt2;
        double dt = 0.0;
        int st = MHD_OK;
        if (dt_fixed > 0.0) dt = dt_fixed;
        else {
            if (kv > 0.0) dt = cfl / kv;
            else if (dt_max > 0.0) dt = dt_max;
            else st = MHD_ERR_ARG;
            if (dt_max > 0.0 && dt > dt_max) dt = dt_max;
        }
        const double cf = dt * kv, cw = dt * ka;
        if (!(cf < 1.0)) st = MHD_ERR_ARG;
        const double X = cw * cw / ((1.0 - cf) * (1.0 - cf)) - 1.0;
        double asi = (X > 0.0) ? X / G.max_kt2 : 0.0;
        if (asi_fixed >= 0.0) asi = asi_fixed;
        ss->dt = dt;
        ss->cf = cf;
        ss->cw = cw;
        ss->alpha_si = (st == MHD_OK) ? asi : 0.0;
        ss->alpha_nu = nu * dt;
        ss->status = st;
    }
}

mhd_status_t coeffs(mhd_grid_s* g, const mhd_params_t* p, const double* vr, const double* vt,
                    const double* vp, const double* br, const double* bt, const double* bp) {
    const Vel<false> v{vr, vt, vp, nullptr, 0.0, g->d.N};
    bt_harmonics(g, bt);
    launch_rows<k_coeffs<true>, k_coeffs<false>>(g, g->stream, (long long)g->d.nr * g->d.nt, kMaxBlocks, g->geo, v, g->bharm, br,
                                                 bt, bp, p->nu, p->cfl, p->dt_fixed, p->dt_max, p->alpha_si_fixed, g->ss,
                                                 g->partials);
    return check_cuda(g, "coeffs");
}

// ------------------------------------------------------------------------------------------
// polar rings
// ------------------------------------------------------------------------------------------
// first-harmonic sums of the rows next to the poles (one CTA per row, fixed-order reduction):
// out[2 b] = sum_k a_k cos(phi_c_k), out[2 b + 1] = sum_k a_k sin(phi_c_k), b = i (north row at
// off_n + i stride_i) or nr + i (south row at off_s + i stride_i)
__global__ void k_ring_harm(Dims d, const double* __restrict__ a, long long stride_i, long long off_n,
                            long long off_s, const double* __restrict__ pcs, double* __restrict__ out) {
    const int i = blockIdx.x % d.nr;
    const int south = blockIdx.x / d.nr;
    const double* row = a + (long long)i * stride_i + (south ? off_s : off_n);
    double sc = 0.0, ss = 0.0;
    for (int k = threadIdx.x; k < d.np; k += blockDim.x) {
        sc = fma(row[k], pcs[k], sc);
        ss = fma(row[k], pcs[d.np + k], ss);
    }
    __shared__ double sm[2][kThreads / 32];
    for (int o = 16; o > 0; o >>= 1) {
        sc += __shfl_xor_sync(0xffffffffu, sc, o);
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
    }
    if ((threadIdx.x & 31) == 0) {
        sm[0][threadIdx.x >> 5] = sc;
        sm[1][threadIdx.x >> 5] = ss;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double tc = 0.0, ts = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            tc += sm[0][w];
            ts += sm[1][w];
        }
        out[2 * blockIdx.x] = tc;
        out[2 * blockIdx.x + 1] = ts;
    }
}

// polar ring sums of a cell-centred array, one CTA per ring: out[i] (north), out[nr + i] (south). done (may be null):
// a solve's flag
__global__ void __launch_bounds__(kThreads) k_ring_sum(Dims d, const double* __restrict__ a, double* __restrict__ out,
                                                       const int* __restrict__ done) {
    if (done && *done) return;
    const int i = blockIdx.x % d.nr, south = blockIdx.x / d.nr;
    const double* row = a + ix(d, i, south ? d.nt - 1 : 0, 0);
    double s = 0.0;
    for (int k = threadIdx.x; k < d.np; k += kThreads) s += row[k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double sm[kThreads / 32];
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        s = sm[0];
        for (int w = 1; w < kThreads / 32; w++) s += sm[w];
        out[blockIdx.x] = s;
    }
}

void ring_harmonics(mhd_grid_s* g, const double* a, long long stride_i, long long off_n, long long off_s,
                    double* out, cudaStream_t st) {
    k_ring_harm<<<2 * g->d.nr, kThreads, 0, st ? st : g->stream>>>(g->d, a, stride_i, off_n, off_s, g->geo.pcs,
                                                                   out);
}

void bt_harmonics(mhd_grid_s* g, const double* bt, cudaStream_t st) {
    const Dims d = g->d;
    ring_harmonics(g, bt, (long long)(d.nt + 1) * d.np, d.np, (long long)(d.nt - 1) * d.np, g->bharm, st);
}

// ------------------------------------------------------------------------------------------
// current density on edges
// ------------------------------------------------------------------------------------------
// J on all edges in one launch, a group of lanes per row; a polar radial row takes its ring's sum of B_phi itself (the cap
// circulation) unless it comes in ring, and with bh the warps of the first 2 nr rows form the harmonics of the B_theta rings beside the
// poles. walls_zero: the resistive operator's current, 0 on the tangential edges of r0 and r1. done (may be null):
// a solve's flag, nothing is formed once it is set.
template <bool WHOLE>
__global__ void __launch_bounds__(kThreads) k_current(Dims d, RowMap map, const double* __restrict__ cr,
                                                      const double* __restrict__ ct, const double* __restrict__ cp,
                                                      const double* __restrict__ br, const double* __restrict__ bt,
                                                      const double* __restrict__ bp, double* __restrict__ jr,
                                                      double* __restrict__ jt, double* __restrict__ jp,
                                                      const double* __restrict__ pcs, double* __restrict__ bh,
                                                      int walls_zero, const int* __restrict__ done,
                                                      const double* __restrict__ ring) {
    if (done && *done) return;
    const unsigned int n_h = bh ? 2u * d.nr : 0u, n_r = (unsigned int)(d.nr * (d.nt + 1)),
                       n_t = (unsigned int)((d.nr + 1) * d.nt), n_p = (unsigned int)((d.nr + 1) * (d.nt + 1));
    const int np = d.np;
    const RowMap M = map.fixed<WHOLE>(d.np);
    const Lanes L(M);
    for (unsigned int it = L.first; it < (n_h + n_r + n_t + n_p) * M.parts; it += L.stride) {
        const Part S(M, L, it, np);
        const unsigned int w = S.row;
        if (w < n_h) {
            if (S.part) continue;
            const int i = (int)(w % d.nr), south = (int)(w / d.nr);
            const double* row = bt + ixt(d, i, south ? d.nt - 1 : 1, 0);
            double c = 0.0, s = 0.0;
            for (int k = L.lane; k < np; k += L.n) {
                c = fma(row[k], pcs[k], c);
                s = fma(row[k], pcs[np + k], s);
            }
            c = L.sum(c);
            s = L.sum(s);
            if (L.lane == 0) {
                bh[2 * w] = c;
                bh[2 * w + 1] = s;
            }
        } else if (w < n_h + n_r) {
            const unsigned int q = w - n_h;
            const int i = (int)(q / (d.nt + 1)), j = (int)(q - (unsigned int)i * (d.nt + 1));
            const double* c = cr + 4 * (size_t)q;
            double* out = jr + (long long)q * np;
            if (j == 0 || j == d.nt) {
                const double* row = bp + ix(d, i, j == 0 ? 0 : d.nt - 1, 0);
                double s = 0.0;
                if (!WHOLE && ring) {
                    s = ring[j == 0 ? i : d.nr + i];
                } else {
                    for (int k = L.lane; k < np; k += L.n) s += row[k];
                    s = L.sum(s);
                }
                s *= j == 0 ? c[3] : -c[3];   // cap circulation / cap area
                for (int k = S.lo; k < S.hi; k += L.n) out[k] = s;
            } else {
                const double c0 = c[0], c1 = c[1], c2 = c[2];
                const double *b = bp + ix(d, i, j, 0), *a = b - np, *t = bt + ixt(d, i, j, 0);
#pragma unroll 4
                for (int k = S.lo; k < S.hi; k += L.n) out[k] = c0 * b[k] - c1 * a[k] - c2 * (t[k] - t[km1(d, k)]);
            }
        } else if (w < n_h + n_r + n_t) {
            const unsigned int q = w - n_h - n_r;
            const int i = (int)(q / d.nt), j = (int)(q - (unsigned int)i * d.nt);
            const bool wall = walls_zero && (i == 0 || i == d.nr);
            // ghost B_phi beyond r0 / r1 = the first interior value (at the mirrored radius in the table)
            const double *lo = bp + ix(d, i > 0 ? i - 1 : 0, j, 0), *hi = bp + ix(d, i < d.nr ? i : d.nr - 1, j, 0);
            const double* b = br + ix(d, i, j, 0);
            const double* c = ct + 3 * (size_t)q;
            const double c0 = c[0], c1 = c[1], c2 = c[2];
            double* out = jt + (long long)q * np;
#pragma unroll 4
            for (int k = S.lo; k < S.hi; k += L.n)
                out[k] = wall ? 0.0 : c0 * lo[k] + c1 * (b[k] - b[km1(d, k)]) - c2 * hi[k];
        } else {
            const unsigned int q = w - n_h - n_r - n_t;
            const int i = (int)(q / (d.nt + 1)), j = (int)(q - (unsigned int)i * (d.nt + 1));
            double* out = jp + (long long)q * np;
            if (j == 0 || j == d.nt || (walls_zero && (i == 0 || i == d.nr))) {
                for (int k = S.lo; k < S.hi; k += L.n) out[k] = 0.0;
            } else {
                const double *lo = bt + ixt(d, i > 0 ? i - 1 : 0, j, 0), *hi = bt + ixt(d, i < d.nr ? i : d.nr - 1, j, 0);
                const double *b = br + ix(d, i, j, 0), *a = b - np;
                const double* c = cp + 3 * (size_t)q;
                const double c0 = c[0], c1 = c[1], c2 = c[2];
#pragma unroll 4
                for (int k = S.lo; k < S.hi; k += L.n) out[k] = c0 * (a[k] - b[k]) + c1 * hi[k] - c2 * lo[k];
            }
        }
    }
}

namespace {

// Rows cut into parts, and long: every part of a polar radial row would take its ring's sum itself, a chain of np / 32
// additions, so the sums and the harmonics are launches of their own, a CTA per ring (us of an induction with
// resistivity, without / with: 4x4x8192 122 / 70, 16x16x4096 194 / 187).
bool rings_apart(const mhd_grid_s* g) {
    return g->d.np >= 2048 && row_launch(g, (long long)g->d.nr * g->d.nt, 2).m.parts > 1;
}
// the ring sums of a cell-centred array where they are launched apart, else null
const double* ring_sums(mhd_grid_s* g, const double* a, const int* done, cudaStream_t st) {
    if (!rings_apart(g)) return nullptr;
    k_ring_sum<<<2 * g->d.nr, kThreads, 0, st>>>(g->d, a, g->ring, done);
    return g->ring;
}

void edge_current(mhd_grid_s* g, const double* cr, const double* ct, const double* cp, const double* br, const double* bt,
                  const double* bp, double* bh, bool walls_zero, const int* done, cudaStream_t st) {
    const Dims d = g->d;
    const double* ring = ring_sums(g, bp, done, st);
    if (ring && bh) {
        bt_harmonics(g, bt, st);
        bh = nullptr;
    }
    const long long rows = (bh ? 2ll * d.nr : 0ll) + (long long)d.nr * (d.nt + 1) + (long long)(d.nr + 1) * d.nt +
                           (long long)(d.nr + 1) * (d.nt + 1);
    launch_rows<k_current<true>, k_current<false>>(g, st, rows, kMaxBlocks, cr, ct, cp, br, bt, bp, g->er, g->et, g->ep,
                                                   g->geo.pcs, bh, walls_zero ? 1 : 0, done, ring);
}

void current_and_harmonics(mhd_grid_s* g, const double* br, const double* bt, const double* bp, double* bh, cudaStream_t st) {
    edge_current(g, g->ex.jr, g->ex.jt, g->ex.jp, br, bt, bp, bh, false, nullptr, st);
}

}  // namespace

void current_edges(mhd_grid_s* g, const double* br, const double* bt, const double* bp) {
    current_and_harmonics(g, br, bt, bp, nullptr, g->stream);
}

void res_edge_current(mhd_grid_s* g, const double* cr, const double* ct, const double* cp, const double* br, const double* bt,
                      const double* bp, const int* done, cudaStream_t st) {
    edge_current(g, cr, ct, cp, br, bt, bp, nullptr, true, done, st);
}

// ------------------------------------------------------------------------------------------
// momentum force
// ------------------------------------------------------------------------------------------
// AVG: the mean with the force in b_avg
template <bool DLT, bool AVG, bool WHOLE>
__global__ void __launch_bounds__(kThreads) k_force(Dims d, RowMap map, Geo G, ExTab X, Vel<DLT> v, const double* __restrict__ bh,
                                                    const double* __restrict__ br,
                                                    const double* __restrict__ bt, const double* __restrict__ bp,
                                                    const double* __restrict__ jr, const double* __restrict__ jt,
                                                    const double* __restrict__ jp, const double* __restrict__ dt_dev,
                                                    double dt_host, const double* __restrict__ b_avg,
                                                    double* __restrict__ b) {
    const double dt = dt_dev ? *dt_dev : dt_host;
    const unsigned int rows = (unsigned int)(d.nr * d.nt);
    const long long plane = (long long)d.nt * d.np;
    const RowMap M = map.fixed<WHOLE>(d.np);
    const Lanes L(M);
    for (unsigned int it = L.first; it < rows * M.parts; it += L.stride) {
        const Part S(M, L, it, d.np);
        const unsigned int ij = S.row;
        const int i = (int)(ij / d.nt), j = (int)(ij - (unsigned int)i * d.nt);
        const FaceRow F(d, G, bh, br, bt, bp, i, j);
        const EdgeRow E(d, jr, jt, jp, i, j);
        // per-shell reciprocals: 1/d_lo, 1/d_hi, 1/rc, 1/rho, 1/(rc dth); 8 J x B is what the sums give
        const double* sh = X.sh + 5 * (size_t)i;
        const double ir_lo = sh[0], ir_hi = sh[1], irc = sh[2], irho8 = 0.125 * sh[3], iht = sh[4];
        const double ihp = X.ihp[ij], cot = X.cot[j];
        const double s = (AVG ? 0.5 : 1.0) * (G.rhoV[ij] * dt);
        // upwind neighbours: none beyond r1 and the poles (the cell itself: difference 0); the Dirichlet mirror
        // ghost -u at r0
        const long long c_row = (long long)ij * d.np;
        const long long r_lo = i > 0 ? -plane : 0, r_hi = i < d.nr - 1 ? plane : 0;
        const long long t_lo = j > 0 ? -d.np : 0, t_hi = j < d.nt - 1 ? d.np : 0;
        F.over([&](auto polar) {
#pragma unroll 1
            for (int k = S.lo; k < S.hi; k += L.n) {
                const long long c = c_row + k;
                const int kp = kp1(d, k), km = km1(d, k);
                double u[3], n[3], adv[3], B[3], J[3];
                v.at(c, u);
                const bool ur = positive(u[0]), ut = positive(u[1]), up = positive(u[2]);
                F.twice<decltype(polar)::value>(k, kp, B);
                E.four(k, kp, J);
                {
                    v.at(c + (ur ? r_lo : r_hi), n);
                    // (the ghost's sign by its bit: three negations would be FP64 instructions of every row)
                    const long long ghost = i == 0 && ur ? (long long)0x8000000000000000ull : 0ll;
#pragma unroll
                    for (int m = 0; m < 3; m++) n[m] = __longlong_as_double(__double_as_longlong(n[m]) ^ ghost);
                    const double a = fabs(u[0]) * (ur ? ir_lo : ir_hi);
#pragma unroll
                    for (int m = 0; m < 3; m++) adv[m] = a * (u[m] - n[m]);
                }
                {
                    v.at(c + (ut ? t_lo : t_hi), n);
                    const double a = fabs(u[1]) * iht;
#pragma unroll
                    for (int m = 0; m < 3; m++) adv[m] = fma(a, u[m] - n[m], adv[m]);
                }
                {
                    v.at(c_row + (up ? km : kp), n);
                    const double a = fabs(u[2]) * ihp;
#pragma unroll
                    for (int m = 0; m < 3; m++) adv[m] = fma(a, u[m] - n[m], adv[m]);
                }
                // spherical curvature terms
                const double a1 = u[1] * irc, a2 = u[2] * irc, c2 = u[2] * cot;
                adv[0] = fma(-u[1], a1, fma(-u[2], a2, adv[0]));
                adv[1] = fma(u[0], a1, fma(-c2, a2, adv[1]));
                adv[2] = fma(u[0], a2, fma(c2, a1, adv[2]));
                double f0 = s * fma(J[1] * B[2] - J[2] * B[1], irho8, -adv[0]);
                double f1 = s * fma(J[2] * B[0] - J[0] * B[2], irho8, -adv[1]);
                double f2 = s * fma(J[0] * B[1] - J[1] * B[0], irho8, -adv[2]);
                if constexpr (AVG) {
                    f0 = fma(0.5, b_avg[c], f0);
                    f1 = fma(0.5, b_avg[d.N + c], f1);
                    f2 = fma(0.5, b_avg[2 * d.N + c], f2);
                }
                b[c] = f0;
                b[d.N + c] = f1;
                b[2 * d.N + c] = f2;
            }
        });
    }
}

namespace {
template <bool DLT, bool AVG>
void force_launch(mhd_grid_s* g, const Vel<DLT>& v, const double* br, const double* bt, const double* bp,
                  const double* dt_dev, double dt_host, const double* b_avg, double* b) {
    launch_rows<k_force<DLT, AVG, true>, k_force<DLT, AVG, false>>(g, g->stream, (long long)g->d.nr * g->d.nt, kMaxBlocks, g->geo,
                                                                   g->ex, v, g->bharm, br, bt, bp, g->er, g->et, g->ep, dt_dev,
                                                                   dt_host, b_avg, b);
}
}  // namespace

void force(mhd_grid_s* g, const double* vr, const double* vt, const double* vp, const double* dlt, double dfac,
           const double* br, const double* bt, const double* bp, const double* dt_dev, double dt_host,
           const double* b_avg, double* b) {
    current_and_harmonics(g, br, bt, bp, g->bharm, g->stream);
    const Vel<false> v{vr, vt, vp, nullptr, 0.0, g->d.N};
    const Vel<true> w{vr, vt, vp, dlt, dfac, g->d.N};
    if (dlt && b_avg) force_launch<true, true>(g, w, br, bt, bp, dt_dev, dt_host, b_avg, b);
    else if (dlt) force_launch<true, false>(g, w, br, bt, bp, dt_dev, dt_host, b_avg, b);
    else if (b_avg) force_launch<false, true>(g, v, br, bt, bp, dt_dev, dt_host, b_avg, b);
    else force_launch<false, false>(g, v, br, bt, bp, dt_dev, dt_host, b_avg, b);
}

// ------------------------------------------------------------------------------------------
// electric field and constrained transport
// ------------------------------------------------------------------------------------------
// twice E at the cell centres; ETA: with the resistive part
template <bool DLT, bool ETA, bool WHOLE>
__global__ void __launch_bounds__(kThreads) k_ecentre(Dims d, RowMap map, Geo G, Vel<DLT> v, const double* __restrict__ bh,
                                                      const double* __restrict__ br,
                                                      const double* __restrict__ bt, const double* __restrict__ bp,
                                                      const double* __restrict__ jr, const double* __restrict__ jt,
                                                      const double* __restrict__ jp, double eta,
                                                      double* __restrict__ ec) {
    const unsigned int rows = (unsigned int)(d.nr * d.nt);
    const double eta_h = 0.5 * eta;   // of four times J
    const RowMap M = map.fixed<WHOLE>(d.np);
    const Lanes L(M);
    for (unsigned int it = L.first; it < rows * M.parts; it += L.stride) {
        const Part S(M, L, it, d.np);
        const unsigned int ij = S.row;
        const int i = (int)(ij / d.nt), j = (int)(ij - (unsigned int)i * d.nt);
        const FaceRow F(d, G, bh, br, bt, bp, i, j);
        const EdgeRow E(d, jr, jt, jp, i, j);
        F.over([&](auto polar) {
#pragma unroll 2
            for (int k = S.lo; k < S.hi; k += L.n) {
                const long long c = (long long)ij * d.np + k;
                const int kp = kp1(d, k);
                double u[3], B[3];
                v.at(c, u);
                F.twice<decltype(polar)::value>(k, kp, B);
                double e0 = u[2] * B[1] - u[1] * B[2];
                double e1 = u[0] * B[2] - u[2] * B[0];
                double e2 = u[1] * B[0] - u[0] * B[1];
                if constexpr (ETA) {
                    double J[3];
                    E.four(k, kp, J);
                    e0 = fma(eta_h, J[0], e0);
                    e1 = fma(eta_h, J[1], e1);
                    e2 = fma(eta_h, J[2], e2);
                }
                ec[c] = e0;
                ec[d.N + c] = e1;
                ec[2 * d.N + c] = e2;
            }
        });
    }
}

// eight times E on the edges, from twice E at the centres (kEdgeScale undoes it)
constexpr double kEdgeScale = 0.125;
template <bool WHOLE>
__global__ void __launch_bounds__(kThreads) k_eedges(Dims d, RowMap map, const double* __restrict__ ec, double* __restrict__ er,
                                                     double* __restrict__ et, double* __restrict__ ep,
                                                     const double* __restrict__ ring) {
    const unsigned int n_r = (unsigned int)(d.nr * (d.nt + 1)), n_t = (unsigned int)((d.nr + 1) * d.nt),
                       n_p = (unsigned int)((d.nr + 1) * (d.nt + 1));
    const int np = d.np;
    const RowMap M = map.fixed<WHOLE>(d.np);
    const Lanes L(M);
    for (unsigned int it = L.first; it < (n_r + n_t + n_p) * M.parts; it += L.stride) {
        const Part S(M, L, it, np);
        const unsigned int w = S.row;
        if (w < n_r) {
            const int i = (int)(w / (d.nt + 1)), j = (int)(w - (unsigned int)i * (d.nt + 1));
            double* out = er + (long long)w * np;
            if (j == 0 || j == d.nt) {
                // the polar radial edge: the mean of the polar ring
                const double* row = ec + ix(d, i, j == 0 ? 0 : d.nt - 1, 0);
                double s = 0.0;
                if (!WHOLE && ring) {
                    s = ring[j == 0 ? i : d.nr + i];
                } else {
                    for (int k = L.lane; k < np; k += L.n) s += row[k];
                    s = L.sum(s);
                }
                s = 4.0 * (s / np);
                for (int k = S.lo; k < S.hi; k += L.n) out[k] = s;
            } else {
                const double *b = ec + ix(d, i, j, 0), *a = b - np;
#pragma unroll 4
                for (int k = S.lo; k < S.hi; k += L.n) {
                    const int km = km1(d, k);
                    out[k] = (a[km] + a[k]) + (b[km] + b[k]);
                }
            }
        } else if (w < n_r + n_t) {
            const unsigned int q = w - n_r;
            const int i = (int)(q / d.nt), j = (int)(q - (unsigned int)i * d.nt);
            double* out = et + (long long)q * np;
            // r0: 0 (line-tied); r1: the mean of the two interior cells
            const double *a = ec + d.N + ix(d, i > 0 ? i - 1 : 0, j, 0), *b = ec + d.N + ix(d, i < d.nr ? i : d.nr - 1, j, 0);
#pragma unroll 4
            for (int k = S.lo; k < S.hi; k += L.n) {
                const int km = km1(d, k);
                out[k] = i == 0 ? 0.0 : (a[km] + a[k]) + (b[km] + b[k]);
            }
        } else {
            const unsigned int q = w - n_r - n_t;
            const int i = (int)(q / (d.nt + 1)), j = (int)(q - (unsigned int)i * (d.nt + 1));
            double* out = ep + (long long)q * np;
            if (j == 0 || j == d.nt || i == 0) {
                for (int k = S.lo; k < S.hi; k += L.n) out[k] = 0.0;
            } else {
                const double *a = ec + 2 * d.N + ix(d, i - 1, j, 0), *b = ec + 2 * d.N + ix(d, i < d.nr ? i : d.nr - 1, j, 0);
#pragma unroll 4
                for (int k = S.lo; k < S.hi; k += L.n) out[k] = (a[k - np] + a[k]) + (b[k - np] + b[k]);
            }
        }
    }
}

// B -= scale dt curl_h of the edge arrays
template <bool WHOLE>
__global__ void __launch_bounds__(kThreads) k_ct(Dims d, RowMap map, ExTab X, const double* __restrict__ er,
                                                 const double* __restrict__ et, const double* __restrict__ ep,
                                                 const double* __restrict__ dt_dev, double dt_host, double scale,
                                                 double* __restrict__ br, double* __restrict__ bt,
                                                 double* __restrict__ bp) {
    const double dt = scale * (dt_dev ? *dt_dev : dt_host);
    const unsigned int n_r = (unsigned int)((d.nr + 1) * d.nt), n_t = (unsigned int)(d.nr * (d.nt + 1)),
                       n_p = (unsigned int)(d.nr * d.nt);
    const int np = d.np;
    const RowMap M = map.fixed<WHOLE>(d.np);
    const Lanes L(M);
    for (unsigned int it = L.first; it < (n_r + n_t + n_p) * M.parts; it += L.stride) {
        const Part S(M, L, it, np);
        const unsigned int w = S.row;
        if (w < n_r) {
            const int i = (int)(w / d.nt), j = (int)(w - (unsigned int)i * d.nt);
            const double* c = X.fr + 3 * (size_t)w;
            const double c0 = c[0], c1 = c[1], c2 = c[2];
            const double *t = et + ix(d, i, j, 0), *p0 = ep + ixt(d, i, j, 0), *p1 = p0 + np;
            double* out = br + (long long)w * np;
#pragma unroll 4
            for (int k = S.lo; k < S.hi; k += L.n) {
                const double circ = c0 * (t[k] - t[kp1(d, k)]) + c1 * p1[k] - c2 * p0[k];
                out[k] -= dt * circ;
            }
        } else if (w < n_r + n_t) {
            const unsigned int q = w - n_r;
            const int i = (int)(q / (d.nt + 1)), j = (int)(q - (unsigned int)i * (d.nt + 1));
            if (j == 0 || j == d.nt) continue;
            const double* c = X.ft + 3 * (size_t)q;
            const double c0 = c[0], c1 = c[1], c2 = c[2];
            const double *r = er + ixt(d, i, j, 0), *p0 = ep + ixt(d, i, j, 0), *p1 = ep + ixt(d, i + 1, j, 0);
            double* out = bt + (long long)q * np;
#pragma unroll 4
            for (int k = S.lo; k < S.hi; k += L.n) {
                const double circ = c0 * p0[k] + c1 * (r[kp1(d, k)] - r[k]) - c2 * p1[k];
                out[k] -= dt * circ;
            }
        } else {
            const unsigned int q = w - n_r - n_t;
            const int i = (int)(q / d.nt), j = (int)(q - (unsigned int)i * d.nt);
            const double* c = X.fp + 3 * (size_t)q;
            const double c0 = c[0], c1 = c[1], c2 = c[2];
            const double *r0 = er + ixt(d, i, j, 0), *r1 = r0 + np, *t0 = et + ix(d, i, j, 0), *t1 = et + ix(d, i + 1, j, 0);
            double* out = bp + (long long)q * np;
#pragma unroll 4
            for (int k = S.lo; k < S.hi; k += L.n) {
                const double circ = c0 * (r0[k] - r1[k]) + c1 * t1[k] - c2 * t0[k];
                out[k] -= dt * circ;
            }
        }
    }
}

namespace {
template <bool DLT, bool ETA>
void ecentre_launch(mhd_grid_s* g, const Vel<DLT>& v, const double* br, const double* bt, const double* bp, double eta) {
    launch_rows<k_ecentre<DLT, ETA, true>, k_ecentre<DLT, ETA, false>>(g, g->stream, (long long)g->d.nr * g->d.nt, kMaxBlocks,
                                                                       g->geo, v, g->bharm, br, bt, bp, g->er, g->et, g->ep, eta,
                                                                       g->ec);
}
void ct_launch(mhd_grid_s* g, const double* dt_dev, double dt_host, double scale, double* br, double* bt, double* bp) {
    const Dims d = g->d;
    const long long rows = (long long)(d.nr + 1) * d.nt + (long long)d.nr * (d.nt + 1) + (long long)d.nr * d.nt;
    launch_rows<k_ct<true>, k_ct<false>>(g, g->stream, rows, kMaxBlocks, g->ex, g->er, g->et, g->ep, dt_dev, dt_host, scale, br,
                                         bt, bp);
}
}  // namespace

void induction(mhd_grid_s* g, const double* vr, const double* vt, const double* vp, const double* dlt, double dfac,
               double eta, const double* dt_dev, double dt_host, double* br, double* bt, double* bp, bool current_ready) {
    const Dims d = g->d;
    if (!current_ready) {
        if (eta != 0.0) current_and_harmonics(g, br, bt, bp, g->bharm, g->stream);
        else bt_harmonics(g, bt);
    }
    const Vel<false> v{vr, vt, vp, nullptr, 0.0, d.N};
    const Vel<true> w{vr, vt, vp, dlt, dfac, d.N};
    if (dlt && eta != 0.0) ecentre_launch<true, true>(g, w, br, bt, bp, eta);
    else if (dlt) ecentre_launch<true, false>(g, w, br, bt, bp, eta);
    else if (eta != 0.0) ecentre_launch<false, true>(g, v, br, bt, bp, eta);
    else ecentre_launch<false, false>(g, v, br, bt, bp, eta);
    const long long rows = (long long)d.nr * (d.nt + 1) + (long long)(d.nr + 1) * d.nt + (long long)(d.nr + 1) * (d.nt + 1);
    const double* ring = ring_sums(g, g->ec, nullptr, g->stream);
    launch_rows<k_eedges<true>, k_eedges<false>>(g, g->stream, rows, kMaxBlocks, g->ec, g->er, g->et, g->ep, ring);
    ct_launch(g, dt_dev, dt_host, kEdgeScale, br, bt, bp);
}

void ct_apply(mhd_grid_s* g, const double* dt_dev, double* br, double* bt, double* bp) {
    ct_launch(g, dt_dev, 0.0, 1.0, br, bt, bp);
}

// ------------------------------------------------------------------------------------------
// field diagnostics (Sec. 3.1 validates runs by integrated energies and by |J x B| and |J . B|):
// out[0..3] = magnetic energy, kinetic energy, sum |J_c x B_c| V_c, sum |J_c . B_c| V_c; out[4] =
// max |div_h B| (net outward flux over the cell volume). B_c and J_c as in the momentum force.
// ------------------------------------------------------------------------------------------
template <bool WHOLE>
__global__ void __launch_bounds__(kThreads) k_diag(Dims d, RowMap map, Geo G, ExTab X, Vel<false> v, const double* __restrict__ bh,
                                                   const double* __restrict__ br, const double* __restrict__ bt,
                                                   const double* __restrict__ bp, const double* __restrict__ jr,
                                                   const double* __restrict__ jt, const double* __restrict__ jp,
                                                   unsigned int* count, unsigned int* count_max,
                                                   double* __restrict__ partials, double* __restrict__ out) {
    double em = 0.0, ek = 0.0, jxb = 0.0, jdb = 0.0, dmax = 0.0;
    const unsigned int rows = (unsigned int)(d.nr * d.nt);
    const RowMap M = map.fixed<WHOLE>(d.np);
    const Lanes L(M);
    for (unsigned int it = L.first; it < rows * M.parts; it += L.stride) {
        const Part S(M, L, it, d.np);
        const unsigned int ij = S.row;
        const int i = (int)(ij / d.nt), j = (int)(ij - (unsigned int)i * d.nt);
        const FaceRow F(d, G, bh, br, bt, bp, i, j);
        const EdgeRow E(d, jr, jt, jp, i, j);
        const double *t0 = bt + ixt(d, i, j, 0), *t1 = t0 + d.np;
        // face areas and volume of the row's cells
        const double ri = G.r[i], ro = G.r[i + 1];
        const double ring = 0.5 * (ro * ro - ri * ri), band = (G.cn[j] - G.cn[j + 1]) * G.dph;
        const double ari = ri * ri * band, aro = ro * ro * band;
        const double atj = G.sn[j] * ring * G.dph, atj1 = G.sn[j + 1] * ring * G.dph;
        const double ap = ring * G.dth, V = G.rhoV[ij] * X.sh[5 * (size_t)i + 3];
        double sb = 0.0, su = 0.0, sx = 0.0, sd = 0.0;
        long long mf = 0;
        F.over([&](auto polar) {
#pragma unroll 1
            for (int k = S.lo; k < S.hi; k += L.n) {
                const int kp = kp1(d, k);
                double u[3], B[3], J[3];
                v.at((long long)ij * d.np + k, u);
                F.twice<decltype(polar)::value>(k, kp, B);
                E.four(k, kp, J);
                const double x0 = J[1] * B[2] - J[2] * B[1], x1 = J[2] * B[0] - J[0] * B[2], x2 = J[0] * B[1] - J[1] * B[0];
                sb = fma(B[0], B[0], fma(B[1], B[1], fma(B[2], B[2], sb)));
                su = fma(u[0], u[0], fma(u[1], u[1], fma(u[2], u[2], su)));
                sx += sqrt(x0 * x0 + x1 * x1 + x2 * x2);
                sd += fabs(J[0] * B[0] + J[1] * B[1] + J[2] * B[2]);
                max_abs(mf, F.r1[k] * aro - F.r0[k] * ari + t1[k] * atj1 - t0[k] * atj + (F.p0[kp] - F.p0[k]) * ap);
            }
        });
        // the sums hold 4 B^2 and 8 times the products of J and B
        em = fma(0.125 * V, sb, em);
        ek = fma(0.5 * G.rho[i] * V, su, ek);
        jxb = fma(0.125 * V, sx, jxb);
        jdb = fma(0.125 * V, sd, jdb);
        dmax = fmax(dmax, __longlong_as_double(mf) / V);
    }
    double val[4] = {em, ek, jxb, jdb}, o[4];
    if (reduce_last<4>(val, partials, count, o) && threadIdx.x == 0)
        for (int q = 0; q < 4; q++) out[q] = o[q];
    double vm[1] = {dmax}, om[1];
    if (reduce_last<1, OpMax>(vm, partials + 4 * (size_t)gridDim.x, count_max, om) && threadIdx.x == 0) out[4] = om[0];
}

// out (device, 5 doubles): the diagnostics of the fields; enqueued on the grid's stream
void diagnostics(mhd_grid_s* g, const double* vr, const double* vt, const double* vp, const double* br,
                 const double* bt, const double* bp, double* out) {
    const Dims d = g->d;
    current_and_harmonics(g, br, bt, bp, g->bharm, g->stream);
    const Vel<false> v{vr, vt, vp, nullptr, 0.0, d.N};
    // two reductions: 5 partials a CTA in the array's 4 kMaxBlocks, and a ticket each (the solver's is idle here)
    launch_rows<k_diag<true>, k_diag<false>>(g, g->stream, (long long)d.nr * d.nt, kMaxBlocks * kPartialsPerBlock / 5, g->geo, g->ex, v,
                                             g->bharm, br, bt, bp, g->er, g->et, g->ep, &g->ss->count, &g->sc->count, g->partials,
                                             out);
}

// ------------------------------------------------------------------------------------------
// v** = v + dlt (in place) and b = rho V v**
// ------------------------------------------------------------------------------------------
__global__ void k_vstar(Dims d, Geo G, double* __restrict__ vr, double* __restrict__ vt, double* __restrict__ vp,
                        const double* __restrict__ dlt, double* __restrict__ b) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < d.N;
         c += (long long)gridDim.x * blockDim.x) {
        const double w = G.rhoV[(unsigned int)c / (unsigned int)d.np];
        const double a = vr[c] + dlt[c], e = vt[c] + dlt[d.N + c], f = vp[c] + dlt[2 * d.N + c];
        vr[c] = a;
        vt[c] = e;
        vp[c] = f;
        b[c] = w * a;
        b[d.N + c] = w * e;
        b[2 * d.N + c] = w * f;
    }
}

void vstar_rhs(mhd_grid_s* g, double* vr, double* vt, double* vp, const double* dlt, double* b) {
    k_vstar<<<grid_blocks(g, g->d.N, 8), kThreads, 0, g->stream>>>(g->d, g->geo, vr, vt, vp, dlt, b);
}

}  // namespace mhd
