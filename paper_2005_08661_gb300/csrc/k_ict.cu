// k_ict.cu -- IC with a drop tolerance (Sec. III-B: the paper's L_t and the preconditioner
// of its NCG-MLS-IC; FM_PC_ICT).
//
// The paper zeroes every factor entry whose magnitude is below tau = droptol * H_max, H_max
// being the largest |H_jk| of the outer iteration's H = diag(d) + beta C'C.  Unlike IC(0)
// this keeps fill-in.  Eliminating an earlier neighbour k of two voxels i > j couples them:
// in natural order the first fill lands at the three "level-1" offsets (x+1, y-1, z),
// (x+1, y, z-1) and (x, y+1, z-1) from a row's voxel.  The kernels here hold the pattern P
// of IC(0)'s offsets a = (-1,0,0), b = (0,-1,0), c = (0,0,-1) plus those fill offsets
// d = (1,-1,0), e = (1,0,-1), f = (0,1,-1); row i of L has L_ii and L_{i,i+o}, o in P.
//
// Row i, in increasing column order c, e, f, b, d, a (each entry needs the row's earlier
// entries and the neighbour row j = i + o):
//   L_{i,j} = (H_ij - sum_{k < j} L_ik L_jk) / L_jj, set to 0 if |L_{i,j}| < tau,
//   L_ii = sqrt(H_ii - sum_o L_{i,i+o}^2),
// where the sums run over the common earlier neighbours inside P -- by offset arithmetic
// a: (b, d), (c, e); b: (c, f); c: none; d: (b, a), (e, f); e: (c, a); f: (c, b), (e, d),
// each pair (p1, p2) meaning L_{i,i+p1} L_{j,j+p2}.  The forward substitution L y = g is
// fused with the factorisation; the back substitution solves L' x = y.
//
// Schedule.  The fill offsets d, e, f link voxels of one x + y + z hyperplane, so the IC(0)
// wavefront does not apply.  With level t = x + 2y + 3z every offset in P points to a strictly
// lower level (t(a) = t(d) = t(f) = -1, t(b) = t(e) = -2, t(c) = -3).  Groups of 32 rows walk along x, a
// lane two steps behind the lane below, and hand their records on as they go ("row wavefront"
// below), or, where planes follow each other faster that way, a grid barrier separates the levels
// ("level sweeps"); the back substitution is the walk mirrored.  The factor stores 1 / L_ii, so every entry
// costs a multiply.
//
// Deeper fill.  When the tolerance keeps entries beyond level 1, the pattern P grows: the host
// holds any set of offsets (up to kIctMaxOffsets), builds the correction pairs of each offset
// by the same offset arithmetic (pairs (p1, p2) with o_p1 - o_p2 = o) and a level function
// t = x + B y + C z under which every held offset points to a lower level, and the
// table-driven kernels k_ictg_fwd / k_ictg_bwd sweep it: one persistent kernel, thread <-> (y, z)
// column, voxel x = t - B y - C z, with a barrier between levels (the bounded grid barrier of a
// cooperative launch, or a block barrier when one block holds every column).
//
// Exactness.  The held factor is the exact drop-tolerance factor as long as no entry outside
// the held pattern survives.  With the factor in hand, k_ict_check forms every would-be entry
// just outside it -- at each offset q = o_p1 - o_p2 (p1, p2 held, q not held, pointing to an
// earlier voxel) -- and flags the offsets where one reaches tau.  If none does, no entry
// outside the pattern ever appears (by induction over the columns); otherwise the first
// column where one does sees exactly this value, since all earlier columns agree.  Holding a
// flagged offset where the exact factor turns out to drop every entry changes nothing (the
// entries are computed and dropped exactly as the definition does), so the host adds every
// flagged offset and factors again until nothing is flagged.  For the base pattern the
// candidates are (-1,1,-1): (c,d); (-1,2,-1): (f,d); (0,2,-1): (f,b); (1,1,-1): (e,b), (f,a);
// (2,-1,0): (d,a); (2,0,-1): (e,a).
//
// A pivot <= 0 is reported (FM_ERR_NOT_PD) by the back sweep, after the check, so that
// FM_ERR_FILL wins when fill outside the held pattern is the cause.
//
// Arithmetic is double in both precision modes (the voxel type only for d, g and p): the
// sweeps are latency-bound, not bound by the FP64 pipe.
#include "fm_internal.h"

namespace fm {

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// ------------------------------------------------------------------ tau = droptol * H_max

template <typename T>
__global__ void __launch_bounds__(kThreads) k_ict_tau(DataArgs a, double droptol) {
    __shared__ double sbuf[32];
    __shared__ bool s_last;
    const T* d = (const T*)a.d;
    const double beta = a.beta;
    const long long nm = a.istate[I_NMASK];
    double m = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nm;
         k += (long long)gridDim.x * blockDim.x) {
        const long long j = a.vlist[k];
        const int n = __popc((unsigned)(a.nb[j] >> 1) & 0x3fu);
        m = fmax(m, fabs((double)d[j] + beta * (double)n));  // H_jj
        if (n > 0) m = fmax(m, fabs(beta));                 // H_jk = -beta
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    m = warp_max(m);
    if (lane == 0) sbuf[wid] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < nw; ++w) m = fmax(m, sbuf[w]);
        a.partials[blockIdx.x] = m;
        __threadfence();
        const unsigned prev = atomicAdd((unsigned*)(a.istate + I_DONE0), 1u);
        s_last = prev == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double h = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += blockDim.x) h = fmax(h, __ldcg(a.partials + i));
    h = warp_max(h);
    __syncthreads();
    if (lane == 0) sbuf[wid] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < nw; ++w) h = fmax(h, sbuf[w]);
        a.scal[S_ICT_TAU] = droptol * h;
        a.istate[I_DONE0] = 0;
        if (!isfinite(h)) set_err(a.istate, FM_ERR_NONFINITE);
    }
}

// ------------------------------------------------------------------ the sweeps

// Plane indices of the factor storage.
enum : int { PL_R = 0, PL_A, PL_B, PL_C, PL_D1, PL_E, PL_F, PL_Y };  // PL_R: 1 / L_ii

// 1 / sqrt(s) for s > 0 in double: a float seed refined by two Newton-Raphson steps
// r <- r (3 - s r^2) / 2, each of which squares the relative error (about 2^-22 for the
// seed, so the second step reaches double rounding).  The GB300 FP64 pipe issues about
// 1/64 as fast as FP32, and this chain sits on every row's critical path.
__device__ __forceinline__ double rsqrt_nr(double s) {
    double r = (double)rsqrtf((float)s);
    const double hs = 0.5 * s;
    r = r * fma(-hs * r, r, 1.5);
    r = r * fma(-hs * r, r, 1.5);
    return r;
}

// A value another thread wrote at an earlier level: with one block the writer shares this
// SM's L1 and the block barrier orders the two, so a plain (L1-cached) load is safe; across
// blocks the load must bypass L1.
__device__ __forceinline__ double ld_level(const double* p) { return gridDim.x == 1 ? *p : __ldcg(p); }

// Separates two levels: a block barrier when one block holds every column, else the
// bounded grid barrier (every block is resident: cooperative launch, grid sized by occupancy).
__device__ __forceinline__ bool level_sync(const IctArgs& a) {
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    return grid_barrier(a.istate, a.spin_limit);
}

// ------------------------------------------------------------------ level sweeps (base pattern)
//
// For volumes whose planes follow each other faster by levels than by rows (ict_form), and those without
// the row wavefront's buffer: thread <-> (y, z) column, voxel x = t - 2y - 3z, a barrier between the levels
// t = x + 2y + 3z.  A level is FP64 arithmetic on the active columns, so the blocks are sized to spread the
// columns over every SM (a volume with few columns runs one-warp blocks).  Each row issues all of its
// loads from the earlier rows before the dependency chain starts.

template <typename T>
__global__ void __launch_bounds__(kIctThreads) k_ict_fwd(IctArgs a) {
    const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz;
    const long long nxy = (long long)nx * ny, nv = a.geo.nv;
    double* Lp = a.L;
    auto P = [&](int k, long long j) -> double* { return Lp + (size_t)k * nv + j; };
    const T* d = (const T*)a.d;
    const T* g = (const T*)a.g;
    T* ipo = (T*)a.ip_out;
    const bool factor = d != nullptr;
    const double beta = a.beta;
    const double tau = factor ? a.scal[S_ICT_TAU] : 0.0;
    const int npair = ny * nz;
    const int tmax = (nx - 1) + 2 * (ny - 1) + 3 * (nz - 1);
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
    bool bad = false;
    for (int t = 0; t <= tmax; ++t) {
        for (int pr = gtid; pr < npair; pr += nthr) {
            const int y = pr % ny, z = pr / ny, x = t - 2 * y - 3 * z;
            if (x < 0 || x >= nx) continue;
            const long long i = x + (long long)nx * y + nxy * z;
            const uint8_t b = a.nb[i];
            if (!(b & NB_IN)) continue;
            const long long ja = i - 1, jb = i - nx, jc = i - nxy, jd = i + 1 - nx, je = i + 1 - nxy, jf = i + nx - nxy;
            const bool ha = b & NB_XM, hb = b & NB_YM, hc = b & NB_ZM;
            const bool hd = x + 1 < nx && y > 0 && (a.nb[jd] & NB_IN);
            const bool he = x + 1 < nx && z > 0 && (a.nb[je] & NB_IN);
            const bool hf = y + 1 < ny && z > 0 && (a.nb[jf] & NB_IN);
            auto ld = [&](bool h, int k, long long j) { return h ? ld_level(P(k, j)) : 0.0; };
            // every value from the earlier rows first (independent loads), then the chain
            const double yc = ld(hc, PL_Y, jc), ye = ld(he, PL_Y, je), yf = ld(hf, PL_Y, jf),
                         yb = ld(hb, PL_Y, jb), yd = ld(hd, PL_Y, jd), ya = ld(ha, PL_Y, ja);
            double la, lb, lc, l_d, le, lf, rii;
            if (factor) {
                const double rc = ld(hc, PL_R, jc), re = ld(he, PL_R, je), rf = ld(hf, PL_R, jf),
                             rb = ld(hb, PL_R, jb), rd = ld(hd, PL_R, jd), ra = ld(ha, PL_R, ja);
                const double e_a = ld(he, PL_A, je), f_b = ld(hf, PL_B, jf), f_d = ld(hf, PL_D1, jf),
                             b_f = ld(hb, PL_F, jb), d_a = ld(hd, PL_A, jd), d_f = ld(hd, PL_F, jd),
                             a_d = ld(ha, PL_D1, ja), a_e = ld(ha, PL_E, ja);
                auto keep = [&](bool h, double v) { return h && fabs(v) >= tau ? v : 0.0; };
                lc = keep(hc, -beta * rc);
                le = keep(he, -(lc * e_a) * re);
                lf = keep(hf, -(lc * f_b + le * f_d) * rf);
                lb = keep(hb, (-beta - lc * b_f) * rb);
                l_d = keep(hd, -(lb * d_a + le * d_f) * rd);
                la = keep(ha, (-beta - lb * a_d - lc * a_e) * ra);
                const double h = (double)d[i] + beta * (double)__popc((unsigned)(b >> 1) & 0x3fu);
                const double s = h - (((la * la + lb * lb) + (lc * lc + l_d * l_d)) + (le * le + lf * lf));
                if (!(s > 0.0)) bad = true;
                rii = s > 0.0 ? rsqrt_nr(s) : 1.0;  // the error is reported; keep the arithmetic finite
                *P(PL_R, i) = rii;
                *P(PL_A, i) = la;
                *P(PL_B, i) = lb;
                *P(PL_C, i) = lc;
                *P(PL_D1, i) = l_d;
                *P(PL_E, i) = le;
                *P(PL_F, i) = lf;
                if (ipo) ipo[i] = (T)(rii * rii);
            } else {
                rii = *P(PL_R, i);
                la = *P(PL_A, i);
                lb = *P(PL_B, i);
                lc = *P(PL_C, i);
                l_d = *P(PL_D1, i);
                le = *P(PL_E, i);
                lf = *P(PL_F, i);
            }
            const double acc = (double)g[i] - ((lc * yc + le * ye) + (lf * yf + lb * yb) + (l_d * yd + la * ya));
            *P(PL_Y, i) = acc * rii;
        }
        if (t < tmax && !level_sync(a)) return;
    }
    // reported by the back sweep, after k_ict_check: fill beyond the held pattern (which can
    // itself make a pivot of the restricted factor non-positive) takes precedence
    if (bad) atomicExch(a.istate + I_ICT_BAD, 1);
}

template <typename T>
__global__ void __launch_bounds__(kIctThreads) k_ict_bwd(IctArgs a) {
    __shared__ double sbuf[2 * 32];
    const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz;
    const long long nxy = (long long)nx * ny, nv = a.geo.nv;
    double* Lp = a.L;
    auto P = [&](int k, long long j) -> double* { return Lp + (size_t)k * nv + j; };
    T* p = (T*)a.p;
    const T* gd = (const T*)a.gdot;
    const T* gpd = (const T*)a.gpdot;
    const int npair = ny * nz;
    const int tmax = (nx - 1) + 2 * (ny - 1) + 3 * (nz - 1);
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
    double acc2[2] = {0.0, 0.0};
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.istate[I_ICT_BAD]) {
        set_err(a.istate, FM_ERR_NOT_PD);
        a.istate[I_ICT_BAD] = 0;
    }
    for (int t = tmax; t >= 0; --t) {
        for (int pr = gtid; pr < npair; pr += nthr) {
            const int y = pr % ny, z = pr / ny, x = t - 2 * y - 3 * z;
            if (x < 0 || x >= nx) continue;
            const long long i = x + (long long)nx * y + nxy * z;
            const uint8_t b = a.nb[i];
            if (!(b & NB_IN)) {
                p[i] = T(0);
                continue;
            }
            // the later rows r = i - o that hold an entry in column i: L_{r,i} = plane o of row r
            const long long ra = i + 1, rb = i + nx, rc = i + nxy, rd = i - 1 + nx, re = i - 1 + nxy, rf = i - nx + nxy;
            const bool ha = b & NB_XP, hb = b & NB_YP, hc = b & NB_ZP;
            const bool hd = x > 0 && y + 1 < ny && (a.nb[rd] & NB_IN);
            const bool he = x > 0 && z + 1 < nz && (a.nb[re] & NB_IN);
            const bool hf = y > 0 && z + 1 < nz && (a.nb[rf] & NB_IN);
            auto ld = [&](bool h, int k, long long j) { return h ? ld_level(P(k, j)) : 0.0; };
            const double s = *P(PL_Y, i) - ((ld(ha, PL_A, ra) * ld(ha, PL_Y, ra) + ld(hd, PL_D1, rd) * ld(hd, PL_Y, rd)) +
                                            (ld(hf, PL_F, rf) * ld(hf, PL_Y, rf) + ld(hb, PL_B, rb) * ld(hb, PL_Y, rb)) +
                                            (ld(he, PL_E, re) * ld(he, PL_Y, re) + ld(hc, PL_C, rc) * ld(hc, PL_Y, rc)));
            const double xi = s * *P(PL_R, i);
            *P(PL_Y, i) = xi;  // y_i becomes x_i: every row that still needs y_i is this one
            p[i] = (T)xi;
            if (gd) acc2[0] += (double)gd[i] * (double)(T)xi;
            if (gpd) acc2[1] += (double)gpd[i] * (double)(T)xi;
        }
        if (t > 0 && !level_sync(a)) return;
    }
    if (gd || gpd) {
        double out[2];
        if (last_block_reduce<2>(acc2, a.partials, (unsigned*)(a.istate + I_DONE0), out, sbuf)) {
            if (threadIdx.x == 0) {
                a.scal[S_GP] = out[0];
                a.scal[S_GPREVP] = out[1];
                if (!isfinite(out[0]) || !isfinite(out[1])) set_err(a.istate, FM_ERR_NONFINITE);
            }
        }
    }
}

// ------------------------------------------------------------------ row wavefront (base pattern)
//
// The two substitutions of the base pattern without level barriers.  A one-warp block holds 32
// consecutive rows (lane = y) of one plane z and walks them along x, each lane two steps behind the
// lane below: row y's voxel x is computed at step s = x + 2 lane, so that the -y neighbours b = (x, y-1)
// and d = (x+1, y-1) are the lower lane's values of two steps and one step ago (shuffles) and
// a = (x-1, y) is the lane's own.  The rows c = (x, y), e = (x+1, y), f = (x, y+1) of plane z-1 come
// from the block that holds that plane: e is one record per lane and step, c is the e of the step
// before, f the upper lane's e of the next step.  Records of a step go to an exchange buffer as they
// are computed and are their own ready signal, as the IC(0) sweeps' face entries are: an entry
// holds an all-ones pattern that is never stored until its value arrives, its one reader polls it
// (bounded), and sets it back.  Two more kinds of record cross between the row groups of a plane:
// the last lane's to the next group (its b and d), the first lane's to the group below in plane
// z+1 (the last lane's f).  Blocks claim their rows through a ticket in (z, y) order, so whom a
// block waits for has claimed before it.  Only steps that reach a mask voxel are walked and handed
// over.  The back substitution is the same walk mirrored.
//
// No barrier is left, and a block runs as far behind plane z-1 as the hand-off takes: 74 x 74 x 10 voxels,
// 32 coils, factor + forward 1012 -> 606 us, back substitution 904 -> 254; the level sweeps pay about 4 us
// on each of 247 levels.  A step of the factor takes about 2.5 us (512 x 512 x 1 voxels: 4.0 ms for a walk of
// 1520 steps), of which its chain of FP64 operations (one warp per SM: 16 cycles an operation, 600 cycles)
// is 0.3.  The rest is not taken apart; beside the chain a step loads its inputs two steps ahead and stores
// seven planes, at addresses a row apart from lane to lane.

constexpr int kRec = 6;  // doubles of a record: R, Y, A, B, D, F (1/L_ii, y and the entries others use)

struct IctwGeo {
    int nyb, nsteps;  // row groups per plane, steps of a group (nx + 62)
};
__device__ __forceinline__ IctwGeo ictw_geo(const Geo& g) { return {(g.ny + 31) / 32, g.nx + 62}; }

__device__ __forceinline__ double2 ldx(const double* p) {
    double2 v;
    asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ double keep_clear(double x) {  // a value that is never the unset pattern
    return __double_as_longlong(x) == -1LL ? __longlong_as_double(0x7fffffffffffffffLL) : x;
}
__device__ __forceinline__ void stx(double* p, double a, double b) {
    asm volatile("st.relaxed.gpu.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(keep_clear(a)), "d"(keep_clear(b)) : "memory");
}
__device__ __forceinline__ void stx_unset(double* p) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %1};" ::"l"(p), "l"(-1LL) : "memory");
}
__device__ __forceinline__ bool is_unset(double2 v) {
    return __double_as_longlong(v.x) == -1LL || __double_as_longlong(v.y) == -1LL;
}

// A record's N double2 at p, wanted or 0.  issue() starts the loads, take() waits for the values
// (bounded), hands the entry back and returns them.
template <int N>
struct Pending {
    double2 v[N];
    double* p;  // null: nothing wanted
    __device__ __forceinline__ void issue(double* at, bool want) {
        p = want ? at : nullptr;
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = want ? ldx(at + 2 * k) : double2{0.0, 0.0};
    }
    __device__ __forceinline__ bool missing() const {
        bool m = false;
#pragma unroll
        for (int k = 0; k < N; ++k) m |= is_unset(v[k]);
        return p && m;
    }
    __device__ __forceinline__ void take(const IctArgs& a, bool& ok) {
        long long n = 0;
        while (__any_sync(0xffffffffu, missing())) {
            if (!ok || ++n > a.spin_limit) {
                ok = false;
                if (missing()) {
                    p = nullptr;
#pragma unroll
                    for (int k = 0; k < N; ++k) v[k] = double2{0.0, 0.0};
                }
                continue;
            }
            if (missing()) {
                __nanosleep(20);
#pragma unroll
                for (int k = 0; k < N; ++k) v[k] = ldx(p + 2 * k);
            }
        }
        if (p) {
#pragma unroll
            for (int k = 0; k < N; ++k) stx_unset(p + 2 * k);
        }
    }
};

// Steps of a row group that reach a mask voxel (first > last: none).
struct Span {
    int lo, hi;
    __device__ __forceinline__ bool has(int s) const { return s >= lo && s <= hi; }
};
__device__ __forceinline__ Span ictw_span(const int4* rows, bool there, int u, bool fwd) {
    if (!there) return {1 << 30, -(1 << 30)};
    const int4 r = rows[u];
    return fwd ? Span{r.x, r.y} : Span{r.z, r.w};
}

// Exchange buffer: plane records [unit][step][lane] of kRec doubles, then edge records
// [unit][step][2] (0: the first lane's for the group below in the next plane, 1: the last lane's for
// the next group) of kRec doubles.  The substitution-only walks use the first two doubles.
__device__ __forceinline__ double* plane_rec(const IctArgs& a, const IctwGeo& w, int u, int s, int lane) {
    return a.xch + (((long long)u * w.nsteps + s) * 32 + lane) * kRec;
}
__device__ __forceinline__ double* edge_rec(const IctArgs& a, const IctwGeo& w, int u, int s, int which) {
    const long long units = (long long)w.nyb * a.geo.nz;
    return a.xch + units * w.nsteps * 32 * kRec + (((long long)u * w.nsteps + s) * 2 + which) * kRec;
}

__device__ __forceinline__ double up1(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ double down1(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// Factor (FACTOR) or apply, with the forward substitution.
template <typename T, bool FACTOR>
__global__ void __launch_bounds__(32) k_ictw_fwd(IctArgs a) {
    constexpr int C = 2;               // steps whose incoming records are in flight ahead
    constexpr int N = FACTOR ? 3 : 1;  // double2 of a record that are used
    const Geo geo = a.geo;
    const IctwGeo w = ictw_geo(geo);
    const int nx = geo.nx, ny = geo.ny, lane = threadIdx.x;
    const long long nv = geo.nv;
    const int units = w.nyb * geo.nz;
    const T* d = (const T*)a.d;
    const T* g = (const T*)a.g;
    T* ipo = (T*)a.ip_out;
    const double beta = a.beta, tau = FACTOR ? a.scal[S_ICT_TAU] : 0.0;
    double* L = a.L;
    bool bad = false, ok = true;
    for (;;) {
        int u = lane == 0 ? atomicAdd(a.ticket, 1) : 0;
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= units) break;
        const int z = u / w.nyb, yb = u % w.nyb, y = yb * 32 + lane;
        const Span me = ictw_span(a.rows, true, u, true);
        if (me.lo > me.hi) continue;
        // whom this group reads, and who reads it
        const Span rz = ictw_span(a.rows, z > 0, u - w.nyb, true), rf = ictw_span(a.rows, z > 0 && yb + 1 < w.nyb, u - w.nyb + 1, true),
                   ry = ictw_span(a.rows, yb > 0, u - 1, true);
        const Span uz = ictw_span(a.rows, z + 1 < geo.nz, u + w.nyb, true), uf = ictw_span(a.rows, z + 1 < geo.nz && yb > 0, u + w.nyb - 1, true),
                   uy = ictw_span(a.rows, yb + 1 < w.nyb, u + 1, true);
        const long long row = ((long long)z * ny + y) * nx;
        const bool row_in = y < ny;
        // plane record of producer step sp; edge record of this lane (lane 31: f at step s; lane 0: d at s)
        auto want_z = [&](int sp) { return sp <= me.hi + 2 && rz.has(sp); };
        auto issue_e = [&](Pending<N>& q, int sp) { q.issue(want_z(sp) ? plane_rec(a, w, u - w.nyb, sp, lane) : nullptr, want_z(sp)); };
        auto issue_x = [&](Pending<N>& q, int s) {
            const bool wf = lane == 31 && s <= me.hi && s >= me.lo && rf.has(s - 62), wy = lane == 0 && s <= me.hi && ry.has(s + 63);
            q.issue(wf ? edge_rec(a, w, u - w.nyb + 1, s - 62, 0) : wy ? edge_rec(a, w, u - 1, s + 63, 1) : nullptr, wf | wy);
        };
        double oR = 0, oY = 0, oA = 0, oD = 0, oE = 0, oF = 0;      // this lane's row of the step before
        double dR = 0, dY = 0, dF = 0;                              // the lower lane's, last step's d: now b
        double cR, cY, eR, eY, eA;                                  // plane z-1: c, e of this step
        {
            Pending<N> p0, p1, x0;
            issue_e(p0, me.lo);
            issue_e(p1, me.lo + 1);
            issue_x(x0, me.lo - 1);
            p0.take(a, ok);
            p1.take(a, ok);
            x0.take(a, ok);
            cR = p0.v[0].x; cY = p0.v[0].y;
            eR = p1.v[0].x; eY = p1.v[0].y; eA = N > 1 ? p1.v[N > 1 ? 1 : 0].x : 0.0;
            if (lane == 0) { dR = x0.v[0].x; dY = x0.v[0].y; dF = N > 2 ? x0.v[N - 1].y : 0.0; }
        }
        Pending<N> e[C], xr[C];
        T gv[C], dv[C];
        uint8_t nbv[C];
        double lp[C][FACTOR ? 1 : 7];  // apply: the stored row
        auto issue_own = [&](int s0) {
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const int x = s0 + q - 2 * lane;
                const bool in = row_in && (unsigned)x < (unsigned)nx;
                const long long i = row + x;
                nbv[q] = in ? a.nb[i] : (uint8_t)0;
                gv[q] = in ? g[i] : T(0);
                dv[q] = FACTOR && in ? d[i] : T(0);
                if (!FACTOR)
#pragma unroll
                    for (int k = 0; k < (FACTOR ? 1 : 7); ++k) lp[q][k] = in ? L[(size_t)k * nv + i] : 0.0;
            }
        };
#pragma unroll
        for (int q = 0; q < C; ++q) {
            issue_e(e[q], me.lo + q + 2);
            issue_x(xr[q], me.lo + q);
        }
        issue_own(me.lo);
        for (int s0 = me.lo; s0 <= me.hi; s0 += C) {
            // this chunk's incoming records and inputs; the next chunk's loads start
            double nR[C], nY[C], nA[C], nB[C], nD[C], xR[C], xY[C], xA[C], xB[C], xD[C], xF[C];
            T gg[C], dd[C];
            uint8_t bb[C];
            double ll[C][FACTOR ? 1 : 7];
#pragma unroll
            for (int q = 0; q < C; ++q) {
                e[q].take(a, ok);
                xr[q].take(a, ok);
                nR[q] = e[q].v[0].x; nY[q] = e[q].v[0].y;
                xR[q] = xr[q].v[0].x; xY[q] = xr[q].v[0].y;
                if constexpr (FACTOR) {
                    nA[q] = e[q].v[1].x; nB[q] = e[q].v[1].y; nD[q] = e[q].v[2].x;
                    xA[q] = xr[q].v[1].x; xB[q] = xr[q].v[1].y; xD[q] = xr[q].v[2].x; xF[q] = xr[q].v[2].y;
                }
                gg[q] = gv[q]; dd[q] = dv[q]; bb[q] = nbv[q];
#pragma unroll
                for (int k = 0; k < (FACTOR ? 1 : 7); ++k) ll[q][k] = lp[q][k];
            }
#pragma unroll
            for (int q = 0; q < C; ++q) {
                issue_e(e[q], s0 + C + q + 2);
                issue_x(xr[q], s0 + C + q);
            }
            issue_own(s0 + C);
#pragma unroll
            for (int q = 0; q < C; ++q) {
                const int s = s0 + q, x = s - 2 * lane;
                const long long i = row + x;
                const bool in = bb[q] & NB_IN;
                // roles: a own, d / b the lower lane's of one and two steps ago, c, e, f plane z-1
                const double aR = oR, aY = oY, bR = dR, bY = dY;
                double uR = up1(oR), uY = up1(oY), fR = down1(nR[q]), fY = down1(nY[q]);
                dR = lane == 0 ? xR[q] : uR;
                dY = lane == 0 ? xY[q] : uY;
                if (lane == 31) { fR = xR[q]; fY = xY[q]; }
                double la, lb, lc, l_d, le, lf, rii;
                if constexpr (FACTOR) {
                    const double a_d = oD, a_e = oE, b_f = dF, e_a = eA;
                    const double uA = up1(oA), uF = up1(oF);
                    double f_b = down1(nB[q]), f_d = down1(nD[q]);
                    const double d_a = lane == 0 ? xA[q] : uA;
                    dF = lane == 0 ? xF[q] : uF;
                    const double d_f = dF;
                    if (lane == 31) { f_b = xB[q]; f_d = xD[q]; }
                    auto kp = [&](double v) { return fabs(v) >= tau ? v : 0.0; };
                    lc = cR != 0.0 ? kp(-beta * cR) : 0.0;
                    le = kp(-(lc * e_a) * eR);
                    lf = kp(-(lc * f_b + le * f_d) * fR);
                    lb = bR != 0.0 ? kp((-beta - lc * b_f) * bR) : 0.0;
                    l_d = kp(-(lb * d_a + le * d_f) * dR);
                    la = aR != 0.0 ? kp((-beta - lb * a_d - lc * a_e) * aR) : 0.0;
                    const double h = (double)dd[q] + beta * (double)__popc((unsigned)(bb[q] >> 1) & 0x3fu);
                    const double sq = h - (((la * la + lb * lb) + (lc * lc + l_d * l_d)) + (le * le + lf * lf));
                    if (in && !(sq > 0.0)) bad = true;
                    rii = sq > 0.0 ? rsqrt_nr(sq) : 1.0;  // the error is reported; keep the arithmetic finite
                } else {
                    rii = ll[q][PL_R];
                    la = ll[q][FACTOR ? 0 : PL_A];
                    lb = ll[q][FACTOR ? 0 : PL_B];
                    lc = ll[q][FACTOR ? 0 : PL_C];
                    l_d = ll[q][FACTOR ? 0 : PL_D1];
                    le = ll[q][FACTOR ? 0 : PL_E];
                    lf = ll[q][FACTOR ? 0 : PL_F];
                }
                const double acc = (double)gg[q] - ((lc * cY + le * eY) + (lf * fY + lb * bY) + (l_d * dY + la * aY));
                // a row outside the mask reads as 0 everywhere
                oR = in ? rii : 0.0;
                oY = in ? acc * rii : 0.0;
                if constexpr (FACTOR) {
                    oA = in ? la : 0.0;
                    oD = in ? l_d : 0.0;
                    oE = in ? le : 0.0;
                    oF = in ? lf : 0.0;
                    lb = in ? lb : 0.0;
                }
                if (in) {
                    if (FACTOR) {
                        L[(size_t)PL_R * nv + i] = rii;
                        L[(size_t)PL_A * nv + i] = la;
                        L[(size_t)PL_B * nv + i] = lb;
                        L[(size_t)PL_C * nv + i] = lc;
                        L[(size_t)PL_D1 * nv + i] = l_d;
                        L[(size_t)PL_E * nv + i] = le;
                        L[(size_t)PL_F * nv + i] = lf;
                        if (ipo) ipo[i] = (T)(rii * rii);
                    }
                    L[(size_t)PL_Y * nv + i] = oY;
                }
                // hand over what is read: consumer steps s - 2 .. (plane), s + 62 and s - 63 (edges)
                if (s <= me.hi) {
                    if (s >= uz.lo && s <= uz.hi + 2) {
                        double* r = plane_rec(a, w, u, s, lane);
                        stx(r, oR, oY);
                        if constexpr (FACTOR) {
                            stx(r + 2, oA, lb);
                            stx(r + 4, oD, oF);
                        }
                    }
                    const bool gf = lane == 0 && uf.has(s + 62), gy = lane == 31 && s - 63 >= uy.lo - 1 && s - 63 <= uy.hi;
                    if (gf | gy) {
                        double* r = edge_rec(a, w, u, s, gf ? 0 : 1);
                        stx(r, oR, oY);
                        if constexpr (FACTOR) {
                            stx(r + 2, oA, lb);
                            stx(r + 4, oD, oF);
                        }
                    }
                }
                cR = eR; cY = eY;
                eR = nR[q]; eY = nY[q];
                if constexpr (FACTOR) eA = nA[q];
            }
        }
    }
    if (bad) atomicExch(a.istate + I_ICT_BAD, 1);
    if (!ok) set_err(a.istate, FM_ERR_TIMEOUT);
}

// The mirrored walk: lane l holds row y = 32 yb + 31 - l and walks x = nx - 1 - (s - 2 l), solving
// L' x = y with the entries of the later rows a = (x+1, y), b = (x, y+1), d = (x-1, y+1) of this plane and
// c, e, f of plane z+1; then p and its dot products, summed per row group and added in order.
template <typename T>
__global__ void __launch_bounds__(32) k_ictw_bwd(IctArgs a) {
    constexpr int C = 2;
    const Geo geo = a.geo;
    const IctwGeo w = ictw_geo(geo);
    const int nx = geo.nx, ny = geo.ny, lane = threadIdx.x;
    const long long nv = geo.nv, nxy = (long long)nx * ny;
    const int units = w.nyb * geo.nz;
    const double* L = a.L;
    T* p = (T*)a.p;
    const T* gd = (const T*)a.gdot;
    const T* gpd = (const T*)a.gpdot;
    bool ok = true;
    if (blockIdx.x == 0 && lane == 0 && a.istate[I_ICT_BAD]) {
        set_err(a.istate, FM_ERR_NOT_PD);
        a.istate[I_ICT_BAD] = 0;
    }
    for (;;) {
        int u = lane == 0 ? atomicAdd(a.ticket, 1) : 0;
        u = units - 1 - __shfl_sync(0xffffffffu, u, 0);
        if (u < 0) break;
        const int z = u / w.nyb, yb = u % w.nyb, y = yb * 32 + 31 - lane;
        const Span me = ictw_span(a.rows, true, u, false);
        double acc0 = 0.0, acc1 = 0.0;
        if (me.lo <= me.hi) {
            const bool zp = z + 1 < geo.nz, zm = z > 0;
            const Span rz = ictw_span(a.rows, zp, u + w.nyb, false), rf = ictw_span(a.rows, zp && yb > 0, u + w.nyb - 1, false),
                       ry = ictw_span(a.rows, yb + 1 < w.nyb, u + 1, false);
            const Span uz = ictw_span(a.rows, zm, u - w.nyb, false), uf = ictw_span(a.rows, zm && yb + 1 < w.nyb, u - w.nyb + 1, false),
                       uy = ictw_span(a.rows, yb > 0, u - 1, false);
            const long long row = ((long long)z * ny + y) * nx;
            const bool row_in = y < ny;
            auto want_z = [&](int sp) { return sp <= me.hi + 2 && rz.has(sp); };
            auto issue_e = [&](Pending<1>& q, int sp) { q.issue(want_z(sp) ? plane_rec(a, w, u + w.nyb, sp, lane) : nullptr, want_z(sp)); };
            auto issue_x = [&](Pending<1>& q, int s) {
                const bool wf = lane == 31 && s <= me.hi && s >= me.lo && rf.has(s - 62), wy = lane == 0 && s <= me.hi && ry.has(s + 63);
                q.issue(wf ? edge_rec(a, w, u + w.nyb - 1, s - 62, 0) : wy ? edge_rec(a, w, u + 1, s + 63, 1) : nullptr, wf | wy);
            };
            double o = 0.0, dv = 0.0, cv, ev;
            {
                Pending<1> p0, p1, x0;
                issue_e(p0, me.lo);
                issue_e(p1, me.lo + 1);
                issue_x(x0, me.lo - 1);
                p0.take(a, ok);
                p1.take(a, ok);
                x0.take(a, ok);
                cv = p0.v[0].x;
                ev = p1.v[0].x;
                if (lane == 0) dv = x0.v[0].x;
            }
            Pending<1> e[C], xr[C];
            // the entries that multiply the neighbours' values, this row's y and 1/L_ii, g and g_prev
            double lp[C][8];
            T gv[C], gpv[C];
            bool inq[C];
            auto issue_own = [&](int s0) {
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int x = nx - 1 - (s0 + q - 2 * lane);
                    const bool in = row_in && (unsigned)x < (unsigned)nx;
                    const long long i = row + x;
                    const bool ym = y > 0, yp = y + 1 < ny, xm = x > 0, xp = x + 1 < nx;
                    auto ld = [&](bool h, int pl, long long j) { return in && h ? L[(size_t)pl * nv + j] : 0.0; };
                    inq[q] = in && (a.nb[i] & NB_IN);
                    lp[q][0] = ld(xp, PL_A, i + 1);
                    lp[q][1] = ld(yp, PL_B, i + nx);
                    lp[q][2] = ld(zp, PL_C, i + nxy);
                    lp[q][3] = ld(yp && xm, PL_D1, i + nx - 1);
                    lp[q][4] = ld(zp && xm, PL_E, i + nxy - 1);
                    lp[q][5] = ld(zp && ym, PL_F, i + nxy - nx);
                    lp[q][6] = ld(true, PL_Y, i);
                    lp[q][7] = ld(true, PL_R, i);
                    gv[q] = gd && in ? gd[i] : T(0);
                    gpv[q] = gpd && in ? gpd[i] : T(0);
                }
            };
#pragma unroll
            for (int q = 0; q < C; ++q) {
                issue_e(e[q], me.lo + q + 2);
                issue_x(xr[q], me.lo + q);
            }
            issue_own(me.lo);
            for (int s0 = me.lo; s0 <= me.hi; s0 += C) {
                double nv_[C], xv[C], ll[C][8];
                T gg[C], gp[C];
                bool in_[C];
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    e[q].take(a, ok);
                    xr[q].take(a, ok);
                    nv_[q] = e[q].v[0].x;
                    xv[q] = xr[q].v[0].x;
                    gg[q] = gv[q];
                    gp[q] = gpv[q];
                    in_[q] = inq[q];
#pragma unroll
                    for (int k = 0; k < 8; ++k) ll[q][k] = lp[q][k];
                }
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    issue_e(e[q], s0 + C + q + 2);
                    issue_x(xr[q], s0 + C + q);
                }
                issue_own(s0 + C);
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int s = s0 + q;
                    const double av = o, bv = dv, uv = up1(o), fdn = down1(nv_[q]);
                    dv = lane == 0 ? xv[q] : uv;
                    const double fv = lane == 31 ? xv[q] : fdn;
                    const double t = ll[q][6] - ((ll[q][0] * av + ll[q][3] * dv) + (ll[q][5] * fv + ll[q][1] * bv) +
                                                 (ll[q][4] * ev + ll[q][2] * cv));
                    const double xi = t * ll[q][7];
                    o = in_[q] ? xi : 0.0;
                    if (in_[q]) {
                        p[row + nx - 1 - (s - 2 * lane)] = (T)xi;
                        acc0 += (double)gg[q] * (double)(T)xi;
                        acc1 += (double)gp[q] * (double)(T)xi;
                    }
                    if (s <= me.hi) {
                        if (s >= uz.lo && s <= uz.hi + 2) stx(plane_rec(a, w, u, s, lane), o, 0.0);
                        const bool gf = lane == 0 && uf.has(s + 62), gy = lane == 31 && s - 63 >= uy.lo - 1 && s - 63 <= uy.hi;
                        if (gf | gy) stx(edge_rec(a, w, u, s, gf ? 0 : 1), o, 0.0);
                    }
                    cv = ev;
                    ev = nv_[q];
                }
            }
        }
        if (gd || gpd) {
            acc0 = warp_sum(acc0);
            acc1 = warp_sum(acc1);
            int last = 0;
            if (lane == 0) {
                a.part[u] = acc0;
                a.part[units + u] = acc1;
                __threadfence();
                last = atomicAdd(a.done, 1) == units - 1;
                if (last) __threadfence();
            }
            if (__shfl_sync(0xffffffffu, last, 0)) {
                double t0 = 0.0, t1 = 0.0;
                for (int k = lane; k < units; k += 32) {
                    t0 += __ldcg(a.part + k);
                    t1 += __ldcg(a.part + units + k);
                }
                t0 = warp_sum(t0);
                t1 = warp_sum(t1);
                if (lane == 0) {
                    a.scal[S_GP] = t0;
                    a.scal[S_GPREVP] = t1;
                    if (!isfinite(t0) || !isfinite(t1)) set_err(a.istate, FM_ERR_NONFINITE);
                }
            }
        }
    }
    if (!ok) set_err(a.istate, FM_ERR_TIMEOUT);
}

// ------------------------------------------------------------------ table-driven sweeps

// Voxel at offset (dx, dy, dz) from (x, y, z), or -1 when it lies outside the grid or the mask.
__device__ __forceinline__ long long ict_nbr(const IctArgs& a, int x, int y, int z, int dx, int dy, int dz) {
    const int xj = x + dx, yj = y + dy, zj = z + dz;
    if ((unsigned)xj >= (unsigned)a.geo.nx || (unsigned)yj >= (unsigned)a.geo.ny || (unsigned)zj >= (unsigned)a.geo.nz)
        return -1;
    const long long j = xj + (long long)a.geo.nx * (yj + (long long)a.geo.ny * zj);
    return (a.nb[j] & NB_IN) ? j : -1;
}

// The factorisation and substitutions for any held pattern (a.tb), used for the grown ones: row i's
// entries in increasing column order, L_{i,j} = (H_ij - sum over the pairs (p1, p2) of o of L_{i,i+o_p1} L_{j,j+o_p2}) / L_jj, dropped below tau, then L_ii and y_i.
// Level t = x + B y + C z, with B and C chosen by the host so that every held offset points
// to a strictly lower level.
template <typename T>
__global__ void __launch_bounds__(kIctThreads) k_ictg_fwd(IctArgs a) {
    const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz;
    const long long nxy = (long long)nx * ny, nv = a.geo.nv;
    const IctTables tb = a.tb;
    const int nh = tb.nh, PY = 1 + nh;
    double* Lp = a.L;
    auto P = [&](int k, long long j) -> double* { return Lp + (size_t)k * nv + j; };
    const T* d = (const T*)a.d;
    const T* g = (const T*)a.g;
    T* ipo = (T*)a.ip_out;
    const bool factor = d != nullptr;
    const double beta = a.beta;
    const double tau = factor ? a.scal[S_ICT_TAU] : 0.0;
    const int npair = ny * nz;
    const int tmax = (nx - 1) + tb.B * (ny - 1) + tb.C * (nz - 1);
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
    bool bad = false;
    double lrow[kIctMaxOffsets];
    for (int t = 0; t <= tmax; ++t) {
        for (int pr = gtid; pr < npair; pr += nthr) {
            const int y = pr % ny, z = pr / ny, x = t - tb.B * y - tb.C * z;
            if (x < 0 || x >= nx) continue;
            const long long i = x + (long long)nx * y + nxy * z;
            const uint8_t b = a.nb[i];
            if (!(b & NB_IN)) continue;
            double rii;
            if (factor) {
                for (int k = 0; k < nh; ++k) {
                    const int h = tb.ord[k];
                    const long long j = ict_nbr(a, x, y, z, tb.off[3 * h], tb.off[3 * h + 1], tb.off[3 * h + 2]);
                    if (j < 0) {
                        lrow[h] = 0.0;
                        continue;
                    }
                    double sj = tb.hs[h] ? -beta : 0.0;
                    for (int q = tb.pp[h]; q < tb.pp[h + 1]; ++q) {
                        const double l1 = lrow[tb.pr[2 * q]];
                        if (l1 != 0.0) sj -= l1 * ld_level(P(1 + tb.pr[2 * q + 1], j));
                    }
                    const double v = sj * ld_level(P(0, j));
                    lrow[h] = fabs(v) >= tau ? v : 0.0;
                }
                double sq = 0.0;
                for (int h = 0; h < nh; ++h) sq += lrow[h] * lrow[h];
                const double sdiag = (double)d[i] + beta * (double)__popc((unsigned)(b >> 1) & 0x3fu) - sq;
                if (!(sdiag > 0.0)) bad = true;
                rii = sdiag > 0.0 ? rsqrt_nr(sdiag) : 1.0;  // the error is reported; keep the arithmetic finite
                *P(0, i) = rii;
                for (int h = 0; h < nh; ++h) *P(1 + h, i) = lrow[h];
                if (ipo) ipo[i] = (T)(rii * rii);
            } else {
                rii = *P(0, i);
                for (int h = 0; h < nh; ++h) lrow[h] = *P(1 + h, i);
            }
            double acc = (double)g[i];
            for (int h = 0; h < nh; ++h) {
                if (lrow[h] == 0.0) continue;
                const long long j = ict_nbr(a, x, y, z, tb.off[3 * h], tb.off[3 * h + 1], tb.off[3 * h + 2]);
                acc -= lrow[h] * ld_level(P(PY, j));
            }
            *P(PY, i) = acc * rii;
        }
        if (t < tmax && !level_sync(a)) return;
    }
    if (bad) atomicExch(a.istate + I_ICT_BAD, 1);
}

template <typename T>
__global__ void __launch_bounds__(kIctThreads) k_ictg_bwd(IctArgs a) {
    __shared__ double sbuf[2 * 32];
    const int nx = a.geo.nx, ny = a.geo.ny, nz = a.geo.nz;
    const long long nxy = (long long)nx * ny, nv = a.geo.nv;
    const IctTables tb = a.tb;
    const int nh = tb.nh, PY = 1 + nh;
    double* Lp = a.L;
    auto P = [&](int k, long long j) -> double* { return Lp + (size_t)k * nv + j; };
    T* p = (T*)a.p;
    const T* gd = (const T*)a.gdot;
    const T* gpd = (const T*)a.gpdot;
    const int npair = ny * nz;
    const int tmax = (nx - 1) + tb.B * (ny - 1) + tb.C * (nz - 1);
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
    double acc2[2] = {0.0, 0.0};
    if (blockIdx.x == 0 && threadIdx.x == 0 && a.istate[I_ICT_BAD]) {
        set_err(a.istate, FM_ERR_NOT_PD);
        a.istate[I_ICT_BAD] = 0;
    }
    for (int t = tmax; t >= 0; --t) {
        for (int pr = gtid; pr < npair; pr += nthr) {
            const int y = pr % ny, z = pr / ny, x = t - tb.B * y - tb.C * z;
            if (x < 0 || x >= nx) continue;
            const long long i = x + (long long)nx * y + nxy * z;
            if (!(a.nb[i] & NB_IN)) {
                p[i] = T(0);
                continue;
            }
            // the later rows r = i - o_h that hold an entry in column i: L_{r,i} = plane h of row r
            double sacc = *P(PY, i);
            for (int h = 0; h < nh; ++h) {
                const long long r = ict_nbr(a, x, y, z, -tb.off[3 * h], -tb.off[3 * h + 1], -tb.off[3 * h + 2]);
                if (r < 0) continue;
                const double l = ld_level(P(1 + h, r));
                if (l != 0.0) sacc -= l * ld_level(P(PY, r));
            }
            const double xi = sacc * *P(0, i);
            *P(PY, i) = xi;  // y_i becomes x_i: every row that still needs y_i is this one
            p[i] = (T)xi;
            if (gd) acc2[0] += (double)gd[i] * (double)(T)xi;
            if (gpd) acc2[1] += (double)gpd[i] * (double)(T)xi;
        }
        if (t > 0 && !level_sync(a)) return;
    }
    if (gd || gpd) {
        double out[2];
        if (last_block_reduce<2>(acc2, a.partials, (unsigned*)(a.istate + I_DONE0), out, sbuf)) {
            if (threadIdx.x == 0) {
                a.scal[S_GP] = out[0];
                a.scal[S_GPREVP] = out[1];
                if (!isfinite(out[0]) || !isfinite(out[1])) set_err(a.istate, FM_ERR_NONFINITE);
            }
        }
    }
}

// ------------------------------------------------------------------ fill beyond the held pattern

// Every would-be entry just outside the held pattern: at each candidate offset q (q = o_p1 -
// o_p2 for held p1, p2, pointing to an earlier voxel, not held), -(sum over its pairs of
// L_{i,i+o_p1} L_{j,j+o_p2}) / L_jj with j = i + q.  One that reaches tau sets its bit in
// tb.qflags and reports FM_ERR_FILL; the host then holds those offsets too and factors again.
// With nothing flagged no entry outside the pattern ever appears (by induction over the
// columns), so the held factor is the exact drop-tolerance factor.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_ict_check(IctArgs a) {
    const int nx = a.geo.nx, ny = a.geo.ny;
    const long long nxy = (long long)nx * ny, nv = a.geo.nv;
    const double* Lp = a.L;
    auto P = [&](int k, long long j) -> double { return Lp[(size_t)k * nv + j]; };
    const IctTables tb = a.tb;
    const double tau = a.scal[S_ICT_TAU];
    const long long nm = a.istate[I_NMASK];
    bool fill = false;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nm;
         k += (long long)gridDim.x * blockDim.x) {
        const long long i = a.vlist[k];
        const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / nxy);
        for (int q = 0; q < tb.nq; ++q) {
            double sq = 0.0;
            long long j = -2;
            for (int e = tb.qp[q]; e < tb.qp[q + 1]; ++e) {
                const double l1 = P(1 + tb.qpr[2 * e], i);
                if (l1 == 0.0) continue;
                if (j == -2) j = ict_nbr(a, x, y, z, tb.qoff[3 * q], tb.qoff[3 * q + 1], tb.qoff[3 * q + 2]);
                if (j < 0) break;
                sq += l1 * P(1 + tb.qpr[2 * e + 1], j);
            }
            if (j >= 0 && sq != 0.0 && fabs(sq * P(0, j)) >= tau) {
                atomicOr(tb.qflags + (q >> 5), 1u << (q & 31));
                fill = true;
            }
        }
    }
    if (fill) set_err(a.istate, FM_ERR_FILL);
}

// ------------------------------------------------------------------ launches

template <typename T>
int ictg_max_blocks_per_sm(int block) {
    int f = 0, b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f, k_ictg_fwd<T>, block, 0) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_ictg_bwd<T>, block, 0) != cudaSuccess) return 0;
    return f < b ? f : b;
}

template <typename T>
int ict_max_blocks_per_sm(int block) {
    int f = 0, b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&f, k_ict_fwd<T>, block, 0) != cudaSuccess) return 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_ict_bwd<T>, block, 0) != cudaSuccess) return 0;
    return f < b ? f : b;
}

template <typename T>
cudaError_t launch_ict_tau(const DataArgs& a, double droptol, int grid, cudaStream_t s) {
    k_ict_tau<T><<<grid, kThreads, 0, s>>>(a, droptol);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_ictw_fwd(const IctArgs& a, int grid, cudaStream_t s) {
    if (a.d) k_ictw_fwd<T, true><<<grid, 32, 0, s>>>(a);
    else k_ictw_fwd<T, false><<<grid, 32, 0, s>>>(a);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_ictw_bwd(const IctArgs& a, int grid, cudaStream_t s) {
    k_ictw_bwd<T><<<grid, 32, 0, s>>>(a);
    return cudaGetLastError();
}
int ictw_units(const Geo& geo) { return (geo.ny + 31) / 32 * geo.nz; }
size_t ictw_exchange_bytes(const Geo& geo) {
    return (size_t)ictw_units(geo) * (geo.nx + 62) * (32 + 2) * kRec * sizeof(double);
}
// The level sweeps wait at a grid barrier, so every block must be resident at once.  A
// cooperative launch guarantees that (or refuses the launch) even when other kernels run
// beside the sweep, e.g. the other volumes' branches of a batched graph.
template <typename T>
cudaError_t launch_ict_fwd(const IctArgs& a, int grid, int block, cudaStream_t s) {
    IctArgs copy = a;
    void* args[] = {&copy};
    return cudaLaunchCooperativeKernel((const void*)k_ict_fwd<T>, dim3(grid), dim3(block), args, 0, s);
}
template <typename T>
cudaError_t launch_ict_bwd(const IctArgs& a, int grid, int block, cudaStream_t s) {
    IctArgs copy = a;
    void* args[] = {&copy};
    return cudaLaunchCooperativeKernel((const void*)k_ict_bwd<T>, dim3(grid), dim3(block), args, 0, s);
}
template <typename T>
cudaError_t launch_ictg_fwd(const IctArgs& a, int grid, int block, cudaStream_t s) {
    IctArgs copy = a;
    void* args[] = {&copy};
    return cudaLaunchCooperativeKernel((const void*)k_ictg_fwd<T>, dim3(grid), dim3(block), args, 0, s);
}
template <typename T>
cudaError_t launch_ictg_bwd(const IctArgs& a, int grid, int block, cudaStream_t s) {
    IctArgs copy = a;
    void* args[] = {&copy};
    return cudaLaunchCooperativeKernel((const void*)k_ictg_bwd<T>, dim3(grid), dim3(block), args, 0, s);
}
template <typename T>
cudaError_t launch_ict_check(const IctArgs& a, int grid, cudaStream_t s) {
    k_ict_check<T><<<grid, kThreads, 0, s>>>(a);
    return cudaGetLastError();
}

#define FM_ICT_INST(T)                                                                   \
    template cudaError_t launch_ict_tau<T>(const DataArgs&, double, int, cudaStream_t); \
    template cudaError_t launch_ictw_fwd<T>(const IctArgs&, int, cudaStream_t);         \
    template cudaError_t launch_ictw_bwd<T>(const IctArgs&, int, cudaStream_t);         \
    template cudaError_t launch_ict_check<T>(const IctArgs&, int, cudaStream_t);        \
    template cudaError_t launch_ict_fwd<T>(const IctArgs&, int, int, cudaStream_t);     \
    template cudaError_t launch_ict_bwd<T>(const IctArgs&, int, int, cudaStream_t);     \
    template cudaError_t launch_ictg_fwd<T>(const IctArgs&, int, int, cudaStream_t);    \
    template cudaError_t launch_ictg_bwd<T>(const IctArgs&, int, int, cudaStream_t);    \
    template int ict_max_blocks_per_sm<T>(int);                                         \
    template int ictg_max_blocks_per_sm<T>(int);
FM_ICT_INST(float)
FM_ICT_INST(double)

}  // namespace fm
