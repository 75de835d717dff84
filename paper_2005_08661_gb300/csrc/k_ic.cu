// k_ic.cu -- IC(0) factorisation and triangular solves in the natural (x fastest, then y,
// then z) order, as tile wavefronts (Sec. III-B, Eq. 12; the "precondition" step of the
// Algorithm box).
//
// H = diag(d) + beta C'C on the mask voxels has, in natural order, the strictly lower
// entries E_jk = -beta for the in-mask neighbours k in {j-1, j-nx, j-nx*ny}.  The 6-neighbour
// grid graph has no triangles, so IC(0) (zero fill-in) only changes the diagonal:
//   pi_j = H_jj - sum_{k lower nbr} E_jk^2 / pi_k = d_j + beta n_j - beta^2 sum_k 1/pi_k,
//   L = (Pi + E) Pi^{-1/2},   L L' = H on H's nonzero set.
// Forward (fused with the pivots): (Pi + E) v = g  ->  v_j = (g_j + beta sum_{k lower} v_k) / pi_j.
// Back:                           (Pi + E') p = Pi v  ->  p_j = v_j + beta/pi_j sum_{k upper} p_k.
// Voxels outside the mask are identity rows with 1/pi = v = p = 0, so every sum may run over
// all grid neighbours: an outside neighbour contributes exactly 0.
//
// Parallel schedule: voxel (x, y, z) depends on (x-1, y, z), (x, y-1, z), (x, y, z-1).  The grid
// is cut into 64 x 16 x 8 tiles; a CTA claims tiles through an atomic ticket in a
// dependency-respecting order (a tile's predecessors always hold smaller tickets, so no
// co-residency is assumed) and starts the asynchronous copy of the tile's inputs into shared
// memory.  A warp holds 16 rows (lane & 15 = y) of two planes (lane >> 4), and each thread walks
// its x row one voxel per step, every row one step behind its -y neighbour and the upper plane
// one step behind the lower: the -y and -z values come from the neighbouring lanes by shuffle,
// the -x value from the thread's own register.  The four warps (z pairs) run a chunk of steps
// plus one behind each other, so that what a warp needs from the warp below was computed a whole
// chunk earlier: one barrier per chunk, none per step.  Voxel (lx, ly, lz) is computed at step
// lx + ly + tz(lz).  The back substitution is the same sweep in mirrored coordinates.  In both
// sweeps faces stream between tiles while they sweep (see "streamed faces" below): a tile runs a
// fixed number of steps behind its predecessors instead of waiting for them to finish.  The
// row-coalesced write-back of the whole tile follows the sweep.
//
// What bounds the sweeps is latency: the steps of the longest chain of voxels through the tiles
// times the time of a step, plus a hand-off (about 1.3 us) per tile on it; no pipe is more than a
// few percent busy.  A step of one warp is a chain of about 25 dependent operations (two shuffles'
// 24 cycles, the FP32 adds' 4.6 each, the reciprocal), so what a step holds beside that chain decides:
// measured on one tile, a barrier per step cost 21 to 57 cycles, a branch (a face store under an if) 20 to
// 35, a load that must follow the step's stores 30.  So a step is registers, shuffles and stores
// only: everything from outside is loaded per chunk, one record per row and step goes to a ring in
// shared memory, and a warp of its own publishes the faces from there.  Per step: forward 440 ->
// 195 cycles, back substitution 200 -> 120, against 32 x 32 x 8 tiles with a warp per plane and a
// barrier per step.  More than one CTA per SM slows the steps (780 -> 1010 cycles per forward chunk)
// more than the extra slots give: 256 x 256 x 128, forward 149 us at two, 122 at one.  The long x
// side keeps the lanes busy (64 of 95 steps) and makes hand-offs along x rare.
//
// Support mask.  A voxel outside the mask has 1/pi = v = p = 0 whatever its neighbours hold, so
// the sweeps leave out what the mask leaves empty.  fm_set_data records, per tile, the first
// and last step of each sweep that reaches a mask voxel and lists the tiles that hold any
// (ic_tiles.h).  Only listed tiles are claimed, a tile sweeps its own steps only, and
// a face entry is handed over only where the producer's and the consumer's steps both
// reach it (both sides evaluate the same test); every other incoming entry is 0.  An ellipsoid
// mask fills a quarter of its grid, and the chain through it is about half as long as the
// grid's: 256 x 256 x 128 voxels, forward 271 -> 128 us, back substitution 194 -> 118 us (with the
// 32 x 32 x 8 tiles of the time; 122 and 109 us now).
// Without a mask every tile keeps all of its steps.
//
// Pivot arithmetic.  FP64 mode uses IEEE double.  FP32 mode carries each inverse pivot as
// an unevaluated pair a + b of floats (about 46 significant bits, like double-float), but
// arranged so that the hi part a is exactly the float recurrence a_j = 1/fl(H - beta^2 sum a_k)
// -- a short dependency chain -- while b, the first-order correction, is formed from
// error-free residuals (two-sum / two-product) of that chain and the neighbours' b:
//   pi = pi_f + dpi,  dpi = (rounding residuals of pi_f) + H_lo - beta^2 (sum b_k + sum errors),
//   1/pi = a (1 + e_r - dpi a) + O(eps^2),  e_r = 1 - pi_f a  (exact by FMA),
// so b = a (e_r - dpi a) with a relative truncation of order (dpi/pi)^2 ~ 1e-14.  The GB300
// FP64 pipe issues at about 1/64 of the FP32 rate and would sit on the sweep's critical path.
#include <type_traits>

#include "fm_internal.h"
#include "ic_tiles.h"

namespace fm {

// ------------------------------------------------------------------ split pivot (FP32 mode)

__device__ __forceinline__ void two_sum(float x, float y, float& s, float& e) {
    s = __fadd_rn(x, y);
    const float bb = __fsub_rn(s, x);
    e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, bb)), __fsub_rn(y, bb));
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

struct PivScal {     // beta-derived constants of the pivot recurrence
    float bh, bl;    // beta = bh + bl
    float b2h, b2l;  // beta^2 = b2h + b2l
};

// What the forward sweep carries of a voxel and hands on: the inverse pivot (FP32: hi + lo) and
// v.  FP32 leaves its fourth float 0.  The apply-only sweep carries v alone (Ent = T).
template <typename T> struct EntOf;
template <> struct EntOf<float> { using t = float4; };   // 1/pi hi, 1/pi lo, v, 0
template <> struct EntOf<double> { using t = double2; }; // 1/pi, v

// H_jj = d_j + beta n_j of a mask voxel with n in-mask neighbours; FP32 as hH + hL (n <= 6, so
// bh * n has one rounding, recovered by FMA).
__device__ __forceinline__ double form_h(double d, int n, double beta, const PivScal&, double&) {
    return d + beta * (double)n;
}
__device__ __forceinline__ float form_h(float d, int n, double, const PivScal& c, float& hL) {
    const float fn = (float)n;
    const float bn = __fmul_rn(c.bh, fn);
    const float bn_e = __fmaf_rn(c.bh, fn, -bn);
    float hH, hE;
    two_sum(d, bn, hH, hE);
    hL = __fadd_rn(hE, __fmaf_rn(c.bl, fn, bn_e));
    return hH;
}

// 1/pi_j = 1/(H_jj - beta^2 sum_k 1/pi_k) into o, and 0 where the pivot is not positive: outside
// the mask (H = -1), or not positive definite (returns false with H >= 0).
__device__ __forceinline__ bool pivot(double hH, double, double beta, const PivScal&, double2 x, double2 y, double2 z,
                                      double2& o) {
    const double piv = hH - beta * beta * ((x.x + y.x) + z.x);
    const bool ok = piv > 0.0;
    o.x = ok ? 1.0 / piv : 0.0;
    return ok;
}
__device__ __forceinline__ bool pivot(float hH, float hL, double, const PivScal& c, float4 x, float4 y, float4 z,
                                      float4& o) {
    // hi chain: S = (a_x + a_y) + a_z, pi_f = hH - b2h S, a ~ 1/pi_f
    float s1, e1, S, e2;
    two_sum(x.x, y.x, s1, e1);
    two_sum(s1, z.x, S, e2);
    const float th = __fmul_rn(c.b2h, S);
    const float tl = __fmaf_rn(c.b2h, S, -th);
    float pf, pe;
    two_sum(hH, -th, pf, pe);
    const bool ok = pf > 0.0f;
    const float a = rcp_approx(pf);
    const float er = __fmaf_rn(-pf, a, 1.0f);  // exact residual of the reciprocal
    // lo: dpi = pe + hL - tl - b2l S - b2h (e1 + e2 + sum b)
    const float base = __fsub_rn(__fadd_rn(pe, hL), __fmaf_rn(c.b2l, S, tl));
    const float sb = __fadd_rn(__fadd_rn(__fadd_rn(x.y, y.y), z.y), __fadd_rn(e1, e2));
    const float dpi = __fmaf_rn(-c.b2h, sb, base);
    const float b = __fmul_rn(a, __fmaf_rn(-dpi, a, er));
    o.x = ok ? a : 0.0f;
    o.y = ok ? b : 0.0f;
    return ok;
}

// ------------------------------------------------------------------ asynchronous staging

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void cp4(void* s, const void* g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp8(void* s, const void* g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp16(void* s, const void* g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(s)), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_wait_all() {
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// ------------------------------------------------------------------ tile geometry

template <int C> struct Steps {
    static constexpr int n = kTX + kTY - 1 + tz<C>(kTZ - 1), chunks = (n + C - 1) / C;
    static_assert(n < 255 && chunks <= 64, "steps in a byte, chunks in a mask");
};

// Shared memory position of voxel (x, row), rows of 64; odd planes are turned by 16, so that the
// 32 lanes of a warp -- neighbouring rows at neighbouring x -- meet on two banks at most once.
__device__ __forceinline__ int vox(int x, int row) { return row * kTX + ((x + 16 * (row / kTY & 1)) & (kTX - 1)); }

// Face layout per tile (counts of values), in the sweep's own (back substitution: mirrored)
// coordinates: x face (lz, ly), y face (lz, lx), z face (t, ly) by its diagonals t = lx + ly, so
// that the entries of one step are contiguous.  The same in the global face buffer and in shared
// memory.
struct FN {
    static constexpr int x = 0, y = kTZ * kTY, z = y + kTZ * kTX, n = z + (kTX + kTY - 1) * kTY;
};
// Shared memory: two tiles of T (forward: g -> v, d -> 1/pi; back substitution: v -> p, 1/pi), the
// incoming faces, and the records of every row at the steps of the last two chunks (the z
// exchange between the warps, and what the publishing warp hands on).
template <typename T>
struct FwdSmem {
    static constexpr size_t bytes = 2 * kVox * sizeof(T) + (FN::n + 2 * kCSF * kRows) * 16;
};
template <typename T>
struct BwdSmem {
    static constexpr size_t bytes = 2 * kVox * sizeof(T) + (FN::n + 2 * kCSB * kRows) * sizeof(T);
};

// Per-tile face buffer (device): the forward sweep's records [n] (v alone in the apply-only
// sweep), then the back substitution's p [n].
template <typename T>
__host__ __device__ constexpr size_t face_bytes_per_tile() {
    return (size_t)FN::n * (16 + sizeof(T));
}
static_assert(sizeof(EntOf<float>::t) == 16 && sizeof(EntOf<double>::t) == 16, "face records of 16 bytes");

// Stage one array's tile: 16-byte copies along x where whole 16-byte pieces of an aligned row are
// inside the grid (nx a multiple of 4 floats / 2 doubles), else one element per lane.  Rows and
// columns outside the grid read 0.  kRows threads; completion by cp_wait_all.
template <typename T>
__device__ __forceinline__ void stage_tile(T* s, const T* g, int x0, int y0, int z0, const Geo& geo) {
    const int nvalid = min(kTX, geo.nx - x0);
    constexpr int per = 16 / sizeof(T), cols = kTX / per;
    if (geo.nx % per == 0 && (reinterpret_cast<uintptr_t>(g) & 15) == 0) {
#pragma unroll 8
        for (int i = threadIdx.x; i < kRows * cols; i += kRows) {
            const int r = i / cols, x = (i % cols) * per, y = y0 + r % kTY, z = z0 + r / kTY;
            T* to = s + vox(x, r);
            if (x < nvalid && y < geo.ny && z < geo.nz) {
                cp16(to, g + ((long long)z * geo.ny + y) * geo.nx + x0 + x);
            } else {
#pragma unroll
                for (int k = 0; k < per; ++k) to[k] = T(0);
            }
        }
    } else {
#pragma unroll 8
        for (int i = threadIdx.x; i < kVox; i += kRows) {
            const int r = i / kTX, x = i % kTX, y = y0 + r % kTY, z = z0 + r / kTY;
            T* to = s + vox(x, r);
            if (x < nvalid && y < geo.ny && z < geo.nz) {
                const T* from = g + ((long long)z * geo.ny + y) * geo.nx + x0 + x;
                if (sizeof(T) == 4) cp4(to, from);
                else cp8(to, from);
            } else {
                *to = T(0);
            }
        }
    }
}
// Steps of a tile's sweeps that reach a mask voxel, a byte each: first and last of the forward
// sweep, first and last of the back substitution; an empty tile has first 255, last 0.
struct Range {
    int lo, hi;
    __device__ __forceinline__ bool has(int s) const { return s >= lo && s <= hi; }
};
template <bool FWD>
__device__ __forceinline__ Range tile_range(const unsigned* range, int tile) {
    if (tile < 0) return {255, 0};
    const unsigned r = range[tile] >> (FWD ? 0 : 16);
    return {(int)(r & 255u), (int)(r >> 8 & 255u)};
}

// The lists anew, for another claim order of the same mask.
__global__ void __launch_bounds__(1024) k_ic_order(TileLists a) { list_tiles(a, blockIdx.x); }

// ------------------------------------------------------------------ streamed faces
//
// A forward tile's sweep does not wait for its predecessor tiles to finish: every voxel of a
// tile's three outgoing faces is written to the face buffer as soon as it is computed.  A
// successor's step s needs, from its -x, -y and -z neighbours, face values those tiles produce
// at their step s + 63, s + 15 and s + tz(7).  So a successor runs those many steps (and one
// hand-off) behind its predecessors instead of a whole tile behind.
//
// The face entries are their own ready signal.  Between launches every forward face entry
// holds an all-ones bit pattern -- a NaN that no FP32 / FP64 operation produces (arithmetic
// returns the canonical NaN) and that a producer never writes (canon).  A successor polls the
// entries themselves with relaxed loads: an entry that no longer holds the pattern has its
// final value for this launch (each entry is written once, element by element, with relaxed
// stores).  This spares the producer a release fence and the consumer a flag round trip
// before the data round trip: the hand-off is one store's propagation plus the poll.  Each
// entry has exactly one reader (the neighbour across that face), which writes the pattern
// back after reading it, so the buffer is ready for the next launch; the host fills it with
// the pattern when the context is created and after a device error.
//
// Extra warps per CTA fetch the faces: chunk by chunk (a few steps each), they poll the
// entries the chunk needs (bounded, with a short sleep), copy them into shared memory and
// hand the chunk to the compute warps through an mbarrier.  The compute warps synchronise
// among themselves with a named barrier and never poll global memory.

template <int NT>
__device__ __forceinline__ void bar_warps() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }
template <int NT>
__device__ __forceinline__ void bar_warps2() { asm volatile("bar.sync 2, %0;" ::"n"(NT) : "memory"); }
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

// the unset pattern of a face entry, and values kept clear of it
__device__ __forceinline__ bool unset(float x) { return __float_as_uint(x) == 0xffffffffu; }
__device__ __forceinline__ bool unset(double x) { return __double_as_longlong(x) == -1LL; }
__device__ __forceinline__ bool unset(float4 e) { return unset(e.x) || unset(e.y) || unset(e.z) || unset(e.w); }
__device__ __forceinline__ bool unset(double2 e) { return unset(e.x) || unset(e.y); }
__device__ __forceinline__ float canon(float x) { return unset(x) ? __uint_as_float(0x7fffffffu) : x; }
__device__ __forceinline__ double canon(double x) {
    return unset(x) ? __longlong_as_double(0x7fffffffffffffffLL) : x;
}
// an inverse pivot is finite by construction (0 where the pivot is not positive), and v is the
// result of a multiplication: the canonical NaN in FP32, while FP64 may carry an operand's NaN on
__device__ __forceinline__ float4 canon(float4 e) { return e; }
__device__ __forceinline__ double2 canon(double2 e) { e.y = canon(e.y); return e; }

// relaxed (gpu scope) loads and stores of face entries; a record's components are ordered by
// nothing but their own values, and unset() looks at each
__device__ __forceinline__ float ld_rlx(const float* p) {
    float v;
    asm volatile("ld.relaxed.gpu.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double ld_rlx(const double* p) {
    double v;
    asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_rlx(const float4* p) {
    float4 v;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ld_rlx(const double2* p) {
    double2 v;
    asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ void st_unset(float* p) {
    asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(-1) : "memory");
}
__device__ __forceinline__ void st_unset(double* p) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(-1LL) : "memory");
}
__device__ __forceinline__ void st_unset(float4* p) {
    asm volatile("st.relaxed.gpu.global.v4.b32 [%0], {%1, %1, %1, %1};" ::"l"(p), "r"(-1) : "memory");
}
__device__ __forceinline__ void st_unset(double2* p) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %1};" ::"l"(p), "l"(-1LL) : "memory");
}
__device__ __forceinline__ float zero_ent(const float*) { return 0.f; }
__device__ __forceinline__ double zero_ent(const double*) { return 0.0; }
__device__ __forceinline__ float4 zero_ent(const float4*) { return {0.f, 0.f, 0.f, 0.f}; }
__device__ __forceinline__ double2 zero_ent(const double2*) { return {0.0, 0.0}; }

// relaxed stores of outgoing face entries (no compiler memory clobber: nothing in the kernel reads
// the entry back)
__device__ __forceinline__ void st_rlx(float* a, float v) {
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" ::"l"(a), "f"(v));
}
__device__ __forceinline__ void st_rlx(double* a, double v) {
    asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(a), "d"(v));
}
__device__ __forceinline__ void st_rlx(float4* a, float4 v) {
    asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
}
__device__ __forceinline__ void st_rlx(double2* a, double2 v) {
    asm volatile("st.relaxed.gpu.global.v2.f64 [%0], {%1, %2};" ::"l"(a), "d"(v.x), "d"(v.y));
}

// Chunk hand-off from the fetch warp to the compute warps: one mbarrier per chunk with an
// arrival count of 1, completing one phase per tile that has the chunk.  Tiles sweep their own steps
// only, so the chunks' barriers run on by themselves: the wait parity is bit c of `par`, flipped with
// each tile that had chunk c.  The fetch warp's lane 0 arrives (release) once the chunk's faces are in shared
// memory; the compute warps wait with try_wait (acquire), which suspends the warp instead of
// spinning and, unlike an acquire load, does not wait for the warp's own outstanding global
// stores to drain.
__device__ __forceinline__ void mbar_init(unsigned long long* m, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(m)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* m) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.release.cta.shared::cta.b64 st, [%0];\n\t}"
                 ::"r"(smem_u32(m)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long* m, unsigned parity) {
    unsigned ok;
    // suspend hint 1000 ns: each call returns within about a microsecond, so spin_limit calls
    // bound the wait
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, 1000;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(m)), "r"(parity) : "memory");
    return ok != 0;
}
// Compute warps: wait until a chunk of the incoming faces is in shared memory (bounded).
__device__ __forceinline__ void wait_chunk(unsigned long long* m, unsigned parity, long long limit, int* istate) {
    long long n = 0;
    while (!mbar_try_wait(m, parity)) {
        if (++n > limit) {
            set_err(istate, FM_ERR_TIMEOUT);
            break;
        }
    }
}

// Which face entry lane `lane` of a fetch or publishing warp handles at step s: lanes 0..15 the
// z face (ly = lane), lanes 16..23 the x face of plane lane - 16, lanes 24..31 the y face of
// plane lane - 24.  With k = s - first (0 <= k < count) the entry is base + k * pitch.
template <int C>
struct FaceLane {
    int cls, lz, first, count, base, pitch;
    __device__ __forceinline__ explicit FaceLane(int lane) {
        cls = lane < 16 ? 2 : lane < 24 ? 0 : 1;
        lz = lane & 7;
        first = cls == 2 ? lane : tz<C>(lz);
        count = cls == 0 ? kTY : kTX;
        base = cls == 2 ? FN::z + lane * (kTY + 1) : cls == 0 ? FN::x + lz * kTY : FN::y + lz * kTX;
        pitch = cls == 2 ? kTY : 1;
    }
    // steps between the producer's and the consumer's use of an entry
    __device__ __forceinline__ int lag() const { return cls == 2 ? tz<C>(kTZ - 1) : cls == 0 ? kTX - 1 : kTY - 1; }
    template <typename V> __device__ __forceinline__ V pick(V x, V y, V z) const { return cls == 2 ? z : cls == 0 ? x : y; }
};

// Fetch warp `w` of `nw`: brings the incoming face entries of chunks w, w + nw, .. into shared
// memory from the neighbours' face records (tiles px, py, pz; -1: none).
template <int C, bool FWD, typename Ent, typename Face>
__device__ __forceinline__ void fetch_faces(Ent* f_in, const IcArgs& a, Face face, int px, int py, int pz, Range rg, int nch,
                                            int w, int nw, unsigned long long* mbar) {
    const FaceLane<C> fl(threadIdx.x & 31);
    const int tile = fl.pick(px, py, pz);
    const Ent* from = tile >= 0 ? face(tile) : nullptr;
    const Range rs = tile_range<FWD>(a.range, tile);
    const int lag = fl.lag();
    bool ok = true;
    for (int c = w; c < nch; c += nw) {
        Ent e[C];
        int at[C];
        unsigned todo = 0;
#pragma unroll
        for (int q = 0; q < C; ++q) {
            const int s = rg.lo + c * C + q, k = s - fl.first;
            at[q] = (unsigned)k < (unsigned)fl.count ? fl.base + k * fl.pitch : -1;
            e[q] = zero_ent((const Ent*)nullptr);  // stays 0 where the neighbour hands nothing over
            if (at[q] >= 0 && s <= rg.hi && rs.has(s + lag)) todo |= 1u << q;
        }
        // poll until every wanted entry is set (all of a round's loads are in flight together); a
        // wait that gives up leaves zeros and reports the timeout
        if (!ok) todo = 0u;
        long long tries = 0;
        while (__any_sync(0xffffffffu, todo != 0u)) {
#pragma unroll
            for (int q = 0; q < C; ++q)
                if (todo & (1u << q)) e[q] = ld_rlx(from + at[q]);
#pragma unroll
            for (int q = 0; q < C; ++q)
                if ((todo & (1u << q)) && !unset(e[q])) todo &= ~(1u << q);
            if (++tries > a.spin_limit && __any_sync(0xffffffffu, todo != 0u)) {
                ok = false;
#pragma unroll
                for (int q = 0; q < C; ++q)
                    if (todo & (1u << q)) e[q] = zero_ent((const Ent*)nullptr);
                todo = 0u;
            } else if (todo != 0u) {
                __nanosleep(20);
            }
        }
#pragma unroll
        for (int q = 0; q < C; ++q)
            if (at[q] >= 0) f_in[at[q]] = e[q];
        __syncwarp();
        if (lane_id() == 0) mbar_arrive(&mbar[c]);
    }
    if (!ok) set_err(a.istate, FM_ERR_TIMEOUT);  // the host resets the faces with the error
}

// Publishing warp: after each chunk, the face entries that the successors (tiles sx, sy, sz; -1:
// none) read go from the ring of step records to this tile's face records.  A compute warp that
// stores them itself spends 10 to 20 cycles a step on each face's predicate, address and store.
template <int C, bool FWD, typename Ent>
__device__ __forceinline__ void publish_faces(const Ent* ring, Ent* out, const IcArgs& a, int sx, int sy, int sz, Range rg,
                                              int nch) {
    const FaceLane<C> fl(threadIdx.x & 31);
    const Range r = tile_range<FWD>(a.range, fl.pick(sx, sy, sz));
    const int lag = fl.lag();
    // entry k is made at step first + lag + k by the row of the face (x face: row of entry k)
    const int lane = threadIdx.x & 31;
    const int row0 = fl.pick(fl.lz * kTY, fl.lz * kTY + kTY - 1, (kTZ - 1) * kTY + lane), drow = fl.cls == 0 ? 1 : 0;
    for (int c = 0; c < nch; ++c) {
        bar_warps<kSweep>();
#pragma unroll
        for (int q = 0; q < C; ++q) {
            const int s = rg.lo + c * C + q, k = s - lag - fl.first;
            const bool go = (unsigned)k < (unsigned)fl.count && s <= rg.hi && r.has(s - lag);
            if (go) st_rlx(out + fl.base + k * fl.pitch, canon(ring[((c & 1) * C + q) * kRows + row0 + k * drow]));
        }
    }
}

// After a tile's sweep every entry of its incoming faces has been read (the compute warps
// waited for every chunk), so they return to the unset pattern for the next launch: the x
// neighbour's x face, the y neighbour's y face and the z neighbour's z face are contiguous
// ranges of those tiles' face buffers.
template <typename E>
__device__ __forceinline__ void unset_faces(E* fx, E* fy, E* fz) {
    for (int i = threadIdx.x; i < FN::n; i += blockDim.x) {
        E* f = i < FN::y ? fx : i < FN::z ? fy : fz;
        if (f) st_unset(f + i);
    }
}

__device__ __forceinline__ float shfl_up(float v, int n) { return __shfl_up_sync(0xffffffffu, v, n); }
__device__ __forceinline__ double shfl_up(double v, int n) { return __shfl_up_sync(0xffffffffu, v, n); }

__device__ __forceinline__ float v_of(float4 e) { return e.z; }
__device__ __forceinline__ double v_of(double2 e) { return e.y; }
__device__ __forceinline__ float v_of(float e) { return e; }
__device__ __forceinline__ double v_of(double e) { return e; }

// MODE 0: pivots from d (factor + forward); MODE 1: stored 1/pi (forward only); MODE 2: as 0, and
// FP32's low parts of the inverse pivots go out too (the inspection call)
template <typename T, int MODE>
__global__ void __launch_bounds__(kThreadsF, sizeof(T) == 4 ? 2 : 1) k_ic_fwd(IcArgs a, PivScal pc) {
    using Ent = std::conditional_t<MODE != 1, typename EntOf<T>::t, T>;
    constexpr int C = kCSF;
    extern __shared__ __align__(16) unsigned char smem[];
    T* sg = (T*)smem;                 // g, then v
    T* sd = sg + kVox;                // d, then 1/pi; or stored 1/pi
    Ent* f_in = (Ent*)(sd + kVox);    // incoming faces
    Ent* ring = f_in + FN::n;         // step records [2][C][kRows]
    __shared__ int s_tile;
    __shared__ __align__(8) unsigned long long s_mbar[Steps<C>::chunks];

    const Geo geo = a.geo;
    const int nx = geo.nx, ny = geo.ny, nz = geo.nz;
    const long long nxy = (long long)nx * ny;
    const int tid = threadIdx.x, lane = tid & 31, wz = tid >> 5;
    T* v = (T*)a.v;
    T* ipo = (T*)a.ip_out;
    const T betaT = (T)a.beta;
    auto face = [&](int t) { return (Ent*)((unsigned char*)a.face + (size_t)t * face_bytes_per_tile<T>()); };

    if (tid == 0)
        for (int c = 0; c < Steps<C>::chunks; ++c) mbar_init(&s_mbar[c], 1);
    const int ntile = a.istate[I_NTILE];
    unsigned long long par = 0;  // bit c: phase parity of chunk c's barrier (one phase per tile that has the chunk)
    for (;;) {
        if (tid == 0) {
            const int t = atomicAdd(a.ticket, 1);
            s_tile = t < ntile ? a.order[t] : -1;
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int X = tile % a.ntx, Y = (tile / a.ntx) % a.nty, Z = tile / (a.ntx * a.nty);
        const int x0 = X * kTX, y0 = Y * kTY, z0 = Z * kTZ;
        const Range rg = tile_range<true>(a.range, tile);
        const int nch = (rg.hi - rg.lo) / C + 1, nvalid = min(kTX, nx - x0);
        const int px = X > 0 ? tile - 1 : -1, py = Y > 0 ? tile - a.ntx : -1, pz = Z > 0 ? tile - a.ntx * a.nty : -1;

        if (wz > kWarps) {
            fetch_faces<C, true>(f_in, a, face, px, py, pz, rg, nch, wz - kWarps - 1, kFetchF, s_mbar);
        } else if (wz == kWarps) {
            publish_faces<C, true>(ring, face(tile), a, X + 1 < a.ntx ? tile + 1 : -1, Y + 1 < a.nty ? tile + a.ntx : -1,
                                   Z + 1 < a.ntz ? tile + a.ntx * a.nty : -1, rg, nch);
        } else {
            const int ly = lane & 15, up = lane >> 4, lz = 2 * wz + up, row = lz * kTY + ly;
            // stage this tile's inputs while the predecessors are still running
            stage_tile<T>(sg, (const T*)a.g, x0, y0, z0, geo);
            stage_tile<T>(sd, (const T*)(MODE != 1 ? a.d : a.ip_in), x0, y0, z0, geo);
            // steps before the first are 0: the z exchange starts from that
            for (int i = tid; i < 2 * C * kRows; i += kRows) ring[i] = zero_ent((const Ent*)nullptr);
            // the row's neighbour bits, read one chunk ahead
            const bool row_in = y0 + ly < ny && z0 + lz < nz;
            const uint8_t* nbp = a.nb + (long long)(z0 + lz) * nxy + (long long)(y0 + ly) * nx + x0;
            unsigned nbq[C];
            auto load_bits = [&](int lx) {
#pragma unroll
                for (int q = 0; q < C; ++q) nbq[q] = row_in && (unsigned)(lx + q) < (unsigned)nvalid ? nbp[lx + q] : 0u;
            };
            if (MODE != 1) load_bits(rg.lo - ly - tz<C>(lz));
            cp_wait_all();
            bar_warps2<kRows>();

            // A step touches registers, shuffles and stores only -- a branch, or a load that has to
            // follow the step's stores, costs more than its arithmetic -- so that the compiler can run
            // one step's low parts under the next one's chain.  A lane outside its row (lx not in
            // [0, 64)) computes on the wrapped index lx & 63 and only active lanes store; an inactive
            // lane's outputs are read by no active lane at the next step.  A last chunk runs to its
            // end: steps after the last reach no mask voxel, and their entries are not handed over.
            Ent o = zero_ent((const Ent*)nullptr);  // this thread's values of the step before
            bool bad = false;
            for (int c = 0; c < nch; ++c) {
                // a row's entries belong to this thread alone, so the chunk's inputs are read, and its
                // H_jj formed, ahead of the chain
                const int s0 = rg.lo + c * C, lx0 = s0 - ly - tz<C>(lz);
                T gg[C], hH[C], hL[C];
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int i = vox(lx0 + q, row);
                    gg[q] = sg[i];
                    hH[q] = sd[i];
                    if constexpr (MODE != 1) {
                        const T h = form_h(hH[q], __popc((nbq[q] >> 1) & 0x3fu), a.beta, pc, hL[q]);
                        hH[q] = nbq[q] & NB_IN ? h : T(-1);
                    }
                }
                if (MODE != 1) load_bits(lx0 + C);
                wait_chunk(&s_mbar[c], (unsigned)(par >> c) & 1u, a.spin_limit, a.istate);
                // neighbours from outside the warp: the x-face record (used at lx = 0, in the chunk whose
                // fetch brought it), the y face (lanes ly = 0), and for the lower plane the z face or
                // what the warp below left one chunk ago
                const Ent fx = f_in[FN::x + row];
                const Ent* zp = wz == 0 ? f_in + FN::z + s0 * kTY + ly
                                        : ring + ((c + 1) & 1) * C * kRows + (2 * wz - 1) * kTY + ly;
                const int zpitch = wz == 0 ? kTY : kRows;
                Ent fy[C], fz[C];
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    fy[q] = f_in[FN::y + lz * kTX + ((lx0 + q + ly) & (kTX - 1))];
                    fz[q] = zp[q * zpitch];
                }
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int lx = lx0 + q, i = vox(lx, row);
                    const bool act = (unsigned)lx < (unsigned)kTX, first = lx == 0;
                    auto ny_ = [&](T f, T own) { const T u = shfl_up(own, 1); return ly == 0 ? f : u; };
                    auto nz_ = [&](T f, T own) { const T u = shfl_up(own, 16); return up == 0 ? f : u; };
                    if constexpr (MODE != 1) {
                        const Ent in = o;
                        Ent x, y, z;
                        x.x = first ? fx.x : in.x;
                        y.x = ny_(fy[q].x, in.x);
                        z.x = nz_(fz[q].x, in.x);
                        if constexpr (sizeof(T) == 4) {
                            x.y = first ? fx.y : in.y;
                            y.y = ny_(fy[q].y, in.y);
                            z.y = nz_(fz[q].y, in.y);
                        }
                        const T vx = first ? v_of(fx) : v_of(in), vy = ny_(v_of(fy[q]), v_of(in)), vz = nz_(v_of(fz[q]), v_of(in));
                        const T rhs = gg[q] + betaT * ((vx + vy) + vz);
                        const bool ok = pivot(hH[q], hL[q], a.beta, pc, x, y, z, o);
                        bad |= act & !ok & (hH[q] >= T(0));
                        const T vj = rhs * o.x;
                        if constexpr (sizeof(T) == 4) o.z = vj;
                        else o.y = vj;
                        if (act) sd[i] = o.x;
                        if constexpr (sizeof(T) == 4 && MODE == 2) {
                            if (act && hH[q] >= 0.f)
                                a.ip_lo_out[(long long)(z0 + lz) * nxy + (long long)(y0 + ly) * nx + x0 + lx] = o.y;
                        }
                    } else {
                        const T vx = first ? fx : o, vy = ny_(fy[q], o), vz = nz_(fz[q], o);
                        o = (gg[q] + betaT * ((vx + vy) + vz)) * hH[q];  // stored 1/pi
                    }
                    if (act) sg[i] = v_of(o);
                    ring[((c & 1) * C + q) * kRows + row] = o;
                }
                bar_warps<kSweep>();
            }
            if (bad) set_err(a.istate, FM_ERR_NOT_PD);
        }
        __syncthreads();
        // every warp: faces back to unset, then write back row-coalesced (lane = x); a voxel on a step
        // that was not swept lies outside the mask
        unset_faces<Ent>(px >= 0 ? face(px) : nullptr, py >= 0 ? face(py) : nullptr, pz >= 0 ? face(pz) : nullptr);
#pragma unroll 4
        for (int r = wz; r < kRows; r += kThreadsF / 32) {
            const int y = y0 + r % kTY, z = z0 + r / kTY;
            if (y >= ny || z >= nz) continue;
            const long long j = (long long)z * nxy + (long long)y * nx + x0;
#pragma unroll
            for (int x = lane; x < kTX; x += 32) {
                if (x >= nvalid) break;
                const bool in = rg.has(x + r % kTY + tz<C>(r / kTY));
                v[j + x] = in ? sg[vox(x, r)] : T(0);
                if (MODE != 1 && ipo) ipo[j + x] = in ? sd[vox(x, r)] : T(0);
            }
        }
        __syncthreads();
        par ^= (2ull << (nch - 1)) - 1ull;
    }
}

// Sums of the two lists part[q * n + i] over i, in the order of a block of 320 threads (thread i
// adds i, i + 320, .., then a tree over lanes and over the ten warps), whatever the block's size:
// the sums decide the step sizes, and a fixed order keeps every solve reproducible bit for bit.
// Result valid in thread 0.
__device__ __forceinline__ void sum_columns(const double* part, int n, double (&out)[2], double* sbuf /* >= 64 */) {
    constexpr int kOrder = 320;
    const int lane = threadIdx.x & 31;
    for (int w = threadIdx.x >> 5; w < kOrder / 32; w += blockDim.x >> 5) {
        double v[2] = {0.0, 0.0};
        for (int i = w * 32 + lane; i < n; i += kOrder) {
            v[0] += __ldcg(part + i);
            v[1] += __ldcg(part + n + i);
        }
        v[0] = warp_sum(v[0]);
        v[1] = warp_sum(v[1]);
        if (lane == 0) {
            sbuf[w] = v[0];
            sbuf[32 + w] = v[1];
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        out[0] = warp_sum(lane < kOrder / 32 ? sbuf[lane] : 0.0);
        out[1] = warp_sum(lane < kOrder / 32 ? sbuf[32 + lane] : 0.0);
    }
}

// Waits (bounded) for a tile's p to be in memory.
__device__ __forceinline__ bool wait_written(const int* flag, long long limit) {
    long long n = 0;
    while (ld_acquire(flag) == 0) {
        if (++n > limit) return false;
        __nanosleep(20);
    }
    return true;
}

// s + x y with Kahan compensation c, every operation rounded as written (a compiler that may
// contract across the first, zero terms would give a sum that depends on the unrolling).
__device__ __forceinline__ void kahan_add(float& s, float& c, float x, float y) {
    const float a = __fmaf_rn(x, y, -c), t = __fadd_rn(s, a);
    c = __fsub_rn(__fsub_rn(t, s), a);
    s = t;
}
__device__ __forceinline__ void kahan_add(double& s, double& c, double x, double y) {
    const double a = __fma_rn(x, y, -c), t = __dadd_rn(s, a);
    c = __dsub_rn(__dsub_rn(t, s), a);
    s = t;
}

// The dot products g'p and g_prev'p of half a unit (32 x 32 x 8 voxels at x0, y0, z0), a warp to a
// plane: each lane sums a column of 32 voxels along y in order, in T with Kahan compensation, and
// converts it to double once (per-product FP64 additions would queue on GB300's narrow FP64 pipe,
// about 1/64 of the FP32 rate); the columns are added in double.  All of a column's loads are in
// flight together.  p comes from other blocks of this launch, and only where they swept: of the
// unit's two tiles one may hold no mask voxel, and nothing has written p there.  Its rows (outside
// y in [ylo, yhi)) count as the zeros they stand for.
template <typename T>
__device__ __forceinline__ void unit_dots(const T* p, const T* g, const T* gp, int x0, int y0, int z0, int ylo, int yhi,
                                          const Geo& geo, double (&acc)[2]) {
    constexpr int B = sizeof(T) == 4 ? 32 : 16;  // voxels in flight
    static_assert(kThreadsB == 32 * kTZ, "one column per thread");
    const int x = x0 + (threadIdx.x & 31), z = z0 + (threadIdx.x >> 5);
    if (x < geo.nx && z < geo.nz) {
        T s0 = 0, c0 = 0, s1 = 0, c1 = 0;
#pragma unroll
        for (int r0 = 0; r0 < 32; r0 += B) {
            T pv[B], gv[B], qv[B];
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const int y = y0 + r0 + k;
                const long long j = ((long long)z * geo.ny + y) * geo.nx + x;
                const bool in = y >= ylo && y < yhi;
                pv[k] = in ? __ldcg(p + j) : T(0);
                gv[k] = in && g ? g[j] : T(0);
                qv[k] = in && gp ? gp[j] : T(0);
            }
#pragma unroll
            for (int k = 0; k < B; ++k) {
                kahan_add(s0, c0, gv[k], pv[k]);
                kahan_add(s1, c1, qv[k], pv[k]);
            }
        }
        acc[0] = (double)s0 - (double)c0;
        acc[1] = (double)s1 - (double)c1;
    }
}

// Back substitution: the same sweep in mirrored coordinates (lx' = 63 - lx, ly' = 15 - ly,
// lz' = 7 - lz), in which the +x, +y, +z neighbours are the predecessors.  A CTA that finds no
// more tiles turns to the dot products, a unit at a time, as soon as the unit's tiles are written
// back: most CTAs are idle by then, and a tile does not hold its CTA for them (9 us of tail after a
// 7 us sweep when it did).  A column of 32 voxels spans two tiles, so the sums wait for both: they
// end about 8 us after the last sweep.
template <typename T>
__global__ void __launch_bounds__(kThreadsB, sizeof(T) == 4 ? 2 : 1) k_ic_bwd(IcArgs a) {
    constexpr int C = kCSB;
    extern __shared__ __align__(16) unsigned char smem[];
    T* sv = (T*)smem;            // v, then p
    T* sip = sv + kVox;          // 1/pi
    T* f_in = sip + kVox;        // incoming faces
    T* ring = f_in + FN::n;      // step records [2][C][kRows]
    __shared__ int s_tile, s_yhi;
    __shared__ __align__(8) unsigned long long s_mbar[Steps<C>::chunks];
    __shared__ bool s_last;
    __shared__ double sbuf[2 * 32];

    const Geo geo = a.geo;
    const int nx = geo.nx, ny = geo.ny, nz = geo.nz;
    const long long nxy = (long long)nx * ny;
    const int tid = threadIdx.x, lane = tid & 31, wz = tid >> 5;
    T* p = (T*)a.p;
    const T* gd = (const T*)a.gdot;
    const T* gpd = (const T*)a.gpdot;
    const T beta = (T)a.beta;
    // backward faces live after each tile's forward records
    auto face = [&](int t) {
        return (T*)((unsigned char*)a.face + (size_t)t * face_bytes_per_tile<T>() + (size_t)FN::n * 16);
    };

    const int ntile = a.istate[I_NTILE];
    if (tid == 0) {
        for (int c = 0; c < Steps<C>::chunks; ++c) mbar_init(&s_mbar[c], 1);
        if (ntile == 0 && blockIdx.x == 0 && a.tile_part) a.scal[S_GP] = a.scal[S_GPREVP] = 0.0;  // empty mask
    }
    unsigned long long par = 0;  // bit c: phase parity of chunk c's barrier
    for (;;) {
        if (tid == 0) {
            const int t = atomicAdd(a.ticket, 1);
            s_tile = t < ntile ? a.order[ntile - 1 - t] : -1;
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int X = tile % a.ntx, Y = (tile / a.ntx) % a.nty, Z = tile / (a.ntx * a.nty);
        const int x0 = X * kTX, y0 = Y * kTY, z0 = Z * kTZ;
        const Range rg = tile_range<false>(a.range, tile);
        const int nch = (rg.hi - rg.lo) / C + 1, nvalid = min(kTX, nx - x0);
        const int px = X + 1 < a.ntx ? tile + 1 : -1, py = Y + 1 < a.nty ? tile + a.ntx : -1,
                  pz = Z + 1 < a.ntz ? tile + a.ntx * a.nty : -1;

        if (wz > kWarps) {
            fetch_faces<C, false>(f_in, a, face, px, py, pz, rg, nch, wz - kWarps - 1, kFetchB, s_mbar);
        } else if (wz == kWarps) {
            publish_faces<C, false>(ring, face(tile), a, X > 0 ? tile - 1 : -1, Y > 0 ? tile - a.ntx : -1,
                                    Z > 0 ? tile - a.ntx * a.nty : -1, rg, nch);
        } else {
            stage_tile<T>(sv, (const T*)a.vin, x0, y0, z0, geo);
            stage_tile<T>(sip, (const T*)a.ipb, x0, y0, z0, geo);
            for (int i = tid; i < 2 * C * kRows; i += kRows) ring[i] = T(0);
            cp_wait_all();
            bar_warps2<kRows>();

            // mirrored row (ly, lz) of the sweep and the actual row it stands for
            const int ly = lane & 15, up = lane >> 4, lz = 2 * wz + up, mrow = lz * kTY + ly, row = kRows - 1 - mrow;
            T o = 0;
            T vv[C], bi[C];
            auto load_chunk = [&](int lx) {
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int i = vox(kTX - 1 - lx - q, row);
                    vv[q] = sv[i];
                    bi[q] = beta * sip[i];
                }
            };
            load_chunk(rg.lo - ly - tz<C>(lz));
            for (int c = 0; c < nch; ++c) {
                const int s0 = rg.lo + c * C, lx0 = s0 - ly - tz<C>(lz);
                wait_chunk(&s_mbar[c], (unsigned)(par >> c) & 1u, a.spin_limit, a.istate);
                const T fx = f_in[FN::x + mrow];
                const T* zp = wz == 0 ? f_in + FN::z + s0 * kTY + ly
                                      : ring + ((c + 1) & 1) * C * kRows + (2 * wz - 1) * kTY + ly;
                const int zpitch = wz == 0 ? kTY : kRows;
                T fy[C], fz[C];
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    fy[q] = f_in[FN::y + lz * kTX + ((lx0 + q + ly) & (kTX - 1))];
                    fz[q] = zp[q * zpitch];
                }
                T v1[C], b1[C];
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    v1[q] = vv[q];
                    b1[q] = bi[q];
                }
                load_chunk(lx0 + C);
#pragma unroll
                for (int q = 0; q < C; ++q) {
                    const int lx = lx0 + q;
                    const T yu = shfl_up(o, 1), zu = shfl_up(o, 16);
                    const T x = lx == 0 ? fx : o, y = ly == 0 ? fy[q] : yu, z = up == 0 ? fz[q] : zu;
                    o = v1[q] + b1[q] * ((x + y) + z);
                    if ((unsigned)lx < (unsigned)kTX) sv[vox(kTX - 1 - lx, row)] = o;
                    ring[((c & 1) * C + q) * kRows + mrow] = o;
                }
                bar_warps<kSweep>();
            }
        }
        __syncthreads();
        // every warp: faces back to unset and write-back of p
        unset_faces<T>(px >= 0 ? face(px) : nullptr, py >= 0 ? face(py) : nullptr, pz >= 0 ? face(pz) : nullptr);
#pragma unroll 4
        for (int r = wz; r < kRows; r += kThreadsB / 32) {
            const int y = y0 + r % kTY, z = z0 + r / kTY;
            if (y >= ny || z >= nz) continue;
            const long long j = (long long)z * nxy + (long long)y * nx + x0;
#pragma unroll
            for (int x = lane; x < kTX; x += 32)
                if (x < nvalid) p[j + x] = sv[vox(x, r)];
        }
        __syncthreads();
        if (a.tile_part && tid == 0) {  // the tile's p is in memory: its unit may be summed
            __threadfence();
            st_release(a.written + tile, 1);
        }
        par ^= (2ull << (nch - 1)) - 1ull;
    }
    if (!a.tile_part) return;
    const int nhalf = 2 * a.istate[I_NUNIT];  // every unit in two halves along x
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            const int u = atomicAdd(a.unit_ticket, 1);
            s_tile = u < nhalf ? u : -1;
            if (u < nhalf) {
                const int t = a.unit[nhalf / 2 - 1 - u / 2], Y = (t / a.ntx) % a.nty;
                const bool both = !(Y & 1) && Y + 1 < a.nty && (a.range[t + a.ntx] & 255u) != 255u;
                s_yhi = min(ny, (Y + (both ? 2 : 1)) * kTY);
                bool ok = wait_written(a.written + t, a.spin_limit);
                if (both) ok = wait_written(a.written + t + a.ntx, a.spin_limit) && ok;
                if (!ok) set_err(a.istate, FM_ERR_TIMEOUT);
            }
        }
        __syncthreads();
        const int u = s_tile;
        if (u < 0) break;
        const int t = a.unit[nhalf / 2 - 1 - u / 2], X = t % a.ntx, Y = (t / a.ntx) % a.nty, Z = t / (a.ntx * a.nty);
        double acc[2] = {0.0, 0.0};
        unit_dots<T>(p, gd, gpd, X * kTX + 32 * (u & 1), (Y & ~1) * kTY, Z * kTZ, Y * kTY, s_yhi, geo, acc);
        block_sum<2>(acc, sbuf);
        if (tid == 0) {
            // by place, in blocks of 32 x 32 x 8 voxels (blocks outside the mask stay 0)
            const int n32 = (nx + 31) / 32, m32 = (ny + 31) / 32, x32 = 2 * X + (u & 1);
            const int at = x32 + n32 * ((Y >> 1) + m32 * Z);
            if (x32 < n32) {
                a.tile_part[at] = acc[0];
                a.tile_part[a.npart + at] = acc[1];
            }
            __threadfence();
            const int prev = atomicAdd(a.done, 1);
            s_last = (prev == nhalf - 1);
            if (s_last) __threadfence();
        }
        __syncthreads();
        if (s_last) {
            double tot[2];
            sum_columns(a.tile_part, a.npart, tot, sbuf);
            if (tid == 0) {
                a.scal[S_GP] = tot[0];
                a.scal[S_GPREVP] = tot[1];
                if (!isfinite(tot[0]) || !isfinite(tot[1])) set_err(a.istate, FM_ERR_NONFINITE);
            }
        }
    }
}

cudaError_t launch_ic_order(const TileLists& a, cudaStream_t s) {
    k_ic_order<<<3, 1024, 0, s>>>(a);
    return cudaGetLastError();
}

template <typename T> int ic_tz() { return kTZ; }
template <typename T> size_t ic_face_bytes_per_tile() { return face_bytes_per_tile<T>(); }

template <typename T>
static cudaError_t prep() {
    static bool done = false;  // attributes are per function, set once per process
    if (done) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_ic_fwd<T, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)FwdSmem<T>::bytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_ic_fwd<T, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FwdSmem<T>::bytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_ic_fwd<T, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FwdSmem<T>::bytes);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_ic_bwd<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)BwdSmem<T>::bytes);
    if (e == cudaSuccess) done = true;
    return e;
}

template <typename T>
int ic_max_blocks_per_sm(bool bwd) {
    if (prep<T>() != cudaSuccess) return 0;
    int n = 0;
    const cudaError_t e =
        bwd ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ic_bwd<T>, kThreadsB, BwdSmem<T>::bytes)
            : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ic_fwd<T, 0>, kThreadsF, FwdSmem<T>::bytes);
    return e == cudaSuccess ? n : 0;
}

static PivScal piv_scal(double beta) {
    PivScal c;
    c.bh = (float)beta;
    c.bl = (float)(beta - (double)c.bh);
    const double b2 = beta * beta;
    c.b2h = (float)b2;
    c.b2l = (float)(b2 - (double)c.b2h);
    return c;
}

template <typename T>
cudaError_t launch_ic_fwd(const IcArgs& a, int grid, cudaStream_t s) {
    cudaError_t e = prep<T>();
    if (e != cudaSuccess) return e;
    if (a.d && a.ip_lo_out)
        k_ic_fwd<T, 2><<<grid, kThreadsF, FwdSmem<T>::bytes, s>>>(a, piv_scal(a.beta));
    else if (a.d)
        k_ic_fwd<T, 0><<<grid, kThreadsF, FwdSmem<T>::bytes, s>>>(a, piv_scal(a.beta));
    else
        k_ic_fwd<T, 1><<<grid, kThreadsF, FwdSmem<T>::bytes, s>>>(a, piv_scal(a.beta));
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_ic_bwd(const IcArgs& a, int grid, cudaStream_t s) {
    cudaError_t e = prep<T>();
    if (e != cudaSuccess) return e;
    k_ic_bwd<T><<<grid, kThreadsB, BwdSmem<T>::bytes, s>>>(a);
    return cudaGetLastError();
}

// 1/pi = hi + lo as one double (FP32 mode's pivot pair, for inspection), 0 outside the mask
__global__ void k_inv_pivot64(const float* hi, const float* lo, double* out, const uint8_t* nb, long long nv) {
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < nv; j += (long long)gridDim.x * blockDim.x)
        out[j] = nb[j] & NB_IN ? (double)hi[j] + (double)lo[j] : 0.0;
}

cudaError_t launch_inv_pivot64(const float* hi, const float* lo, double* out, const uint8_t* nb, long long nv, int grid,
                               cudaStream_t s) {
    k_inv_pivot64<<<grid, kThreads, 0, s>>>(hi, lo, out, nb, nv);
    return cudaGetLastError();
}

#define FM_INST(T)                                                            \
    template cudaError_t launch_ic_fwd<T>(const IcArgs&, int, cudaStream_t);  \
    template cudaError_t launch_ic_bwd<T>(const IcArgs&, int, cudaStream_t);  \
    template int ic_tz<T>();                                                  \
    template size_t ic_face_bytes_per_tile<T>();                              \
    template int ic_max_blocks_per_sm<T>(bool);
FM_INST(float)
FM_INST(double)

}  // namespace fm
