// lbm_pass.cuh -- a pass: K time steps of a D2Q5 lattice (crack along +x, or
// none) in one launch, with the fields on chip between the steps.
//
// One step per launch moves the whole state through HBM (or L2) and pays a
// launch, a memory round trip and a ramp per step, whatever the arithmetic
// needs.  A pass instead gives each CTA a tile of the lattice with a halo of
// K sites (a site's value K steps on depends on the sites at most K away),
// loads it once into registers, advances it K steps -- the outermost ring of
// sites that is still right shrinks by one site per step, so after K steps
// exactly the tile's own sites are left -- and stores those.  The arithmetic
// of every site is the single step's, operation for operation, so a pass
// gives the same bits as K single steps.
//
// Tile: 8 warps (small FP64 lattices: 4) on top of one another, a warp spans 32 16-byte vectors of
// columns (128 FP32 columns), a thread holds RPT rows of one vector (w and
// wdot: 64 registers at 8 rows).  East and west neighbours come by shuffles
// within the warp, the rows between warps through shared memory (16-byte
// vectors, double buffered, one barrier per step).  With K = 8 and RPT = 8 a
// 128 x 64 tile keeps 112 x 48 sites: 1.5 times the arithmetic of a single
// step, for an eighth of its memory traffic and launches.
//
// Measured, one GB300, time per step of a run against one launch per step:
// 4096 x 2048 FP32, K-criterion 20.0 -> 6.9 us; the same on nine velocities
// 25.8 -> 9.3 us; 8192 x 8192 BF16 wdot 149 -> 36 us; 16384 x 16384 leapfrog 575
// -> 166 us; 1001 x 777 FP16 wdot, periodic sides 6.0 -> 2.3 us; 512 x 192 with
// the edge rule and two tips 11.6 -> 3.1 us; 128 x 128 FP64 10.9 -> 3.2 us.
// What bounds a bulk tile is instruction issue: half the issue slots and 45 %
// of the FMA pipes are busy, DRAM half of its copy rate.  With scalar FP32 and
// the rows moved back after each step the leapfrog kernel issued 85.7 M
// instructions per 4096^2 pass (120 us), without the moves 69.8 M (110 us),
// packed 50.7 M (98 us).  Loading the next tile's rows during a tile's steps
// (asynchronous copies, persistent CTAs) was slower (8192^2 FP32 32.8 -> 36.3
// us per step): the second resident CTA hides the loads already.  A strip
// tile's step takes 1250 cycles, an edge tile's 700 (chains of a few shuffles,
// one barrier and the rules); small lattices are bound by these.
//
// The crack strip.  The rows within 16 - K of the crack line form tiles of
// their own (32 rows, the line between warps 3 and 4), which apply the cuts
// and the crack-face rule and run the crack step of Alg. 1 before each of
// their K updates.  Their column boundaries are moved away from the tips
// (pass_boundary), so that every tile whose sites can see a link that a step
// of this pass severs also holds the K window behind that tip: such a tile
// runs the crack step itself, and all reach the same decision; the one that
// owns the tip's column records it.
#pragma once

#include "lbm_barrier.cuh"
#include "lbm_crack.cuh"
#include "lbm_d2q9.cuh"
#include "lbm_internal.cuh"
#include "lbm_rows.cuh"
#include "lbm_window.h"

#include <cstddef>
#include <type_traits>

namespace lbm {

constexpr int kPassSteps = 8;     // most steps of a pass (and no more than a tile has warps)
constexpr int kStripRpt = 4;      // rows per thread of a strip tile

// FP64 storage taken one column a thread (32-column tiles of four warps): FP64
// runs at two results a cycle and SM, so a pass lasts as long as its busiest
// SM's tile, and on small lattices the tiles have to be many and small (128^2
// with a stationary crack: 4.4 -> 3.2 us per step, 256^2 prescribed 5.9 -> 4.8).
// Where the decisions need no K, a strip tile lies anywhere (PassPlan::free):
// 32 columns would not hold the zones around the tips.
struct NarrowF64 {
    double v;
};
template <> struct WdIO<NarrowF64> {
    typedef Row<double, 1> Raw;
    static __device__ __forceinline__ void fetch(const NarrowF64 *p, Raw &r) { r.v[0] = p->v; }
    static __device__ __forceinline__ void unpack(const Raw &q, Row<double, 1> &r, double) { r = q; }
    static __device__ __forceinline__ void store(NarrowF64 *p, const Row<double, 1> &r, double) { p->v = r.v[0]; }
    static __device__ __forceinline__ void put(NarrowF64 *p, double v, double) { p->v = v; }
};
template <typename T, typename D> struct PassVec { static constexpr int N = Vec<T>::N; };
template <> struct PassVec<double, NarrowF64> { static constexpr int N = 1; };
__device__ __forceinline__ void ldg_row(const double *p, Row<double, 1> &r) { r.v[0] = __ldg(p); }
__device__ __forceinline__ void ld_row(const double *p, Row<double, 1> &r) { r.v[0] = *p; }
__device__ __forceinline__ void stg_row(double *p, const Row<double, 1> &r) { *p = r.v[0]; }

// One site's wdot as the next step reads it back from storage.
template <typename D, typename T> __device__ __forceinline__ T wd_round(T v, T, T) { return v; }
template <> __device__ __forceinline__ float wd_round<__nv_bfloat16, float>(float v, float, float)
{
    return __bfloat162float(__float2bfloat16_rn(v));
}
template <> __device__ __forceinline__ float wd_round<__half, float>(float v, float scale, float inv)
{
    return __half2float(__float2half_rn(v * scale)) * inv;
}
template <typename D, typename T, int N>
__device__ __forceinline__ void wd_store(D *p, const Row<T, N> &r, T scale)
{
    if constexpr (std::is_same<D, Lf>::value) stg_row(reinterpret_cast<float *>(p), r);
    else WdIO<D>::store(p, r, scale);
}
template <typename D, typename T> __device__ __forceinline__ void wd_put(D *p, T v, T scale)
{
    if constexpr (std::is_same<D, Lf>::value) p->v = v;
    else WdIO<D>::put(p, v, scale);
}

// Two neighbouring ones at once: the packed conversions run at the ALU's
// rate, the scalar ones at an eighth of it (8192 x 8192 BF16: 68 us a step
// with those, against 32 us for FP32 wdot).
template <typename D> __device__ __forceinline__ void wd_round2(float &a, float &b, float scale, float inv)
{
    if constexpr (std::is_same<D, __nv_bfloat16>::value) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
        const uint32_t u = *reinterpret_cast<const uint32_t *>(&h);
        a = __uint_as_float(u << 16);
        b = __uint_as_float(u & 0xffff0000u);
    } else if constexpr (std::is_same<D, __half>::value) {
        const float2 f = __half22float2(__floats2half2_rn(a * scale, b * scale));
        a = f.x * inv;
        b = f.y * inv;
    }
}

// Two FP32 operations in one instruction (each rounded as the scalar one).
// They do not raise the FP32 rate, but halve the instructions a row issues,
// and a tile is bound by instruction issue.
__device__ __forceinline__ uint64_t pk2(float a, float b)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void up2(uint64_t v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// (new - old) / dt; exact without the division where dt = 1.  The division is
// a call of its own, so that it is not computed and dropped there (inlined, it
// was: with the slow path it takes for zeros, the crack-face rule of a strip
// tile cost 850 cycles a step).
template <typename T> static __device__ __noinline__ T div_dt(T d, T dt) { return d / dt; }
template <typename T, int N> __device__ __forceinline__ Row<T, N> rate_of(const Row<T, N> &wn, const Row<T, N> &w0, T dt)
{
    Row<T, N> d;
#pragma unroll
    for (int k = 0; k < N; ++k) d.v[k] = wn.v[k] - w0.v[k];
    if (dt != (T)1) {
#pragma unroll
        for (int k = 0; k < N; ++k) d.v[k] = div_dt(d.v[k], dt);
    }
    return d;
}

// What the row next to an edge receives over it: its own values (free), 2 w* -
// w (Dirichlet).
template <typename T, int N>
__device__ __forceinline__ Row<T, N> edge_image(const Row<T, N> &w, bool dirichlet, T two_ws)
{
    Row<T, N> o;
#pragma unroll
    for (int k = 0; k < N; ++k) o.v[k] = dirichlet ? two_ws - w.v[k] : w.v[k];
    return o;
}

// The update of one row segment (site_update of each of its sites): cu the
// row, up and dn the rows above and below, hs the sums of the east and west
// neighbours; d: wdot, updated in place as storage rounds it (leapfrog: the
// w before, left alone).
template <typename T, typename D, int N>
__device__ __forceinline__ void row_sites(const Row<T, N> &cu, const Row<T, N> &up, const Row<T, N> &dn, const Row<T, N> &hs,
                                          Row<T, N> &d, T g, T dt, T wd_scale, T wd_inv, Row<T, N> &out)
{
    constexpr bool kLf = std::is_same<D, Lf>::value;
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int k = 0; k < N; k += 2) {
            const uint64_t c = pk2(cu.v[k], cu.v[k + 1]);
            const uint64_t v = add2(pk2(up.v[k], up.v[k + 1]), pk2(dn.v[k], dn.v[k + 1]));
            const uint64_t lap = fma2(pk2(-4.0f, -4.0f), c, add2(v, pk2(hs.v[k], hs.v[k + 1])));
            if constexpr (kLf) {
                // w + ((w - w_{n-1}) + (g dt) lap)
                const uint64_t e = fma2(pk2(-1.0f, -1.0f), pk2(d.v[k], d.v[k + 1]), c);
                const float gd = g * dt;
                up2(add2(c, fma2(pk2(gd, gd), lap, e)), out.v[k], out.v[k + 1]);
            } else {
                const uint64_t dn2 = fma2(pk2(g, g), lap, pk2(d.v[k], d.v[k + 1]));
                up2(fma2(pk2(dt, dt), dn2, c), out.v[k], out.v[k + 1]);
                up2(dn2, d.v[k], d.v[k + 1]);
                wd_round2<D>(d.v[k], d.v[k + 1], wd_scale, wd_inv);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const T lap = ((up.v[k] + dn.v[k]) + hs.v[k]) - (T)4 * cu.v[k];
            T wn, dn_;
            site_update<T, D>(cu.v[k], d.v[k], lap, g, dt, wn, dn_);
            d.v[k] = dn_;
            out.v[k] = wn;
        }
    }
}

// The same with eight neighbours: axis and diag hold the sums over the axis
// and the diagonal neighbours.
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
template <typename T, int N>
__device__ __forceinline__ void row_sites9(const Row<T, N> &cu, const Row<T, N> &axis, const Row<T, N> &diag, Row<T, N> &d, T ga,
                                           T gd, T dt, Row<T, N> &out)
{
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int k = 0; k < N; k += 2) {
            const uint64_t c = pk2(cu.v[k], cu.v[k + 1]), m4 = pk2(-4.0f, -4.0f);
            const uint64_t ax = fma2(m4, c, pk2(axis.v[k], axis.v[k + 1])), di = fma2(m4, c, pk2(diag.v[k], diag.v[k + 1]));
            // d9_rate and d9_integrate
            const uint64_t r = add2(pk2(d.v[k], d.v[k + 1]), fma2(pk2(ga, ga), ax, mul2(pk2(gd, gd), di)));
            up2(r, d.v[k], d.v[k + 1]);
            up2(fma2(pk2(dt, dt), r, c), out.v[k], out.v[k + 1]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const T ax = axis.v[k] - (T)4 * cu.v[k], di = diag.v[k] - (T)4 * cu.v[k];
            d.v[k] = d9_rate(d.v[k], ax, di, ga, gd);
            out.v[k] = d9_integrate(cu.v[k], d.v[k], dt);
        }
    }
}

// The crack state in force during one update of a pass, and the records of
// the crack step before it (lazy: its K and pairs are formed at the end).
struct PassTip {
    int64_t tr, tl;
    double vr, vl, Kr, Kl, vp_r, vp_l;   // vp: the speed before it (its window's, eq. r(v))
    int32_t f, l, npr, npl;
    int32_t arr_r, arr_l, lazy, pad;
};

template <typename T, int NW, int N = Vec<T>::N>
struct PassShared {
    static constexpr int W = 32 * N;
    alignas(16) T top[2][NW][W];    // each warp's last row, by step parity
    alignas(16) T bot[2][NW][W];    // each warp's first row
    alignas(16) T pair[kPassSteps][2][W];   // rows jc - 1 and jc of a strip tile at each step
    T ws[4][kPassSteps + 1], ws2[4][kPassSteps + 1];   // w* of the Dirichlet edges at t_n .. t_{n+K}, and twice that
    PassTip log[kPassSteps + 1];
    CrackState in;                          // the state the pass starts from
    CrackState S;
    int32_t reach[2];
};

// What a pass of the adjoint's recording (kRecord) or sweep (kAdjoint) keeps
// besides: the tile's sensors, in ascending order, and their values at each
// step (recording: w; sweep: the sources 2 r).
template <typename T, int MODE> struct PassSensors {
    int32_t n;
    int32_t i[2 * kPassSensors], j[2 * kPassSensors], k[2 * kPassSensors];
    T v[kPassSteps][2 * kPassSensors];
};
template <typename T> struct PassSensors<T, kForward> {};
template <typename T> struct PassSensors<T, kNine> {};

struct TileGeo {
    int xl, x0, x1, yl, y0, y1;   // first column held, own columns [x0, x1); first row held, own rows [y0, y1)
};

__device__ __forceinline__ int pass_floor(int x, int n) { return x >= 0 ? x / n * n : -((-x + n - 1) / n * n); }
__device__ __forceinline__ int pass_ceil(int x, int n) { return -pass_floor(-x, n); }

// The columns of the two tips: where the next link of each end would be cut.
__device__ __forceinline__ int tip_col_r(int i_first, int i_last, int nx)
{
    return min(max(max(i_last + 1, i_first), 0), nx - 1);
}
__device__ __forceinline__ int tip_col_l(int i_first, int i_last, int nx)
{
    return min(max(min(i_first - 1, i_last), 0), nx - 1);
}

// Boundary b of the strip's column tiles, moved out of the zones around the
// tips: a tile left of a boundary inside the zone ahead of a tip would see
// the cuts without the K window behind it.  lo / hi: the forbidden
// boundaries of each tip (one interval where they overlap).
template <int N>
__device__ __forceinline__ int pass_boundary(int b, int nx, bool per, int lo0, int hi0, int lo1, int hi1, bool two)
{
    for (int sh = per ? -1 : 0; sh <= (per ? 1 : 0); ++sh) {
        const int o = sh * nx;
        if (b >= lo0 + o && b <= hi0 + o) {
            const int l = pass_floor(lo0 + o - 1, N), h = pass_ceil(hi0 + o + 1, N);
            b = b - l <= h - b ? l : h;
            break;
        }
        if (two && b >= lo1 + o && b <= hi1 + o) {
            const int l = pass_floor(lo1 + o - 1, N), h = pass_ceil(hi1 + o + 1, N);
            b = b - l <= h - b ? l : h;
            break;
        }
    }
    if (!per) {
        if (b < 4) b = 0;
        if (nx - b < 4) b = nx;
    }
    return b;
}

// The one pair a K window of at most one spacing can hold: the nearest column
// at least lo_q behind the tip, d its distance (units of 2^-32 dh).
struct PassPair {
    int32_t col, in;
    int64_t d;
};
__device__ __forceinline__ PassPair pass_pair(int dir, int64_t tip, int64_t lo_q, int64_t hi_q, int f, int l)
{
    const int64_t half = (int64_t)1 << (kQBits - 1);
    const int64_t i = dir > 0 ? (tip - lo_q - half) >> kQBits : (tip + lo_q - half + ((int64_t)1 << kQBits) - 1) >> kQBits;
    const int64_t xq = (2 * i + 1) * half;
    PassPair r;
    r.d = dir > 0 ? tip - xq : xq - tip;
    r.in = r.d >= lo_q && r.d < hi_q && i >= f && i <= l;
    r.col = (int)i;
    return r;
}

// sqrt(r / 2 pi) of a pair, and K from it (the sums of crack_eval_pairs over one pair).
__device__ __forceinline__ double pass_sf(const CrackParams &p, int64_t d)
{
    const double r_h = (double)d * kTwoM32;
    const double r = p.dh == 1.0 ? r_h : r_h * p.dh;
    return sqrt(div_known(r, 2.0 * kPi, 1.0 / (2.0 * kPi)));
}
template <typename T>
__device__ __forceinline__ CrackSums pass_sums(double sf, T above, T below, double r_min)
{
    const double delta = (double)above - (double)below;
    return CrackSums{delta * sf, sf * sf, r_min, 1};
}
__device__ __forceinline__ double pass_K(const CrackParams &p, const CrackSums &c)
{
    return c.np > 0 ? p.mu / 4.0 * c.num / c.den : 0.0;
}

// What a lane of warp 0 keeps to see that an end at rest stays at rest: the
// column of its pair of the K window (lanes 0-15 the right end, 16-31 the
// left; -1: none) and the pair's weight in K, in FP32.
struct PassWindow {
    int64_t tip;     // the tip they belong to
    float coef;
    int32_t col;
};

// The window of an end at rest (v = 0).  Its bounds are exact: r = d 2^-32
// for the integer distance d between tip and column, and lo_q, hi_q are the
// least integers with d 2^-32 >= r_min, >= r_min + W.
__device__ __forceinline__ void pass_window(const PassPlan &q, const CrackState &S, int org, bool ev,
                                            PassWindow &w)
{
    const int lane = threadIdx.x & 31, l = lane & 15;
    const bool right = lane < 16;
    const int64_t tip = right ? S.r.tip_q : S.l.tip_q, half = (int64_t)1 << (kQBits - 1);
    const int64_t i = right ? ((tip - q.lo_q - half) >> kQBits) - l
                            : ((tip + q.lo_q - half + ((int64_t)1 << kQBits) - 1) >> kQBits) + l;
    const int64_t xq = (2 * i + 1) * half, d = right ? tip - xq : xq - tip;
    const bool in = ev && d >= q.lo_q && d < q.hi_q && i >= S.i_first && i <= S.i_last;
    const float r = in ? (float)d : 0.0f;
    const float sf = sqrtf(r);
    float den = r;
    int np = in ? 1 : 0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        den += __shfl_xor_sync(0xffffffffu, den, o);
        np += __shfl_xor_sync(0xffffffffu, np, o);
    }
    // |K| <= sum |coef delta| <= np max |coef delta|, K = mu / 4 sum(delta sf) / sum(sf^2), sf = sqrt(r / 2 pi)
    w.tip = tip;
    w.col = in ? (int)(i - org) : -1;
    w.coef = in ? (float)np * q.k_unit * sf / den : 0.0f;
}

// One K-criterion crack step of a strip tile by warp 0 (all 32 lanes): the
// ends this tile follows, from the pair rows of the current fields.  below /
// above: rows jc - 1 and jc of the tile, column i at i - org (org_l for the
// left end).  An end at rest whose K is below K_C by a margin far larger
// than FP32 rounding stays at rest: that costs one product and a vote, and
// its K, which decides nothing, is formed for the history at the end of the
// pass (the exact step is a chain of FP64 divisions, roots and a tanh: 64
// cycles per operation on GB300, 1.5 us at rest and 3.7 us growing).
template <typename T, int W>
__device__ __forceinline__ void pass_crack_step(const CrackParams &p, const PassPlan &q, const T *below, const T *above,
                                                int org_r, int org_l, CrackState &S, PassTip &rec, bool ev_r, bool ev_l,
                                                PassWindow &win)
{
    const int lane = threadIdx.x & 31;
    const bool act_r = ev_r && !S.r.decided, act_l = ev_l && !S.l.decided;
    // lanes 0-15 the right end, 16-31 the left: both criteria on the state before either advances
    const int dir = lane < 16 ? +1 : -1;
    const TipState &E = dir > 0 ? S.r : S.l;
    const int org = dir > 0 ? org_r : org_l;
    const bool act = dir > 0 ? act_r : act_l;
    const bool rest = (__double_as_longlong(E.v_prev) << 1) == 0;   // v_prev = 0
    if (__any_sync(0xffffffffu, act && rest && E.tip_q != win.tip)) pass_window(q, S, org, dir > 0 ? ev_r : ev_l, win);
    float t = 0.0f;
    if (win.col >= 0 && win.col < W) t = fabsf(win.coef * (float)(above[win.col] - below[win.col]));
    const bool hot = act && !(rest && (E.arrested || t < q.k_rest));
    const bool pending = !S.r.decided;
    if (!__any_sync(0xffffffffu, hot)) {
        __syncwarp();
        if (lane == 0) {
            if (act_r) {
                S.r.v = 0.0;
                S.r.grew = 0;
            }
            if (act_l) {
                S.l.v = 0.0;
                S.l.grew = 0;
            }
            rec.lazy = 1;
            rec.vr = rec.vl = 0.0;
        }
    } else {
        CrackSums c = {0.0, 0.0, 0.0, 0};
        CrackDecision d = {};
        const bool head = (lane & 15) == 0 && act;
        bool full = !q.one_pair || !q.unit;
        if (!full && head) {
            // dh = dt = 1 and a window of at most one pair: its column from
            // r_min in FP32 (exact unless a column lies within the slack of the
            // window's ends), and no FP64 operation that does not decide
            const float lo = rest ? q.lo_f : window_start(q.lo_f, E.v_prev);
            const int64_t lo_q = (int64_t)(lo * 4294967296.0f);
            const PassPair w = pass_pair(dir, E.tip_q, lo_q, lo_q + ((int64_t)1 << kQBits), S.i_first, S.i_last);
            const int64_t past = w.d - lo_q;   // in [0, 2^32)
            full = !(lo < q.lo_max) || (uint32_t)past + q.slack < 2u * q.slack || (uint32_t)(past - q.w_q) + q.slack < 2u * q.slack;
            const int k = w.col - org;
            if (w.in && past < q.w_q && k >= 0 && k < W) c = pass_sums<T>(pass_sf(p, w.d), above[k], below[k], 0.0);
            if (!full) {
                // crack_decide for K-criterion growth
                d.K = pass_K(p, c);
                d.flags = E.flags;
                const double Ka = fabs(d.K);
                if (c.np > 0 && Ka > p.K_C) {
                    const double ratio = div_known(Ka, p.K_C, q.k_inv);
                    d.propagate = 1;
                    d.v = p.v_max * tanh(sqrt(ratio * ratio * ratio * ratio - 1.0));   // eq. v-tanh
                }
                full = huge_K(Ka);
                if (E.arrested) {
                    d.propagate = 0;
                    d.v = 0.0;
                }
                if (d.propagate) d.dq = __double2ll_rn(d.v * p.cs * 4294967296.0);
            }
        }
        if (__any_sync(0xffffffffu, full)) {
            c = crack_eval_pairs<T, 16>(p, E.tip_q, E.v_prev, S.i_first, S.i_last, dir, [&](int i, T &a, T &b) {
                const int k = i - org;
                if (k < 0 || k >= W) return false;   // an end this tile does not follow
                a = above[k];
                b = below[k];
                return true;
            });
            if (head) d = crack_decide(p, S, dir, c);
        }
        if (lane == 0) rec.vp_r = S.r.v_prev;
        if (lane == 16) rec.vp_l = S.l.v_prev;
        const History none = {};
        __syncwarp();
        if (lane == 0 && act_r) crack_commit(p, nullptr, none, S, +1, false, c, d);
        __syncwarp();
        if (lane == 16 && act_l) crack_commit(p, nullptr, none, S, -1, false, c, d);
        __syncwarp();
        if (lane == 0) {
            rec.lazy = 0;
            rec.vr = S.r.v;
            rec.vl = S.l.v;
            rec.Kr = S.r.K;
            rec.Kl = S.l.K;
            rec.npr = S.r.npairs;
            rec.npl = S.l.npairs;
        }
    }
    if (lane == 0) {
        rec.tr = S.r.tip_q;
        rec.tl = S.l.tip_q;
        rec.f = S.i_first;
        rec.l = S.i_last;
        S.hist_n += pending ? 1 : 0;
        S.r.decided = 0;
        S.l.decided = 0;
    }
    __syncwarp();
}

// The crack steps of a pass whose decisions need no K, one after another by
// one thread: the state in force during each update.
static __device__ __noinline__ void pass_known_serial(const CrackParams &p, CrackState S, PassTip *log, int K)
{
    const History none = {};
    for (int s = 0; s <= K; ++s) {
        log[s].tr = S.r.tip_q;
        log[s].tl = S.l.tip_q;
        log[s].vr = S.r.v;
        log[s].vl = S.l.v;
        log[s].f = S.i_first;
        log[s].l = S.i_last;
        log[s].arr_r = S.r.arrested;
        log[s].arr_l = S.l.arrested;
        log[s].lazy = 1;
        if (s == K) break;
        const bool grow = p.mode == CRACK_PRESCRIBED;
        const CrackSums c = {0.0, 0.0, 0.0, 0};
        for (int dir = 1; dir >= (p.two_tips ? -1 : 1); dir -= 2) {
            TipState &E = dir > 0 ? S.r : S.l;
            if (E.decided) continue;
            CrackDecision d;
            d.K = E.K;
            d.v = grow && !E.arrested ? p.v_rel : 0.0;
            d.dq = p.dq_prescribed;
            d.propagate = grow && !E.arrested ? 1 : 0;
            d.flags = E.flags;
            crack_commit(p, nullptr, none, S, dir, false, c, d);
        }
        S.r.decided = 0;
        S.l.decided = 0;
    }
}

// The same in closed form, entry s by lane s of a warp (0 <= s <= K): an end
// that grows has advanced s times by the prescribed distance or stopped at
// the body's side.  For a crack that has links (first <= last): the ends do
// not touch each other's columns.
__device__ __forceinline__ void pass_known_lane(const CrackParams &p, const CrackState *st, int s, PassTip &t)
{
    const int64_t half = (int64_t)1 << (kQBits - 1);
    const bool grow = p.mode == CRACK_PRESCRIBED;
    t.f = st->i_first;
    t.l = st->i_last;
    t.lazy = 1;
    {
        const int64_t tip = st->r.tip_q, m = max(0, s - (st->r.decided ? 1 : 0)), dq = p.dq_prescribed;
        const bool arr = st->r.arrested != 0, go = grow && !arr;
        int64_t q = go ? tip + m * dq : tip;
        const bool stop = go && m > 0 && q >= p.clamp_q, before = arr || (go && m > 1 && tip + (m - 1) * dq >= p.clamp_q);
        if (stop) q = p.clamp_q;
        t.tr = q;
        t.arr_r = arr || stop;
        t.vr = grow && !before ? p.v_rel : 0.0;
        if (q > tip) t.l = max(t.l, min((int)((q - half) >> kQBits), p.nx - 1));
    }
    t.tl = st->l.tip_q;
    t.arr_l = 0;
    t.vl = 0.0;
    if (p.two_tips) {
        const int64_t tip = st->l.tip_q, m = max(0, s - (st->l.decided ? 1 : 0)), dq = p.dq_prescribed;
        const bool arr = st->l.arrested != 0, go = grow && !arr;
        int64_t q = go ? tip - m * dq : tip;
        const bool stop = go && m > 0 && q <= 0, before = arr || (go && m > 1 && tip - (m - 1) * dq <= 0);
        if (stop) q = 0;
        t.tl = q;
        t.arr_l = arr || stop;
        t.vl = grow && !before ? p.v_rel : 0.0;
        if (q < tip) t.f = min(t.f, max((int)((q - half + ((int64_t)1 << kQBits) - 1) >> kQBits), 0));
    }
}

// A column index taken around a lattice with periodic sides.
__device__ __forceinline__ int wrap_col(int c, int nx)
{
    c %= nx;
    return c < 0 ? c + nx : c;
}

// Rows and values that an earlier pass of the same launch may have written:
// from L2, past the L1 caches.
__device__ __forceinline__ void cg_row(const float *p, Row<float, 4> &r)
{
    const float4 q = __ldcg(reinterpret_cast<const float4 *>(p));
    r.v[0] = q.x; r.v[1] = q.y; r.v[2] = q.z; r.v[3] = q.w;
}
__device__ __forceinline__ void cg_row(const double *p, Row<double, 1> &r) { r.v[0] = __ldcg(p); }
__device__ __forceinline__ void cg_row(const double *p, Row<double, 2> &r)
{
    const double2 q = __ldcg(reinterpret_cast<const double2 *>(p));
    r.v[0] = q.x; r.v[1] = q.y;
}
template <typename D, typename Raw> __device__ __forceinline__ void cg_raw(const D *p, Raw &r)
{
    if constexpr (std::is_same<D, Lf>::value) cg_row(reinterpret_cast<const float *>(p), r);
    else if constexpr (std::is_same<D, NarrowF64>::value) cg_row(reinterpret_cast<const double *>(p), r);
    else if constexpr (sizeof(D) == 2) r = __ldcg(reinterpret_cast<const uint2 *>(p));
    else cg_row(p, r);
}
template <typename T> __device__ __forceinline__ T cg_get(const T *p) { return __ldcg(p); }
template <typename D, typename T> __device__ __forceinline__ T cg_rate_get(const D *p, T inv)
{
    if constexpr (std::is_same<D, Lf>::value) return __ldcg(reinterpret_cast<const float *>(p));
    else if constexpr (std::is_same<D, NarrowF64>::value) return __ldcg(reinterpret_cast<const double *>(p));
    else if constexpr (sizeof(D) == 2) {
        const unsigned short u = __ldcg(reinterpret_cast<const unsigned short *>(p));
        if constexpr (std::is_same<D, __half>::value) return __half2float(__ushort_as_half(u)) * inv;
        else return __uint_as_float((uint32_t)u << 16);
    } else return __ldcg(p);
}

// The buffers of one pass, and what write_pads reads of them.
template <typename T, typename D> struct PassBuf {
    const T *w_in;
    const D *wd_in;
    T *w_out;
    D *wd;
    const CrackState *s_in;
    CrackState *s_out;
    const int64_t *cnt_in;   // adjoint: the step counter
    int64_t *cnt_out;
};
template <typename T> struct PassPads {
    T *w_out;
    int64_t pitch;
    int32_t nx, ny;
    int32_t edge[4];
};

// What a thread knows about its tile.
struct PassCtx {
    TileGeo g;
    int lane, warp, x0, jb;
    bool per;
    bool is_l;                  // element 0 is column 0 (no periodic sides)
    int kr;                     // the element that is column nx - 1, else -1
    bool side;                  // the warp holds column 0 or nx - 1
    // the warp's rows: its last is ny - 1, its first 0; rows 0 or ny - 1 lie
    // inside them, or nx - 1 inside a vector
    bool has_t, has_b, odd;
    // strip tiles: whether the pass's decisions need no K; the ends this tile
    // follows (a link it can see may be cut in this pass); the ends whose
    // records it writes; the lattice column of its column 0 as seen from each
    // end; the severed columns at the start
    bool known, ev_r, ev_l, own_r, own_l, follow;
    int org_r, org_l, f0, l0;
    bool senses;                // a sensor of the tile's list lies on one of the thread's sites
    bool on_edge;               // adjoint: the warp holds row 0 or ny - 1
    int64_t n;                  // adjoint: the transposed step the pass starts with
};

// The fields of a thread: RPT rows of one vector.  Each update writes the
// new rows where the next one reads them, so that no register is copied from
// step to step: leapfrog storage writes w_{n+1} over w_{n-1} and the two
// planes change places; the other forms shift the rows of w by one slot, up
// in one step (PH = 0, rows swept upwards) and down in the next (PH = 1).
template <typename T, typename D, int RPT> struct PassRows {
    static constexpr int N = PassVec<T, D>::N;
    typedef Row<T, N> R;
    static constexpr bool kLf = std::is_same<D, Lf>::value;
    R a[RPT + (kLf ? 0 : 1)];
    R b[RPT];
    // row r of w before a step of phase PH, and where the step writes it
    template <int PH> __device__ __forceinline__ R &cur(int r)
    {
        if constexpr (kLf) return PH == 0 ? a[r] : b[r];
        else return PH == 0 ? a[r + 1] : a[r];
    }
    template <int PH> __device__ __forceinline__ R &next(int r)
    {
        if constexpr (kLf) return PH == 0 ? b[r] : a[r];
        else return PH == 0 ? a[r] : a[r + 1];
    }
    // row r of wdot (leapfrog: of the w before, which the step overwrites)
    template <int PH> __device__ __forceinline__ R &rate(int r)
    {
        if constexpr (kLf) return PH == 0 ? b[r] : a[r];
        else return b[r];
    }
};

// Adjoint: the values of m next to the Dirichlet edges before step s, which a
// reduction over all steps turns into the load gradient (summed here, in FP64,
// they would cost the tiles along an edge as much as a step).
template <typename T, typename D, int RPT, typename F>
__device__ __forceinline__ void pass_edge_rows(const PassArgs<T, D> &A, const PassCtx &c, int s, F &&row)
{
    constexpr int N = PassVec<T, D>::N;
    const PassAdj<T> &d = A.adj;
    const int64_t n = c.n - s;
    if (n < 0 || n >= d.n_steps || !(c.on_edge || c.side)) return;
    const StepArgs<T, D> &a = A.s;
    T *at = d.edge_m + (n % d.edge_ring) * 4 * d.edge_len;
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const int j = c.jb + r;
        if (j < c.g.y0 || j >= c.g.y1) continue;
        const Row<T, N> w = row(r);
        if (c.on_edge) {
#pragma unroll
            for (int e = BOTTOM; e <= TOP; ++e) {
                if (j != (e == BOTTOM ? 0 : a.ny - 1) || a.edge[e] != EDGE_DIRICHLET) continue;
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    int q = c.x0 + k;
                    if (q < c.g.x0 || q >= c.g.x1) continue;
                    if (c.per) q = wrap_col(q, a.nx);
                    at[e * d.edge_len + q] = w.v[k];
                }
            }
        }
        if (c.is_l && a.edge[LEFT] == EDGE_DIRICHLET && c.g.x0 == 0) at[LEFT * d.edge_len + j] = w.v[0];
        if (c.kr >= 0 && a.edge[RIGHT] == EDGE_DIRICHLET && c.g.x1 == a.nx) {
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (k == c.kr) at[RIGHT * d.edge_len + j] = w.v[k];
        }
    }
}

// One time step of a tile.
template <typename T, typename D, int NW, int RPT, int KIND, int PH, int MODE>
__device__ __forceinline__ void pass_step(const PassArgs<T, D> &A, const PassCtx &c, int s, PassRows<T, D, RPT> &F,
                                          PassShared<T, NW, PassVec<T, D>::N> &sh, PassSensors<T, MODE> &sen, PassWindow &win)
{
    constexpr int N = PassVec<T, D>::N;
    constexpr int kBelowWarp = NW / 2 - 1;   // strip: the warp whose last row is jc - 1; the next one's first is jc
    constexpr bool kLf = std::is_same<D, Lf>::value;
    typedef Row<T, N> R;
    const unsigned kFull = 0xffffffffu;
    const StepArgs<T, D> &a = A.s;
    const CrackParams &p = a.p;
    const int lane = c.lane, warp = c.warp, x0 = c.x0, jb = c.jb, nx = a.nx, ny = a.ny;
    const T gg = a.g, dt = a.dt, wd_inv = a.wd_inv, wd_scale = a.wd_scale;
    const int b = s & 1;
    stg_row(&sh.top[b][warp][lane * N], F.template cur<PH>(RPT - 1));
    stg_row(&sh.bot[b][warp][lane * N], F.template cur<PH>(0));
    const bool face = KIND == 2 && (warp == kBelowWarp || warp == kBelowWarp + 1), below = warp == kBelowWarp;
    if (MODE == kAdjoint && KIND != 0) pass_edge_rows<T, D, RPT>(A, c, s, [&](int r) { return F.template cur<PH>(r); });
    if (MODE != kAdjoint && KIND == 2 && face) stg_row(&sh.pair[s][below ? 0 : 1][lane * N], F.template cur<PH>(below ? RPT - 1 : 0));

    const bool dir_l = KIND != 0 && a.edge[LEFT] == EDGE_DIRICHLET, dir_r = KIND != 0 && a.edge[RIGHT] == EDGE_DIRICHLET;
    constexpr bool kNineQ = MODE == kNine;
    const bool em = (MODE == kForward || kNineQ) && KIND != 0 && A.q.edge_macro != 0, em_side = em && c.side;
    const bool last_r = KIND != 0 && c.kr == N - 1;
    T tl = (T)0, tr = (T)0;
    R first, last;                                         // the first and last rows before the update
    T el[KIND != 0 ? RPT : 1], er[KIND != 0 ? RPT : 1];   // edge rule: the edge columns before the update
    if (KIND != 0) {
        if (dir_l) tl = sh.ws2[LEFT][s];
        if (dir_r) tr = sh.ws2[RIGHT][s];
        first = F.template cur<PH>(0);
        last = F.template cur<PH>(RPT - 1);
        if (c.odd || em_side) {
            // the images of edge sites inside a warp's rows or a thread's
            // columns, as neighbours: the row update itself knows no edge
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                if (kNineQ) break;   // (a D2Q9 diagonal sends back its own site's value, not its neighbour's)
                if (r + 1 < RPT && jb + r == ny - 1)
                    F.template cur<PH>(r + 1 < RPT ? r + 1 : r) =
                        edge_image<T, N>(F.template cur<PH>(r), a.edge[TOP] == EDGE_DIRICHLET, sh.ws2[TOP][s]);
                if (r > 0 && jb + r == 0)
                    F.template cur<PH>(r > 0 ? r - 1 : r) =
                        edge_image<T, N>(F.template cur<PH>(r), a.edge[BOTTOM] == EDGE_DIRICHLET, sh.ws2[BOTTOM][s]);
            }
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                R &w = F.template cur<PH>(r);
#pragma unroll
                for (int k = 0; k + 1 < N; ++k) w.v[k + 1] = k == c.kr ? (dir_r ? tr - w.v[k] : w.v[k]) : w.v[k + 1];
                el[r] = w.v[0];
                er[r] = el[r];
#pragma unroll
                for (int k = 1; k < N; ++k) er[r] = k == c.kr ? w.v[k] : er[r];
            }
        }
    }
    // the sums of a row's east and west neighbours, before the barrier
    auto sides = [&](const R &cu) {
        T left0 = __shfl_up_sync(kFull, cu.v[N - 1], 1);
        T rightN = __shfl_down_sync(kFull, cu.v[0], 1);
        if (KIND != 0) {
            // no branches here: they would keep the rows' latencies from
            // overlapping (FP64: two instructions of 64 cycles cost more)
            if (sizeof(T) == 4 || c.side) {
                T il = cu.v[0], ir = cu.v[N - 1];
                if (dir_l) il = tl - il;
                if (dir_r) ir = tr - ir;
                left0 = c.is_l ? il : left0;
                rightN = last_r ? ir : rightN;
            }
        }
        R hs;
#pragma unroll
        for (int k = 0; k < N; ++k)
            hs.v[k] = (k == 0 ? left0 : cu.v[k > 0 ? k - 1 : 0]) + (k == N - 1 ? rightN : cu.v[k < N - 1 ? k + 1 : k]);
        return hs;
    };
    // Rows that need no other warp's: tiles of four rows a warp, which wait
    // on latency more than on issue, update them before the barrier (row 1's
    // new values take the slot of row 0, whose old values and neighbour are
    // kept); larger ones sweep all rows after it.
    constexpr bool kEarly = RPT <= 4 && !kNineQ;
    R old0, old1, hs0, hsT;
    if (kEarly && PH == 0) {
        old0 = F.template cur<PH>(0);
        old1 = F.template cur<PH>(1);
        hs0 = sides(F.template cur<PH>(0));
        hsT = sides(F.template cur<PH>(RPT - 1));
#pragma unroll
        for (int r = 1; r + 1 < RPT; ++r) {
            const R cu = F.template cur<PH>(r), up = F.template cur<PH>(r + 1), dn = r == 1 ? old0 : F.template cur<PH>(r - 1);
            const R hs = sides(cu);
            R out;
            row_sites<T, D, N>(cu, up, dn, hs, F.template rate<PH>(r), gg, dt, wd_scale, wd_inv, out);
            F.template next<PH>(r) = out;
        }
    }
    __syncthreads();
    if (MODE != kAdjoint && KIND == 2 && c.follow) {
        const bool reach = sh.reach[b] != 0;
        if (warp == 0) {
            pass_crack_step<T, PassShared<T, NW, PassVec<T, D>::N>::W>(p, A.q, sh.top[b][kBelowWarp], sh.bot[b][kBelowWarp + 1], c.org_r,
                                                     c.org_l, sh.S, sh.log[s + 1], c.ev_r, c.ev_l, win);
            // (D2Q9: any advance can pass a diagonal crossing)
            if (lane == 0) sh.reach[b ^ 1] = kNineQ || crack_cut_in_reach(p, sh.S) ? 1 : 0;
        }
        // rows next to the crack wait for the decision only where it can cut a link
        if (reach) __syncthreads();
    }
    R dnx, upx;
    ld_row(&sh.top[b][warp > 0 ? warp - 1 : 0][lane * N], dnx);
    ld_row(&sh.bot[b][warp < NW - 1 ? warp + 1 : warp][lane * N], upx);
    if (KIND != 0 && !kNineQ && (c.has_t || c.has_b)) {
        // the images beyond the bottom and top rows
        if (c.has_t) upx = edge_image<T, N>(last, a.edge[TOP] == EDGE_DIRICHLET, sh.ws2[TOP][s]);
        if (c.has_b) dnx = edge_image<T, N>(first, a.edge[BOTTOM] == EDGE_DIRICHLET, sh.ws2[BOTTOM][s]);
    }
    bool cut[N], cutp[N];   // cutp (adjoint): severed in the forward step before
#pragma unroll
    for (int k = 0; k < N; ++k) cut[k] = cutp[k] = false;
    if (KIND == 2 && face) {
        const int e = MODE == kAdjoint ? s : s + 1;
        const int f = c.known ? sh.log[e].f : (c.ev_l ? sh.S.i_first : c.f0);
        const int l = c.known ? sh.log[e].l : (c.ev_r ? sh.S.i_last : c.l0);
        const int fp = MODE == kAdjoint ? sh.log[s + 1].f : 0, lp = MODE == kAdjoint ? sh.log[s + 1].l : -1;
        // a severed link sends the site's own value back
#pragma unroll
        for (int k = 0; k < N; ++k) {
            int q = x0 + k;
            if (c.per) q = q < 0 ? q + nx : (q >= nx ? q - nx : q);
            cut[k] = q >= f && q <= l;
            cutp[k] = q >= fp && q <= lp;
            if (!kNineQ) {
                upx.v[k] = cut[k] && below ? last.v[k] : upx.v[k];
                dnx.v[k] = cut[k] && !below ? first.v[k] : dnx.v[k];
            }
        }
    }
    if constexpr (kNineQ) {
        const T ga = gg * (T)(2.0 / 3.0), gd = gg * (T)(1.0 / 6.0);
        // the severed diagonals: crossings of the crack line between the tips
        // in force, left and right of each column
        bool dl[N], dr[N];
#pragma unroll
        for (int k = 0; k < N; ++k) dl[k] = dr[k] = false;
        if (KIND == 2 && face) {
            const int64_t rq = c.known ? sh.log[s + 1].tr : (c.ev_r ? sh.S.r.tip_q : sh.in.r.tip_q);
            const int64_t lq = !p.two_tips ? p.start_q : (c.known ? sh.log[s + 1].tl : (c.ev_l ? sh.S.l.tip_q : sh.in.l.tip_q));
#pragma unroll
            for (int k = 0; k < N; ++k) {
                int q = x0 + k;
                if (c.per) q = q < 0 ? q + nx : (q >= nx ? q - nx : q);
                const int64_t ml = (int64_t)q << kQBits, mr = (int64_t)(q + 1) << kQBits;
                dl[k] = q >= 1 && lq <= ml && ml <= rq;
                dr[k] = q + 1 <= nx - 1 && lq <= mr && mr <= rq;
            }
        }
        const TwoWs<T> two_ws{sh.ws2[LEFT][s], sh.ws2[RIGHT][s], sh.ws2[BOTTOM][s], sh.ws2[TOP][s]};
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = PH == 0 ? q : RPT - 1 - q, j = jb + r;
            const R cu = F.template cur<PH>(r);
            const R up = r + 1 < RPT ? F.template cur<PH>(r + 1 < RPT ? r + 1 : r) : upx;
            const R dn = r > 0 ? F.template cur<PH>(r > 0 ? r - 1 : r) : dnx;
            const bool crow = KIND == 2 && face && r == (below ? RPT - 1 : 0);
            const bool top = KIND != 0 && j == ny - 1, bot = KIND != 0 && j == 0;
            R axis, diag;
            if (KIND != 0 && (crow || top || bot || c.odd)) {
                // a row with links that leave the body or cross the crack:
                // each diagonal by itself
                const T lc = __shfl_up_sync(kFull, cu.v[N - 1], 1), rc = __shfl_down_sync(kFull, cu.v[0], 1);
                const T la = __shfl_up_sync(kFull, up.v[N - 1], 1), ra = __shfl_down_sync(kFull, up.v[0], 1);
                const T lb = __shfl_up_sync(kFull, dn.v[N - 1], 1), rb = __shfl_down_sync(kFull, dn.v[0], 1);
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    const T w0 = cu.v[k];
                    const bool lft = c.is_l && k == 0, rgt = k == c.kr;
                    T wl = k == 0 ? lc : cu.v[k > 0 ? k - 1 : 0], wr = k == N - 1 ? rc : cu.v[k < N - 1 ? k + 1 : k];
                    T al = k == 0 ? la : up.v[k > 0 ? k - 1 : 0], ar = k == N - 1 ? ra : up.v[k < N - 1 ? k + 1 : k];
                    T bl = k == 0 ? lb : dn.v[k > 0 ? k - 1 : 0], br = k == N - 1 ? rb : dn.v[k < N - 1 ? k + 1 : k];
                    T u = up.v[k], v = dn.v[k];
                    if (lft) wl = leaving(a.edge, two_ws, true, false, -1, 0, w0);
                    if (rgt) wr = leaving(a.edge, two_ws, true, false, 1, 0, w0);
                    if (top) u = leaving(a.edge, two_ws, false, true, 0, 1, w0);
                    else if (crow && below && cut[k]) u = w0;
                    if (bot) v = leaving(a.edge, two_ws, false, true, 0, -1, w0);
                    else if (crow && !below && cut[k]) v = w0;
                    if (crow && below && dl[k]) al = w0;
                    else if (lft || top) al = leaving(a.edge, two_ws, lft, top, -1, 1, w0);
                    if (crow && below && dr[k]) ar = w0;
                    else if (rgt || top) ar = leaving(a.edge, two_ws, rgt, top, 1, 1, w0);
                    if (crow && !below && dl[k]) bl = w0;
                    else if (lft || bot) bl = leaving(a.edge, two_ws, lft, bot, -1, -1, w0);
                    if (crow && !below && dr[k]) br = w0;
                    else if (rgt || bot) br = leaving(a.edge, two_ws, rgt, bot, 1, -1, w0);
                    axis.v[k] = (u + v) + (wl + wr);
                    diag.v[k] = (al + bl) + (ar + br);
                }
            } else {
                // from the column sums of the rows above and below
                R sc;
#pragma unroll
                for (int k = 0; k < N; ++k) sc.v[k] = up.v[k] + dn.v[k];
                T sl = __shfl_up_sync(kFull, sc.v[N - 1], 1), sr = __shfl_down_sync(kFull, sc.v[0], 1);
                if (KIND != 0) {
                    T il = cu.v[0], ir = cu.v[N - 1];
                    if (dir_l) il = tl - il;
                    if (dir_r) ir = tr - ir;
                    sl = c.is_l ? il + il : sl;
                    sr = last_r ? ir + ir : sr;
                }
                const R hs = sides(cu);
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    axis.v[k] = sc.v[k] + hs.v[k];
                    diag.v[k] = (k == 0 ? sl : sc.v[k > 0 ? k - 1 : 0]) + (k == N - 1 ? sr : sc.v[k < N - 1 ? k + 1 : k]);
                }
            }
            R out;
            row_sites9<T, N>(cu, axis, diag, F.b[r], ga, gd, dt, out);
            F.template next<PH>(r) = out;
        }
#pragma unroll
        for (int k = 0; k < N; ++k) cut[k] = cut[k] || dl[k] || dr[k];   // the crack-face points
    }
    if constexpr (kNineQ) {
    } else if (kEarly && PH == 0) {
        R out;
        row_sites<T, D, N>(old0, old1, dnx, hs0, F.template rate<PH>(0), gg, dt, wd_scale, wd_inv, out);
        // the last row: its old values and its neighbour's are still in place
        const R cuT = F.template cur<PH>(RPT - 1), dnT = std::is_same<D, Lf>::value || RPT > 2 ? F.template cur<PH>(RPT - 2) : old0;
        R outT;
        row_sites<T, D, N>(cuT, upx, dnT, hsT, F.template rate<PH>(RPT - 1), gg, dt, wd_scale, wd_inv, outT);
        F.template next<PH>(0) = out;
        F.template next<PH>(RPT - 1) = outT;
    } else {
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = PH == 0 ? q : RPT - 1 - q;
            const R cu = F.template cur<PH>(r);
            // the row whose slot this row's new values take is read first
            const R up = r + 1 < RPT ? F.template cur<PH>(r + 1 < RPT ? r + 1 : r) : upx;
            const R dn = r > 0 ? F.template cur<PH>(r > 0 ? r - 1 : r) : dnx;
            const R hs = sides(cu);
            R out;
            row_sites<T, D, N>(cu, up, dn, hs, F.template rate<PH>(r), gg, dt, wd_scale, wd_inv, out);
            F.template next<PH>(r) = out;
        }
    }
    if constexpr (MODE == kAdjoint) {
        // the sensor sources of the state this step belongs to
        if (c.senses)
            for (int e = 0; e < sen.n; ++e) {
                const int r0 = sen.j[e] - jb, k0 = sen.i[e] - x0;
                const T v = sen.v[s][e];
#pragma unroll
                for (int r = 0; r < RPT; ++r)
#pragma unroll
                    for (int k = 0; k < N; ++k)
                        if (r == r0 && k == k0) {
                            F.template rate<PH>(r).v[k] += v;
                            F.template next<PH>(r).v[k] = fma_rn(dt, v, F.template next<PH>(r).v[k]);
                        }
            }
        if (KIND == 2 && p.macro && face) {
            // the transposed crack-face rule of the columns severed before
            const T inv_dt = dt == (T)1 ? (T)1 : div_dt((T)1, dt);
#pragma unroll
            for (int k = 0; k < N; ++k) {
                T &oT = F.template next<PH>(RPT - 1).v[k], &oT1 = F.template next<PH>(RPT - 2).v[k], &oT2 = F.template next<PH>(RPT - 3).v[k];
                T &oB = F.template next<PH>(0).v[k], &oB1 = F.template next<PH>(1).v[k], &oB2 = F.template next<PH>(2).v[k];
                T &aT = F.b[RPT - 1].v[k], &aT1 = F.b[RPT - 2].v[k], &aT2 = F.b[RPT - 3].v[k];
                T &aB = F.b[0].v[k], &aB1 = F.b[1].v[k], &aB2 = F.b[2].v[k];
                if (cutp[k] && below) face_transposed(inv_dt, oT, aT, oT1, aT1, oT2, aT2);
                if (cutp[k] && !below) face_transposed(inv_dt, oB, aB, oB1, aB1, oB2, aB2);
            }
        }
    }
    if (MODE != kAdjoint && KIND == 2 && p.macro && face) {
        // the crack-face rule: w_B from the two new values further from the crack
        R wB, w0;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const T w2 = below ? F.template next<PH>(RPT - 2).v[k] : F.template next<PH>(1).v[k];
            const T w3 = below ? F.template next<PH>(RPT - 3).v[k] : F.template next<PH>(2).v[k];
            wB.v[k] = face_value(w2, w3);
            w0.v[k] = below ? last.v[k] : first.v[k];
        }
        R rt = wB;
        if (kNineQ) {
            // (the D2Q9 face rule multiplies by 1 / dt)
            const T inv_dt = dt == (T)1 ? (T)1 : div_dt((T)1, dt);
#pragma unroll
            for (int k = 0; k < N; ++k) rt.v[k] = (wB.v[k] - w0.v[k]) * inv_dt;
        } else if (!kLf) {
            rt = rate_of(wB, w0, dt);
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {
            if (!kLf) {
                const T v = wd_round<D, T>(rt.v[k], wd_scale, wd_inv);
                F.b[RPT - 1].v[k] = cut[k] && below ? v : F.b[RPT - 1].v[k];
                F.b[0].v[k] = cut[k] && !below ? v : F.b[0].v[k];
            }
            T &oT = F.template next<PH>(RPT - 1).v[k], &oB = F.template next<PH>(0).v[k];
            oT = cut[k] && below ? wB.v[k] : oT;
            oB = cut[k] && !below ? wB.v[k] : oB;
        }
    }
    if constexpr (N > 1) if (em) {
        // the macroscopic rule on the outer edges (the two levels of
        // edge_rule_at): the edge columns, the crack-face points on
        // them, then the bottom and top rows and the corners
        const bool on_l = a.edge[LEFT] != EDGE_PERIODIC && c.is_l, on_r = a.edge[RIGHT] != EDGE_PERIODIC && c.kr >= 0;
        EdgeRule<T> E;
        E.wn = nullptr;
        E.pitch = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            E.dir[e] = a.edge[e] == EDGE_DIRICHLET;
            E.ws[e] = E.dir[e] ? sh.ws[e][s + 1] : (T)0;
        }
        R in1, in2;         // rows 1, 2 (or ny-2, ny-3) before the edge columns
        const bool has_b = c.has_b, has_t = c.has_t;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            in1.v[k] = has_t ? F.template next<PH>(RPT - 2).v[k] : F.template next<PH>(1).v[k];
            in2.v[k] = has_t ? F.template next<PH>(RPT - 3).v[k] : F.template next<PH>(2).v[k];
        }
        if (em_side) {
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                R &w = F.template next<PH>(r);
                const int j = jb + r;
                const bool row = j >= 1 && j <= ny - 2;
                const T p1 = __shfl_up_sync(kFull, w.v[N - 1], 1), p2 = __shfl_up_sync(kFull, w.v[N - 2], 1);
                const T n0 = __shfl_down_sync(kFull, w.v[0], 1);
                const T vl = E.rule(LEFT, w.v[1], N > 2 ? w.v[N > 2 ? 2 : 0] : n0);
                T wI = p1, wII = p2;
#pragma unroll
                for (int k = 1; k < N; ++k) {
                    wI = k == c.kr ? w.v[k - 1] : wI;
                    wII = k == c.kr ? (k >= 2 ? w.v[k >= 2 ? k - 2 : 0] : p1) : wII;
                }
                const T vr = E.rule(RIGHT, wI, wII);
                Row<T, 2> wn, wo;
                wn.v[0] = vl;
                wn.v[1] = vr;
                wo.v[0] = el[r];
                wo.v[1] = er[r];
                w.v[0] = row && on_l ? vl : w.v[0];
#pragma unroll
                for (int k = 0; k < N; ++k) w.v[k] = row && on_r && k == c.kr ? vr : w.v[k];
                if (!kLf) {
                    // wdot of the sites that took the rule (crack-face points again below)
                    const Row<T, 2> rt = rate_of(wn, wo, dt);
                    const T rl = wd_round<D, T>(rt.v[0], wd_scale, wd_inv), rr = wd_round<D, T>(rt.v[1], wd_scale, wd_inv);
                    F.b[r].v[0] = row && on_l ? rl : F.b[r].v[0];
#pragma unroll
                    for (int k = 0; k < N; ++k) F.b[r].v[k] = row && on_r && k == c.kr ? rr : F.b[r].v[k];
                }
            }
            if (KIND == 2 && face && p.macro) {
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    if (!(cut[k] && ((on_l && k == 0) || (on_r && k == c.kr)))) continue;
                    const T v1 = below ? F.template next<PH>(RPT - 2).v[k] : F.template next<PH>(1).v[k];
                    const T v2 = below ? F.template next<PH>(RPT - 3).v[k] : F.template next<PH>(2).v[k];
                    const T v = face_value(v1, v2);
                    Row<T, 1> wn, wo;
                    wn.v[0] = v;
                    wo.v[0] = below ? last.v[k] : first.v[k];
                    const T rt = wd_round<D, T>(rate_of(wn, wo, dt).v[0], wd_scale, wd_inv);
                    if (below) {
                        F.template next<PH>(RPT - 1).v[k] = v;
                        if (!kLf) F.b[RPT - 1].v[k] = rt;
                    } else {
                        F.template next<PH>(0).v[k] = v;
                        if (!kLf) F.b[0].v[k] = rt;
                    }
                }
            }
        }
        if (has_b || has_t) {
            const int ev = has_t ? TOP : BOTTOM;
            R o;
#pragma unroll
            for (int k = 0; k < N; ++k) o.v[k] = E.rule(ev, in1.v[k], in2.v[k]);
            if (em_side) {
                // corners: along the bottom / top edge's normal from the edge
                // columns, or (its side Dirichlet, ev not) along the row from
                // the points of edge ev
                const T q1 = __shfl_up_sync(kFull, o.v[N - 1], 1), q2 = __shfl_up_sync(kFull, o.v[N - 2], 1);
                const T m0 = __shfl_down_sync(kFull, o.v[0], 1);
                R e1, e2;   // the rows one and two from the edge, after the edge columns
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    e1.v[k] = has_t ? F.template next<PH>(RPT - 2).v[k] : F.template next<PH>(1).v[k];
                    e2.v[k] = has_t ? F.template next<PH>(RPT - 3).v[k] : F.template next<PH>(2).v[k];
                }
                const T cl = E.dir[LEFT] && !E.dir[ev] ? E.rule(LEFT, o.v[1], N > 2 ? o.v[N > 2 ? 2 : 0] : m0)
                                                       : E.rule(ev, e1.v[0], e2.v[0]);
                T oI = q1, oII = q2, c1 = (T)0, c2 = (T)0;
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if (k == c.kr) {
                        if (k >= 1) oI = o.v[k >= 1 ? k - 1 : 0];
                        if (k >= 1) oII = k >= 2 ? o.v[k >= 2 ? k - 2 : 0] : q1;
                        c1 = e1.v[k];
                        c2 = e2.v[k];
                    }
                const T cr = E.dir[RIGHT] && !E.dir[ev] ? E.rule(RIGHT, oI, oII) : E.rule(ev, c1, c2);
                o.v[0] = on_l ? cl : o.v[0];
#pragma unroll
                for (int k = 0; k < N; ++k) o.v[k] = on_r && k == c.kr ? cr : o.v[k];
            }
            R w0;
#pragma unroll
            for (int k = 0; k < N; ++k) w0.v[k] = has_t ? last.v[k] : first.v[k];
            const R rt = kLf ? o : rate_of(o, w0, dt);
#pragma unroll
            for (int k = 0; k < N; ++k) {
                const T v = kLf ? rt.v[k] : wd_round<D, T>(rt.v[k], wd_scale, wd_inv);
                if (has_t) {
                    F.template next<PH>(RPT - 1).v[k] = o.v[k];
                    if (!kLf) F.b[RPT - 1].v[k] = v;
                } else {
                    F.template next<PH>(0).v[k] = o.v[k];
                    if (!kLf) F.b[0].v[k] = v;
                }
            }
        }
    }
    if constexpr (MODE == kRecord)
        for (int e = 0; c.senses && e < sen.n; ++e) {
            const int r0 = sen.j[e] - jb, k0 = sen.i[e] - x0;
            if (r0 < 0 || r0 >= RPT || k0 < 0 || k0 >= N) continue;
            T v = (T)0;
#pragma unroll
            for (int r = 0; r < RPT; ++r)
#pragma unroll
                for (int k = 0; k < N; ++k) v = r == r0 && k == k0 ? F.template next<PH>(r).v[k] : v;
            sen.v[s][e] = v;
        }
}

// The sensors of a tile, in ascending order (warp 0): recording, those among
// its own sites; adjoint, those among all the sites it holds (a halo site's
// source reaches the tile's own sites) and their sources at each step.
template <typename T, typename D, int NW, int RPT, int MODE>
__device__ __forceinline__ void pass_sensors(const PassArgs<T, D> &A, const PassBuf<T, D> &B, const TileGeo &g, int64_t n,
                                             PassSensors<T, MODE> &sen)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const int ns = MODE == kRecord ? A.rec.ns : A.adj.ns;
    const int32_t *si = MODE == kRecord ? A.rec.s_i : A.adj.s_i, *sj = MODE == kRecord ? A.rec.s_j : A.adj.s_j;
    const int nx = A.s.nx;
    const int i0 = MODE == kRecord ? g.x0 : g.xl, i1 = MODE == kRecord ? g.x1 : g.x1 + A.q.hc;
    const int j0 = MODE == kRecord ? g.y0 : g.yl, j1 = MODE == kRecord ? g.y1 : g.yl + NW * RPT;
    const bool per = A.s.edge[LEFT] == EDGE_PERIODIC;
    if (tid < 32) {
        int cnt = 0;
        for (int img = 0; img < (per ? 3 : 1); ++img) {   // (periodic sides: the columns' images too)
            const int o = img == 0 ? 0 : (img == 1 ? -nx : nx);
            for (int q0 = 0; q0 < ns; q0 += 32) {
                const int q = q0 + lane;
                int i = 0, j = -1;
                if (q < ns) {
                    i = si[q] + o;
                    j = sj[q];
                }
                const bool mine = q < ns && j >= j0 && j < j1 && i >= i0 && i < i1;
                const unsigned m = __ballot_sync(0xffffffffu, mine);
                const int at = cnt + __popc(m & ((1u << lane) - 1u));
                if (mine && at < 2 * kPassSensors) {
                    sen.i[at] = i;
                    sen.j[at] = j;
                    sen.k[at] = q;
                }
                cnt += __popc(m);
            }
        }
        __syncwarp();
        cnt = min(cnt, 2 * kPassSensors);   // (with images; a tile of a narrow lattice holds at most two of a column)
        if (lane == 0) sen.n = cnt;
        if (MODE == kAdjoint) {
            for (int q = lane; q < cnt * A.q.K; q += 32) {
                const int e = q % cnt, s = q / cnt;
                // step n - s adds the sources of state n - s (none before the first)
                const int64_t t = n - s - 1;
                sen.v[s][e] = t >= 0 ? (T)(2.0 * A.adj.resid[(t % A.adj.ring) * ns + sen.k[e]]) : (T)0;
            }
        }
    }
}

// The misfits of a recording pass's states, and their squares added to the
// loss step by step.
template <typename T, typename D, int NW>
__device__ __forceinline__ void pass_misfits(const PassArgs<T, D> &A, const PassBuf<T, D> &B, PassSensors<T, kRecord> &sen)
{
    __syncthreads();
    const RecArgs &r = A.rec;
    const int64_t t0 = __ldcg(&B.s_in->step) - *r.n0;
    for (int e = threadIdx.x; e < sen.n; e += 32 * NW) {
        const int k = sen.k[e];
        double sum = r.acc_loss ? __ldcg(&r.loss[k]) : 0.0;
        double tg[kPassSteps];
#pragma unroll
        for (int s = 0; s < kPassSteps; ++s) tg[s] = s < A.q.K && t0 + s < r.n_steps ? r.target[(t0 + s) * r.ns + k] : 0.0;
#pragma unroll
        for (int s = 0; s < kPassSteps; ++s) {
            const int64_t t = t0 + s;
            if (s >= A.q.K || t < 0 || t >= r.n_steps) continue;
            const double res = (double)sen.v[s][e] - tg[s];
            r.resid[(t % r.ring) * r.ns + k] = res;
            sum += res * res;
        }
        if (r.acc_loss) __stcg(&r.loss[k], sum);
    }
}

// A tile.  KIND: 0 one none of whose sites sees an edge or the crack, 1 with
// outer edges, 2 a crack-strip tile (with edges where it meets them).
template <typename T, typename D, int NW, int RPT, int KIND, bool COOP, int MODE>
__device__ __forceinline__ void pass_tile(const PassArgs<T, D> &A, const PassBuf<T, D> &B, const TileGeo g,
                                          PassShared<T, NW, PassVec<T, D>::N> &sh, PassSensors<T, MODE> &sen)
{
    constexpr int N = PassVec<T, D>::N;
    constexpr int W = PassShared<T, NW, PassVec<T, D>::N>::W;
    typedef Row<T, N> R;
    const unsigned kFull = 0xffffffffu;
    const StepArgs<T, D> &a = A.s;
    const CrackParams &p = a.p;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nx = a.nx, ny = a.ny, K = A.q.K;
    const int64_t P = a.pitch;
    const T wd_inv = a.wd_inv, wd_scale = a.wd_scale;
    PassCtx c;
    c.g = g;
    c.lane = lane;
    c.warp = warp;
    c.x0 = g.xl + lane * N;
    c.jb = g.yl + warp * RPT;
    c.per = KIND != 0 && a.edge[LEFT] == EDGE_PERIODIC;
    const int x0 = c.x0, jb = c.jb;
    const bool per = c.per;

    PassRows<T, D, RPT> F;
    {
        const T *wp = B.w_in + (int64_t)jb * P + x0;
        const D *dp = B.wd_in + (int64_t)jb * P + x0;
        const bool whole = KIND == 0 ? x0 < nx : (x0 >= 0 && x0 + N <= nx);
        // every load before any conversion, so that they are in flight together
        typename WdIO<D>::Raw raw[RPT];
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            R &w = F.template cur<0>(r);
#pragma unroll
            for (int k = 0; k < N; ++k) w.v[k] = (T)0;
            raw[r] = typename WdIO<D>::Raw{};
            const int j = jb + r;
            if (whole && j >= 0 && j < ny) {
                if (COOP) {
                    cg_row(wp + (int64_t)r * P, w);
                    cg_raw(dp + (int64_t)r * P, raw[r]);
                } else {
                    ldg_row(wp + (int64_t)r * P, w);
                    WdIO<D>::fetch(dp + (int64_t)r * P, raw[r]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RPT; ++r) WdIO<D>::unpack(raw[r], F.b[r], wd_inv);
        if (KIND != 0 && !whole) {
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int j = jb + r;
                if (j < 0 || j >= ny) continue;
                R &w = F.template cur<0>(r), &d = F.b[r];
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    int q = x0 + k;
                    if (per) q = wrap_col(q, nx);
                    if (q < 0 || q >= nx) continue;
                    w.v[k] = cg_get(B.w_in + (int64_t)j * P + q);
                    d.v[k] = cg_rate_get(B.wd_in + (int64_t)j * P + q, wd_inv);
                }
            }
        }
    }

    int rec0 = 0;
    int64_t hist0 = 0;
    c.known = true;
    c.ev_r = c.ev_l = c.own_r = c.own_l = c.follow = false;
    c.org_r = c.org_l = g.xl;
    c.f0 = 0;
    c.l0 = -1;
    PassWindow win = {-1, 0.0f, -1};
    int64_t fit_tip = 0;
    PassPair fit_pair = {0, 0, 0};
    double fit_sf = 0.0;
    c.senses = false;
    c.n = 0;
    if (MODE == kAdjoint) {
        c.n = __ldcg(B.cnt_in);
        if (KIND == 2 && tid <= K) {
            // the columns severed in forward step n - tid
            const int64_t q = c.n - tid, qc = q < A.adj.n_steps ? q : A.adj.n_steps - 1;
            sh.log[tid].f = q >= 0 ? A.adj.i_first[qc] : 1;
            sh.log[tid].l = q >= 0 ? A.adj.i_last[qc] : 0;
        }
    }
    if constexpr (MODE == kRecord || MODE == kAdjoint) pass_sensors<T, D, NW, RPT, MODE>(A, B, g, c.n, sen);
    if (MODE != kAdjoint && KIND == 2) {
        c.known = p.mode != CRACK_KCRIT;
        c.f0 = sh.in.i_first;
        c.l0 = sh.in.i_last;
        hist0 = p.hist_cap > 0 ? sh.in.hist_n % p.hist_cap : 0;   // the ring slot of the first record
        rec0 = sh.in.r.decided ? 1 : 0;   // the first update whose crack step is still to run
        const int cr = tip_col_r(c.f0, c.l0, nx), cl = tip_col_l(c.f0, c.l0, nx);
        const int hc = A.q.hc, grow = A.q.grow, back = A.q.back;
        // (periodic sides: the column itself, then its images beyond either side)
        for (int q = 0; q < (per ? 3 : 1); ++q) {
            const int o = q == 0 ? 0 : (q == 1 ? -nx : nx);
            if (cr + o >= g.x0 && cr + o < g.x1) c.own_r = true;
            if (p.two_tips && cl + o >= g.x0 && cl + o < g.x1) c.own_l = true;
            if (!c.ev_r && g.x0 - hc <= cr + o + grow && g.x1 + hc > cr + o - back) {
                c.ev_r = true;
                c.org_r = g.xl - o;
            }
            if (p.two_tips && !c.ev_l && g.x0 - hc <= cl + o + back && g.x1 + hc > cl + o - grow) {
                c.ev_l = true;
                c.org_l = g.xl - o;
            }
        }
        c.follow = !c.known && (c.ev_r || c.ev_l);
        if (c.known) {
            // every tile of the strip forms the cuts of the whole pass
            if (c.f0 <= c.l0) {
                if (tid <= K) pass_known_lane(p, &sh.in, tid, sh.log[tid]);
            } else if (tid == 0) {
                pass_known_serial(p, sh.in, sh.log, K);
            }
        } else {
            if (tid == 0) {
                sh.S = sh.in;
                sh.reach[0] = MODE == kNine || crack_cut_in_reach(p, sh.S) ? 1 : 0;
                sh.log[0].tr = sh.S.r.tip_q;
                sh.log[0].tl = sh.S.l.tip_q;
                sh.log[0].f = c.f0;
                sh.log[0].l = c.l0;
            }
            if (c.follow && warp == 0) {
                __syncwarp();
                pass_window(A.q, sh.S, lane < 16 ? c.org_r : c.org_l, lane < 16 ? c.ev_r : c.ev_l, win);
            }
        }
        if ((c.own_r || c.own_l || (N == 1 && A.q.free)) && A.q.one_pair && warp == 1 && lane < 2 * kPassSteps) {
            // the part of the K fits that needs no fields (an FP64 root and
            // division), while the loads are under way: lane st of the right
            // end, st + 8 of the left, for the tip before update st (K-
            // criterion: the tip at rest where it starts)
            const int st = lane & (kPassSteps - 1), dir = lane < kPassSteps ? +1 : -1;
            PassTip t;
            if (c.known && c.f0 <= c.l0) {
                pass_known_lane(p, &sh.in, st, t);
            } else {
                t.tr = sh.in.r.tip_q;
                t.tl = sh.in.l.tip_q;
                t.f = c.f0;
                t.l = c.l0;
            }
            fit_tip = dir > 0 ? t.tr : t.tl;
            fit_pair = pass_pair(dir, fit_tip, A.q.lo_q, A.q.hi_q, t.f, t.l);
            fit_sf = fit_pair.in ? pass_sf(p, fit_pair.d) : 0.0;
        }
    }
    if (MODE == kAdjoint && KIND != 0 && tid < 4 * (kPassSteps + 1)) sh.ws2[tid / (kPassSteps + 1)][tid % (kPassSteps + 1)] = (T)0;
    if (MODE != kAdjoint && KIND != 0) {
        // w* of the Dirichlet edges this tile meets, in the arithmetic's
        // precision once (a conversion from FP64 costs a warp 64 cycles)
        if (tid < 4 * (kPassSteps + 1)) {
            const int e = tid / (kPassSteps + 1), q = tid % (kPassSteps + 1);
            const bool meets = e == LEFT ? g.xl <= 0 : e == RIGHT ? g.xl + W >= nx : e == BOTTOM ? g.yl <= 0 : g.yl + NW * RPT >= ny;
            if (q <= K && meets && a.edge[e] == EDGE_DIRICHLET) {
                const T v = a.load[e].kind == LOAD_CONST ? (T)a.load[e].amp
                          : a.load[e].kind == LOAD_ZERO  ? (T)0
                                                         : (T)load_value(a.load[e], __ldcg(&B.s_in->step) + q, (double)p.dt);
                sh.ws[e][q] = v;
                sh.ws2[e][q] = (T)2 * v;
            }
        }
    }
    c.is_l = KIND != 0 && !per && x0 == 0;
    c.kr = KIND != 0 && !per && nx - 1 - x0 >= 0 && nx - 1 - x0 < N ? nx - 1 - x0 : -1;

    c.side = KIND != 0 && __any_sync(kFull, c.is_l || c.kr >= 0);
    c.has_t = KIND != 0 && jb + RPT == ny;
    c.has_b = KIND != 0 && jb == 0;
    c.odd = KIND != 0 && ((jb < 0 && jb + RPT > 0) || (jb < ny && jb + RPT > ny) ||
                          __any_sync(kFull, c.kr >= 0 && c.kr < N - 1));
    if (KIND != 0 || MODE == kRecord || MODE == kAdjoint) __syncthreads();   // w*, the cuts of the pass, the sensors
    if constexpr (MODE == kRecord || MODE == kAdjoint) {
        for (int e = 0; e < sen.n; ++e) {
            const int r0 = sen.j[e] - jb, k0 = sen.i[e] - x0;
            c.senses |= r0 >= 0 && r0 < RPT && k0 >= 0 && k0 < N;
        }
    }
    c.on_edge = KIND != 0 && ((jb <= 0 && jb + RPT > 0) || (jb <= ny - 1 && jb + RPT > ny - 1));
    // bulk tiles: two steps an iteration (PassRows); an odd last step leaves
    // the rows where a step of phase 0 writes them.  The other tiles, whose
    // step is far longer code, take every step in phase 0 and move the rows
    // back: unrolled twice, it ran out of the instruction cache.
    int s = 0;
    if (KIND == 0) {
        for (; s + 2 <= K; s += 2) {
            pass_step<T, D, NW, RPT, KIND, 0, MODE>(A, c, s, F, sh, sen, win);
            pass_step<T, D, NW, RPT, KIND, 1, MODE>(A, c, s + 1, F, sh, sen, win);
        }
    }
    for (; s < K; ++s) {
        pass_step<T, D, NW, RPT, KIND, 0, MODE>(A, c, s, F, sh, sen, win);
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = RPT - 1 - q;
            if constexpr (std::is_same<D, Lf>::value) {
                const R t = F.a[r];
                F.a[r] = F.b[r];
                F.b[r] = t;
            } else {
                F.a[r + 1] = F.a[r];
            }
        }
    }

    // the tile's own sites
    const PassPads<T> pads = {B.w_out, P, nx, ny, {a.edge[0], a.edge[1], a.edge[2], a.edge[3]}};
    T acc = (T)0;
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const R &w = F.template cur<0>(r), &d = F.b[r];
        const int j = jb + r;
        if (j < g.y0 || j >= g.y1) continue;
        if (x0 + N <= g.x0 || x0 >= g.x1) continue;
        const int64_t o = (int64_t)j * P + x0;
        if (KIND == 0 || (x0 >= g.x0 && x0 + N <= g.x1 && x0 >= 0 && x0 + N <= nx)) {
            stg_row(B.w_out + o, w);
            wd_store(B.wd + o, d, wd_scale);
            if (KIND != 0) write_pads(pads, x0, j, w);
            acc += w.v[0];
        } else {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                int q = x0 + k;
                if (q < g.x0 || q >= g.x1) continue;
                if (per) q = wrap_col(q, nx);
                if (q < 0 || q >= nx) continue;
                T *row = B.w_out + (int64_t)j * P;
                const T v = w.v[k];
                row[q] = v;
                wd_put(B.wd + (int64_t)j * P + q, d.v[k], wd_scale);
                if (q == 0) {
                    if (a.edge[LEFT] == EDGE_FREE) row[-1] = v;
                    else if (per) row[nx] = v;
                }
                if (q == nx - 1) {
                    if (a.edge[RIGHT] == EDGE_FREE) row[nx] = v;
                    else if (per) row[-1] = v;
                }
                if (j == 0 && a.edge[BOTTOM] == EDGE_FREE) row[q - P] = v;
                if (j == ny - 1 && a.edge[TOP] == EDGE_FREE) row[q + P] = v;
                acc += v;
            }
        }
    }
    if (__any_sync(kFull, !isfinite(acc)) && lane == 0) atomicOr(a.err, (uint32_t)ERR_NONFINITE);

    if constexpr (MODE == kRecord) pass_misfits<T, D, NW>(A, B, sen);
    if (MODE != kAdjoint && KIND == 2 && (c.own_r || c.own_l || (N == 1 && A.q.free))) {
        __syncthreads();   // the last crack step
        // the records of the pass's crack steps, and the K fits their decisions
        // did not wait for.  A window of one spacing holds at most one pair, so
        // one warp forms the fits of all steps, a lane each (an FP64
        // instruction takes a warp 64 cycles whatever its active lanes); a
        // wider one takes a warp per step.
        auto fit = [&](int st, int dir, double v_prev, double &Kf, int &np, double &r_min) {
            const PassTip &q = sh.log[st];
            const int org = dir > 0 ? c.org_r : c.org_l;
            const CrackSums f = crack_eval_pairs<T, 32>(
                p, dir > 0 ? q.tr : q.tl, v_prev, q.f, q.l, dir, [&](int i, T &ab, T &be) {
                    const int e = i - org;
                    if (e < 0 || e >= W) return false;
                    ab = sh.pair[st][1][e];
                    be = sh.pair[st][0][e];
                    return true;
                });
            np = f.np;
            Kf = np > 0 ? p.mu / 4.0 * f.num / f.den : 0.0;
            r_min = f.r_min;
        };
        auto record = [&](int st, int dir, double Kf, int np, double r_min) {
            const PassTip &q1 = sh.log[st + 1];
            if (q1.lazy) {
                if (!isfinite(Kf)) atomicOr(a.err, (uint32_t)ERR_NONFINITE);
                if (st == K - 1) {
                    TipState &O = dir > 0 ? B.s_out->r : B.s_out->l;
                    O.K = Kf;
                    O.r_min = r_min;
                    O.npairs = np;
                }
            } else {
                Kf = dir > 0 ? q1.Kr : q1.Kl;
                np = dir > 0 ? q1.npr : q1.npl;
            }
            if (p.hist_cap > 0) {
                int64_t h = hist0 + (st - rec0);   // the ring slot
                h -= h >= p.hist_cap ? p.hist_cap : 0;
                (dir > 0 ? a.hist.K : a.hist.Kl)[h] = Kf;
                (dir > 0 ? a.hist.v : a.hist.vl)[h] = dir > 0 ? q1.vr : q1.vl;
                (dir > 0 ? a.hist.tip : a.hist.tipl)[h] = dir > 0 ? q1.tr : q1.tl;
                (dir > 0 ? a.hist.np : a.hist.npl)[h] = np;
            }
        };
        const double v_prev = p.mode == CRACK_PRESCRIBED ? p.v_rel : 0.0;
        if (A.q.one_pair) {
            const int st = lane & (kPassSteps - 1), dir = lane < kPassSteps ? +1 : -1;
            if constexpr (N == 1) {
                bool mine = dir > 0 ? c.own_r : c.own_l;
                if (warp == 1 && lane < 2 * kPassSteps && st >= rec0 && st < K && (mine || (A.q.free && (dir > 0 || p.two_tips)))) {
                    double Kf = 0.0;
                    int np = 0;
                    if (sh.log[st + 1].lazy) {
                        const PassTip &q = sh.log[st];
                        const int64_t tip = dir > 0 ? q.tr : q.tl;
                        PassPair w = pass_pair(dir, tip, A.q.lo_q, A.q.hi_q, q.f, q.l);
                        if (tip != fit_tip || w.in != fit_pair.in) fit_sf = w.in ? pass_sf(p, w.d) : 0.0;   // it has moved since
                        // (free: the tile that owns the step's pair forms it, whichever tile owns the tip)
                        if (A.q.free && w.in) mine = w.col >= g.x0 && w.col < g.x1;
                        const int e = w.col - (A.q.free ? g.xl : (dir > 0 ? c.org_r : c.org_l));
                        if (w.in && e >= 0 && e < W) {
                            const CrackSums f = pass_sums<T>(fit_sf, sh.pair[st][1][e], sh.pair[st][0][e], 0.0);
                            Kf = pass_K(p, f);
                            np = 1;
                        }
                    }
                    if (mine) record(st, dir, Kf, np, A.q.r_min);
                }
            } else {
                if (warp == 1 && lane < 2 * kPassSteps && st >= rec0 && st < K && (dir > 0 ? c.own_r : c.own_l)) {
                    double Kf = 0.0;
                    int np = 0;
                    if (sh.log[st + 1].lazy) {
                        const PassTip &q = sh.log[st];
                        const int64_t tip = dir > 0 ? q.tr : q.tl;
                        PassPair w = pass_pair(dir, tip, A.q.lo_q, A.q.hi_q, q.f, q.l);
                        if (tip != fit_tip || w.in != fit_pair.in) fit_sf = w.in ? pass_sf(p, w.d) : 0.0;   // it has moved since
                        const int e = w.col - (dir > 0 ? c.org_r : c.org_l);
                        if (w.in && e >= 0 && e < W) {
                            const CrackSums f = pass_sums<T>(fit_sf, sh.pair[st][1][e], sh.pair[st][0][e], 0.0);
                            Kf = pass_K(p, f);
                            np = 1;
                        }
                    }
                    record(st, dir, Kf, np, A.q.r_min);
                }
            }
        } else if (warp >= rec0 && warp < K) {
            for (int dir = 1; dir >= (c.own_l ? -1 : 1); dir -= 2) {
                if (dir > 0 && !c.own_r) continue;
                double Kf = 0.0, r_min = 0.0;
                int np = 0;
                if (sh.log[warp + 1].lazy) fit(warp, dir, v_prev, Kf, np, r_min);
                if (lane == 0) record(warp, dir, Kf, np, r_min);
            }
        }
        if (MODE == kRecord && tid < K) {
            // the columns severed in each step, for the adjoint
            const int64_t t = sh.in.step + tid - *A.rec.n0;
            if (t >= 0 && t < A.rec.n_steps) {
                if (c.own_r) A.rec.i_last[t] = sh.log[tid + 1].l;
                if (c.own_l || (c.own_r && !p.two_tips)) A.rec.i_first[t] = sh.log[tid + 1].f;
            }
        }
        if (tid == 0) {
            CrackState *o = B.s_out;
            const PassTip &e = sh.log[K], &e1 = sh.log[K - 1];
            auto r_min_at = [&](double v) { return p.r_min_fixed > 0.0 ? p.r_min_fixed : (v == 0.0 ? p.r0 : p.r0 / (1.0 - v)); };
            // an end's decision after the pass (modes that need no K)
            auto known_end = [&](const TipState &s0, int64_t tip, int64_t tip1, int arr, double v, TipState &t) {
                t = s0;
                t.flags |= arr && !s0.arrested ? FLAG_CLAMPED : 0;
                t.tip_q = tip;
                t.arrested = arr;
                t.grew = tip != tip1;
                t.v = v;
                t.v_prev = p.mode == CRACK_PRESCRIBED ? p.v_rel : 0.0;
            };
            if (c.own_r) {
                o->step = sh.in.step + K;
                o->hist_n = sh.in.hist_n + K - rec0;
                o->i_last = e.l;
                if (!p.two_tips) o->i_first = e.f;
                if (c.known) {
                    TipState t;
                    known_end(sh.in.r, e.tr, e1.tr, e.arr_r, e.vr, t);
                    copy_tip_decision(o->r, t);
                } else {
                    copy_tip_decision(o->r, sh.S.r);
                }
                if (!e.lazy) {
                    o->r.K = sh.S.r.K;
                    o->r.r_min = r_min_at(e.vp_r);
                    o->r.npairs = sh.S.r.npairs;
                }
                o->r.decided = 0;
                for (int i = c.l0 + 1; i <= e.l; ++i)
                    if (i >= c.f0) atomicOr(&a.cut_v[(int64_t)(p.jc - 1) * p.words + (i >> 5)], 1u << (i & 31));
            }
            if (c.own_l) {
                o->i_first = e.f;
                if (c.known) {
                    TipState t;
                    known_end(sh.in.l, e.tl, e1.tl, e.arr_l, e.vl, t);
                    copy_tip_decision(o->l, t);
                } else {
                    copy_tip_decision(o->l, sh.S.l);
                }
                if (!e.lazy) {
                    o->l.K = sh.S.l.K;
                    o->l.r_min = r_min_at(e.vp_l);
                    o->l.npairs = sh.S.l.npairs;
                }
                o->l.decided = 0;
                for (int i = e.f; i < c.f0; ++i)
                    if (i <= c.l0) atomicOr(&a.cut_v[(int64_t)(p.jc - 1) * p.words + (i >> 5)], 1u << (i & 31));
            }
        }
    }
}

// Where the i-th of the tiles of `len` items begins, the first `more` of them of one more.
__device__ __forceinline__ int pass_split(int i, int len, int more) { return i * len + min(i, more); }

// Tile t of a pass.
template <typename T, typename D, int NW, int RPT, bool COOP, int MODE>
__device__ __forceinline__ void pass_cta(const PassArgs<T, D> &A, const PassBuf<T, D> &B, int t, PassShared<T, NW, PassVec<T, D>::N> &sh,
                                         PassSensors<T, MODE> &sen)
{
    constexpr int N = PassVec<T, D>::N;
    const StepArgs<T, D> &a = A.s;
    const PassPlan &q = A.q;
    const int nx = a.nx, ny = a.ny;
    const bool per = a.edge[LEFT] == EDGE_PERIODIC;
    const int tid = threadIdx.x;
    auto read_state = [&](CrackState &S) {
        constexpr int kWords = (int)(sizeof(CrackState) / 4);
        for (int k = tid; k < kWords; k += 32 * NW)
            reinterpret_cast<uint32_t *>(&S)[k] = __ldcg(reinterpret_cast<const uint32_t *>(B.s_in) + k);
        __syncthreads();
    };
    if (MODE == kAdjoint) {
        if (t == q.tiles - 1 && tid == 0) __stcg(B.cnt_out, __ldcg(B.cnt_in) - q.K);
    } else if (t == q.tiles - 1 && a.p.mode == CRACK_NONE) {
        // without a crack, the state only counts steps
        read_state(sh.in);
        if (tid == 0) {
            CrackState S = sh.in;
            S.step += q.K;
            S.r.decided = 1;
            S.l.decided = 1;
            for (int e = 0; e < 4; ++e)
                S.wstar[e] = a.edge[e] == EDGE_DIRICHLET ? load_value(a.load[e], S.step, (double)a.p.dt) : 0.0;
            *B.s_out = S;
        }
    } else if (t == q.tiles - 1 && tid < 4) {
        // the Dirichlet values after the pass (single steps read them)
        const int64_t n1 = __ldcg(&B.s_in->step) + q.K;
        B.s_out->wstar[tid] = a.edge[tid] == EDGE_DIRICHLET ? load_value(a.load[tid], n1, (double)a.p.dt) : 0.0;
    }
    TileGeo g;
    if (MODE == kAdjoint && t < q.ms) {
        // the recorded cuts need no tips: columns as the bulk splits them
        g.x0 = N * pass_split(t, q.px, q.ex);
        g.x1 = min(N * pass_split(t + 1, q.px, q.ex), nx);
        g.xl = g.x0 == 0 && !per ? 0 : g.x0 - q.hc;
        g.yl = a.p.jc - NW * kStripRpt / 2;
        g.y0 = q.jb;
        g.y1 = q.jt;
        pass_tile<T, D, NW, kStripRpt, 2, COOP, MODE>(A, B, g, sh, sen);
        return;
    }
    if (MODE != kAdjoint && t < q.ms) {
        read_state(sh.in);
        const int f = sh.in.i_first, l = sh.in.i_last;
        const int cr = tip_col_r(f, l, nx), cl = tip_col_l(f, l, nx);
        int lo0 = cr - q.zb, hi0 = cr + q.za, lo1 = cl + 1 - q.za, hi1 = cl + q.zb;
        bool two = a.p.two_tips != 0;
        if (two && lo0 <= hi1 + N && lo1 <= hi0 + N) {   // one zone around both tips
            lo0 = min(lo0, lo1);
            hi0 = max(hi0, hi1);
            two = false;
        }
        if (N == 1 && q.free) {
            g.x0 = N * pass_split(t, q.px, q.ex);
            g.x1 = min(N * pass_split(t + 1, q.px, q.ex), nx);
        } else {
            g.x0 = t == 0 && !per ? 0 : pass_boundary<N>(t * q.ps, nx, per, lo0, hi0, lo1, hi1, two);
            if (t + 1 < q.ms) g.x1 = pass_boundary<N>((t + 1) * q.ps, nx, per, lo0, hi0, lo1, hi1, two);
            else g.x1 = per ? nx + pass_boundary<N>(0, nx, per, lo0, hi0, lo1, hi1, two) : nx;
        }
        if (q.ms == 1) {
            g.x0 = 0;
            g.x1 = nx;
        }
        if (g.x0 >= g.x1) return;
        g.xl = g.x0 == 0 && !per ? 0 : g.x0 - q.hc;
        g.yl = a.p.jc - NW * kStripRpt / 2;
        g.y0 = q.jb;
        g.y1 = q.jt;
        pass_tile<T, D, NW, kStripRpt, 2, COOP, MODE>(A, B, g, sh, sen);
        return;
    }
    t -= q.ms;
    const int cx = t % q.mx, ry = t / q.mx;
    g.x0 = N * pass_split(cx, q.px, q.ex);
    g.x1 = min(N * pass_split(cx + 1, q.px, q.ex), nx);
    if (ry < q.mb) {
        g.y0 = pass_split(ry, q.pb, q.eb);
        g.y1 = pass_split(ry + 1, q.pb, q.eb);
    } else {
        g.y0 = q.jt + pass_split(ry - q.mb, q.pt, q.et);
        g.y1 = q.jt + pass_split(ry - q.mb + 1, q.pt, q.et);
    }
    g.xl = g.x0 == 0 && !per ? 0 : g.x0 - q.hc;
    g.yl = g.y0 == 0 ? 0 : (g.y1 == ny ? ny - NW * RPT : g.y0 - q.K);
    const bool plain = g.x0 >= q.K && g.x1 + q.K <= nx && g.y0 >= q.K && g.y1 + q.K <= ny && g.xl >= 0;
    if (plain) pass_tile<T, D, NW, RPT, 0, COOP, MODE>(A, B, g, sh, sen);
    else pass_tile<T, D, NW, RPT, 1, COOP, MODE>(A, B, g, sh, sen);
}

// One pass, a CTA per tile.
template <typename T, typename D, int NW, int RPT, int MODE>
__global__ void __launch_bounds__(32 * NW, 16 / NW) pass_kernel(const __grid_constant__ PassArgs<T, D> a)
{
    __shared__ PassShared<T, NW, PassVec<T, D>::N> sh;
    __shared__ PassSensors<T, MODE> sen;
    pdl_wait();
    pdl_trigger();
    const PassBuf<T, D> B = {a.s.w_in, a.wd_in, a.s.w_out, a.s.wd, a.s.s_in, a.s.s_out, a.adj.cnt_in, a.adj.cnt_out};
    pass_cta<T, D, NW, RPT, false, MODE>(a, B, blockIdx.x, sh, sen);
}

// n_pass passes, alternating between the two buffer sets, as one cooperative
// launch (every tile resident at once) with a grid barrier between passes: on
// lattices of a few hundred tiles a pass takes hardly longer than the launch
// gap, the ramp and the instruction fetches of a cold start.
template <typename T, typename D, int NW, int RPT, int MODE>
__global__ void __launch_bounds__(32 * NW, 16 / NW)
    pass_run_kernel(const __grid_constant__ PassArgs<T, D> a, int n_pass)
{
    __shared__ PassShared<T, NW, PassVec<T, D>::N> sh;
    __shared__ PassSensors<T, MODE> sen;
    for (int it = 0; it < n_pass; ++it) {
        const bool odd = (it & 1) != 0;
        PassBuf<T, D> B;
        B.w_in = odd ? a.w_in1 : a.s.w_in;
        B.wd_in = odd ? a.wd_in1 : a.wd_in;
        B.w_out = odd ? a.w_out1 : a.s.w_out;
        B.wd = odd ? a.wd1 : a.s.wd;
        B.s_in = odd ? a.s.s_out : a.s.s_in;
        B.s_out = odd ? const_cast<CrackState *>(a.s.s_in) : a.s.s_out;
        B.cnt_in = odd ? a.adj.cnt_out : a.adj.cnt_in;
        B.cnt_out = odd ? const_cast<int64_t *>(a.adj.cnt_in) : a.adj.cnt_out;
        pass_cta<T, D, NW, RPT, true, MODE>(a, B, blockIdx.x, sh, sen);
        if (it + 1 < n_pass && !grid_barrier(a.bar, gridDim.x, a.budget, a.s.err)) return;
    }
}

// One pass of every lattice of a batch: CTA u takes tile units[u].cb of
// lattice units[u].inst, with that lattice's arguments (descriptor par + 2
// second of its four) copied to shared memory.  The crack strips' tiles come
// first: a growing end's tile runs a chain of FP64 steps that the bulk tiles
// of all lattices hide.
template <typename T, typename D>
__global__ void __launch_bounds__(256, 2) pass_batch_kernel(const PassArgs<T, D> *descs, const BatchUnit *units, int which)
{
    __shared__ PassShared<T, 8> sh;
    __shared__ PassSensors<T, kForward> sen;
    __shared__ __align__(16) PassArgs<T, D> sa;
    const BatchUnit u = units[blockIdx.x];
    const uint32_t *src = reinterpret_cast<const uint32_t *>(descs + 4 * u.inst + which);
    uint32_t *dst = reinterpret_cast<uint32_t *>(&sa);
    typedef PassArgs<T, D> Args;
    for (int q = threadIdx.x; q < (int)(offsetof(Args, rec) / 4); q += 256) dst[q] = src[q];
    __syncthreads();
    const PassBuf<T, D> B = {sa.s.w_in, sa.wd_in, sa.s.w_out, sa.s.wd, sa.s.s_in, sa.s.s_out, nullptr, nullptr};
    pass_cta<T, D, 8, 8, false, kForward>(sa, B, u.cb, sh, sen);
}

template <typename T, typename D>
cudaError_t launch_pass_batch(const PassArgs<T, D> *descs, const BatchUnit *units, int n_units, int which, cudaStream_t s)
{
    pass_batch_kernel<T, D><<<(unsigned)n_units, 256, 0, s>>>(descs, units, which);
    return cudaGetLastError();
}

template <typename T, typename D, int MODE> const void *pass_kernel_ptr(int nw, int rpt, bool run)
{
    if constexpr (PassVec<T, D>::N == 1)
        return run ? reinterpret_cast<const void *>(&pass_run_kernel<T, D, 4, 4, MODE>)
                   : reinterpret_cast<const void *>(&pass_kernel<T, D, 4, 4, MODE>);
    else if constexpr (sizeof(T) == 8)
        if (nw == 4)
            return run ? reinterpret_cast<const void *>(&pass_run_kernel<T, D, 4, 4, MODE>)
                       : reinterpret_cast<const void *>(&pass_kernel<T, D, 4, 4, MODE>);
    if constexpr (sizeof(T) == 4)
        if (rpt == 4)
            return run ? reinterpret_cast<const void *>(&pass_run_kernel<T, D, 8, 4, MODE>)
                       : reinterpret_cast<const void *>(&pass_kernel<T, D, 8, 4, MODE>);
    if constexpr (PassVec<T, D>::N > 1)
        return run ? reinterpret_cast<const void *>(&pass_run_kernel<T, D, 8, 8, MODE>)
                   : reinterpret_cast<const void *>(&pass_kernel<T, D, 8, 8, MODE>);
}

template <typename T, typename D, int MODE> cudaError_t launch_pass(const PassArgs<T, D> &a, int n_pass, cudaStream_t s)
{
    const bool run = n_pass > 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.q.tiles);
    cfg.blockDim = dim3(32u * (unsigned)a.q.nw);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (run) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = run || a.s.chained ? 1 : 0;
    void *args[] = {(void *)&a, (void *)&n_pass};   // one pass: the first argument only
    return cudaLaunchKernelExC(&cfg, pass_kernel_ptr<T, D, MODE>(a.q.nw, a.q.rpt, run), args);
}

}  // namespace lbm
