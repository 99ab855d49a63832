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
// Tile: 8 warps on top of one another, a warp spans 32 16-byte vectors of
// columns (128 FP32 columns), a thread holds RPT rows of one vector (w and
// wdot: 64 registers at 8 rows).  East and west neighbours come by shuffles
// within the warp, the rows between warps through shared memory (16-byte
// vectors, double buffered, one barrier per step).  With K = 8 and RPT = 8 a
// 128 x 64 tile keeps 112 x 48 sites: 1.5 times the arithmetic of a single
// step, for an eighth of its memory traffic and launches.
//
// Measured, one GB300, time per step of a run against one launch per step:
// 4096 x 2048 FP32, K-criterion 20.0 -> 8.6 us; 8192 x 8192 BF16 wdot 161 ->
// 69 us; 16384 x 16384 leapfrog 575 -> 187 us; 1001 x 777 FP16 wdot, periodic
// sides 6.0 -> 3.4 us; 512 x 192 with the edge rule and two tips 10.7 -> 5.3 us.
// What bounds a bulk tile is instruction issue: with scalar FP32 and the rows
// moved back after each step the leapfrog kernel issued 85.7 M instructions
// per 4096^2 pass (120 us), without the moves 69.8 M (110 us), packed 50.7 M
// (98 us; FP32 pipes 44 % busy, DRAM 27 %).
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

#include "lbm_crack.cuh"
#include "lbm_internal.cuh"
#include "lbm_rows.cuh"

#include <type_traits>

namespace lbm {

constexpr int kPassWarps = 8;
constexpr int kPassThreads = 32 * kPassWarps;
constexpr int kPassSteps = 8;     // most steps of a pass
constexpr int kStripRpt = 4;      // rows per thread of a strip tile
constexpr int kStripHalf = kPassWarps * kStripRpt / 2;   // rows of a strip tile on each side of the crack line
constexpr int kBelowWarp = kPassWarps / 2 - 1;           // the warp whose last row is jc - 1; the next one's first is jc

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
template <typename D, typename T> __device__ __forceinline__ T wd_get(const D *p, T inv)
{
    if constexpr (std::is_same<D, Lf>::value) return p->v;
    else if constexpr (sizeof(D) == 2) return WdIO<D>::get(p, inv);
    else return *p;
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
                float d0, d1;
                up2(dn2, d0, d1);
                d.v[k] = wd_round<D, T>(d0, wd_scale, wd_inv);
                d.v[k + 1] = wd_round<D, T>(d1, wd_scale, wd_inv);
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

// Crack state in force during one step of a pass (modes whose decisions need
// no K: prescribed growth and stationary cracks).
struct PassTip {
    int64_t tr, tl;
    double vr, vl;       // speeds recorded by the crack step before the update
    int32_t f, l;
};

template <typename T>
struct PassShared {
    static constexpr int W = 32 * Vec<T>::N;
    alignas(16) T top[2][kPassWarps][W];    // each warp's last row, by step parity
    alignas(16) T bot[2][kPassWarps][W];    // each warp's first row
    alignas(16) T pair[kPassSteps][2][W];   // rows jc - 1 and jc of a strip tile at each step
    double ws[4][kPassSteps + 1];           // w* of the Dirichlet edges at t_n .. t_{n+K}
    PassTip log[kPassSteps + 1];
    CrackState S;
    int32_t reach[2];
};

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

// One K-criterion crack step of a strip tile by warp 0 (all 32 lanes): the
// ends this tile follows, from the pair rows of the current fields.  below /
// above: rows jc - 1 and jc of the tile, column i at i - org (org_l for the
// left end).
template <typename T>
__device__ __forceinline__ void pass_crack_step(const CrackParams &p, const T *below, const T *above, int org_r, int org_l,
                                                CrackState &S, const History &hist, bool ev_r, bool ev_l, bool commit_r,
                                                bool commit_l)
{
    constexpr int W = PassShared<T>::W;
    const int lane = threadIdx.x & 31;
    const bool act_r = ev_r && !S.r.decided, act_l = ev_l && !S.l.decided;
    // lanes 0-15 the right end, 16-31 the left: both criteria on the state before either advances
    const int dir = lane < 16 ? +1 : -1;
    const TipState &E = dir > 0 ? S.r : S.l;
    const int org = dir > 0 ? org_r : org_l;
    const CrackSums c = crack_eval_pairs<T, 16>(p, E.tip_q, E.v_prev, S.i_first, S.i_last, dir, [&](int i, T &a, T &b) {
        const int q = i - org;
        if (q < 0 || q >= W) return false;   // an end this tile does not follow
        a = above[q];
        b = below[q];
        return true;
    });
    CrackDecision d = {};
    if ((lane & 15) == 0 && (dir > 0 ? act_r : act_l)) d = crack_decide(p, S, dir, c);
    __syncwarp();
    const bool pending = !S.r.decided;
    if (lane == 0 && act_r) crack_commit(p, nullptr, hist, S, +1, commit_r, c, d);
    __syncwarp();
    if (lane == 16 && act_l) crack_commit(p, nullptr, hist, S, -1, commit_l, c, d);
    __syncwarp();
    if (lane == 0) {
        S.hist_n += pending ? 1 : 0;
        S.r.decided = 0;
        S.l.decided = 0;
    }
    __syncwarp();
}

// The crack steps of a pass whose decisions need no K, by one thread: the
// state in force during each update.  S becomes the state after the last.
__device__ __forceinline__ void pass_known_steps(const CrackParams &p, const History &hist, CrackState &S, PassTip *log,
                                                 int K)
{
    log[0].tr = S.r.tip_q;
    log[0].tl = S.l.tip_q;
    log[0].f = S.i_first;
    log[0].l = S.i_last;
    for (int s = 0; s < K; ++s) {
        const bool pending = !S.r.decided;
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
            crack_commit(p, nullptr, hist, S, dir, false, c, d);
        }
        S.hist_n += pending ? 1 : 0;
        S.r.decided = 0;
        S.l.decided = 0;
        log[s + 1].tr = S.r.tip_q;
        log[s + 1].tl = S.l.tip_q;
        log[s + 1].vr = S.r.v;
        log[s + 1].vl = S.l.v;
        log[s + 1].f = S.i_first;
        log[s + 1].l = S.i_last;
    }
}

// A column index taken around a lattice with periodic sides.
__device__ __forceinline__ int wrap_col(int c, int nx)
{
    c %= nx;
    return c < 0 ? c + nx : c;
}

// What a thread knows about its tile.
struct PassCtx {
    TileGeo g;
    int lane, warp, x0, jb;
    bool per;
    bool is_l;                  // element 0 is column 0 (no periodic sides)
    int kr;                     // the element that is column nx - 1, else -1
    bool side;                  // the tile's warps hold column 0 or nx - 1
    // strip tiles: whether the pass's decisions need no K; the ends this tile
    // follows (a link it can see may be cut in this pass); the ends whose
    // records it writes; the lattice column of its column 0 as seen from each
    // end; the severed columns at the start
    bool known, ev_r, ev_l, own_r, own_l, follow;
    int org_r, org_l, f0, l0;
};

// The fields of a thread: RPT rows of one vector.  Each update writes the
// new rows where the next one reads them, so that no register is copied from
// step to step: leapfrog storage writes w_{n+1} over w_{n-1} and the two
// planes change places; the other forms shift the rows of w by one slot, up
// in one step (PH = 0, rows swept upwards) and down in the next (PH = 1).
template <typename T, typename D, int RPT> struct PassRows {
    static constexpr int N = Vec<T>::N;
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

// One time step of a tile.
template <typename T, typename D, int RPT, int KIND, int PH>
__device__ __forceinline__ void pass_step(const PassArgs<T, D> &A, const PassCtx &c, int s, PassRows<T, D, RPT> &F,
                                          PassShared<T> &sh)
{
    constexpr int N = Vec<T>::N;
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
    if (KIND == 2 && c.known && warp == kBelowWarp) stg_row(&sh.pair[s][0][lane * N], F.template cur<PH>(RPT - 1));
    if (KIND == 2 && c.known && warp == kBelowWarp + 1) stg_row(&sh.pair[s][1][lane * N], F.template cur<PH>(0));
    __syncthreads();
    if (KIND == 2 && c.follow) {
        const bool reach = sh.reach[b] != 0;
        if (warp == 0) {
            pass_crack_step<T>(p, sh.top[b][kBelowWarp], sh.bot[b][kBelowWarp + 1], c.org_r, c.org_l, sh.S, a.hist, c.ev_r,
                               c.ev_l, c.own_r, c.own_l);
            if (lane == 0) sh.reach[b ^ 1] = crack_cut_in_reach(p, sh.S) ? 1 : 0;
        }
        // rows next to the crack wait for the decision only where it can cut a link
        if (reach) __syncthreads();
    }
    R dnx, upx;
    ld_row(&sh.top[b][warp > 0 ? warp - 1 : 0][lane * N], dnx);
    ld_row(&sh.bot[b][warp < kPassWarps - 1 ? warp + 1 : warp][lane * N], upx);
    uint32_t cut = 0u;
    if (KIND == 2 && (warp == kBelowWarp || warp == kBelowWarp + 1)) {
        const int f = c.known ? sh.log[s + 1].f : (c.ev_l ? sh.S.i_first : c.f0);
        const int l = c.known ? sh.log[s + 1].l : (c.ev_r ? sh.S.i_last : c.l0);
#pragma unroll
        for (int k = 0; k < N; ++k) {
            int q = x0 + k;
            if (c.per) q = wrap_col(q, nx);
            if (q >= f && q <= l) cut |= 1u << k;
        }
    }
    T tl = (T)0, tr = (T)0, tb = (T)0, tt = (T)0;
    R first, last;                                         // the first and last rows before the update
    T el[KIND != 0 ? RPT : 1], er[KIND != 0 ? RPT : 1];   // edge rule: the edge columns before the update
    const bool em_side = KIND != 0 && A.q.edge_macro && c.side;
    if (KIND != 0) {
        tl = (T)2 * (T)sh.ws[LEFT][s];
        tr = (T)2 * (T)sh.ws[RIGHT][s];
        tb = (T)2 * (T)sh.ws[BOTTOM][s];
        tt = (T)2 * (T)sh.ws[TOP][s];
        first = F.template cur<PH>(0);
        last = F.template cur<PH>(RPT - 1);
        if (em_side) {
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                el[r] = F.template cur<PH>(r).v[0];
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if (k == 0 || k == c.kr) er[r] = F.template cur<PH>(r).v[k];
            }
        }
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int r = PH == 0 ? q : RPT - 1 - q;
        const R cu = F.template cur<PH>(r);
        // the row whose slot this row's new values take is read first
        R up = r + 1 < RPT ? F.template cur<PH>(r + 1 < RPT ? r + 1 : r) : upx;
        R dn = r > 0 ? F.template cur<PH>(r > 0 ? r - 1 : r) : dnx;
        T left0 = __shfl_up_sync(kFull, cu.v[N - 1], 1);
        T rightN = __shfl_down_sync(kFull, cu.v[0], 1);
        if (KIND != 0) {
            const int j = jb + r;
            if (j == ny - 1) {
#pragma unroll
                for (int k = 0; k < N; ++k) up.v[k] = a.edge[TOP] == EDGE_DIRICHLET ? tt - cu.v[k] : cu.v[k];
            }
            if (j == 0) {
#pragma unroll
                for (int k = 0; k < N; ++k) dn.v[k] = a.edge[BOTTOM] == EDGE_DIRICHLET ? tb - cu.v[k] : cu.v[k];
            }
            if (KIND == 2 && r == RPT - 1 && warp == kBelowWarp) {
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if ((cut >> k) & 1u) up.v[k] = cu.v[k];
            }
            if (KIND == 2 && r == 0 && warp == kBelowWarp + 1) {
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if ((cut >> k) & 1u) dn.v[k] = cu.v[k];
            }
            if (c.is_l) left0 = a.edge[LEFT] == EDGE_DIRICHLET ? tl - cu.v[0] : cu.v[0];
        }
        R hs;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const T wl = k == 0 ? left0 : cu.v[k - 1];
            T wr = k == N - 1 ? rightN : cu.v[k + 1];
            if (KIND != 0 && k == c.kr) wr = a.edge[RIGHT] == EDGE_DIRICHLET ? tr - cu.v[k] : cu.v[k];
            hs.v[k] = wl + wr;
        }
        R out;
        row_sites<T, D, N>(cu, up, dn, hs, F.template rate<PH>(r), gg, dt, wd_scale, wd_inv, out);
        F.template next<PH>(r) = out;
    }
    if (KIND == 2 && p.macro && cut) {
        // the crack-face rule: w_B from the two new values further from the crack
        if (warp == kBelowWarp) {
            R &w1 = F.template next<PH>(RPT - 1), &w2 = F.template next<PH>(RPT - 2), &w3 = F.template next<PH>(RPT - 3);
#pragma unroll
            for (int k = 0; k < N; ++k)
                if ((cut >> k) & 1u) {
                    const T wB = (T)1.5 * w2.v[k] - (T)0.5 * w3.v[k];
                    if (!kLf) F.b[RPT - 1].v[k] = wd_round<D, T>((wB - last.v[k]) / dt, wd_scale, wd_inv);
                    w1.v[k] = wB;
                }
        } else {
            R &w1 = F.template next<PH>(0), &w2 = F.template next<PH>(1), &w3 = F.template next<PH>(2);
#pragma unroll
            for (int k = 0; k < N; ++k)
                if ((cut >> k) & 1u) {
                    const T wB = (T)1.5 * w2.v[k] - (T)0.5 * w3.v[k];
                    if (!kLf) F.b[0].v[k] = wd_round<D, T>((wB - first.v[k]) / dt, wd_scale, wd_inv);
                    w1.v[k] = wB;
                }
        }
    }
    if (KIND != 0 && A.q.edge_macro) {
        // the macroscopic rule on the outer edges (the two levels of
        // edge_rule_at): the edge columns, the crack-face points on
        // them, then the bottom and top rows and the corners
        const bool on_l = a.edge[LEFT] != EDGE_PERIODIC, on_r = a.edge[RIGHT] != EDGE_PERIODIC;
        EdgeRule<T> E;
        E.wn = nullptr;
        E.pitch = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            E.dir[e] = a.edge[e] == EDGE_DIRICHLET;
            E.ws[e] = (T)sh.ws[e][s + 1];
        }
        R in1, in2;         // rows 1, 2 (or ny-2, ny-3) before the edge columns
        const bool has_b = jb == 0, has_t = jb + RPT == ny;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            in1.v[k] = has_t ? F.template next<PH>(RPT - 2).v[k] : F.template next<PH>(1).v[k];
            in2.v[k] = has_t ? F.template next<PH>(RPT - 3).v[k] : F.template next<PH>(2).v[k];
        }
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            if (!em_side) break;
            R &w = F.template next<PH>(r);
            const int j = jb + r;
            const T p1 = __shfl_up_sync(kFull, w.v[N - 1], 1), p2 = __shfl_up_sync(kFull, w.v[N - 2], 1);
            const T n0 = __shfl_down_sync(kFull, w.v[0], 1);
            if (j < 1 || j > ny - 2) continue;
            if (c.is_l && on_l) {
                const T v2 = N > 2 ? w.v[N > 2 ? 2 : 0] : n0;
                w.v[0] = E.rule(LEFT, w.v[1], v2);
            }
            if (c.kr >= 0 && on_r) {
                T wI = p1, wII = p2;
#pragma unroll
                for (int k = 1; k < N; ++k)
                    if (k == c.kr) {
                        wI = w.v[k - 1];
                        wII = k >= 2 ? w.v[k >= 2 ? k - 2 : 0] : p1;
                    }
                const T v = E.rule(RIGHT, wI, wII);
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if (k == c.kr) w.v[k] = v;
            }
        }
        if (KIND == 2 && em_side && p.macro && cut && (c.is_l || c.kr >= 0)) {
            const bool be = warp == kBelowWarp;
#pragma unroll
            for (int k = 0; k < N; ++k) {
                if (!((cut >> k) & 1u) || !((c.is_l && on_l && k == 0) || (on_r && k == c.kr))) continue;
                const T v1 = be ? F.template next<PH>(RPT - 2).v[k] : F.template next<PH>(1).v[k];
                const T v2 = be ? F.template next<PH>(RPT - 3).v[k] : F.template next<PH>(2).v[k];
                const T v = (T)1.5 * v1 - (T)0.5 * v2;
                if (be) F.template next<PH>(RPT - 1).v[k] = v;
                else F.template next<PH>(0).v[k] = v;
            }
        }
        if (has_b || has_t) {
            const int ev = has_t ? TOP : BOTTOM;
            R e1, e2;   // the rows one and two from the edge, after the edge columns
#pragma unroll
            for (int k = 0; k < N; ++k) {
                e1.v[k] = has_t ? F.template next<PH>(RPT - 2).v[k] : F.template next<PH>(1).v[k];
                e2.v[k] = has_t ? F.template next<PH>(RPT - 3).v[k] : F.template next<PH>(2).v[k];
            }
            R o;
#pragma unroll
            for (int k = 0; k < N; ++k) o.v[k] = E.rule(ev, in1.v[k], in2.v[k]);
            // corners: along the bottom / top edge's normal from the edge
            // columns, or (its side Dirichlet, ev not) along the row from
            // the points of edge ev
            const T q1 = __shfl_up_sync(kFull, o.v[N - 1], 1), q2 = __shfl_up_sync(kFull, o.v[N - 2], 1);
            const T m0 = __shfl_down_sync(kFull, o.v[0], 1);
            T cl = (T)0, cr = (T)0;
            if (c.is_l && on_l)
                cl = a.edge[LEFT] == EDGE_DIRICHLET && a.edge[ev] != EDGE_DIRICHLET
                         ? E.rule(LEFT, o.v[1], N > 2 ? o.v[N > 2 ? 2 : 0] : m0)
                         : E.rule(ev, e1.v[0], e2.v[0]);
            if (c.kr >= 0 && on_r) {
                T oI = q1, oII = q2, c1 = (T)0, c2 = (T)0;
#pragma unroll
                for (int k = 0; k < N; ++k)
                    if (k == c.kr) {
                        if (k >= 1) oI = o.v[k >= 1 ? k - 1 : 0];
                        if (k >= 1) oII = k >= 2 ? o.v[k >= 2 ? k - 2 : 0] : q1;
                        c1 = e1.v[k];
                        c2 = e2.v[k];
                    }
                cr = a.edge[RIGHT] == EDGE_DIRICHLET && a.edge[ev] != EDGE_DIRICHLET ? E.rule(RIGHT, oI, oII)
                                                                                   : E.rule(ev, c1, c2);
            }
            if (c.is_l && on_l) o.v[0] = cl;
#pragma unroll
            for (int k = 0; k < N; ++k)
                if (on_r && k == c.kr) o.v[k] = cr;
            if (has_t) F.template next<PH>(RPT - 1) = o;
            else F.template next<PH>(0) = o;
        }
        if (!kLf && (em_side || has_b || has_t)) {
            // wdot of the sites that took the rule
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const R &w = F.template next<PH>(r);
                const int j = jb + r;
                if (j == 0 || j == ny - 1) {
                    if ((r == 0 && has_b) || (r == RPT - 1 && has_t)) {
#pragma unroll
                        for (int k = 0; k < N; ++k)
                            F.b[r].v[k] = wd_round<D, T>((w.v[k] - (r == 0 ? first.v[k] : last.v[k])) / dt, wd_scale, wd_inv);
                    }
                    continue;
                }
                if (!em_side) continue;
                if (c.is_l && on_l) F.b[r].v[0] = wd_round<D, T>((w.v[0] - el[r]) / dt, wd_scale, wd_inv);
                if (c.kr >= 0 && on_r) {
#pragma unroll
                    for (int k = 0; k < N; ++k)
                        if (k == c.kr) F.b[r].v[k] = wd_round<D, T>((w.v[k] - er[r]) / dt, wd_scale, wd_inv);
                }
            }
        }
    }
}

// A tile.  KIND: 0 one none of whose sites sees an edge or the crack, 1 with
// outer edges, 2 a crack-strip tile (with edges where it meets them).
template <typename T, typename D, int RPT, int KIND>
__device__ __forceinline__ void pass_tile(const PassArgs<T, D> &A, const TileGeo g, PassShared<T> &sh)
{
    constexpr int N = Vec<T>::N;
    constexpr int W = PassShared<T>::W;
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
        const T *wp = a.w_in + (int64_t)jb * P + x0;
        const D *dp = A.wd_in + (int64_t)jb * P + x0;
        const bool whole = KIND == 0 ? x0 < nx : (x0 >= 0 && x0 + N <= nx);
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            R &w = F.template cur<0>(r), &d = F.b[r];
#pragma unroll
            for (int k = 0; k < N; ++k) w.v[k] = d.v[k] = (T)0;
            const int j = jb + r;
            if (j < 0 || j >= ny) continue;
            if (whole) {
                ldg_row(wp + (int64_t)r * P, w);
                WdIO<D>::load(dp + (int64_t)r * P, d, wd_inv);
            } else if (KIND != 0) {
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    int q = x0 + k;
                    if (per) q = wrap_col(q, nx);
                    if (q < 0 || q >= nx) continue;
                    w.v[k] = a.w_in[(int64_t)j * P + q];
                    d.v[k] = wd_get(A.wd_in + (int64_t)j * P + q, wd_inv);
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
    if (KIND == 2) {
        c.known = p.mode != CRACK_KCRIT;
        c.f0 = a.s_in->i_first;
        c.l0 = a.s_in->i_last;
        hist0 = a.s_in->hist_n;
        rec0 = a.s_in->r.decided ? 1 : 0;   // the first update whose crack step is still to run
        const int cr = tip_col_r(c.f0, c.l0, nx), cl = tip_col_l(c.f0, c.l0, nx);
        const int hc = A.q.hc, grow = A.q.grow;
        // (periodic sides: the column itself, then its images beyond either side)
        for (int q = 0; q < (per ? 3 : 1); ++q) {
            const int o = q == 0 ? 0 : (q == 1 ? -nx : nx);
            if (cr + o >= g.x0 && cr + o < g.x1) c.own_r = true;
            if (p.two_tips && cl + o >= g.x0 && cl + o < g.x1) c.own_l = true;
            if (!c.ev_r && g.x0 - hc <= cr + o + grow && g.x1 + hc > cr + o) {
                c.ev_r = true;
                c.org_r = g.xl - o;
            }
            if (p.two_tips && !c.ev_l && g.x0 - hc <= cl + o && g.x1 + hc > cl + o - grow) {
                c.ev_l = true;
                c.org_l = g.xl - o;
            }
        }
        c.follow = !c.known && (c.ev_r || c.ev_l);
        if (tid == 0) {
            sh.S = *a.s_in;
            if (c.known) pass_known_steps(p, a.hist, sh.S, sh.log, K);
            else sh.reach[0] = crack_cut_in_reach(p, sh.S) ? 1 : 0;
        }
    }
    if (KIND != 0) {
        const int64_t n = a.s_in->step;
        if (tid < 4 * (kPassSteps + 1)) {
            const int e = tid / (kPassSteps + 1), q = tid % (kPassSteps + 1);
            if (q <= K) sh.ws[e][q] = a.edge[e] == EDGE_DIRICHLET ? load_value(a.load[e], n + q, (double)p.dt) : 0.0;
        }
    }
    c.is_l = KIND != 0 && !per && x0 == 0;
    c.kr = KIND != 0 && !per && nx - 1 - x0 >= 0 && nx - 1 - x0 < N ? nx - 1 - x0 : -1;

    c.side = KIND != 0 && __any_sync(kFull, c.is_l || c.kr >= 0);
    // bulk tiles: two steps an iteration (PassRows); an odd last step leaves
    // the rows where a step of phase 0 writes them.  The other tiles, whose
    // step is far longer code, take every step in phase 0 and move the rows
    // back: unrolled twice, it ran out of the instruction cache.
    int s = 0;
    if (KIND == 0) {
        for (; s + 2 <= K; s += 2) {
            pass_step<T, D, RPT, KIND, 0>(A, c, s, F, sh);
            pass_step<T, D, RPT, KIND, 1>(A, c, s + 1, F, sh);
        }
    }
    for (; s < K; ++s) {
        pass_step<T, D, RPT, KIND, 0>(A, c, s, F, sh);
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
    T acc = (T)0;
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
        const R &w = F.template cur<0>(r), &d = F.b[r];
        const int j = jb + r;
        if (j < g.y0 || j >= g.y1) continue;
        if (x0 + N <= g.x0 || x0 >= g.x1) continue;
        const int64_t o = (int64_t)j * P + x0;
        if (KIND == 0 || (x0 >= g.x0 && x0 + N <= g.x1 && x0 >= 0 && x0 + N <= nx)) {
            stg_row(a.w_out + o, w);
            wd_store(a.wd + o, d, wd_scale);
            if (KIND != 0) write_pads(a, x0, j, w);
            acc += w.v[0];
        } else {
#pragma unroll
            for (int k = 0; k < N; ++k) {
                int q = x0 + k;
                if (q < g.x0 || q >= g.x1) continue;
                if (per) q = wrap_col(q, nx);
                if (q < 0 || q >= nx) continue;
                T *row = a.w_out + (int64_t)j * P;
                const T v = w.v[k];
                row[q] = v;
                wd_put(a.wd + (int64_t)j * P + q, d.v[k], wd_scale);
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

    if (KIND == 2 && (c.own_r || c.own_l)) {
        if (c.known) {
            // the K fits of the pass's crack steps, one step per warp: their
            // decisions did not wait for them
            if (warp >= rec0 && warp < K) {
                for (int dir = 1; dir >= (c.own_l ? -1 : 1); dir -= 2) {
                    if (dir > 0 && !c.own_r) continue;
                    const PassTip &q = sh.log[warp], &q1 = sh.log[warp + 1];
                    const int org = dir > 0 ? c.org_r : c.org_l;
                    const double v_prev = p.mode == CRACK_PRESCRIBED ? p.v_rel : 0.0;
                    const CrackSums f = crack_eval_pairs<T, 32>(
                        p, dir > 0 ? q.tr : q.tl, v_prev, q.f, q.l, dir, [&](int i, T &ab, T &be) {
                            const int e = i - org;
                            if (e < 0 || e >= W) return false;
                            ab = sh.pair[warp][1][e];
                            be = sh.pair[warp][0][e];
                            return true;
                        });
                    if (lane == 0) {
                        const double Kf = f.np > 0 ? p.mu / 4.0 * f.num / f.den : 0.0;
                        if (!isfinite(Kf)) atomicOr(a.err, (uint32_t)ERR_NONFINITE);
                        if (p.hist_cap > 0) {
                            const int64_t h = (hist0 + (warp - rec0)) % p.hist_cap;
                            (dir > 0 ? a.hist.K : a.hist.Kl)[h] = Kf;
                            (dir > 0 ? a.hist.v : a.hist.vl)[h] = dir > 0 ? q1.vr : q1.vl;
                            (dir > 0 ? a.hist.tip : a.hist.tipl)[h] = dir > 0 ? q1.tr : q1.tl;
                            (dir > 0 ? a.hist.np : a.hist.npl)[h] = f.np;
                        }
                        if (warp == K - 1) {
                            TipState &O = dir > 0 ? a.s_out->r : a.s_out->l;
                            O.K = Kf;
                            O.r_min = f.r_min;
                            O.npairs = f.np;
                        }
                    }
                }
            }
        } else {
            __syncthreads();   // the last crack step
        }
        if (tid == 0) {
            CrackState *o = a.s_out;
            const CrackState &S = sh.S;
            if (c.own_r) {
                o->step = S.step + K;
                o->hist_n = S.hist_n;
                o->i_last = S.i_last;
                if (!p.two_tips) o->i_first = S.i_first;
                copy_tip_decision(o->r, S.r);
                if (!c.known) {
                    o->r.K = S.r.K;
                    o->r.r_min = S.r.r_min;
                    o->r.npairs = S.r.npairs;
                }
                o->r.decided = 0;
                for (int i = c.l0 + 1; i <= S.i_last; ++i)
                    if (i >= c.f0) atomicOr(&a.cut_v[(int64_t)(p.jc - 1) * p.words + (i >> 5)], 1u << (i & 31));
            }
            if (c.own_l) {
                o->i_first = S.i_first;
                copy_tip_decision(o->l, S.l);
                if (!c.known) {
                    o->l.K = S.l.K;
                    o->l.r_min = S.l.r_min;
                    o->l.npairs = S.l.npairs;
                }
                o->l.decided = 0;
                for (int i = S.i_first; i < c.f0; ++i)
                    if (i <= c.l0) atomicOr(&a.cut_v[(int64_t)(p.jc - 1) * p.words + (i >> 5)], 1u << (i & 31));
            }
        }
    }
}

// Tile t of a pass.
template <typename T, typename D, int RPT>
__device__ __forceinline__ void pass_cta(const PassArgs<T, D> &A, int t, PassShared<T> &sh)
{
    constexpr int N = Vec<T>::N;
    const StepArgs<T, D> &a = A.s;
    const PassPlan &q = A.q;
    const int nx = a.nx, ny = a.ny;
    const bool per = a.edge[LEFT] == EDGE_PERIODIC;
    const int tid = threadIdx.x;
    // the next pass's Dirichlet values (and, without a crack, its state): the last tile
    if (t == q.tiles - 1 && tid < 4) {
        const int64_t n1 = a.s_in->step + q.K;
        if (tid == 0 && a.p.mode == CRACK_NONE) {
            CrackState S = *a.s_in;
            S.step = n1;
            S.r.decided = 1;
            S.l.decided = 1;
            for (int e = 0; e < 4; ++e)
                S.wstar[e] = a.edge[e] == EDGE_DIRICHLET ? load_value(a.load[e], n1, (double)a.p.dt) : 0.0;
            *a.s_out = S;
        } else if (a.p.mode != CRACK_NONE) {
            a.s_out->wstar[tid] = a.edge[tid] == EDGE_DIRICHLET ? load_value(a.load[tid], n1, (double)a.p.dt) : 0.0;
        }
    }
    TileGeo g;
    if (t < q.ms) {
        const int f = a.s_in->i_first, l = a.s_in->i_last;
        const int cr = tip_col_r(f, l, nx), cl = tip_col_l(f, l, nx);
        int lo0 = cr - q.zb, hi0 = cr + q.za, lo1 = cl + 1 - q.za, hi1 = cl + q.zb;
        bool two = a.p.two_tips != 0;
        if (two && lo0 <= hi1 + N && lo1 <= hi0 + N) {   // one zone around both tips
            lo0 = min(lo0, lo1);
            hi0 = max(hi0, hi1);
            two = false;
        }
        g.x0 = t == 0 && !per ? 0 : pass_boundary<N>(t * q.ps, nx, per, lo0, hi0, lo1, hi1, two);
        if (t + 1 < q.ms) g.x1 = pass_boundary<N>((t + 1) * q.ps, nx, per, lo0, hi0, lo1, hi1, two);
        else g.x1 = per ? nx + pass_boundary<N>(0, nx, per, lo0, hi0, lo1, hi1, two) : nx;
        if (q.ms == 1) {
            g.x0 = 0;
            g.x1 = nx;
        }
        if (g.x0 >= g.x1) return;
        g.xl = g.x0 == 0 && !per ? 0 : g.x0 - q.hc;
        g.yl = a.p.jc - kStripHalf;
        g.y0 = q.jb;
        g.y1 = q.jt;
        pass_tile<T, D, kStripRpt, 2>(A, g, sh);
        return;
    }
    t -= q.ms;
    const int cx = t % q.mx, ry = t / q.mx;
    g.x0 = cx * q.px;
    g.x1 = min(g.x0 + q.px, nx);
    if (ry < q.mb) {
        g.y0 = ry * q.pb;
        g.y1 = min(g.y0 + q.pb, q.jb);
    } else {
        g.y0 = q.jt + (ry - q.mb) * q.pt;
        g.y1 = min(g.y0 + q.pt, ny);
    }
    g.xl = g.x0 == 0 && !per ? 0 : g.x0 - q.hc;
    g.yl = g.y0 == 0 ? 0 : (g.y1 == ny ? ny - kPassWarps * RPT : g.y0 - q.K);
    const bool plain = g.x0 >= q.K && g.x1 + q.K <= nx && g.y0 >= q.K && g.y1 + q.K <= ny && g.xl >= 0;
    if (plain) pass_tile<T, D, RPT, 0>(A, g, sh);
    else pass_tile<T, D, RPT, 1>(A, g, sh);
}

template <typename T, typename D, int RPT>
__global__ void __launch_bounds__(kPassThreads, 2) pass_kernel(const __grid_constant__ PassArgs<T, D> a)
{
    __shared__ PassShared<T> sh;
    pdl_wait();
    pdl_trigger();
    pass_cta<T, D, RPT>(a, blockIdx.x, sh);
}

template <typename T, typename D> cudaError_t launch_pass(const PassArgs<T, D> &a, int rpt, cudaStream_t s)
{
    const dim3 grid((unsigned)a.q.tiles), block(kPassThreads);
    const bool ch = a.s.chained != 0;
    return rpt == 8 ? launch_chained(pass_kernel<T, D, 8>, grid, block, 0, s, ch, a)
                    : launch_chained(pass_kernel<T, D, 4>, grid, block, 0, s, ch, a);
}

}  // namespace lbm
