// lbm_pass_plan.cu -- host side of the passes (lbm_pass.cuh): how the
// lattice is split into tiles for a pass of K steps.
#include "lbm_host.h"
#include "lbm_window.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace lbm {
namespace host {

namespace {

int ceil_div(int a, int b) { return (a + b - 1) / b; }
int round_up(int a, int n) { return ceil_div(a, n) * n; }

// FP64 runs at two results a cycle and SM, so recomputed halos cost more than
// saved launches and traffic give once every SM has its tile.  Time per step
// in passes and (in parentheses) in single steps.  Above kPass64Small sites:
// the K-criterion 512^2 10.1 (13.3), 640^2 11.6 (12.6), 724^2 18.4 us (14.2 us)
// and nine velocities 512^2 16.4 (24.8), 640^2 18.6 (26.8), 724^2 30.5 us (29.7
// us): passes of four steps while there are no more tiles of eight warps than
// SMs.  Prescribed growth 600^2 10.0 (10.1), 1500 x 90 10.0 (8.7), periodic sides
// 1500 x 90 9.3 us (5.8 us) and the edge rule 512^2 19.9 us (16.1 us): single
// steps.  Up to kPass64Small sites, in tiles of four warps: 362^2 7.3 (9.0), K-
// criterion 10.4 (11.1), nine velocities 13.0 (18.4), the edge rule 9.7 us (13.7
// us) on 1000 x 120.  Up to kPass64Narrow they are one column a thread (128^2,
// stationary crack: 3.2 us, two columns a thread 4.4 us, single steps 10.9 us).
constexpr int64_t kPass64Small = (int64_t)1 << 17, kPass64Narrow = (int64_t)1 << 16;

// n items in m tiles: of p, the first e of one more.
void even(int n, int m, int &p, int &e)
{
    p = m > 0 ? n / m : 0;
    e = m > 0 ? n % m : 0;
}

// Row tiles of H held rows, K of them halo on each side that is no lattice
// edge, over a region of `len` rows; at least `least` tiles.  Even: the rules
// next to an edge span three rows of a tile.
void split_rows(int len, int H, int K, bool edge0, bool edge1, int least, int &m, int &p, int &e)
{
    m = 0;
    if (len > 0) {
        const int one = H - (edge0 ? 0 : K) - (edge1 ? 0 : K);
        if (len <= one) m = 1;
        else if (edge0 && edge1 && len <= 2 * (H - K)) m = 2;
        else m = ceil_div(len, H - 2 * K);
        m = std::max(m, std::min(least, len));
    }
    even(len, m, p, e);
}

}  // namespace

bool pass_plan(const lbm_handle *h, int K, int nw, int rpt, PassPlan &q, bool adjoint, bool narrow)
{
    const int nx = h->grid.nx, ny = h->grid.ny;
    const int N = narrow ? 1 : (int)(16 / h->esize), W = 32 * N, H = nw * rpt;
    const int strip_half = nw * 4 / 2;   // kStripRpt rows a warp
    const bool per = h->grid.edge[LBM_LEFT] == LBM_EDGE_PERIODIC;
    const bool crack = h->cp.mode != CRACK_NONE;
    const CrackParams &p = h->cp;
    if (K < 2 || K > nw || 2 * K > strip_half) return false;
    if (per && nx < 16) return false;   // a halo holds at most one image of a column
    if (crack && p.hist_cap > 0 && p.hist_cap < K) return false;   // a pass's records go around the ring once at most
    std::memset(&q, 0, sizeof q);
    q.K = K;
    q.nw = nw;
    q.rpt = rpt;
    q.hc = round_up(K, N);
    q.edge_macro = h->edge_macro ? 1 : 0;

    // bulk columns
    const int ow = W - 2 * q.hc;
    if (nx + (per ? 2 * q.hc : 0) <= W) q.mx = 1;
    else q.mx = !per && nx <= 2 * (W - q.hc) ? 2 : ceil_div(nx, ow);
    if (N == 1) {
        even(nx, q.mx, q.px, q.ex);
    } else {
        q.px = ceil_div(ceil_div(nx, q.mx), N);
        // no last tile narrower than the columns the rules next to an edge span
        while (nx - (ceil_div(nx, q.px * N) - 1) * q.px * N < 4 && q.px > 1) --q.px;
        q.mx = ceil_div(nx, q.px * N);
    }

    // rows: the crack strip, and the bulk below and above it (all of it without a crack)
    const int so = strip_half - K;
    // the transposed crack-face rule reaches two rows further from the crack
    if (adjoint && crack && p.macro && so < K + 2) return false;
    int region0 = 0, region1 = ny;
    if (crack) {
        region0 = std::max(0, p.jc - so);
        region1 = std::min(ny, p.jc + so);
        q.jb = region0;
        q.jt = region1;
        split_rows(q.jb, H, K, true, false, 1, q.mb, q.pb, q.eb);
        split_rows(ny - q.jt, H, K, false, true, 1, q.mt, q.pt, q.et);
    } else {
        split_rows(ny, H, K, true, true, h->edge_macro ? 2 : 1, q.mt, q.pt, q.et);
    }
    // the edge rule is applied by tiles whose rows 0 .. 2 (or ny-1 .. ny-3) lie
    // in one thread: tiles held from row 0 or up to row ny - 1, not the strip
    if (h->edge_macro && (crack ? p.jc < strip_half + 3 || ny - p.jc < strip_half + 3 : ny < 64)) return false;
    if (h->edge_macro && nx < 4) return false;

    if (crack && adjoint) {
        q.ms = q.mx;
    } else if (crack) {
        // columns an end can cut in a pass, and the reach of its K window
        const int64_t dq = p.mode == CRACK_KCRIT ? p.dq_max : p.mode == CRACK_PRESCRIBED ? p.dq_prescribed : 0;
        // (D2Q9: a diagonal crossing lies up to half a spacing behind the next
        // vertical link and belongs to the columns on both of its sides)
        const int d9 = h->q == 9 ? 2 : 0;
        q.grow = (int)((dq * K) >> kQBits) + 2 + d9;
        q.back = d9;
        const double v = p.mode == CRACK_KCRIT ? p.v_max : p.mode == CRACK_PRESCRIBED ? p.v_rel : 0.0;
        const double r_min = p.r_min_fixed > 0.0 ? p.r_min_fixed : p.r0 / (1.0 - v);
        const double reach = (r_min + p.fit_width) / p.dh;
        // the window of an end at rest (prescribed growth: at its speed), as
        // crack_eval_pairs bounds it, in whole units
        const double v0 = p.mode == CRACK_PRESCRIBED ? p.v_rel : 0.0;
        q.r_min = p.r_min_fixed > 0.0 ? p.r_min_fixed : (v0 == 0.0 ? p.r0 : p.r0 / (1.0 - v0));
        const double lo = p.dh == 1.0 ? q.r_min : q.r_min / p.dh;
        const double hi = p.dh == 1.0 ? q.r_min + p.fit_width : (q.r_min + p.fit_width) / p.dh;
        q.lo_q = (int64_t)std::ceil(std::min(lo, 1e6) * 4294967296.0);
        q.hi_q = (int64_t)std::ceil(std::min(hi, 1e6) * 4294967296.0);
        q.one_pair = p.fit_width <= p.dh && q.hi_q - q.lo_q <= ((int64_t)1 << kQBits);
        // (a fixed r_min does not follow the speed: the general step)
        q.unit = p.dh == 1.0 && p.dt == 1.0 && !(p.r_min_fixed > 0.0) && known_divisor(p.K_C) && p.r0 >= kWindowR0;
        q.lo_f = (float)p.r0;
        q.lo_max = (float)std::min((double)kWindowLo, 1.001 * p.r0 / (1.0 - p.v_max));
        q.slack = q.unit ? (uint32_t)window_slack(q.lo_f, q.lo_max) : 0u;
        q.w_q = (int64_t)std::llrint(std::min(p.fit_width / p.dh, 1e6) * 4294967296.0);
        q.k_inv = known_inverse(p.K_C);
        // the FP32 test that an end at rest stays there has a margin of 1e-3: taken
        // where neither its factors nor an FP64 jump too small for FP32 (off by
        // 2^-150 at most, times up to 16 units) round by as much; else an end is
        // never seen to rest by it
        const double unit = p.mu / 4.0 * std::sqrt(2.0 * kPi / p.dh) * 65536.0;
        q.k_unit = (float)unit;
        q.k_rest = unit >= 0x1p-60 && unit <= 0x1p90 && p.K_C >= 0x1p-100 && p.K_C >= unit * 0x1p-135 ? (float)(p.K_C * 0.999) : 0.0f;
        // both ends are fitted at once by half a warp each: at most 16 columns
        if (!(p.fit_width / p.dh <= 12.0)) return false;
        q.free = narrow && p.mode != CRACK_KCRIT && q.one_pair;
        if (q.free) {
            q.ms = q.mx;
        } else if (nx + (per ? 2 * q.hc : 0) <= W) {
            q.ms = 1;
            q.ps = nx;
        } else {
            if (!(reach < (double)W)) return false;
            q.zb = std::max((int)std::ceil(reach) + 4 + K - q.hc, q.hc) + 1 + d9;
            q.za = q.grow + q.hc + 1;
            const int Z = q.zb + q.za + 1;
            const int moved = p.two_tips ? Z + 2 * N : Z / 2 + N;   // how much wider moved boundaries can make a tile
            const int most = (ow - moved - 4) / N * N;
            if (most < 4 * N) return false;
            q.ms = ceil_div(nx, most);
            q.ps = round_up(ceil_div(nx, q.ms), N);
            // one boundary at most in the zones (or zone) around the tips
            const int zone = p.two_tips ? 2 * Z + N : Z;
            if (q.ps <= zone) q.ps = most;
            q.ms = ceil_div(nx, q.ps);
            if (q.ms > 2 && q.ps <= zone) return false;
            if (per && q.ps <= zone) return false;
        }
    }
    q.tiles = q.ms + q.mx * (q.mb + q.mt);
    return true;
}

void choose_pass(lbm_handle *h)
{
    h->pass_k = 0;
    h->pass_narrow = false;
    if (!h->alt[0]) return;
    const int64_t sites = (int64_t)h->grid.nx * h->grid.ny;
    const bool f64 = h->esize == 8;
    if (f64 && sites > kPass64Small && (h->edge_macro || (h->q == 5 && h->cp.mode != CRACK_KCRIT))) return;
    auto feasible = [&](int K, bool narrow) {
        PassPlan q;
        h->pass_nw = f64 && (narrow || sites <= kPass64Small) ? 4 : 8;
        h->pass_rpt = h->pass_nw == 4 ? 4 : 8;
        if (!pass_plan(h, K, h->pass_nw, h->pass_rpt, q, false, narrow)) return false;
        if (f64 && sites > kPass64Small && (K < 4 || q.tiles > h->sms)) return false;
        // shorter tiles while the taller ones would leave a good part of the SMs
        // with one: four and (in parentheses) eight rows a thread, prescribed
        // growth, 512 x 192 1.32 (1.38), 1024^2 1.74 (1.76), 1400 x 1024 2.09
        // (1.89), 1600 x 1400 2.83 us (2.26 us); FP16 rates, periodic sides 1001 x
        // 777 2.29 (2.90), 1400 x 1024 2.99 us (2.82 us)
        if (!f64 && q.tiles < 7 * h->sms / 4) h->pass_rpt = 4;
        bool all = true;   // every shorter pass too: a call's last passes
        for (int k = K; k >= 2; --k) all = all && pass_plan(h, k, h->pass_nw, h->pass_rpt, q, false, narrow);
        return all;
    };
    // (the edge rule, nine velocities and a tape's passes take two columns a thread)
    if (f64 && sites <= kPass64Narrow && !h->edge_macro && h->q == 5 && feasible(4, true) && feasible(4, false)) {
        h->pass_k = 4;
        h->pass_narrow = true;
    }
    for (int K = f64 ? 4 : 8; K >= 2 && !h->pass_k; --K)
        if (feasible(K, false)) h->pass_k = K;
    if (!h->pass_k) return;
    const int nw = h->pass_nw, rpt = h->pass_rpt;
    const void *fn = h->q == 9 ? (f64 ? pass_kernel_ptr<double, double, kNine>(nw, rpt, true)
                                      : pass_kernel_ptr<float, float, kNine>(nw, rpt, true))
                     : h->pass_narrow                     ? pass_kernel_ptr<double, NarrowF64>(nw, rpt, true)
                     : h->lat.storage == LBM_F64          ? pass_kernel_ptr<double, double>(nw, rpt, true)
                     : h->lat.storage == LBM_F32_WD_BF16  ? pass_kernel_ptr<float, __nv_bfloat16>(nw, rpt, true)
                     : h->lat.storage == LBM_F32_WD_F16   ? pass_kernel_ptr<float, __half>(nw, rpt, true)
                     : h->lat.storage == LBM_F32_LEAPFROG ? pass_kernel_ptr<float, Lf>(nw, rpt, true)
                                                          : pass_kernel_ptr<float, float>(nw, rpt, true);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * nw, 0) != cudaSuccess || per_sm < 1) {
        h->pass_k = 0;
        return;
    }
    h->pass_slots = per_sm * h->sms;
}

}  // namespace host
}  // namespace lbm
