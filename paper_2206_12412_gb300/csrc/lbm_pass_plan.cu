// lbm_pass_plan.cu -- host side of the passes (lbm_pass.cuh): how the
// lattice is split into tiles for a pass of K steps.
#include "lbm_host.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace lbm {
namespace host {

namespace {

int ceil_div(int a, int b) { return (a + b - 1) / b; }
int round_up(int a, int n) { return ceil_div(a, n) * n; }

// FP64 lattices up to kPass64Sites sites are stepped in passes, those up to
// kPass64Small in tiles of four warps.
constexpr int64_t kPass64Sites = (int64_t)1 << 19, kPass64Small = (int64_t)1 << 17;

// Row tiles of H held rows, K of them halo on each side that is no lattice
// edge, over a region of `len` rows; at least `least` tiles.
void split_rows(int len, int H, int K, bool edge0, bool edge1, int least, int &m, int &p)
{
    m = 0;
    p = 1;
    if (len <= 0) return;
    const int one = H - (edge0 ? 0 : K) - (edge1 ? 0 : K);
    if (len <= one) m = 1;
    else if (edge0 && edge1 && len <= 2 * (H - K)) m = 2;
    else m = ceil_div(len, H - 2 * K);
    m = std::max(m, std::min(least, len));
    p = ceil_div(len, m);
    // no last tile thinner than the three rows the rules next to an edge span
    while (m > 1 && p > 3 && len - (ceil_div(len, p) - 1) * p < 3) --p;
    m = ceil_div(len, p);
}

}  // namespace

bool pass_plan(const lbm_handle *h, int K, int nw, int rpt, PassPlan &q, bool adjoint)
{
    const int nx = h->grid.nx, ny = h->grid.ny;
    const int N = (int)(16 / h->esize), W = 32 * N, H = nw * rpt;
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
    if (nx + (per ? 2 * q.hc : 0) <= W) {
        q.mx = 1;
        q.px = nx;
    } else {
        q.mx = !per && nx <= 2 * (W - q.hc) ? 2 : ceil_div(nx, ow);
        q.px = round_up(ceil_div(nx, q.mx), N);
        // no last tile narrower than the columns the rules next to an edge span
        while (nx - (ceil_div(nx, q.px) - 1) * q.px < 4 && q.px > N) q.px -= N;
        q.mx = ceil_div(nx, q.px);
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
        split_rows(q.jb, H, K, true, false, 1, q.mb, q.pb);
        split_rows(ny - q.jt, H, K, false, true, 1, q.mt, q.pt);
    } else {
        split_rows(ny, H, K, true, true, h->edge_macro ? 2 : 1, q.mt, q.pt);
    }
    // the edge rule is applied by tiles whose rows 0 .. 2 (or ny-1 .. ny-3) lie
    // in one thread: tiles held from row 0 or up to row ny - 1, not the strip
    if (h->edge_macro && (crack ? p.jc < strip_half + 3 || ny - p.jc < strip_half + 3 : ny < 64)) return false;
    if (h->edge_macro && nx < 4) return false;

    if (crack && adjoint) {
        q.ms = q.mx;
        q.ps = q.px;
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
        q.unit = p.dh == 1.0 && p.dt == 1.0 && !(p.r_min_fixed > 0.0);
        q.lo_f = (float)p.r0;
        q.w_q = (int64_t)std::llrint(std::min(p.fit_width / p.dh, 1e6) * 4294967296.0);
        q.k_inv = p.K_C > 0.0 ? 1.0 / p.K_C : 0.0;
        q.k_unit = (float)(p.mu / 4.0 * std::sqrt(2.0 * kPi / p.dh) * 65536.0);
        q.k_rest = (float)(p.K_C * 0.999);
        // both ends are fitted at once by half a warp each: at most 16 columns
        if (!(p.fit_width / p.dh <= 12.0)) return false;
        if (nx + (per ? 2 * q.hc : 0) <= W) {
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
    if (!h->alt[0]) return;
    const int64_t sites = (int64_t)h->grid.nx * h->grid.ny;
    // FP64: two results per cycle and SM, so recomputed halos cost more than
    // launches save on large lattices, and on small ones the tiles have to be
    // many and small (see kPass64*)
    if (h->esize == 8 && sites > kPass64Sites) return;
    h->pass_nw = h->esize == 8 && sites <= kPass64Small ? 4 : 8;
    const int kmax = h->esize == 8 ? 4 : 8;
    for (int K = kmax; K >= 2; --K) {
        PassPlan q;
        h->pass_rpt = h->pass_nw == 4 ? 4 : 8;
        if (!pass_plan(h, K, h->pass_nw, h->pass_rpt, q)) continue;
        if (h->esize == 4 && q.tiles < 2 * h->sms) h->pass_rpt = 4;
        bool shorter = true;   // every shorter pass too: a call's last passes
        for (int k = K; k >= 2; --k) shorter = shorter && pass_plan(h, k, h->pass_nw, h->pass_rpt, q);
        if (!shorter) continue;
        const void *fn = h->q == 9 ? (h->esize == 8 ? pass_kernel_ptr<double, double, kNine>(h->pass_nw, h->pass_rpt, true)
                                                    : pass_kernel_ptr<float, float, kNine>(h->pass_nw, h->pass_rpt, true))
                         : h->lat.storage == LBM_F64           ? pass_kernel_ptr<double, double>(h->pass_nw, h->pass_rpt, true)
                         : h->lat.storage == LBM_F32_WD_BF16 ? pass_kernel_ptr<float, __nv_bfloat16>(h->pass_nw, h->pass_rpt, true)
                         : h->lat.storage == LBM_F32_WD_F16  ? pass_kernel_ptr<float, __half>(h->pass_nw, h->pass_rpt, true)
                         : h->lat.storage == LBM_F32_LEAPFROG ? pass_kernel_ptr<float, Lf>(h->pass_nw, h->pass_rpt, true)
                                                              : pass_kernel_ptr<float, float>(h->pass_nw, h->pass_rpt, true);
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, 32 * h->pass_nw, 0) != cudaSuccess || per_sm < 1)
            return;
        h->pass_slots = per_sm * h->sms;
        h->pass_k = K;
        return;
    }
}

}  // namespace host
}  // namespace lbm
