// Host-side schedule of the row-stream decode kernel (gemm_row.cu): pure integer arithmetic.
#pragma once
#include <cstddef>
#include <cstdint>

#include "plan.h"

namespace bd {

constexpr int kRowStageK = 1024;     // reduction extent of a stage: 128 k for each of the eight consumer warps
constexpr int kRowMaxM = 8;          // tokens per tenant
constexpr int kRowMaxStages = 4;

struct RowPlan {
    int tpt;       // tenants whose tokens share an 8-column activation tile (8 / m, or a power of two that covers all of them)
    int nt;        // activation tiles of a unit: 1, 2 or 4
    int TB;        // tenants of a unit (box of the sign words)
    int rows;      // weight rows of a unit (even, at most 16)
    int tiles, groups, units, grid, stages, k_stages;
    uint32_t s_off, x_off, stage_bytes, smem_bytes;
    bool ok;
};

inline RowPlan make_row_plan(int B, int m, int N, int K, int num_sms) {
    RowPlan p{};
    if (B <= 0 || m <= 0 || m > kRowMaxM || N <= 0 || K <= 0 || (K % kPairK) != 0) return p;
    // (every tenant column of a tile is computed, without tests)
    p.tpt = m == 1 ? 8 : m == 2 ? 4 : m <= 4 ? 2 : 1;
    for (int c = 1; c < p.tpt; c *= 2)
        if (c >= B) p.tpt = c;
    const int nt_max = 8 / p.tpt < 4 ? 8 / p.tpt : 4;             // at most eight tenants a unit, four activation tiles
    const int need = (B + p.tpt - 1) / p.tpt;
    p.nt = need < nt_max ? (need == 3 ? 4 : need) : nt_max;
    p.TB = p.tpt * p.nt < B ? p.tpt * p.nt : B;
    p.groups = (B + p.tpt * p.nt - 1) / (p.tpt * p.nt);
    // Rows: full rounds of units over the multiprocessors, each a little under sixteen rows, instead of a nearly empty last one.
    const long long t16 = ((long long)N + 15) / 16;
    const long long rounds = (t16 * p.groups + num_sms - 1) / num_sms;
    long long tiles = rounds * num_sms / p.groups;
    if (tiles < 1) tiles = 1;
    int r = (int)((N + tiles - 1) / tiles);
    r = (r + 1) / 2 * 2;
    p.rows = r < 2 ? 2 : r > 16 ? 16 : r;
    p.tiles = (int)(((long long)N + p.rows - 1) / p.rows);
    if ((long long)p.tiles * p.groups >= (1ll << 30)) return p;
    p.units = p.tiles * p.groups;
    p.grid = p.units < num_sms ? p.units : num_sms;
    p.k_stages = (K + kRowStageK - 1) / kRowStageK;
    p.s_off = (uint32_t)p.rows * 128u * 16u;
    p.x_off = p.s_off + (uint32_t)round_up(p.TB * p.rows * 128, 1024);
    p.stage_bytes = p.x_off + (uint32_t)p.nt * 16384u;
    const int red = (p.nt < 4 ? 2 : 1) * p.nt * 8 * 128 * 4 + 1024;   // the warps' partial results (of two units in turn); barriers
    int st = (kSmemBudget - 1024 - red) / (int)p.stage_bytes;
    if (st > kRowMaxStages) st = kRowMaxStages;
    if (st < 2) return p;
    const long long total = (long long)((p.units + p.grid - 1) / p.grid) * p.k_stages;
    p.stages = total < st ? (int)total : st;
    p.smem_bytes = 1024u + (uint32_t)p.stages * p.stage_bytes + (uint32_t)red;
    p.ok = true;
    return p;
}

// Where the row-stream kernel is taken by default: one or two tenants, or up to 48 M signs including the tenant columns computed
// for nothing.  Its MMAs cost ~1.1 us per tenant at 4096 x 4096, the others' latencies are the same whatever the size.
// Measured (us, row-stream / the others, in a graph): 1 x 1 x 4096 x 4096 8.4 / 10.5, 1 x 8 x 4096 x 11008 15.7 / 21.6, 2 x 1 x 4096 x 4096
// 9.6 / 11.0, 2 x 8 10.6 / 13.0, 8 x 1 x 2048 x 2048 6.3 / 13.4, 8 x 8 x 1024 x 1024 3.5 / 12.6, 4 x 2 x 5632 x 2048 9.9 / 18.4,
// 16 x 1 x 2048 x 768 5.2 / 14.1; beyond: 4 x 1 x 4096 x 4096 12.1 / 11.7, 8 x 1 16.5 / 14.2, 28 x 1 x 6400 x 816 23.2 / 19.9.
// (In the other direction some are left to the others that it would win: 32 x 1 x 2048 x 1024 9.3 / 16.7.)
// Calls with options or binary16 operands have the slower 8-bit kernel as the alternative: up to 68 M (binary16, bias, gate: 4 x 1 x
// 4096 x 4096 12.8 / 14.6, 4 x 8 16.6 / 21.5; beyond, 28 x 1 x 6400 x 816 23.5 / 19.5).  Where the 4-bit kernel's clusters of two or four
// blocks apply (`cluster`), it is ahead from 32 M on (3 x 1 x 2048 x 4096 8.3 / 7.8, 4 x 1 x 2816 x 4096 10.0 / 9.3; without clusters
// 8 x 1 x 2048 x 2816 9.8 / 14.9).
// Within that, three kinds of call are left to the others (`cols`: token columns x rows computed, in whole rounds, x K in whole stages):
//   * units of four activation tiles in more than seven rounds: a unit's two barriers and its partial sums cost ~1 us (19 x 5 x 512 x
//     3642 15.9 / 11.2, 9 x 6 x 512 x 7192 18.9 / 16.0; in seven rounds 11 x 8 x 1024 x 4804 16.8 / 17.8);
//   * a second round that is mostly empty, with much to compute (binary16 and gate, 12 x 1 x 3200 x 1220 14.1 / 13.0);
//   * two tenants of five tokens and more (options: eight), large, with the last round partly empty: ~1 us of MMA time per stage,
//     whatever the rows (2 x 8 x 11008 x 5632 31.2 / 28.9, 2 x 6 x 8192 x 8192 31.3 / 29.3; full rounds: 2 x 8 x 14336 x 11008 62.0 / 67.5).
inline bool row_kernel_pays(const RowPlan& p, int B, int m, int N, int K, bool plain, int cluster) {
    if (!p.ok) return false;
    const long long rounds = (p.units + p.grid - 1) / p.grid, rows = rounds * 16 * p.grid;
    const long long cols = (long long)p.tpt * p.nt * rows * p.k_stages * kRowStageK;
    if (B <= 2) return !(B == 2 && m >= (plain ? 5 : 8) && rounds >= 3 && 10ll * N < 9 * rows && cols > 110000000ll);
    if ((p.nt == 4 && rounds > 7) || (rounds >= 2 && cols > 140000000ll)) return false;
    const long long limit = !plain ? 68000000ll : (cluster == 2 || cluster == 4) ? 32000000ll : 48000000ll;
    return (long long)p.tpt * p.nt * p.groups * N * K <= limit;
}

}  // namespace bd
