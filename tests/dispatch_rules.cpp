// The rules by which launches choose their kernels, for tests without a GPU.
#include "wash_internal.h"

extern "C" {

int rule_copies_in_bulk(int has_status, unsigned pn_pad, unsigned group_lo, unsigned group_hi, unsigned groups, int n_models, int bytes_a, int bytes_b, float share)
{
    uint32_t word = 0;
    wash::ShuffleArgs args = {};
    args.status = has_status ? &word : nullptr;
    args.pn_pad = pn_pad;
    args.group_lo = group_lo;
    args.group_hi = group_hi;
    args.pop.N = n_models;
    args.expected_share = share;
    return wash::copies_in_bulk(args, groups, bytes_a, bytes_b) ? 1 : 0;
}

int rule_fetch_half_lines(int layout, int n_models, float share, int by_warps, int bytes_a, int bytes_b)
{
    wash::ShuffleArgs args = {};
    args.pop.layout = layout;
    args.pop.N = n_models;
    args.expected_share = share;
    return wash::fetch_half_lines(args, by_warps != 0, bytes_a, bytes_b) ? 1 : 0;
}

int rule_half_wave_serves(int layout, int n_models, int stacks, double expected, double by_load, unsigned resident, unsigned n_wtiles)
{
    return wash::half_wave_serves(layout, n_models, stacks, expected, by_load, resident, n_wtiles) ? 1 : 0;
}

int rule_stored_together(int layout, int n_models) { return wash::stored_together(layout, n_models); }

unsigned rule_dense_threshold(int n_models, int two_stacks, int all_f32) { return wash::dense_threshold(n_models, two_stacks != 0, all_f32 != 0); }

unsigned rule_report_grid(unsigned long long n_tiles, unsigned long long resident) { return wash::report_grid(n_tiles, resident); }
int rule_stat_slots() { return wash::kStatSlots; }

}
