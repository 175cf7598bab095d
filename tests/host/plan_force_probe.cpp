// Host run of the evaluation planner with forced values: for each line
// "ntiles pcap tpi jsplit m" read from stdin, prints the plan's threads per particle,
// particles per tile, tiles per j-chunk, j-chunks and work items.
#include <stdio.h>

#include "hg_internal.cuh"

int main()
{
    long long ntiles, pcap, m;
    int tpi, jsplit;
    while (scanf("%lld %lld %d %d %lld", &ntiles, &pcap, &tpi, &jsplit, &m) == 5) {
        hg::PlanParams q{};
        q.tj = hg::kTJMixed;
        q.i_per_thread = q.ipt1 = hg::kIMixed;
        q.ntiles = ntiles;
        q.pcap = pcap;
        q.grid = q.grid1 = 3 * 152;
        q.tpi_force = tpi;
        q.b_force = jsplit;
        q.c_tile = 2;
        q.c_item = 24;
        q.variants = 1;
        q.weight1 = q.weight1_one = 100;
        for (int k = 0; k < hg::kTuneBuckets; ++k) q.tuned[k] = -1;
        const hg::Plan p = hg::make_plan(m, q);
        printf("%d %d %lld %d %lld\n", p.tpi, p.ti, (long long)p.tiles_per_split, p.b, (long long)p.n_items);
    }
    return 0;
}
