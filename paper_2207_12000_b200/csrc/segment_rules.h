// What plan construction decides about segments by arithmetic alone: plain C++ that host and device share, and that a test can
// compile for the CPU.
#pragma once

#include <algorithm>
#include <cstdint>

#ifdef __CUDACC__
#define GNNPRE_HOST_DEVICE __host__ __device__
#else
#define GNNPRE_HOST_DEVICE
#endif

namespace gnnpre {

constexpr int kOrderBuckets = 1024;  // of segments inside one row, by their middle column

// The bucket of a column of n.  A column that nobody has checked (GNNPRE_FLAG_SKIP_VALIDATION) may be any 31-bit number: what
// is out of range goes to the last bucket, so that it is never an index out of a table's range.
GNNPRE_HOST_DEVICE inline int column_bucket(uint32_t col, int64_t n) {
    const int64_t bucket = (int64_t)col * kOrderBuckets / n;
    return bucket < kOrderBuckets ? (int)bucket : kOrderBuckets - 1;
}

// Whether a segment of this row whose middle column this is reads rows numbered like its own, within a thirty-second of all.
GNNPRE_HOST_DEVICE inline bool near_diagonal(uint32_t row, uint32_t col, int64_t n) {
    const int apart = column_bucket(row, n) - column_bucket(col, n);
    return apart <= kOrderBuckets / 32 && apart >= -kOrderBuckets / 32;
}

// Segments of `edges` edges in m edges cut into `blocks` blocks: block l holds the edges [floor(l m / blocks),
// floor((l + 1) m / blocks)), that is, m mod blocks of them one more than the others.
inline int64_t count_segments(int64_t m, int64_t blocks, int64_t edges) {
    const int64_t q = m / blocks, longer = m % blocks;
    return (blocks - longer) * ((q + edges - 1) / edges) + longer * ((q + edges) / edges);
}

// Edges per segment of a plan that was not given any.  m: edges that one launch covers, in how many blocks; bulk_copy: summed by the bulk-copy kernel;
// beyond: the rows gathered from are on the device and more than the L2 holds (a streamed plan waits for the host's link and keeps
// the longer segments, which need fewer scratch rows); whole_hops: one launch covers a hop.
inline int32_t auto_segment_edges(int64_t slab_width, int64_t m, int64_t blocks, bool bulk_copy, bool beyond, bool whole_hops, int num_sms) {
    if (bulk_copy) {
        // persistent warps walk whole segments with a two-stage pipeline that drains at every segment end: long segments, but
        // at least ~4 per resident warp so the tail stays short, and short enough that half the edges lie in segments of a
        // single row (k_segment_order; 124 M edges, 100 columns, us per hop at 256 / 512 / 1024 / 2048 edges
        // 3843 / 3651 / 3637 / 3745; without such rows, 90 M edges, 6365 at 1024 and 6260 at 4096).  Blocks launched singly gain
        // as much by the shorter tail (124 M edges in one block 4410 at 4096 and 4425 at 1024, in two 4890 and 4445).
        const int64_t per_warp = m / ((int64_t)std::max(num_sms, 1) * 16 * 4);
        int32_t p = 256;
        while ((int64_t)p * 2 <= per_warp && p < (beyond ? 1024 : 4096)) p *= 2;
        return p;
    }
    const int64_t f4 = std::min<int64_t>(std::max<int64_t>(slab_width, 4), 128) / 4;
    const int64_t lanes = f4 <= 4 ? 4 : f4 <= 8 ? 8 : f4 <= 16 ? 16 : 32;
    const int64_t groups = (int64_t)std::max(num_sms, 1) * (28 * 32 / lanes);  // lane groups the device holds at a time
    const int64_t per_group = m / groups;
    // Register kernel, a hop of few waves over a matrix that the L2 holds: a last wave that is nearly empty costs as much as a
    // full one, so segments are as long as makes the waves whole - one wave while that leaves them even enough.  us per hop at
    // segments of a power of two (two or three per group) / so, R-MAT graphs, mean operator: 600,000 edges, 16 columns
    // 12.4 / 12.2, 32 15.4 / 13.6, 64 20.7 / 17.7, 128 31.1 / 24.7; 1.2 M 20.8 / 18.2, 24.2 / 21.3, 34.8 / 31.2; 2.4 M
    // 34.2 / 31.0, 39.4 / 36.1, 61.0 / 59.5; 4.8 M, 16 columns 58.2 / 52.5, 32 71.0 / 67.6 (two waves); 10 M 108.0 / 102.6 (two),
    // 132.3 / 125.8 (four); 24 M, 16 columns 209 / 198 (four).  Where the epilogue reads rows too, long segments are uneven: 64
    // columns, 2.4 M edges, ten hops with a teleport term and their sum 1155 at 80 edges, 1241 in one wave; 128 columns, 1.2 M
    // edges 843 at 64, 888 at 160, and without the epilogue 170 / 162; so those stay at 96 edges, and at one wave of 160.
    // Every edge block ends with a segment of its own, so the segments are counted: where a longer one makes the wave whole it is
    // taken, else one more wave.  GCN, 256 blocks, us for two hops, blocks not counted / counted: 150,000 nodes, 2.3 M edges, 32 columns
    // 90.4 / 81.9; 56,000 nodes, 870,000 edges, 32 columns 40.7 / 38.9, 64 columns 56.5 / 57.0.
    if (whole_hops && !beyond && slab_width <= 128) {
        const int64_t most = lanes == 4 ? 192 : lanes == 16 ? 96 : 160;
        for (int64_t waves = per_group / most + 1; waves <= (lanes == 32 ? 1 : 4); ++waves)
            for (int64_t L = std::max<int64_t>(16, (m / (groups * waves) + 8) / 8 * 8); L <= most; L += 8)
                if (count_segments(m, blocks, L) <= groups * waves) return (int32_t)L;
    }
    // Wider rows are several column tiles in one launch.  Where all tiles' segments of 16 edges run at once the hop is a chain of
    // latencies, and it takes those; else 32 at least.  us per hop at 16 / 32 edges, GCN and mean: 2,700 nodes, 10,600 edges, 500
    // columns 4.9 / 6.0, 6.4 / 6.7; 3,300 nodes, 9,100 edges, 500 columns 5.0 / 6.1, 6.3 / 7.5; beyond the line the same at 1433
    // columns 11.2 / 11.5, 10.0 / 9.1, 3703 columns 25.6 / 23.0, 22.6 / 22.2; 5,000 nodes, 19,400 edges, 500 columns 12.8 / 11.0,
    // 11.5 / 9.6; 7,600 nodes, 38,700 edges 18.6 / 17.1, 16.3 / 15.2.
    const int64_t tiles = (std::max<int64_t>(slab_width, 4) / 4 + 31) / 32;
    if (whole_hops && (m / 16) * lanes * tiles <= (int64_t)num_sms * 768) return 16;
    // Else segments long enough that few rows are cut, short enough that every lane group gets two (four or eight lanes per
    // group) or three (wider) of them, up to 256 edges.  Beyond 256 edges, up to 1024, only while eight segments per lane
    // group remain (23 M edges, 128 columns: 829 / 744 / 702 us at 64 / 128 / 256, as fast at 1024; 12.8 M edges: 531 at 256,
    // 583 at 1024): what longer segments save there is tables and scratch rows.  Up to 512 for a matrix beyond the L2, where
    // segments of a single row are the better ones (124 M edges, 100 columns, at 128 / 256 / 512 / 1024 edges
    // 4008 / 3898 / 3870 / 3950; GCN, 128 columns 4434 / 4331 / 4295), and blocks launched singly end sooner (GCN, 128 columns, two
    // blocks, 124 M edges 5460 at 1024 and 5330 at 512).
    const int64_t L = std::max(std::min<int64_t>(per_group / (lanes <= 8 ? 2 : 3), 256), per_group / 8);
    int32_t p = 32;
    while ((int64_t)p * 2 <= L && p < (beyond ? 512 : 1024)) p *= 2;
    return p;
}

}  // namespace gnnpre
