// Stacked rows: the M rows of every slice or node of a list, one after the other.  A list has up to 2^31 entries of up to
// 1024 rows each, so their number needs 64 bits; positions are divided once and then moved on in 32 bits.
// Plain C++ on the host, so that the arithmetic is tested there at its limits.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define TT_HD __host__ __device__ __forceinline__
#else
#define TT_HD inline
#endif

struct StackedRow {
    uint32_t node, m;   // entry of the list, row inside it
};

TT_HD uint64_t tt_stacked_rows(uint32_t nodes, int M) { return (uint64_t)nodes * (uint32_t)M; }

TT_HD StackedRow tt_stacked_row(uint64_t row, int M)
{
    StackedRow r;
    r.node = (uint32_t)(row / (uint32_t)M);
    r.m = (uint32_t)(row - (uint64_t)r.node * (uint32_t)M);
    return r;
}

// n rows further on
TT_HD StackedRow tt_stacked_next(StackedRow r, uint32_t n, int M)
{
    const uint32_t m = r.m + n, q = m / (uint32_t)M;
    r.node += q;
    r.m = m - q * (uint32_t)M;
    return r;
}

// CTAs per slice for work of `tiles` tiles a slice at most: they fill the SMs four times over with four CTAs each.  The
// slices of all tables of a handle may be 2^31 and more.
TT_HD int tt_ctas_per_slice(int sm_count, int64_t slices, int64_t tiles)
{
    const int64_t want = ((int64_t)sm_count * 16 + slices - 1) / slices, most = tiles < 65535 ? tiles : 65535;
    return (int)(want < most ? want : most);
}
