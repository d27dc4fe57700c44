// Sizes and indexes of the setup's kernels, on the host and on the device.
#pragma once

#ifdef __CUDACC__
#define AIRG_HD __host__ __device__
#else
#define AIRG_HD
#endif

namespace airg {

// The warp of a launch that a thread belongs to.  In 64 bits: one warp per
// row passes 2^32 threads at 2^27 rows, a size that the setup accepts.
AIRG_HD inline long long warp_index(unsigned block, unsigned block_threads, unsigned thread)
{
    return ((long long)block * block_threads + thread) >> 5;
}

constexpr long long GEMM_MAX_SLOTS = 1LL << 30;   // table offsets are 32-bit

// Slots of the hash table of a row with `products` products in a product of
// n_cols columns: the smallest power of two that leaves half the slots free
// whatever the columns are.  A row has at most n_cols of them, however many
// products it has.  More than GEMM_MAX_SLOTS is for the caller to refuse.
AIRG_HD inline long long gemm_table_slots(long long products, long long n_cols)
{
    const long long most = products < n_cols ? products : n_cols;
    long long size = 1;
    while (size < 2 * most) size <<= 1;
    return size;
}

// Entries that a piece of a product may hold, from the number asked for
inline long long gemm_piece_limit(long long asked)
{
    return asked < 1 ? 1 : (asked < GEMM_MAX_SLOTS ? asked : GEMM_MAX_SLOTS);
}

}  // namespace airg
