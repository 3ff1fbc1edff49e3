// Counts of a clustering round in one 64-bit word, so that a single prefix sum
// and a single load carry both: the clusters that stay in the low 31 bits, the
// merges in the next 31.  A scene has at most 2^31 - 1 triangles and no sum
// counts one twice, so neither field overflows.  The top two bits are free for
// the round's tag, by which a block knows its answer from the one before: never
// 0 (a sector no round has written), and different in consecutive rounds.
#pragma once

#ifdef __CUDACC__
#define LIDAR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define LIDAR_HOST_DEVICE inline
#endif

namespace lidar {

LIDAR_HOST_DEVICE unsigned long long ploc_counts(unsigned merges, unsigned stays)
{
    return (unsigned long long)merges << 31 | stays;
}

LIDAR_HOST_DEVICE unsigned ploc_merges(unsigned long long counts)
{
    return (unsigned)(counts >> 31) & 0x7FFFFFFFu;
}

LIDAR_HOST_DEVICE unsigned ploc_stays(unsigned long long counts)
{
    return (unsigned)counts & 0x7FFFFFFFu;
}

LIDAR_HOST_DEVICE unsigned long long ploc_tagged(unsigned long long counts, unsigned round)
{
    return (unsigned long long)(round % 3u + 1u) << 62 | counts;
}

LIDAR_HOST_DEVICE bool ploc_is_of(unsigned long long word, unsigned round)
{
    return word >> 62 == round % 3u + 1u;
}

LIDAR_HOST_DEVICE unsigned long long ploc_untagged(unsigned long long word)
{
    return word & ((1ull << 62) - 1ull);
}

}  // namespace lidar
