// The chain of chunk maps of the two scans.
#pragma once

namespace hts {

// Chunk ww of a super-chunk maps what comes in behind it, c, to S + P c.  With few chunks every thread walks them all.  With
// many (64 chunks in 16 warps are 2048 loads from shared memory, a clock each) the block's first threads, one per column, walk for
// all of them, eight maps loaded at a time, and leave what goes into a chunk in the place of its S and what comes out of the first
// one in sP[0].  512 x 512, us: advantages 4.33 -> 4.02, V-trace 5.06 -> 4.56; 256 x 5000: advantages 10.6 -> 9.3.
constexpr int kManyChunks = 32;
// The maps of chunk ww are at sS, sP [ww * cols]; c comes in behind the last one.
__device__ __forceinline__ void walk_chunks(float* sS, float* sP, int cols, int chunks, float c)
{
    int ww = chunks - 1;
    for (; ww >= 7; ww -= 8) {
        float S[8], P[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) { S[i] = sS[(ww - i) * cols]; P[i] = sP[(ww - i) * cols]; }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            sS[(ww - i) * cols] = c;
            c = S[i] + P[i] * c;
        }
    }
    for (; ww >= 0; --ww) {
        const float S = sS[ww * cols], P = sP[ww * cols];
        sS[ww * cols] = c;
        c = S + P * c;
    }
    sP[0] = c;
}

}  // namespace hts
