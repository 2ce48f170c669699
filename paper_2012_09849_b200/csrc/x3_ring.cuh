// Who fills, reads and gives back the shared-memory slots of a data gradient's block (x3_dgrad in x3_gemm.cu): the order of its copying
// and its two issuing threads, without what they copy and multiply, so that a test can walk through all of their interleavings.
//
// Barriers count one arrival of the copying thread in "full" and one of each issuing thread in "empty".  An issuing thread waits for
// every slot to be filled, also where the other one multiplies what is in it, and arrives on its "empty" only then.  So an arrival of
// one phase comes after the phase before is over, a phase cannot be completed by two arrivals of one thread (the other's products
// would still read the slot), and no thread is more than one phase away from a barrier: the parity it waits for is that of one phase.
#pragma once

namespace hts {

constexpr int kX3Part = 2;              // stages of an accumulation

struct X3Ring {
    int m_tiles, n_tiles, chunks, taps, tpe, entries, b_stages;
    int first, blocks;                  // a block's tiles: first, first + blocks, ...
#ifdef __CUDACC__
    __host__ __device__
#endif
    bool stay() const { return chunks * taps <= b_stages; }     // the weights of an N tile stay while its M tiles pass
};

#ifdef __CUDACC__
#define HTS_RING_FN __device__ __forceinline__
#else
#define HTS_RING_FN inline
#endif

// The copying thread.  Waits return false where it is to give up.
template <class Io>
HTS_RING_FN void x3_ring_copy(const X3Ring& r, Io io)
{
    const int tiles = r.m_tiles * r.n_tiles, groups = r.taps / r.tpe;      // A entries per chunk
    const bool stay = r.stay();
    int ea = 0, sb = 0, held = -1;
    unsigned pa = 1, pb = 1;                            // parity of the "empty" phase waited for
    for (int t = r.first; t < tiles; t += r.blocks) {   // M fastest, so that blocks running together share B through L2
        const int mt = t % r.m_tiles, nt = t / r.m_tiles;
        const bool load = !stay || nt != held;
        if (stay) { sb = 0; if (load && held >= 0) pb ^= 1u; }
        held = nt;
        for (int c = 0; c < r.chunks; ++c)
            for (int g = 0; g < groups; ++g) {
                if (!io.wait_a_empty(ea, pa)) return;
                io.load_a(ea, mt, c, g);
                if (++ea == r.entries) { ea = 0; pa ^= 1u; }
                for (int j = 0; load && j < r.tpe; ++j) {
                    if (!io.wait_b_empty(sb, pb)) return;
                    io.load_b(sb, nt, c, g + j);
                    if (++sb == r.b_stages && !stay) { sb = 0; pb ^= 1u; }
                }
            }
    }
}

// Issuing thread e: accumulations it = e, e + 2, ... of kX3Part stages each, in accumulator e.
template <class Io>
HTS_RING_FN void x3_ring_issue(const X3Ring& r, int e, Io io)
{
    const int tiles = r.m_tiles * r.n_tiles, groups = r.taps / r.tpe;
    const bool stay = r.stay();
    int ea = 0, sb = 0, it = 0, in = 0;
    unsigned pa = 0, pb = 0;
    int end = r.m_tiles;                                // of the N tile's tiles
    while (stay && end <= r.first) end += r.m_tiles;
    for (int t = r.first; t < tiles; t += r.blocks) {
        if (stay) {
            sb = 0;
            if (t >= end) pb ^= 1u;
            while (end <= t) end += r.m_tiles;
        }
        const bool give = !stay || t + r.blocks >= end;          // the last to read them
        int left = r.chunks * r.taps;
        for (int c = 0; c < r.chunks; ++c)
            for (int g = 0; g < groups; ++g) {
                if (!io.wait_a_full(ea, pa)) return;
                bool used = false;
                for (int j = 0; j < r.tpe; ++j) {
                    const bool mine = (it & 1) == e;
                    --left;
                    const bool last = in == kX3Part - 1 || left == 0;
                    if (!io.wait_b_full(sb, pb)) return;
                    if (mine) {
                        if (in == 0 && !io.wait_d_empty((unsigned)(it >> 1) & 1u ^ 1u)) return;
                        io.multiply(ea, sb, j, in == 0);
                        if (give) io.commit_b_empty(sb);
                        if (last) io.commit_d_full();
                        used = true;
                    } else if (give)
                        io.arrive_b_empty(sb);
                    if (last) { ++it; in = 0; } else ++in;
                    if (++sb == r.b_stages && !stay) { sb = 0; pb ^= 1u; }
                }
                if (used) io.commit_a_empty(ea);
                else io.arrive_a_empty(ea);
                if (++ea == r.entries) { ea = 0; pa ^= 1u; }
            }
    }
}

}  // namespace hts
