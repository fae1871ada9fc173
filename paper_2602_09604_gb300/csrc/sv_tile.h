// Shared-memory tiles of whole 256-byte blocks (staged passes, Pauli strings): address arithmetic.
//
// A tile is 2^fb blocks; block c's 32 real parts lie at float 64 c, its imaginary parts at 64 c + 32,
// both with the in-block positions XOR-ed by a swizzle of c.  Every address is then linear over GF(2)
// in the tile-local index bits.
#pragma once

#include <vector>

#include "sv_internal.h"

namespace svg {

// swizzle of a tile block's in-block positions, linear in the tile block index c: bit i of c XORs
// swz_vec(i) into the position.  A gate whose targets lie below qubit 5 needs other address bits to
// spread a warp over the 32 banks; block bit i then stands in for position bit i (and bits 5-8 for
// mixtures), see lane_bits.  Only block bits 0 and 1 reach position bits 0 and 1, so the order of
// the four floats of a 16-byte chunk depends on c & 3 alone (TileMover: the same for a whole warp).
__host__ __device__ constexpr unsigned swz_vec(int i)
{
    return i < 5 ? 1u << i : (i == 5 ? 20u : i == 6 ? 24u : i == 7 ? 12u : 28u);
}
__host__ __device__ constexpr unsigned swz_of(unsigned c)
{
    unsigned s = 0;
    for (int i = 0; i < 9; ++i) s ^= ((c >> i) & 1u) ? swz_vec(i) : 0u;
    return s;
}

// the four floats of a chunk with position bits 0 and 1 XOR-ed by S
template <int S>
__device__ __forceinline__ float4 perm4(float4 v)
{
    if constexpr (S == 1) return make_float4(v.y, v.x, v.w, v.z);
    else if constexpr (S == 2) return make_float4(v.z, v.w, v.x, v.y);
    else if constexpr (S == 3) return make_float4(v.w, v.z, v.y, v.x);
    else return v;
}

// A tile's geometry in global memory.  Blocks move as 16 chunks of 16 bytes, a half warp each.
constexpr int kTileMaxFb = 7;             // tiles of up to 2^12 amplitudes (32 KB)
struct TileGeom {
    int fb;                               // a tile is 2^fb blocks
    int fpos[kTileMaxFb];                 // their ascending block-index bits
    long long ioff[1 << (kTileMaxFb - 3)];   // float offset of tile block i << 3 (the bits placed at fpos)
};

inline void fill_geom(uint64_t lam, int n, TileGeom *t)
{
    int fb = 0;
    for (int q = 5; q < n; ++q)
        if ((lam >> q) & 1) t->fpos[fb++] = q - 5;
    t->fb = fb;
    for (int i = 0; i < (1 << (kTileMaxFb - 3)); ++i) {
        long long o = 0;
        for (int b = 3; b < fb; ++b)
            if ((i >> (b - 3)) & 1) o |= 64ll << t->fpos[b];
        t->ioff[i] = o;
    }
}

// block index of tile t's first block
__device__ __forceinline__ unsigned long long tile_base(const TileGeom &t, unsigned long long i)
{
    for (int b = 0; b < t.fb; ++b) {
        const unsigned long long low = i & ((1ull << t.fpos[b]) - 1ull);
        i = ((i >> t.fpos[b]) << (t.fpos[b] + 1)) | low;
    }
    return i;
}

// Copies a tile between global and shared memory with T threads.  A thread's tile blocks are
// thread part | i << SH; the warp gives block bits 0 and 1, so the chunk order is uniform in a warp,
// and every address is the thread's own plus (XOR) a constant of i.
template <int T>
struct TileMover {
    static constexpr int SH = T == 128 ? 3 : 5;
    static constexpr int N = 1 << (kTileMaxFb - SH);   // chunks a thread moves
    long long goff;     // float offset of the thread's chunk of its block 0 from the tile's first block
    unsigned soff;      // and in shared memory
    int cthr;
    __device__ __forceinline__ explicit TileMover(const TileGeom &t)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        cthr = (warp & 3) | ((lane >> 4) << 2) | ((warp >> 2) << 3);
        goff = (lane & 15) * 4;
        for (int b = 0; b < t.fb && b < SH; ++b)
            if ((cthr >> b) & 1) goff += 64ll << t.fpos[b];
        soff = (unsigned)(cthr * 64 + (lane & 8) * 4) + ((((unsigned)lane & 7u) ^ (swz_of((unsigned)cthr) >> 2)) << 2);
    }
    static __device__ __forceinline__ constexpr unsigned ivec(int i)
    {
        return (unsigned)(i << SH) * 64u ^ ((swz_of((unsigned)(i << SH)) >> 2) << 2);
    }
    __device__ __forceinline__ bool has(const TileGeom &t, int i) const { return cthr + (i << SH) < (1 << t.fb); }
    template <int S>
    __device__ __forceinline__ void put(const TileGeom &t, float *tile, const float4 (&v)[8 < N ? 8 : N], int i0) const
    {
#pragma unroll
        for (int i = 0; i < (8 < N ? 8 : N); ++i)
            if (has(t, i0 + i)) *reinterpret_cast<float4 *>(tile + (soff ^ ivec(i0 + i))) = perm4<S>(v[i]);
    }
    template <int S>
    __device__ __forceinline__ void get(const TileGeom &t, const float *tile, float *g) const
    {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (has(t, i)) *reinterpret_cast<float4 *>(g + goff + t.ioff[i << (SH - 3)]) =
                               perm4<S>(*reinterpret_cast<const float4 *>(tile + (soff ^ ivec(i))));
    }
    // g: the tile's first block
    __device__ __forceinline__ void load(const TileGeom &t, const float *g, float *tile) const
    {
        constexpr int B = 8 < N ? 8 : N;
        const int w = (threadIdx.x >> 5) & 3;
#pragma unroll
        for (int i0 = 0; i0 < N; i0 += B) {
            float4 v[B];
#pragma unroll
            for (int i = 0; i < B; ++i)
                if (has(t, i0 + i)) v[i] = __ldcs(reinterpret_cast<const float4 *>(g + goff + t.ioff[(i0 + i) << (SH - 3)]));
            if (w == 0) put<0>(t, tile, v, i0);
            else if (w == 1) put<1>(t, tile, v, i0);
            else if (w == 2) put<2>(t, tile, v, i0);
            else put<3>(t, tile, v, i0);
        }
    }
    __device__ __forceinline__ void store(const TileGeom &t, const float *tile, float *g) const
    {
        const int w = (threadIdx.x >> 5) & 3;
        if (w == 0) get<0>(t, tile, g);
        else if (w == 1) get<1>(t, tile, g);
        else if (w == 2) get<2>(t, tile, g);
        else get<3>(t, tile, g);
    }
};

// Address vector (floats into the swizzled tile) of tile-local bit t: position bits 0-4 as they
// are, block bit i moves 64 << i floats and XORs swz_vec(i) into the position.
inline unsigned addr_vec(int t) { return t < 5 ? 1u << t : (64u << (t - 5)) ^ swz_vec(t - 5); }

// Orders the free tile bits so that the first five (a warp's lanes) reach 32 different banks where
// the gate allows it: greedy choice of bits whose bank vectors (address bits 0-4) are linearly
// independent over GF(2), then the rest.
inline void lane_bits(const std::vector<int> &free_bits, std::vector<int> *order)
{
    unsigned basis[5] = {0, 0, 0, 0, 0};
    std::vector<int> rest;
    order->clear();
    for (int t : free_bits) {
        unsigned v = addr_vec(t) & 31u;
        for (int b = 4; b >= 0 && v; --b)
            if ((v >> b) & 1) {
                if (!basis[b]) {
                    basis[b] = v;
                    break;
                }
                v ^= basis[b];
            }
        if (v && order->size() < 5) order->push_back(t);
        else rest.push_back(t);
    }
    order->insert(order->end(), rest.begin(), rest.end());
}

}  // namespace svg
