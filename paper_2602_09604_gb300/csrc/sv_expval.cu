// Expectation values of Pauli strings, <psi|P|psi>, as a read-only reduction over the state.
//
// Section IV runs ExpectationValue with the same group loop as ApplyGate but reduces the result
// instead of storing it back.  For a Pauli string the "matrix-vector product" of a group is a
// signed, phased permutation, so the reduction needs no matrix at all.  Write the string as two
// bit masks over the qubits: x (X or Y on that qubit) and z (Z or Y).  With Y = i X Z,
//     P |j> = i^popc(x & z) (-1)^popc(j & z) |j ^ x>,
//     <psi|P|psi> = i^popc(x & z) * S,   S = sum_j (-1)^popc(j & z) conj(c_(j^x)) c_j.
// P is Hermitian, so the value is real: Re S, -Im S, -Re S or Im S for popc(x & z) = 0, 1, 2, 3
// (mod 4); each string accumulates only the component it needs.
//
// Strings with the same x read the same pairs of amplitudes, so up to kEvMaxStrings of them are
// evaluated in one pass: each amplitude is read once, its term conj(c_(j^x)) c_j is formed once in
// fp32, and every string adds it with its own sign into a float-float accumulator (two-sum); the
// per-thread results are combined in fp64, per CTA and then by the last CTA in a fixed order
// (strided per-thread sums, then a fixed-shape tree), so results are deterministic.
//
// Work unit = one block (x has no bit >= 5) or one pair of blocks b, b ^ (x >> 5) with bit
// `pair_bit` of b clear (otherwise); a warp reads each block's 32 real and 32 imaginary parts with
// coalesced loads, and the partner amplitude j ^ x inside the paired block comes from lane
// (lane ^ (x & 31)) through a shuffle.  A warp takes 32 consecutive units and handles them in
// batches of 8 (eight blocks or pairs of loads in flight per warp).  Signs are bit lookups: for
// unit u of a range starting at u0 (a multiple of 32), parity(b & zb) = parity(u0 & zu) ^ bit
// (u - u0) of a 32-bit parity table of zu's low five bits, where zu is zb with the pair bit
// deleted (b is u with a zero inserted there); these bits are the same in every lane.  The lane
// part parity(lane & zl) is fixed per thread and applied once at the end.  Each string sums a
// batch's signed terms in fp32 (with four or more strings, through one 8-point Walsh-Hadamard
// transform of the batch that serves every string), then adds the batch sum to its float-float
// accumulator.
#include <algorithm>
#include <cstring>
#include <exception>
#include <mutex>
#include <vector>

#include "sv_evplan.h"
#include "sv_internal.h"
#include "sv_tile.h"

namespace svg {
namespace {

constexpr int kEvThreads = 256;
constexpr int kEvMaxStrings = 8;

struct EvArgs {
    long long n_units;        // blocks, or block pairs
    unsigned long long xb;    // x >> 5
    int xl;                   // x & 31
    int pair_bit;             // bit of the block index inserted as 0 to enumerate pairs; -1: no pairing
    unsigned long long zu[kEvMaxStrings];   // z >> 5 with the pair bit deleted (unit-index parity mask)
    unsigned ztab[kEvMaxStrings];           // bit i = parity(i & zu & 31), i < 32
    unsigned zc[kEvMaxStrings];             // zu & 7: the Walsh-Hadamard entry of a batch of 8 units
    unsigned zl[kEvMaxStrings];             // z & 31
    unsigned pairpar[kEvMaxStrings];        // parity((x >> 5) & (z >> 5)): sign change to the paired block
    int comp[kEvMaxStrings];  // 0: accumulate the real part of the term, 1: the imaginary part
    int m;                    // strings in this pass (<= the kernel's M; the rest are padding)
};

struct FF2 {
    float hi, lo;
};

__device__ __forceinline__ void ff_add(FF2 &a, float x)
{
    const float s = a.hi + x;
    const float bp = s - a.hi;
    const float e = (a.hi - (s - bp)) + (x - bp);
    a.hi = s;
    a.lo += e;
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ unsigned long long ins_zero(unsigned long long v, int p)
{
    const unsigned long long low = v & ((1ull << p) - 1ull);
    return ((v >> p) << (p + 1)) | low;
}

constexpr int kEvBatch = 8;     // units per batch

// in place: w[c] <- sum_i (-1)^popc(i & c) w[i]
__device__ __forceinline__ void wht8(float (&w)[8])
{
#pragma unroll
    for (int h = 1; h < 8; h <<= 1)
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (!(i & h)) {
                const float x = w[i], y = w[i + h];
                w[i] = x + y;
                w[i + h] = x - y;
            }
}

// w[c] for a warp-uniform c < 8 without indexing a register array (three levels of selects)
__device__ __forceinline__ float sel8(const float (&w)[8], unsigned c)
{
    const float a0 = (c & 1u) ? w[1] : w[0], a1 = (c & 1u) ? w[3] : w[2];
    const float a2 = (c & 1u) ? w[5] : w[4], a3 = (c & 1u) ? w[7] : w[6];
    const float b0 = (c & 2u) ? a1 : a0, b1 = (c & 2u) ? a3 : a2;
    return (c & 4u) ? b1 : b0;
}
constexpr int kEvRange = 32;    // units per warp range (one parity table)

template <int M, bool PAIRED>
__global__ void __launch_bounds__(kEvThreads, M >= 4 ? 3 : 4) expval_kernel(const float *__restrict__ sv, const __grid_constant__ EvArgs a,
                                                           double *__restrict__ partials, unsigned *__restrict__ counter,
                                                           double *__restrict__ result)
{
    FF2 acc[M];
#pragma unroll
    for (int p = 0; p < M; ++p) acc[p] = FF2{0.f, 0.f};
    const unsigned lane = threadIdx.x & 31u;
    const unsigned plane = lane ^ (unsigned)a.xl;
    const long long n_ranges = (a.n_units + kEvRange - 1) / kEvRange;
    const long long wstride = (long long)gridDim.x * (kEvThreads / 32);
    for (long long r = (long long)blockIdx.x * (kEvThreads / 32) + (threadIdx.x >> 5); r < n_ranges; r += wstride) {
        const long long u0 = r * kEvRange;
        unsigned sgn0[M];   // block-parity sign bit of the range base, per string (warp-uniform)
#pragma unroll
        for (int p = 0; p < M; ++p) sgn0[p] = (unsigned)(__popcll((unsigned long long)u0 & a.zu[p]) & 1) << 31;
#pragma unroll 1
        for (int bt = 0; bt < kEvRange / kEvBatch; ++bt) {
            float ur[kEvBatch], ui[kEvBatch], vr[kEvBatch], vi[kEvBatch];
#pragma unroll
            for (int i = 0; i < kEvBatch; ++i) {
                const long long u = u0 + bt * kEvBatch + i;
                ur[i] = ui[i] = vr[i] = vi[i] = 0.f;
                if (u < a.n_units) {
                    const unsigned long long b = PAIRED ? ins_zero((unsigned long long)u, a.pair_bit) : (unsigned long long)u;
                    ur[i] = __ldcs(sv + b * 64 + lane);
                    ui[i] = __ldcs(sv + b * 64 + 32 + lane);
                    if constexpr (PAIRED) {
                        const unsigned long long b2 = b ^ a.xb;
                        vr[i] = __ldcs(sv + b2 * 64 + lane);
                        vi[i] = __ldcs(sv + b2 * 64 + 32 + lane);
                    }
                }
            }
            float tr[kEvBatch], ti[kEvBatch], sr[kEvBatch], si[kEvBatch];
#pragma unroll
            for (int i = 0; i < kEvBatch; ++i) {
                if constexpr (PAIRED) {
                    const float vpr = __shfl_sync(0xffffffffu, vr[i], plane), vpi = __shfl_sync(0xffffffffu, vi[i], plane);
                    const float upr = __shfl_sync(0xffffffffu, ur[i], plane), upi = __shfl_sync(0xffffffffu, ui[i], plane);
                    // j in block b (partner in b2) and j' in block b2 (partner in b)
                    tr[i] = fmaf(vpr, ur[i], vpi * ui[i]);
                    ti[i] = fmaf(vpr, ui[i], -(vpi * ur[i]));
                    sr[i] = fmaf(upr, vr[i], upi * vi[i]);
                    si[i] = fmaf(upr, vi[i], -(upi * vr[i]));
                } else {
                    const float pr = __shfl_sync(0xffffffffu, ur[i], plane), pi = __shfl_sync(0xffffffffu, ui[i], plane);
                    tr[i] = fmaf(pr, ur[i], pi * ui[i]);
                    ti[i] = fmaf(pr, ui[i], -(pi * ur[i]));
                }
            }
            if constexpr (M >= 4) {
                // many strings: an 8-point Walsh-Hadamard transform of the batch's terms gives,
                // for every mask c of the batch's unit bits, the sum of the terms signed by
                // parity(i & c); string p then takes entry zu & 7, signed by the batch's base parity
                wht8(tr);
                wht8(ti);
                if constexpr (PAIRED) {
                    wht8(sr);
                    wht8(si);
                }
#pragma unroll
                for (int p = 0; p < M; ++p) {
                    const unsigned c = a.zc[p];
                    const unsigned sg = sgn0[p] ^ (((a.ztab[p] >> (bt * kEvBatch)) & 1u) << 31);
                    float v = a.comp[p] ? sel8(ti, c) : sel8(tr, c);
                    if constexpr (PAIRED) {
                        const float w = a.comp[p] ? sel8(si, c) : sel8(sr, c);
                        v += __uint_as_float(__float_as_uint(w) ^ (a.pairpar[p] << 31));
                    }
                    ff_add(acc[p], __uint_as_float(__float_as_uint(v) ^ sg));
                }
            } else {
#pragma unroll
                for (int p = 0; p < M; ++p) {
                    // block-parity sign bits of the batch's units: warp-uniform; the lane's own
                    // parity (lane & zl) is applied once at the end
                    const unsigned tab = a.ztab[p] >> (bt * kEvBatch);
                    float sum = 0.f;
                    if (a.comp[p] == 0) {
#pragma unroll
                        for (int i = 0; i < kEvBatch; ++i) {
                            const unsigned sg = sgn0[p] ^ (((tab >> i) & 1u) << 31);
                            sum += __uint_as_float(__float_as_uint(tr[i]) ^ sg);
                            if constexpr (PAIRED) sum += __uint_as_float(__float_as_uint(sr[i]) ^ sg ^ (a.pairpar[p] << 31));
                        }
                    } else {
#pragma unroll
                        for (int i = 0; i < kEvBatch; ++i) {
                            const unsigned sg = sgn0[p] ^ (((tab >> i) & 1u) << 31);
                            sum += __uint_as_float(__float_as_uint(ti[i]) ^ sg);
                            if constexpr (PAIRED) sum += __uint_as_float(__float_as_uint(si[i]) ^ sg ^ (a.pairpar[p] << 31));
                        }
                    }
                    ff_add(acc[p], sum);
                }
            }
        }
    }
    // the lane's parity(lane & zl) sign, common to every term this thread added
#pragma unroll
    for (int p = 0; p < M; ++p)
        if (__popc(lane & a.zl[p]) & 1) {
            acc[p].hi = -acc[p].hi;
            acc[p].lo = -acc[p].lo;
        }
    __shared__ double ws[kEvThreads / 32][M];
    __shared__ bool last;
#pragma unroll
    for (int p = 0; p < M; ++p) {
        const double v = warp_sum((double)acc[p].hi + (double)acc[p].lo);
        if (lane == 0) ws[threadIdx.x >> 5][p] = v;
    }
    __syncthreads();
    if (threadIdx.x < M) {
        double s = 0.0;
        for (int w = 0; w < kEvThreads / 32; ++w) s += ws[w][threadIdx.x];
        partials[(size_t)blockIdx.x * M + threadIdx.x] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned done = atomicAdd(counter, 1u);
        last = (done == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    // last CTA: every thread sums a fixed strided subset of the partials, then a fixed-shape tree
    __threadfence();
    __shared__ double red[kEvThreads][M];
    {
        const volatile double *pp = partials;
        double s[M];
#pragma unroll
        for (int p = 0; p < M; ++p) s[p] = 0.0;
        for (unsigned i = threadIdx.x; i < gridDim.x; i += kEvThreads)
#pragma unroll
            for (int p = 0; p < M; ++p) s[p] += pp[(size_t)i * M + p];
#pragma unroll
        for (int p = 0; p < M; ++p) red[threadIdx.x][p] = s[p];
    }
    __syncthreads();
    for (int w = kEvThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
#pragma unroll
            for (int p = 0; p < M; ++p) red[threadIdx.x][p] += red[threadIdx.x + w][p];
        __syncthreads();
    }
    if ((int)threadIdx.x < a.m) result[threadIdx.x] = red[0][threadIdx.x];
    if (threadIdx.x == 0) *counter = 0u;   // ready for the next launch
}

// The grid is one wave of resident CTAs (occupancy x SMs), capped by the work and by max_grid:
// every CTA then loops over an equal share of the ranges with no second, partly filled wave.
template <int M>
int launch_ev(const float *sv, const EvArgs &a, double *partials, unsigned *counter, double *result, long long work_ctas,
              int num_sms, int max_grid, cudaStream_t s)
{
    auto kern = a.pair_bit >= 0 ? expval_kernel<M, true> : expval_kernel<M, false>;
    int per_sm = 1;
    SV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kEvThreads, 0));
    long long g = (long long)num_sms * (per_sm > 0 ? per_sm : 1);
    if (g > max_grid) g = max_grid;
    if (g > work_ctas) g = work_ctas;
    if (g < 1) g = 1;
    kern<<<(unsigned)g, kEvThreads, 0, s>>>(sv, a, partials, counter, result);
    SV_CUDA_TRY(cudaGetLastError());
    return SV_OK;
}

// ------------------------------------------------------------------------------------ tiles
// Many strings in one read pass.  The chain Hamiltonians of variational runs hold many strings
// with different x masks, each a read of the whole state for the kernel above.  Here a CTA keeps a
// tile -- 2^12 amplitudes agreeing on the qubits outside a local set that holds qubits 0-4 -- in
// shared memory and evaluates every string whose x mask lies in the local set: per x mask (and
// component) each thread forms 16 terms and takes two 8-point Walsh-Hadamard transforms (every sign
// pattern a z mask can put on three of the four index bits that vary in the thread), and each string
// adds the 128 threads' two entries for its mask, signed by the fourth bit and its thread-index and
// tile parities, in float-float.  z masks may
// name any qubit.  Terms of a pair (j, j ^ x) are equal once signed, so only one of each pair is formed.
constexpr int kEvtThreads = 128;
constexpr int kEvtQubits = 12;
constexpr int kEvtTileFloats = 2 << kEvtQubits;
// Tile passes start here although they are faster from 12 qubits on and no less exact: values are
// returned in 64 bits, the two kernels round in other places, and below this size what they
// return differs by more than 1e-9 even on states without structure (relative 2-norm over a chain's
// strings, random amplitudes on a product state; one-mask / tile time of the XYZ chain, and the largest
// difference of the XYZ and X-ZZ chains):
//     20 qubits   345 /  103 us   6e-9        25 qubits  1781 /  639 us   2e-9
//     23 qubits   725 /  235 us   2e-9        26 qubits  3283 / 1287 us   6e-10
//     24 qubits  1099 /  370 us   2e-9        27 qubits  6359 / 2520 us   6e-10
// On states whose terms repeat in a pattern both are off by up to 1e-7 at every size.  The bound of a
// string's error is 5 * 2^-24 of the sum of |c_(j^x)| |c_j| (two roundings a term, three levels of
// sums); the one-mask kernel's is 6 * 2^-24 with four or more strings a pass and up to 18 * 2^-24 with
// fewer.  Measured against 64 bits on the states above: 20 qubits 1.8e-9 (one-mask) and 1.2e-9
// (tiles), 24 qubits 5.9e-10 and 3.1e-10, 26 qubits 2.4e-10 and 2.0e-10.
constexpr int kEvtMinQubits = 26;
constexpr int kEvtCtas = 4;      // per SM: 53 KB of shared memory, 128 registers a thread
constexpr int kEvtGroups = 32;
constexpr int kEvtStrings = 64;

struct EvtGroup {
    unsigned short xv;        // address XOR to the partner amplitude
    unsigned short ov[12];    // address vectors: 7 thread bits, 4 bits inside the thread, the round bit (x = 0)
    unsigned char rounds;     // 2 when x = 0 (2^12 terms), else 1
    unsigned char comp;       // 0: real part of the term, 1: imaginary part
    unsigned char s0, s1;     // its strings
};
struct EvtString {
    unsigned long long z_out; // z outside the tile
    unsigned char zt, zw, zr; // z on the thread bits, the in-thread bits, the round bit
};
struct EvtArgs {
    TileGeom t;
    long long tiles;
    int n_groups, n_strings;
    EvtGroup g[kEvtGroups];
    EvtString s[kEvtStrings];
};

__device__ __forceinline__ float pick_sign(float v, unsigned odd) { return __uint_as_float(__float_as_uint(v) ^ (odd << 31)); }

__global__ void __launch_bounds__(kEvtThreads, kEvtCtas) expval_tile_kernel(const float *__restrict__ sv, const __grid_constant__ EvtArgs a,
                                                                     double *__restrict__ partials)
{
    extern __shared__ __align__(16) float smem[];
    float *tile = smem;
    float *rb = smem + kEvtTileFloats;                              // 16 x 128 entries
    float2 *acc = reinterpret_cast<float2 *>(rb + 16 * kEvtThreads);   // per string and lane
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const TileMover<kEvtThreads> mv(a.t);
    for (int i = tid; i < a.n_strings * 32; i += kEvtThreads) acc[i] = make_float2(0.f, 0.f);
    for (long long t = blockIdx.x; t < a.tiles; t += gridDim.x) {
        const unsigned long long b0 = tile_base(a.t, (unsigned long long)t);
        __syncthreads();   // the last tile's readers are done
        mv.load(a.t, sv + (long long)(b0 << 6), tile);
        __syncthreads();
        for (int gi = 0; gi < a.n_groups; ++gi) {
            const EvtGroup &g = a.g[gi];
            unsigned bt = 0;
#pragma unroll
            for (int b = 0; b < 7; ++b) bt ^= (0u - ((unsigned)(tid >> b) & 1u)) & (unsigned)g.ov[b];
            for (int r = 0; r < g.rounds; ++r) {
                const unsigned base = r ? bt ^ g.ov[11] : bt;
                float w[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    unsigned o = base;
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if ((i >> b) & 1) o ^= g.ov[7 + b];
                    const unsigned p = o ^ g.xv;
                    const float ur = tile[o], ui = tile[o + 32], vr = tile[p], vi = tile[p + 32];
                    w[i] = g.comp ? fmaf(vr, ui, -(vi * ur)) : fmaf(vr, ur, vi * ui);
                }
#pragma unroll
                for (int h = 1; h < 8; h <<= 1)   // two 8-point transforms: fp32 sums hold eight terms
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (!(i & h)) {
                            const float x = w[i], y = w[i + h];
                            w[i] = x + y;
                            w[i + h] = x - y;
                        }
                __syncthreads();   // the last group's entries have been read
#pragma unroll
                for (int i = 0; i < 16; ++i) rb[i * kEvtThreads + tid] = w[i];
                __syncthreads();
                for (int s = g.s0 + ((warp - g.s0) & 3); s < g.s1; s += 4) {
                    const EvtString &z = a.s[s];
                    const unsigned odd = (unsigned)(__popcll((b0 << 5) & z.z_out) & 1) ^ (r ? z.zr : 0u);
                    const float2 v = acc[s * 32 + lane];
                    FF2 f{v.x, v.y};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int e = lane + 32 * k;
                        const unsigned oe = odd ^ ((unsigned)__popc(e & z.zt) & 1u);
                        ff_add(f, pick_sign(rb[(z.zw & 7) * kEvtThreads + e], oe));
                        ff_add(f, pick_sign(rb[(8 + (z.zw & 7)) * kEvtThreads + e], oe ^ (z.zw >> 3)));
                    }
                    acc[s * 32 + lane] = make_float2(f.hi, f.lo);
                }
            }
        }
    }
    for (int gi = 0; gi < a.n_groups; ++gi)
        for (int s = a.g[gi].s0 + ((warp - a.g[gi].s0) & 3); s < a.g[gi].s1; s += 4) {
            const float2 v = acc[s * 32 + lane];
            const double d = warp_sum((double)v.x + (double)v.y);
            if (lane == 0) partials[(size_t)blockIdx.x * a.n_strings + s] = a.g[gi].xv ? 2.0 * d : d;
        }
}

// one CTA per string: the CTAs' partials in a fixed order
__global__ void __launch_bounds__(128) expval_sum_kernel(const double *__restrict__ partials, int ctas, int n_strings,
                                                         double *__restrict__ result)
{
    __shared__ double red[4];
    double s = 0.0;
    for (int i = threadIdx.x; i < ctas; i += 128) s += partials[(size_t)i * n_strings + blockIdx.x];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) result[blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
}

constexpr int kEvtSmem = (int)sizeof(float) * (kEvtTileFloats + 16 * kEvtThreads) + kEvtStrings * 32 * (int)sizeof(float2);

// The tile pass of the strings order[..] listed in `runs` (each a run of equal x masks); res[i]
// receives the i-th string's sum in the order of `placed`.
void fill_tiles(const std::vector<EvRun> &runs, const std::vector<int> &order, const uint64_t *x_masks, const uint64_t *z_masks, int n,
                uint64_t lam, EvtArgs *a, std::vector<int> *placed)
{
    std::memset(a, 0, sizeof(*a));
    placed->clear();
    int local_of[64], L = 0;
    for (int q = 0; q < n; ++q) {
        local_of[q] = -1;
        if ((lam >> q) & 1) local_of[q] = L++;
    }
    fill_geom(lam, n, &a->t);
    a->tiles = 1ll << (n - L);
    for (const EvRun &run : runs)
        for (int comp = 0; comp < 2; ++comp) {
            EvtGroup &g = a->g[a->n_groups];
            const uint64_t x = x_masks[order[(size_t)run.pos]];
            g.s0 = (unsigned char)placed->size();
            int top = -1;
            g.xv = 0;
            for (int q = 0; q < n; ++q)
                if ((x >> q) & 1) {
                    g.xv = (unsigned short)(g.xv ^ addr_vec(local_of[q]));
                    top = local_of[q];
                }
            std::vector<int> free_bits, ob;
            for (int t = 0; t < L; ++t)
                if (t != top) free_bits.push_back(t);
            lane_bits(free_bits, &ob);
            for (size_t b = 0; b < ob.size(); ++b) g.ov[b] = (unsigned short)addr_vec(ob[b]);
            g.rounds = x ? 1 : 2;
            g.comp = (unsigned char)comp;
            for (int i = 0; i < run.m; ++i) {
                const int s = order[(size_t)(run.pos + i)];
                const uint64_t z = z_masks[s];
                if ((__builtin_popcountll(x & z) & 1) != comp) continue;
                EvtString &o = a->s[placed->size()];
                o.z_out = z & ~lam;
                unsigned bits = 0;   // z on the ordered index bits
                for (size_t b = 0; b < ob.size(); ++b)
                    for (int q = 0; q < n; ++q)
                        if (local_of[q] == ob[b] && ((z >> q) & 1)) bits |= 1u << b;
                o.zt = (unsigned char)(bits & 127u);
                o.zw = (unsigned char)((bits >> 7) & 15u);
                o.zr = (unsigned char)((bits >> 11) & 1u);
                placed->push_back(s);
            }
            g.s1 = (unsigned char)placed->size();
            if (g.s1 > g.s0) ++a->n_groups;
        }
    a->n_strings = (int)placed->size();
}

std::mutex g_evt_mu;
uint64_t g_evt_attr = 0;

int launch_tiles(const float *sv, const EvtArgs &a, double *partials, double *result, int num_sms, cudaStream_t s)
{
    int dev = 0;
    SV_CUDA_TRY(cudaGetDevice(&dev));
    const uint64_t bit = dev >= 0 && dev < 64 ? (1ull << dev) : 0ull;
    {
        std::lock_guard<std::mutex> lk(g_evt_mu);
        if (!(g_evt_attr & bit) || !bit) {
            SV_CUDA_TRY(cudaFuncSetAttribute(expval_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kEvtSmem));
            g_evt_attr |= bit;
        }
    }
    const int grid = (int)std::min<long long>(a.tiles, (long long)kEvtCtas * num_sms);
    const int smem = (int)sizeof(float) * (kEvtTileFloats + 16 * kEvtThreads) + a.n_strings * 32 * (int)sizeof(float2);
    expval_tile_kernel<<<grid, kEvtThreads, smem, s>>>(sv, a, partials);
    SV_CUDA_TRY(cudaGetLastError());
    expval_sum_kernel<<<a.n_strings, 128, 0, s>>>(partials, grid, a.n_strings, result);
    SV_CUDA_TRY(cudaGetLastError());
    return SV_OK;
}

int highest_bit(unsigned long long v)
{
    int h = -1;
    while (v) {
        ++h;
        v >>= 1;
    }
    return h;
}

}  // namespace
}  // namespace svg

using namespace svg;

namespace {

int expval_pauli(const sv_state *st_c, const uint64_t *x_masks, const uint64_t *z_masks, int count, double *out)
{
    sv_state *st = const_cast<sv_state *>(st_c);
    if (!st || count < 0 || (count > 0 && (!x_masks || !z_masks || !out))) { set_error("sv_expval_pauli: bad argument"); return SV_EINVAL; }
    if (st->c128) { set_error("sv_expval_pauli: expectation values need a complex64 state"); return SV_EINVAL; }
    if (count == 0) return SV_OK;
    const int n = st->n;
    const uint64_t valid = n >= 64 ? ~0ull : ((1ull << n) - 1ull);
    for (int i = 0; i < count; ++i)
        if ((x_masks[i] | z_masks[i]) & ~valid) {
            set_error("sv_expval_pauli: string %d acts on a qubit >= n = %d", i, n);
            return SV_EINVAL;
        }
    // workspace: per-CTA partials for one launch, a counter, and one result per string
    const int max_grid = st->num_sms * 8;
    const size_t n_partials = (size_t)st->num_sms * std::max(8 * kEvMaxStrings, kEvtCtas * kEvtStrings);
    if (count > st->ev_capacity) {
        cudaStreamSynchronize(st->stream);
        cudaFree(st->d_ev);
        st->d_ev = nullptr;
        st->ev_capacity = 0;
        const size_t doubles = n_partials + (size_t)count + 1;
        cudaError_t e = cudaMalloc(&st->d_ev, sizeof(double) * doubles);
        if (e == cudaSuccess) e = cudaMemsetAsync(st->d_ev, 0, sizeof(double) * doubles, st->stream);
        if (e != cudaSuccess) { set_error("sv_expval_pauli: workspace allocation failed: %s", cudaGetErrorString(e)); return SV_ENOMEM; }
        st->ev_capacity = count;
    }
    double *partials = st->d_ev;
    double *results = partials + n_partials;
    unsigned *counter = reinterpret_cast<unsigned *>(results + st->ev_capacity);

    // strings grouped by x mask (first-appearance order), at most kEvMaxStrings per pass
    std::vector<int> order((size_t)count);
    for (int i = 0; i < count; ++i) order[(size_t)i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int p, int q) { return x_masks[p] < x_masks[q]; });
    const long long nb = n >= 5 ? (1ll << (n - 5)) : 1ll;
    std::vector<int> slot_of((size_t)count);
    int out_pos = 0;   // next slot of `results`
    // Runs of equal x masks (cut at half a tile pass's strings).  Runs whose masks fit one tile's local
    // qubits share a read of the state; a tile pass is taken when it replaces two or more passes of the
    // kernel above.  26 qubits, tile / one-mask (us): one string 127 / 110, eight of one mask 152 / 160,
    // two masks 149 / 192, 16 of one mask 168 / 297, two masks of eight 206 / 298, seven of eight 435 / 959.
    std::vector<EvRun> runs, left;
    std::vector<uint64_t> run_x;
    for (int p = 0; p < count;) {
        const uint64_t x = x_masks[order[(size_t)p]];
        int m = 0;
        while (p + m < count && m < kEvtStrings / 2 && x_masks[order[(size_t)(p + m)]] == x) ++m;
        runs.push_back(EvRun{p, m});
        run_x.push_back(x);
        p += m;
    }
    if (n >= kEvtMinQubits) {
        std::vector<EvTilePass> tiles;
        plan_tiles(runs, run_x, n, EvTileLimits{kEvtQubits, kEvtStrings, kEvtGroups, 2, kEvMaxStrings}, &tiles, &left);
        for (const EvTilePass &t : tiles) {
            EvtArgs a;
            std::vector<int> placed;
            fill_tiles(t.runs, order, x_masks, z_masks, n, t.lam, &a, &placed);
            SV_TRY(launch_tiles(st->d, a, partials, results + out_pos, st->num_sms, st->stream));
            for (int s : placed) slot_of[(size_t)s] = out_pos++;
        }
    } else {
        left.swap(runs);
    }
    for (const EvRun &run : left)
    for (int pos = run.pos; pos < run.pos + run.m;) {
        const uint64_t x = x_masks[order[(size_t)pos]];
        const int m = std::min(kEvMaxStrings, run.pos + run.m - pos);
        EvArgs a;
        std::memset(&a, 0, sizeof(a));
        a.xb = x >> 5;
        a.xl = (int)(x & 31u);
        a.pair_bit = a.xb ? highest_bit(a.xb) : -1;
        a.n_units = a.xb ? nb / 2 : nb;
        a.m = m;
        for (int p = 0; p < m; ++p) {
            const int s = order[(size_t)(pos + p)];
            const unsigned long long zb = z_masks[s] >> 5;
            unsigned long long zu = zb;
            if (a.pair_bit >= 0) {   // delete the pair bit: b = u with a zero inserted there
                const unsigned long long low = zb & ((1ull << a.pair_bit) - 1ull);
                zu = ((zb >> (a.pair_bit + 1)) << a.pair_bit) | low;
            }
            a.zu[p] = zu;
            unsigned tab = 0;
            for (unsigned i = 0; i < 32; ++i) tab |= (unsigned)(__builtin_popcountll(i & zu & 31ull) & 1) << i;
            a.ztab[p] = tab;
            a.zc[p] = (unsigned)(zu & 7ull);
            a.zl[p] = (unsigned)(z_masks[s] & 31u);
            a.pairpar[p] = (unsigned)(__builtin_popcountll(a.xb & zb) & 1);
            a.comp[p] = __builtin_popcountll(x & z_masks[s]) & 1;
            slot_of[(size_t)s] = out_pos + p;
        }
        const long long ranges = (a.n_units + kEvRange - 1) / kEvRange;
        const long long work = (ranges * 32 + kEvThreads - 1) / kEvThreads;   // CTAs with a range per warp
        const float *sv = st->d;
        double *res = results + out_pos;
        int rc;
        if (m == 1) rc = launch_ev<1>(sv, a, partials, counter, res, work, st->num_sms, max_grid, st->stream);
        else if (m == 2) rc = launch_ev<2>(sv, a, partials, counter, res, work, st->num_sms, max_grid, st->stream);
        else if (m <= 4) rc = launch_ev<4>(sv, a, partials, counter, res, work, st->num_sms, max_grid, st->stream);
        else rc = launch_ev<8>(sv, a, partials, counter, res, work, st->num_sms, max_grid, st->stream);
        if (rc != SV_OK) return rc;
        pos += m;
        out_pos += m;
    }
    std::vector<double> host((size_t)count + kEvMaxStrings);
    SV_CUDA_TRY(cudaMemcpyAsync(host.data(), results, sizeof(double) * (size_t)count, cudaMemcpyDeviceToHost, st->stream));
    SV_CUDA_TRY(cudaStreamSynchronize(st->stream));
    for (int i = 0; i < count; ++i) {
        const double s = host[(size_t)slot_of[(size_t)i]];
        // <psi|P|psi> = i^popc(x & z) * S; the accumulated component is Re S (even) or Im S (odd)
        switch (__builtin_popcountll(x_masks[i] & z_masks[i]) & 3) {
        case 0: out[i] = s; break;
        case 1: out[i] = -s; break;
        case 2: out[i] = -s; break;
        default: out[i] = s; break;
        }
    }
    return SV_OK;
}

}  // namespace

extern "C" int sv_expval_pauli(const sv_state *st, const uint64_t *x_masks, const uint64_t *z_masks, int count, double *out)
{
    clear_error();
    try {
        return expval_pauli(st, x_masks, z_masks, count, out);
    } catch (const std::exception &) {   // the vectors of many strings
        set_error("sv_expval_pauli: out of host memory");
        return SV_ENOMEM;
    }
}
