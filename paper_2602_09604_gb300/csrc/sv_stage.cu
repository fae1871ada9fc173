// Staged passes: several fused gates applied in one pass over the state (CUDA-core fp32 gates).
//
// One launch per fused gate reads and writes the whole state for every gate.  A CUDA-core gate of
// k <= 3 qubits is bound by that traffic (16 bytes an amplitude), and on states that fit the L2 by
// the launch itself.  Here consecutive gates whose qubits fit in one set of kStageQubits local qubits
// (always holding qubits 0-4, so that global memory moves in whole 256-byte blocks) form a pass: a
// CTA copies one tile -- the 2^kStageQubits amplitudes that agree on the other qubits -- into shared
// memory, applies every gate of the pass there and writes the tile back, so the state is read and
// written once per pass instead of once per gate.
//
// A gate joins a pass when no earlier gate left out shares a qubit with it, so it only moves ahead
// of gates on other qubits: the same product, but its roundings fall in another order (96
// Grover circuits of 10 to 25 qubits: errors of 0.25 to 4 times those in circuit order, 0.93 in the
// geometric mean, the largest at 23 qubits with gates of 4: 4.2e-7 against 2.2e-7 over twelve marked
// elements, 24 qubits 4.2e-7 both; grids and quantum volume 0.98 to 1.04).  Every output is formed by the same chain of fused multiply-adds
// as in the one-gate kernels (columns in order; re += ar xr, re -= ai xi, im += ar xi, im += ai xr),
// so passes that keep the circuit's order give the same bits.
//
// What bounds a pass: shared memory moves 2 x 8 bytes an amplitude and gate and the FMA pipe
// 4 * 2^k multiply-adds an amplitude and gate.  The multiply-adds are issued as packed pairs
// (fma.rn.f32x2, two rows of one column).  The pass's descriptors and matrices are copied to shared
// memory ahead of the tile and read there by broadcast 16-byte loads, each of which costs two passes of
// the shared-memory pipe: a thread therefore takes four groups at a time for k <= 3 and two for k = 4,
// so that one such load serves 8 to 16 packed multiply-adds.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <mutex>
#include <queue>

#include "sv_internal.h"
#include "sv_launch.h"
#include "sv_tile.h"

namespace svg {
namespace {

// One gate of a pass.  Tile addresses are float offsets, linear over GF(2) in the tile's index bits.
// Every address is the XOR of addr_vec(t) over some of the tile's 5 + fb local bits t, each used once (as a
// target, a control or a group-index bit): below 64 << fb and with bit 5 clear, so that the real part and
// the imaginary part 32 floats on lie in the tile for every thread, trip and column.
struct alignas(16) StageGate {
    // address vectors of the group-index bits that come from the thread index, two to a word: bit b
    // in the low half of word b, bit b + 5 in the high half
    unsigned lane[5];
    unsigned short step[7];     // address vectors of group-index bits 5-11 (those past the thread index count trips)
    unsigned short pad;
    unsigned short tv[5];       // address vector of target b
    unsigned short cset;        // address of the control bits inside the tile, all 1
    unsigned short moff;        // matrix offset (16-byte units) in the pass's matrices
    unsigned char k, nb;        // targets; group-index bits
    uint64_t cm_out;            // control qubits outside the tile: the gate applies to tiles with all of them 1
};
static_assert(sizeof(StageGate) == 64, "a gate's descriptor is read as 16-byte words");
constexpr int kStageMaxGates = 48;
struct StageArgs {
    TileGeom t;
    int n_gates;
    int units;                  // 16-byte units of the pass's image: descriptors, then matrices
};

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 dup2(float x)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void fma2(f32x2 &d, f32x2 a, f32x2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }

__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)   // a * b + 0: the first step of a chain
{
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(0ull));
    return d;
}

// The thread index's bits as masks, laid out as StageGate::lane.
struct ThreadMasks {
    unsigned m[5];
    __device__ __forceinline__ ThreadMasks()
    {
#pragma unroll
        for (int b = 0; b < 5; ++b)
            m[b] = ((threadIdx.x >> b) & 1u ? 0xffffu : 0u) | ((threadIdx.x >> (b + 5)) & 1u ? 0xffff0000u : 0u);
    }
};

// One gate on the tile: a thread takes V groups (group index bits -> tile address by the XOR of the
// set bits' vectors) at a time, accumulates all rows while the columns stream from shared memory, then
// writes the rows back.  m: column j, row pair p at m[j * D / 2 + p] = (re, re', im, im').
template <int K, int V, int T>
__device__ __forceinline__ void stage_gate(float *__restrict__ tile, const ulonglong2 *__restrict__ m, const StageGate &g, const ThreadMasks &tm)
{
    constexpr int D = 1 << K;
    constexpr int LT = T == 128 ? 7 : 9;
    constexpr int LV = V == 4 ? 2 : V == 2 ? 1 : 0;
    static_assert((T == 128 || T == 512) && (1 << LV) == V, "thread and group counts");
    const int nb = g.nb;
    // group index = thread index + (trip V + v) T, v < V; a gate with fewer groups than that (kept
    // controls) repeats its last ones under v: their address bits are 0, and every copy of a group is
    // read before any is written (one thread holds them all)
    const bool active = nb >= LT || (threadIdx.x >> nb) == 0;
    if (active) {
        unsigned bt = 0;
#pragma unroll
        for (int b = 0; b < 5; ++b) bt ^= tm.m[b] & g.lane[b];
        bt = (bt & 0xffffu) ^ (bt >> 16) ^ g.cset;
        unsigned tv[K], pv[V];
#pragma unroll
        for (int b = 0; b < K; ++b) tv[b] = g.tv[b];
#pragma unroll
        for (int v = 0; v < V; ++v) {
            pv[v] = 0u;
#pragma unroll
            for (int b = 0; b < LV; ++b)
                if ((v >> b) & 1) pv[v] ^= g.step[LT - 5 + b];   // 0 from group-index bit nb on
        }
        const int iters = nb > LT + LV ? 1 << (nb - LT - LV) : 1;
#pragma unroll 1
        for (int it = 0; it < iters; ++it) {
            unsigned base = bt;
            for (int b = LT + LV; b < nb; ++b) base ^= ((it >> (b - LT - LV)) & 1) ? (unsigned)g.step[b - 5] : 0u;
            f32x2 yr[V][D / 2], yi[V][D / 2];
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int p = 0; p < D / 2; ++p) yr[v][p] = yi[v][p] = 0ull;   // dead when K <= 2
            // columns in fours, the fours in a real loop: unrolled whole, the compiler keeps every
            // column's address and operands alive and spills
            constexpr int LJ = K < 2 ? K : 2, JU = 1 << LJ;
#pragma unroll 1
            for (int jh = 0; jh < D / JU; ++jh) {
                unsigned oh = base;
#pragma unroll
                for (int b = LJ; b < K; ++b) oh ^= ((jh >> (b - LJ)) & 1) ? tv[b] : 0u;
                const ulonglong2 *mj = m + jh * (JU * D / 2);
#pragma unroll
                for (int jl = 0; jl < JU; ++jl) {
                    unsigned o = oh;
#pragma unroll
                    for (int b = 0; b < LJ; ++b)
                        if ((jl >> b) & 1) o ^= tv[b];
                    f32x2 xr[V], xi[V], xn[V];
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const unsigned a = o ^ pv[v];
                        const float r = tile[a], i = tile[a + 32];
                        xr[v] = dup2(r);
                        xi[v] = dup2(i);
                        xn[v] = dup2(-i);
                    }
#pragma unroll
                    for (int p = 0; p < D / 2; ++p) {
                        const ulonglong2 u = mj[jl * (D / 2) + p];
#pragma unroll
                        for (int v = 0; v < V; ++v) {
                            if (K <= 2 && jl == 0) {   // one trip: the chains start here
                                yr[v][p] = mul2(u.x, xr[v]);
                                yi[v][p] = mul2(u.x, xi[v]);
                            } else {
                                fma2(yr[v][p], u.x, xr[v]);
                                fma2(yi[v][p], u.x, xi[v]);
                            }
                            fma2(yr[v][p], u.y, xn[v]);
                            fma2(yi[v][p], u.y, xr[v]);
                        }
                    }
                }
            }
#pragma unroll
            for (int p = 0; p < D / 2; ++p) {
                unsigned o = base;
#pragma unroll
                for (int b = 1; b < K; ++b)
                    if ((p >> (b - 1)) & 1) o ^= tv[b];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const unsigned a = o ^ pv[v];
                    float r0, r1, i0, i1;
                    unpack2(yr[v][p], r0, r1);
                    unpack2(yi[v][p], i0, i1);
                    tile[a] = r0;
                    tile[a + 32] = i0;
                    tile[a ^ tv[0]] = r1;
                    tile[(a ^ tv[0]) + 32] = i1;
                }
            }
        }
    }
}

// CTAs per SM of the 128-thread form by the largest gate of the pass: what its registers allow without
// spills that count (28 qubits, 8 cycles, gates of 3: 20.9 ms so; two groups a thread in six CTAs 21.2).
__host__ __device__ constexpr int stage_ctas(int kmax) { return kmax <= 2 ? 5 : kmax <= 4 ? 4 : 3; }

// T threads a CTA, gates of up to KMAX qubits (see launch_stage for the forms).  A kernel per largest
// gate: passes of small gates keep their own register count, so more CTAs share an SM.
template <int T, int KMAX>
__global__ void __launch_bounds__(T, T == 128 ? stage_ctas(KMAX) : 1) stage_kernel(float *__restrict__ sv, const uint4 *__restrict__ image,
                                                                                 const __grid_constant__ StageArgs a)
{
    extern __shared__ __align__(16) float tile[];
    next_may_start();
    uint4 *img = reinterpret_cast<uint4 *>(tile + (64 << a.t.fb));
    for (int i = threadIdx.x; i < a.units; i += T) img[i] = __ldg(image + i);
    const TileMover<T> mv(a.t);
    const ThreadMasks tm;
    const unsigned long long b0 = tile_base(a.t, blockIdx.x);
    float *g0 = sv + (long long)(b0 << 6);
    wait_for_previous();
    mv.load(a.t, g0, tile);
    __syncthreads();
    constexpr bool F = T == 512;   // few tiles: one group at a time, so that more threads have one
    for (int i = 0; i < a.n_gates; ++i) {
        const StageGate &g = reinterpret_cast<const StageGate *>(img)[i];
        if (((b0 << 5) & g.cm_out) == g.cm_out) {
            const ulonglong2 *m = reinterpret_cast<const ulonglong2 *>(img + g.moff);
            const int k = g.k;
            if (k == 1) {
                stage_gate<1, F ? 1 : 4, T>(tile, m, g, tm);
            } else if (KMAX <= 2 || k == 2) {
                stage_gate<2, F ? 1 : 4, T>(tile, m, g, tm);
            } else if constexpr (KMAX >= 3) {
                if (KMAX == 3 || k == 3) {
                    stage_gate<3, F ? 1 : 4, T>(tile, m, g, tm);
                } else if constexpr (KMAX >= 4) {
                    if (KMAX == 4 || k == 4) stage_gate<4, F ? 1 : 2, T>(tile, m, g, tm);
                    else if constexpr (KMAX == 5) stage_gate<5, 1, T>(tile, m, g, tm);
                }
            }
        }
        __syncthreads();
    }
    mv.store(a.t, tile, g0);
}

// ------------------------------------------------------------------------------------ planner
constexpr int kLargeQubits = 21;        // from 512 tiles on (the many-tile form)
constexpr int kStageMatFloats = 4096;   // matrices of one pass: 16 KB, so that four CTAs share an SM

bool stageable(const FusedGate &g)
{
    if (!g.post.empty() || !g.swaps.empty()) return false;
    if (g.path == SV_PATH_CONTROLLED) return g.k >= 1 && g.k <= 3;
    return (g.path == SV_PATH_LOW || g.path == SV_PATH_HIGH || g.path == SV_PATH_MIXED) && g.k >= 1 && g.k <= 5 && g.cmask == 0;
}

// Time of a gate on its own kernel, and its share in a pass, on states past the L2 in units of one read
// and write of the state at the copy rate (k = 1..5; 28 qubits: 1.0 = 0.63 ms).  A pass adds
// kPassCost for its own read and write, partly hidden behind the arithmetic.  Below 28 qubits the same
// figures serve as a rule; measured by it / every pass taken / every gate alone (us, grids of 10
// cycles, gates of 4): 21 qubits 161 / 166 / 185, 23 qubits 567 / 616 / 633, 24 qubits 1229 / 1220 / 1414,
// 26 qubits 5518 / 5572 / 6101.  It loses most, 2 to 3%, on quantum volume with gates of 4 (24 qubits
// 868 / 843 / 980, 26 qubits 3484 / 3400 / 3672), and below 21 qubits it costs up to a third (19 qubits
// 48 / 35 / 83): there every pass is taken.
constexpr double kPassCost = 0.7, kInPass[6] = {0, 0.2, 0.3, 0.5, 1.0, 2.0};
double alone_cost(const FusedGate &g)
{
    static const double high[6] = {0, 0.97, 0.97, 0.97, 1.09, 2.4}, tile[6] = {0, 0.97, 1.0, 1.2, 1.55, 4.0};
    if (g.path == SV_PATH_CONTROLLED) return std::ldexp(1.0, -__builtin_popcountll(g.cmask & ~uint64_t(7)));
    return g.path == SV_PATH_HIGH ? high[g.k] : tile[g.k];
}

uint64_t named(const FusedGate &g)
{
    uint64_t q = g.mask | g.cmask;
    for (const FusedGate::PostTerm &t : g.post) q |= uint64_t(1) << t.q;
    return q;   // a swap network's mask already holds its qubits
}

size_t mat_floats(const FusedGate &g) { return size_t(2) << (2 * g.k); }

constexpr size_t kGateFloats = sizeof(StageGate) / sizeof(float);

// the launch arguments of a pass over gates `idx` with the local qubits `lam` (bits 0-4 set), and its
// image: descriptors, then matrices
void fill_stage(const std::vector<const FusedGate *> &gates, const std::vector<int> &idx, uint64_t lam, int n, StageArgs *a, float *image)
{
    std::memset(a, 0, sizeof(*a));
    int local_of[64];
    int L = 0;
    for (int q = 0; q < n; ++q)
        if ((lam >> q) & 1) local_of[q] = L++;
    fill_geom(lam, n, &a->t);
    a->n_gates = (int)idx.size();
    size_t at = idx.size() * kGateFloats;
    std::vector<int> free_bits, order;
    for (size_t s = 0; s < idx.size(); ++s) {
        const FusedGate &g = *gates[(size_t)idx[s]];
        StageGate o;
        std::memset(&o, 0, sizeof(o));
        o.k = (unsigned char)g.k;
        uint64_t used = 0;   // local bits that are targets or controls
        for (int b = 0; b < g.k; ++b) {
            used |= uint64_t(1) << local_of[g.targets[b]];
            o.tv[b] = (unsigned short)addr_vec(local_of[g.targets[b]]);
        }
        for (int q = 0; q < n; ++q)
            if ((g.cmask >> q) & 1) {
                if ((lam >> q) & 1) {
                    used |= uint64_t(1) << local_of[q];
                    o.cset = (unsigned short)(o.cset ^ addr_vec(local_of[q]));
                } else {
                    o.cm_out |= uint64_t(1) << q;
                }
            }
        free_bits.clear();
        for (int t = 0; t < L; ++t)
            if (!((used >> t) & 1)) free_bits.push_back(t);
        lane_bits(free_bits, &order);
        o.nb = (unsigned char)order.size();
        for (size_t b = 0; b < order.size(); ++b) {
            const unsigned v = addr_vec(order[b]);
            if (b < 10) o.lane[b % 5] |= b < 5 ? v : v << 16;
            if (b >= 5) o.step[b - 5] = (unsigned short)v;
        }
        o.moff = (unsigned short)(at / 4);
        const int D = 1 << g.k;
        for (int j = 0; j < D; ++j)
            for (int p = 0; p < D / 2; ++p, at += 4) {
                const size_t e0 = size_t(2 * p) * D + j, e1 = e0 + D;
                image[at] = g.ur[e0];
                image[at + 1] = g.ur[e1];
                image[at + 2] = g.ui[e0];
                image[at + 3] = g.ui[e1];
            }
        std::memcpy(image + s * kGateFloats, &o, sizeof(o));
    }
    a->units = (int)(at / 4);
}

}  // namespace

void plan_passes(const std::vector<const FusedGate *> &gates, int n, bool keep_order, PassPlan *plan)
{
    plan->steps.clear();
    plan->image_floats = 0;
    const size_t ng = gates.size();
    bool small = true;
    for (const FusedGate *g : gates)
        if (g->k > 2) small = false;
    // Each gate waits for the gates before it on its qubits.  `ready` holds the gates left that wait
    // for none: they share no qubit, so there are at most n of them, and a pass looks at those and at
    // what it takes, not at every gate left (200,000 gates of two on 20 qubits: 0.26 s, 21 s by scans).
    std::vector<int> waits(ng, 0), at(ng + 1, 0), then;   // then[at[g] ..]: the next gate on each of g's qubits
    for (size_t i = 0; i < ng; ++i) at[i + 1] = at[i] + __builtin_popcountll(named(*gates[i]));
    then.assign((size_t)at[ng], -1);
    std::priority_queue<int, std::vector<int>, std::greater<int>> ready;
    {
        int last[64];   // the slot of `then` of each qubit's last gate
        std::fill(last, last + 64, -1);
        for (size_t i = 0; i < ng; ++i) {
            int slot = at[i];
            for (uint64_t q = named(*gates[i]); q; q &= q - 1) {
                int &l = last[__builtin_ctzll(q)];
                if (l >= 0) {
                    then[(size_t)l] = (int)i;
                    ++waits[i];
                }
                l = slot++;
            }
            if (!waits[i]) ready.push((int)i);
        }
    }
    // Large tiles hold more gates a pass; on a small state they leave SMs without a tile, and a pass is
    // then as long as its chain of gates on one tile.  Measured (us, tiles of 2^10 / 2^11 / 2^12; grids of
    // 14 cycles): gates of 2, 16 qubits 47 / 59 / 85, 17 qubits 46 / 60 / 85, 18 qubits 98 / 73 / 98;
    // gates of 4, 16 qubits 61 / 43 / 47, 17 qubits 42 / 42 / 64; gates of 3, 18 qubits 83 / 57 / 77,
    // 19 qubits 204 / 128 / 88, 20 qubits 380 / 226 / 190.
    const int L = std::min(n, n >= 19 ? kStageQubits : n <= 17 && small ? kStageQubits - 2 : kStageQubits - 1);
    std::vector<int> took, held;
    while (!ready.empty()) {
        PassStep st;
        uint64_t lam = 31;
        size_t mats = 0;
        took.clear();
        held.clear();
        // ready gates in circuit order: one that does not join holds back those that wait for it
        while (!ready.empty()) {
            const int i = ready.top();
            ready.pop();
            const FusedGate &g = *gates[(size_t)i];
            const uint64_t with = lam | g.mask;
            const bool joins = n >= 5 && stageable(g) && __builtin_popcountll(with) <= L && (int)took.size() < kStageMaxGates &&
                               mats + mat_floats(g) <= size_t(kStageMatFloats);
            if (!joins && !took.empty()) {
                held.push_back(i);
                if (keep_order) break;
                continue;
            }
            took.push_back(i);
            for (int t = at[(size_t)i]; t < at[(size_t)i + 1]; ++t) {
                const int w = then[(size_t)t];
                if (w >= 0 && --waits[(size_t)w] == 0) ready.push(w);
            }
            if (!joins) break;   // the first gate left runs alone
            lam = with;
            mats += mat_floats(g);
        }
        for (int i : held) ready.push(i);
        // On large states the one-gate kernels of four-qubit gates on high qubits run near the copy rate:
        // a pass of two or three of those alone costs more than it saves.
        bool pass = took.size() > 1;
        if (pass && n >= kLargeQubits) {
            double alone = 0, in = kPassCost;
            for (int t : took) {
                alone += alone_cost(*gates[(size_t)t]);
                in += kInPass[gates[(size_t)t]->k];
            }
            pass = in < alone;
        }
        if (!pass) {
            for (size_t t = 0; t + 1 < took.size(); ++t) {
                PassStep one;
                one.single = took[t];
                plan->steps.push_back(std::move(one));
            }
            st.single = took.back();
        } else {
            for (int q = 5; q < n && __builtin_popcountll(lam) < L; ++q) lam |= uint64_t(1) << q;   // whole tiles: lowest free qubits
            for (int t : took) st.kmax = std::max(st.kmax, gates[(size_t)t]->k);
            st.tiles = 1ll << (n - L);
            st.tile = lam;
            st.gates = took;
            st.image_off = plan->image_floats;
            plan->image_floats += took.size() * kGateFloats + mats;
        }
        plan->steps.push_back(std::move(st));
    }
}

void fill_images(const std::vector<const FusedGate *> &gates, int n, PassPlan *plan, float *image)
{
    for (PassStep &st : plan->steps)
        if (st.single < 0) {
            st.args.assign((sizeof(StageArgs) + 7) / 8, 0);
            fill_stage(gates, st.gates, st.tile, n, reinterpret_cast<StageArgs *>(st.args.data()), image + st.image_off);
        }
}

void pass_block(const PassStep &p, const float *image, std::vector<unsigned char> *out)
{
    const StageArgs *a = reinterpret_cast<const StageArgs *>(p.args.data());
    static_assert(sizeof(StageArgs) == 168, "sv_fused_plan_passes documents the layout");
    out->resize(sizeof(StageArgs) + 16 * (size_t)a->units);
    std::memcpy(out->data(), a, sizeof(StageArgs));
    std::memcpy(out->data() + sizeof(StageArgs), image + p.image_off, 16 * (size_t)a->units);
}

namespace {

std::mutex g_stage_mu;
uint64_t g_stage_attr[2][6] = {};   // by form and largest gate: a bit per device

template <int T, int KMAX>
int launch_form(float *sv, const float *image, const PassStep &p, cudaStream_t stream, int num_sms)
{
    const StageArgs *a = reinterpret_cast<const StageArgs *>(p.args.data());
    auto kern = stage_kernel<T, KMAX>;
    int dev = 0;
    SV_CUDA_TRY(cudaGetDevice(&dev));
    const uint64_t bit = dev >= 0 && dev < 64 ? (1ull << dev) : 0ull;
    {
        uint64_t &slot = g_stage_attr[T == 512][KMAX];
        std::lock_guard<std::mutex> lk(g_stage_mu);
        if (!(slot & bit) || !bit) {
            SV_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (8 << kStageQubits) + kStageMaxGates * (int)sizeof(StageGate) + 4 * kStageMatFloats));
            slot |= bit;
        }
    }
    // A part-filled wave of small CTAs leaves SMs with room, where the next pass's CTAs crowd: with gates of
    // one or two (five CTAs an SM) 21 qubits, 512 tiles, plain / chained: grid 237 / 259 us, quantum volume
    // 236 / 251; from 1024 tiles on 408 / 384. Larger gates fill 512 tiles' wave to 0.84 and more: 193 / 170.
    const bool chained = T == 512 || KMAX > 2 || p.tiles >= (long long)stage_ctas(KMAX) * num_sms;
    return launch_chained(chained, kern, (unsigned)p.tiles, T, (size_t(256) << a->t.fb) + 16 * (size_t)a->units, stream, sv,
                          reinterpret_cast<const uint4 *>(image), *a);
}

template <int T>
int launch_kmax(float *sv, const float *image, const PassStep &p, cudaStream_t stream, int num_sms)
{
    switch (p.kmax) {
    case 1:
    case 2: return launch_form<T, 2>(sv, image, p, stream, num_sms);
    case 3: return launch_form<T, 3>(sv, image, p, stream, num_sms);
    case 4: return launch_form<T, 4>(sv, image, p, stream, num_sms);
    default: return launch_form<T, 5>(sv, image, p, stream, num_sms);
    }
}

}  // namespace

int launch_stage(float *sv, const float *image, const PassStep &p, cudaStream_t stream, int num_sms)
{
    // With few tiles a pass is a chain of short gates, so each tile gets all the threads an SM
    // takes; with many, small CTAs of several groups a thread share an SM and overlap each other's
    // loads, barriers and arithmetic.
    return p.tiles < 2ll * num_sms ? launch_kmax<512>(sv, image + p.image_off, p, stream, num_sms)
                                      : launch_kmax<128>(sv, image + p.image_off, p, stream, num_sms);
}

}  // namespace svg
