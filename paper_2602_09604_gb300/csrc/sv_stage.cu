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
// of gates on other qubits (exact).  Every output is formed by the same chain of fused multiply-adds
// as in the one-gate kernels (columns in order; re += ar xr, re -= ai xi, im += ar xi, im += ai xr),
// so passes that keep the circuit's order give the same bits.
//
// What bounds a pass: shared memory moves 2 x 8 bytes an amplitude and gate and the FMA pipe
// 4 * 2^k multiply-adds an amplitude and gate.  The multiply-adds are issued as packed pairs
// (fma.rn.f32x2, two rows of one column); the matrices travel in the kernel's parameter block and are
// read through the constant bank at a run-time, warp-uniform index.  A loop of this form (k = 4, two
// groups a thread) measured 33.6 T multiply-adds/s on 152 SMs, against 28.4 with the matrices in
// shared memory (a broadcast 16-byte read costs two passes of the shared-memory pipe) and 24-29 with
// scalar multiply-adds.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "sv_internal.h"
#include "sv_tile.h"

namespace svg {
namespace {

// One gate of a pass.  Tile addresses are float offsets, linear over GF(2) in the tile's index bits.
struct StageGate {
    uint64_t cm_out;            // control qubits outside the tile: the gate applies to tiles with all of them 1
    unsigned short tv[5];       // address vector of target b
    unsigned short gv[kStageQubits];   // address vector of group-index bit b (0 from nb on)
    unsigned short cset;        // address of the control bits inside the tile, all 1
    unsigned short moff;        // matrix offset (16-byte units) in the pass's matrices
    unsigned char k, nb;        // targets; group-index bits
};
constexpr int kStageMaxGates = 48;
struct alignas(16) StageHead {
    TileGeom t;
    int n_gates;
    StageGate g[kStageMaxGates];
};
template <int M>
struct StageArgs {
    StageHead h;
    float mat[M];
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

// One gate on the tile: a thread takes V groups (group index bits -> tile address by the XOR of the
// set bits' vectors), accumulates all rows while the columns stream from shared memory, then writes
// the rows back.  m: column j, row pair p at m[j * D / 2 + p] = (re, re', im, im').
template <int K, int V, int T>
__device__ __forceinline__ void stage_gate(float *__restrict__ tile, const ulonglong2 *__restrict__ m, const StageGate &g)
{
    constexpr int D = 1 << K;
    constexpr int LT = T == 128 ? 7 : 9;
    static_assert((1 << LT) == T, "thread count");
    const int np = (V == 2 && g.nb > 0) ? g.nb - 1 : g.nb;
    const unsigned pv = (V == 2 && g.nb > 0) ? g.gv[np] : 0u;
    unsigned bt = g.cset;
#pragma unroll
    for (int b = 0; b < LT; ++b) bt ^= (0u - ((threadIdx.x >> b) & 1u)) & (unsigned)g.gv[b];
    if (np < LT && (threadIdx.x >> np) != 0) return;
    const int iters = np > LT ? 1 << (np - LT) : 1;
    for (int it = 0; it < iters; ++it) {
        unsigned base = bt;
        for (int b = LT; b < np; ++b) base ^= (0u - ((unsigned)(it >> (b - LT)) & 1u)) & (unsigned)g.gv[b];
        f32x2 yr[V][D / 2], yi[V][D / 2];
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int p = 0; p < D / 2; ++p) yr[v][p] = yi[v][p] = 0ull;
        // columns in fours, the fours in a real loop: unrolled whole, the compiler keeps every
        // column's address and operands alive and spills
        constexpr int JU = D < 4 ? D : 4;
#pragma unroll 1
        for (int jh = 0; jh < D / JU; ++jh) {
            unsigned oh = base;
#pragma unroll
            for (int b = 2; b < K; ++b) oh ^= ((jh >> (b - 2)) & 1) ? (unsigned)g.tv[b] : 0u;
            const ulonglong2 *mj = m + jh * (JU * D / 2);
#pragma unroll
            for (int jl = 0; jl < JU; ++jl) {
                unsigned o = oh;
                if (jl & 1) o ^= g.tv[0];
                if (jl & 2) o ^= g.tv[1];
                f32x2 xr[V], xi[V], xn[V];
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    const unsigned a = v ? o ^ pv : o;
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
                        fma2(yr[v][p], u.x, xr[v]);
                        fma2(yr[v][p], u.y, xn[v]);
                        fma2(yi[v][p], u.x, xi[v]);
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
                if ((p >> (b - 1)) & 1) o ^= g.tv[b];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const unsigned a = v ? o ^ pv : o;
                float r0, r1, i0, i1;
                unpack2(yr[v][p], r0, r1);
                unpack2(yi[v][p], i0, i1);
                tile[a] = r0;
                tile[a + 32] = i0;
                tile[a ^ g.tv[0]] = r1;
                tile[(a ^ g.tv[0]) + 32] = i1;
            }
        }
    }
}

// T threads a CTA, V groups a thread, matrices of up to M floats (see launch_stage for the forms).
template <int T, int V, int M>
__global__ void __launch_bounds__(T, T == 128 ? 5 : 1) stage_kernel(float *__restrict__ sv, const __grid_constant__ StageArgs<M> a)
{
    extern __shared__ __align__(16) float tile[];
    const TileMover<T> mv(a.h.t);
    const unsigned long long b0 = tile_base(a.h.t, blockIdx.x);
    float *g0 = sv + (long long)(b0 << 6);
    mv.load(a.h.t, g0, tile);
    __syncthreads();
    for (int i = 0; i < a.h.n_gates; ++i) {
        const StageGate &g = a.h.g[i];
        if (((b0 << 5) & g.cm_out) == g.cm_out) {
            const ulonglong2 *m = reinterpret_cast<const ulonglong2 *>(a.mat + 4 * g.moff);
            switch (g.k) {
            case 1: stage_gate<1, V, T>(tile, m, g); break;
            case 2: stage_gate<2, V, T>(tile, m, g); break;
            case 3: stage_gate<3, V, T>(tile, m, g); break;
            case 4: stage_gate<4, V, T>(tile, m, g); break;
            default: stage_gate<5, 1, T>(tile, m, g); break;
            }
        }
        __syncthreads();
    }
    mv.store(a.h.t, tile, g0);
}

// ------------------------------------------------------------------------------------ planner
// Matrix space of one pass, in the three parameter-block sizes a launch chooses from (a block is
// copied by every launch, so short passes take a short one; the limit is 32,764 bytes).
constexpr int kStageMat[3] = {1024, 2560, 6656};
constexpr int kStageMatFloats = kStageMat[2];

bool stageable(const FusedGate &g)
{
    if (!g.post.empty() || !g.swaps.empty()) return false;
    if (g.path == SV_PATH_CONTROLLED) return g.k >= 1 && g.k <= 3;
    return (g.path == SV_PATH_LOW || g.path == SV_PATH_HIGH || g.path == SV_PATH_MIXED) && g.k >= 1 && g.k <= 5 && g.cmask == 0;
}

uint64_t named(const FusedGate &g)
{
    uint64_t q = g.mask | g.cmask;
    for (const FusedGate::PostTerm &t : g.post) q |= uint64_t(1) << t.q;
    return q;   // a swap network's mask already holds its qubits
}

size_t mat_floats(const FusedGate &g) { return size_t(2) << (2 * g.k); }

// the launch arguments of a pass over gates `idx` with the local qubits `lam` (bits 0-4 set)
void fill_stage(const std::vector<const FusedGate *> &gates, const std::vector<int> &idx, uint64_t lam, int n, StageHead *a,
                float *mat)
{
    std::memset(a, 0, sizeof(*a));
    int local_of[64];
    int L = 0;
    for (int q = 0; q < n; ++q)
        if ((lam >> q) & 1) local_of[q] = L++;
    fill_geom(lam, n, &a->t);
    a->n_gates = (int)idx.size();
    size_t at = 0;
    for (size_t s = 0; s < idx.size(); ++s) {
        const FusedGate &g = *gates[(size_t)idx[s]];
        StageGate &o = a->g[s];
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
        std::vector<int> free_bits, order;
        for (int t = 0; t < L; ++t)
            if (!((used >> t) & 1)) free_bits.push_back(t);
        lane_bits(free_bits, &order);
        o.nb = (unsigned char)order.size();
        for (size_t b = 0; b < order.size(); ++b) o.gv[b] = (unsigned short)addr_vec(order[b]);
        o.moff = (unsigned short)(at / 4);
        const int D = 1 << g.k;
        for (int j = 0; j < D; ++j)
            for (int p = 0; p < D / 2; ++p) {
                const size_t e0 = size_t(2 * p) * D + j, e1 = e0 + D;
                mat[at++] = g.ur[e0];
                mat[at++] = g.ur[e1];
                mat[at++] = g.ui[e0];
                mat[at++] = g.ui[e1];
            }
    }
}

}  // namespace

void plan_passes(const std::vector<const FusedGate *> &gates, int n, PassPlan *plan)
{
    plan->steps.clear();
    std::vector<int> left;
    bool reorder = true;
    for (size_t i = 0; i < gates.size(); ++i) {
        left.push_back((int)i);
        if (gates[i]->path == SV_PATH_TC_TF32 || gates[i]->path == SV_PATH_TC_BF16X3) reorder = false;
    }
    const int L = std::min(n, kStageQubits);
    while (!left.empty()) {
        PassStep st;
        uint64_t lam = 31, blocked = 0;
        size_t mats = 0;
        std::vector<int> took, rest;
        for (size_t s = 0; s < left.size(); ++s) {
            const FusedGate &g = *gates[(size_t)left[s]];
            const uint64_t q = named(g);
            const uint64_t with = lam | g.mask;
            // blocked qubits may appear outside a tile (controls) too, so every named qubit counts
            const bool joins = n >= 5 && stageable(g) && !(q & blocked) && __builtin_popcountll(with) <= L &&
                               (int)took.size() < kStageMaxGates && mats + mat_floats(g) <= size_t(kStageMatFloats);
            if (joins) {
                lam = with;
                mats += mat_floats(g);
                took.push_back(left[s]);
                continue;
            }
            if (took.empty()) {   // the first gate left runs alone
                took.push_back(left[s]);
                rest.insert(rest.end(), left.begin() + (long)s + 1, left.end());
                break;
            }
            blocked |= q;
            rest.push_back(left[s]);
            if (!reorder) {
                rest.insert(rest.end(), left.begin() + (long)s + 1, left.end());
                break;
            }
        }
        if (took.size() == 1) {
            st.single = took[0];
        } else {
            for (int q = 5; q < n && __builtin_popcountll(lam) < L; ++q) lam |= uint64_t(1) << q;   // whole tiles: lowest free qubits
            st.form = mats <= size_t(kStageMat[0]) ? 0 : mats <= size_t(kStageMat[1]) ? 1 : 2;
            st.tiles = 1ll << (n - L);
            st.args.assign((sizeof(StageHead) + sizeof(float) * (size_t)kStageMat[st.form]) / 8, 0);
            StageHead *h = reinterpret_cast<StageHead *>(st.args.data());
            fill_stage(gates, took, lam, n, h, reinterpret_cast<float *>(h + 1));
        }
        plan->steps.push_back(std::move(st));
        left.swap(rest);
    }
}

namespace {

template <int T, int V, int M>
int launch_form(float *sv, const PassStep &p, cudaStream_t stream)
{
    static_assert(sizeof(StageArgs<M>) == sizeof(StageHead) + sizeof(float) * M, "a step's argument block is the kernel's");
    const StageArgs<M> *a = reinterpret_cast<const StageArgs<M> *>(p.args.data());
    const size_t smem = sizeof(float) * (size_t(64) << a->h.t.fb);
    static_assert((8 << kStageQubits) <= 48 * 1024, "tiles need no shared-memory attribute");
    void *args[2] = {&sv, const_cast<StageArgs<M> *>(a)};
    SV_CUDA_TRY(cudaLaunchKernel(reinterpret_cast<const void *>(stage_kernel<T, V, M>), dim3((unsigned)p.tiles), dim3(T), args, smem, stream));
    return SV_OK;
}

template <int M>
int launch_mat(float *sv, const PassStep &p, cudaStream_t stream, int num_sms)
{
    // With few tiles a pass is a chain of short gates, so each tile gets all the threads an SM
    // takes; with many, small CTAs of two groups a thread share an SM and overlap each other's
    // loads, barriers and arithmetic.
    if (p.tiles < 2ll * num_sms) return launch_form<512, 1, M>(sv, p, stream);
    return launch_form<128, 2, M>(sv, p, stream);
}

}  // namespace

int launch_stage(float *sv, const PassStep &p, cudaStream_t stream, int num_sms)
{
    switch (p.form) {
    case 0: return launch_mat<kStageMat[0]>(sv, p, stream, num_sms);
    case 1: return launch_mat<kStageMat[1]>(sv, p, stream, num_sms);
    default: return launch_mat<kStageMat[2]>(sv, p, stream, num_sms);
    }
}

}  // namespace svg
