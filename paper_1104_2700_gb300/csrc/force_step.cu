// Steps 1-4 of a block step of a small system in one launch: the next block
// time and its block, the prediction, and the force on the block.
//
// At a thousand particles a block step's kernels are latency: launches,
// dependent loads, and instructions run once by a cold SM (~13 cycles each in
// straight-line code, where a warm one takes ~1.3).  Beside a force launch of
// ~10 us, select and predictor take 2.5 + 2.4 us of a 22.4 us block step.  Here
// every CTA selects the block itself, and stages the j tiles it sums by
// predicting them: a warp per component, in a loop over 32-particle chunks, so
// that the code is short and fetched once.  A tile is then summed by the CTA's
// four warps: a near tile a quarter of the records each, a far tile (one FP32
// run of 64) whole by one of them.  The price is the select in every CTA and
// the prediction again for every i-group; STEP_MAX_N says where that pays.
#include <math_constants.h>

#include "force_kernel.cuh"
#include "predict.cuh"

namespace nb {
namespace {

constexpr int ST_WARPS = FORCE_WARPS;
constexpr int ST_THREADS = ST_WARPS * 32;
constexpr int ST_TILES = 4;  // tiles staged at a time
static_assert(ST_WARPS == 4, "a warp per component and one for the masses");
static_assert(STEP_MAX_N <= 32 * ST_THREADS, "a mask bit per key of a thread");

// Shared memory: the warps' areas for cta_finish, the staged tiles, one more
// tile for the i particles (its first 32 records), the block.
template <class K>
struct StepSmem {
    // (near pairs' pieces and, after the tiles, the sums share an area)
    static constexpr int SUMS = (K::NV * 32 * 8 + 127) / 128 * 128;
    static constexpr int WARP =
        WarpSmem<K>::BAR_BYTES + (SUMS > K::PIECE_BYTES ? SUMS : K::PIECE_BYTES);
    static constexpr int TILE = TJ * 64;
    static constexpr int TILES = ST_WARPS * WARP;
    static constexpr int LIST = TILES + (ST_TILES + 1) * TILE;
    static constexpr int BYTES = LIST + STEP_MAX_N * (int)sizeof(uint16_t);
};

// Step 1: the smallest next-time key and the particles that have it, ascending,
// in `list`; CTA 0 also publishes them for the corrector.  Thread k owns
// particles k + 128 u: its smallest key and a mask of the u that reach it, then
// one ballot per u and a scan of the per-(u, warp) counts.  Returns n_act (0
// past t_end).
__device__ __forceinline__ int step_select(const ForceParams& f, uint16_t* list,
                                           unsigned long long& key)
{
    __shared__ unsigned long long wmin[ST_WARPS];
    __shared__ int cnt[ST_THREADS];  // 32 u x 4 warps
    __shared__ int wtot[ST_WARPS];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int n = static_cast<int>(f.n);
    const int rows = (n + ST_THREADS - 1) / ST_THREADS;
    const double t_end = f.t_end.get();
    unsigned long long best = ~0ull;
    uint32_t mask = 0u;
#pragma unroll 1
    for (int u0 = 0; u0 < rows; u0 += 8) {
        unsigned long long kk[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const int i = tid + ST_THREADS * (u0 + v);
            kk[v] = i < n ? __ldcg(f.st.nkey + i) : ~0ull;
        }
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            if (kk[v] < best) best = kk[v], mask = 0u;
            if (kk[v] == best) mask |= 1u << (u0 + v);
        }
    }
    unsigned long long low = best;
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, low, o);
        low = other < low ? other : low;
    }
    if (lane == 0) wmin[wid] = low;
    __syncthreads();
    low = wmin[0];
#pragma unroll
    for (int w = 1; w < ST_WARPS; ++w) low = wmin[w] < low ? wmin[w] : low;
    key = low;
    if (best != low || !(dkey_decode(low) <= t_end)) mask = 0u;
    uint32_t bal = 0u;  // lane u: the warp's ballot of row u
#pragma unroll 1
    for (int u = 0; u < rows; ++u) {
        const bool in = ((mask >> u) & 1u) && tid + ST_THREADS * u < n;
        const uint32_t b = __ballot_sync(0xffffffffu, in);
        if (lane == u) bal = b;
    }
    cnt[lane * ST_WARPS + wid] = __popc(bal);
    __syncthreads();
    const int mine = cnt[tid];
    int x = mine;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wtot[wid] = x;
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < ST_WARPS; ++w) {
        before += w < wid ? wtot[w] : 0;
        total += wtot[w];
    }
    cnt[tid] = before + x - mine;
    __syncthreads();
#pragma unroll 1
    for (int u = 0; u < rows; ++u) {
        const uint32_t b = __shfl_sync(0xffffffffu, bal, u);
        if ((b >> lane) & 1u) {
            const int pos = cnt[u * ST_WARPS + wid] + __popc(b & ((1u << lane) - 1u));
            const int i = tid + ST_THREADS * u;
            list[pos] = static_cast<uint16_t>(i);
            if (blockIdx.x == 0) f.sel_idx[pos] = i;
        }
    }
    if (blockIdx.x == 0 && tid == 0) {
        *f.sel_n_act = total;
        *f.sel_tmin = key;
    }
    __syncthreads();
    return total;
}

// Steps 2-3 of `chunks` chunks of 32 particles, particle_of(chunk, lane) (-1: a
// ghost), into chunk % 2 of the tile at tile_of(chunk): the records of the
// predictor kernel, bit for bit, with the tile's box after its second chunk.
template <class P, class T>
__device__ __forceinline__ void step_predict(const ForceParams& f, double t, int chunks,
                                             P particle_of, T tile_of)
{
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    const StateDev& st = f.st;
    const int64_t n = f.n;
    // every chunk's state on its way to this SM before the first is used
#pragma unroll 1
    for (int k = 0; k < chunks; ++k) {
        const int i = particle_of(k, lane);
        if (i < 0) continue;
        const double* p[5] = {st.t + i, st.x + c * n + i, st.v + c * n + i, st.a + c * n + i,
                              st.j + c * n + i};
        if (c == 3) p[0] = st.m + i;
#pragma unroll
        for (int e = 0; e < 5; ++e)
            if (e == 0 || c < 3) asm volatile("prefetch.global.L1 [%0];" ::"l"(p[e]));
    }
    float qx, iqx;
    grid_quantum_f(st.bound[0], qx, iqx);
    float lo_e = CUDART_INF_F, hi_e = -CUDART_INF_F;
#pragma unroll 1
    for (int k = 0; k < chunks; ++k) {
        const int i = particle_of(k, lane);
        float* A = reinterpret_cast<float*>(tile_of(k)) + 4 * (lane + 32 * (k & 1));
        float* B = A + 4 * TJ;
        float* C = B + 4 * TJ;
        float* D = C + 4 * TJ;
        if (c < 3) {
            float hi = static_cast<float>(GHOST_POS), lo = 0.f;
            Dsf v = {0.f, 0.f};
            if (i >= 0) {
                const int64_t e = c * n + i;
                const Dsf h = dsf_of(t - st.t[i]);  // exact: both times are dyadic
                const PredictedComp p =
                    predict_component(st.x[e], st.v[e], st.a[e], st.j[e], h, qx, iqx);
                hi = p.hi, lo = p.lo, v = p.v;
                lo_e = fminf(lo_e, hi), hi_e = fmaxf(hi_e, hi);
            }
            float vh, vl;
            split_velocity<true>(v, 0.f, 0.f, vh, vl);
            A[c] = hi, B[c] = lo, C[c] = vh, D[c] = vl;
        } else {
            const Dsf gm = i >= 0 ? dsf_mass(f.G, st.m[i]) : Dsf{0.f, 0.f};
            const float g = cbrtf(gm.hi);
            A[3] = gm.hi, B[3] = gm.lo, C[3] = g * g;
            if (lane >= 8 || (k & 1)) D[3] = 0.f;
            lo_e = fminf(lo_e, -gm.hi), hi_e = fmaxf(hi_e, g * g);
        }
        if (k & 1) {
#pragma unroll 1
            for (int o = 16; o > 0; o >>= 1) {
                lo_e = fminf(lo_e, __shfl_xor_sync(0xffffffffu, lo_e, o));
                hi_e = fmaxf(hi_e, __shfl_xor_sync(0xffffffffu, hi_e, o));
            }
            float* box = reinterpret_cast<float*>(tile_of(k)) + 12 * TJ + 3;
            if (lane == 0) {
                box[4 * c] = c < 3 ? lo_e : -lo_e;
                box[4 * (4 + c)] = hi_e;
            }
            lo_e = CUDART_INF_F, hi_e = -CUDART_INF_F;
        }
    }
}

template <class K>
__global__ void __launch_bounds__(ST_THREADS, K::MIN_CTAS) step_force_kernel(const ForceParams f)
{
    using M = StepSmem<K>;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    unsigned char* tiles = smem + M::TILES;
    uint16_t* list = reinterpret_cast<uint16_t*>(smem + M::LIST);
    unsigned long long key;
    const int na = step_select(f, list, key);
    if (na == 0) return;
    const double t_now = dkey_decode(key);
    UniformPlan plan;
    plan.template init<32>(f, na);
    const int G = static_cast<int>(plan.G), NT = static_cast<int>(plan.NT);
    // Each group gets R consecutive CTAs, each a stretch of its tile walk; with
    // more groups than CTAs a CTA takes several groups in turn.
    const int P = gridDim.x;
    int R = P / G;
    R = R < 1 ? 1 : R > NT ? NT : R;
    const int slots = P / R;
    const int crank = blockIdx.x % R;
    for (int g = blockIdx.x / R; g < G; g += slots) {
        if (static_cast<int>(blockIdx.x) >= slots * R) break;
        const GroupInfo gi = plan.group(g);
        const int act0 = static_cast<int>(gi.act_begin), acts = static_cast<int>(gi.act_count);
        const int c0 = NT * crank / R, c1 = NT * (crank + 1) / R;
        typename K::I is[1];
        typename K::Acc ac[1];
        ac[0].zero();
        bool guard_any = false;
        for (int b0 = c0; b0 < c1; b0 += ST_TILES) {
            const int nb = c1 - b0 < ST_TILES ? c1 - b0 : ST_TILES;
            const bool first = b0 == c0;
            // j tile of the walk's rank b0 + b; chunk 2 nb: the i particles
            auto jtile = [&](int b) { return static_cast<int>(tile_at(gi, b0 + b)); };
            __syncthreads();  // the last use of the staged tiles is over
            step_predict(
                f, t_now, 2 * nb + (first ? 1 : 0),
                [&](int k, int l) {
                    if (k == 2 * nb) return l < acts ? static_cast<int>(list[act0 + l]) : -1;
                    const int q = jtile(k >> 1) * TJ + 32 * (k & 1) + l;
                    return q < f.n ? q : -1;
                },
                [&](int k) { return tiles + (k == 2 * nb ? ST_TILES : k >> 1) * M::TILE; });
            __syncthreads();
            if (first) {
                const float4* r = reinterpret_cast<const float4*>(tiles + ST_TILES * M::TILE);
                const float4 A = r[lane], B = r[TJ + lane], C = r[2 * TJ + lane],
                             D = r[3 * TJ + lane];
                auto& s = is[0];
                s.p = lane < acts ? static_cast<int>(list[act0 + lane]) : -1;
                if (s.p >= 0) {
                    s.xh = A.x, s.yh = A.y, s.zh = A.z, s.xl = B.x, s.yl = B.y, s.zl = B.z;
                    s.vxh = C.x, s.vyh = C.y, s.vzh = C.z, s.vxl = D.x, s.vyl = D.y, s.vzl = D.z;
                } else {
                    s.xh = s.yh = s.zh = s.xl = s.yl = s.zl = 0.f;
                    s.vxh = s.vyh = s.vzh = s.vxl = s.vyl = s.vzl = 0.f;
                }
                K::limits_i(f, s.p, s);
                guard_any = __any_sync(0xffffffffu, K::guarded(s));
            }
            if (g == 0) {  // the layout in global memory, as the predictor leaves it
                const void* jl[4] = {f.jl0, f.jl1, f.jl2, f.jl3};
                for (int e = threadIdx.x; e < nb * TJ; e += ST_THREADS) {
                    const int64_t q = (int64_t)jtile(e / TJ) * TJ + e % TJ;
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        static_cast<float4*>(const_cast<void*>(jl[k]))[q] =
                            reinterpret_cast<const float4*>(tiles + (e / TJ) * M::TILE)[k * TJ + e % TJ];
                }
            }
#pragma unroll 1
            for (int b = 0; b < nb; ++b) {
                const unsigned char* buf = tiles + b * M::TILE;
                const int64_t j0 = (int64_t)jtile(b) * TJ;
                const bool mask_self =
                    __any_sync(0xffffffffu, is[0].p >= j0 && is[0].p < j0 + TJ);
                const int u0 = wib * (TJ / ST_WARPS), u1 = u0 + TJ / ST_WARPS;
                // (the same answer in every warp of the group: a block names no
                // particle twice, so no other group stores its noise estimate)
                bool far = !mask_self && !guard_any;
                if (far) far = __all_sync(0xffffffffu, K::tile_far(buf, is[0], gi.e2.h));
                if (far) {
                    if (((b0 + b) & 3) == wib) K::template far_tile<1>(buf, gi.e2, is, ac, 0);
                    continue;
                }
                uint32_t nlo[1], nhi[1];
                if (guard_any) {
                    if (mask_self)
                        K::template tile<true, true, 1>(buf, j0, gi.e2, is, ac, 0, u0, u1, nlo, nhi);
                    else
                        K::template tile<false, true, 1>(buf, j0, gi.e2, is, ac, 0, u0, u1, nlo,
                                                         nhi);
                } else {
                    if (mask_self)
                        K::template tile<true, false, 1>(buf, j0, gi.e2, is, ac, 0, u0, u1, nlo,
                                                         nhi);
                    else
                        K::template tile<false, false, 1>(buf, j0, gi.e2, is, ac, 0, u0, u1, nlo,
                                                          nhi);
                }
                K::template near_pass<1>(buf, gi.e2, is, ac, lane, nlo, nhi,
                                         reinterpret_cast<float2*>(smem + wib * M::WARP +
                                                                   WarpSmem<K>::BAR_BYTES));
            }
        }
        // (cta_finish starts with a barrier after its own area's stores; the
        // previous group's last reads of that area lie before the barriers above)
        cta_finish<K, 1, 1, M::WARP>(f, smem, is, ac, gi, g, R, crank);
    }
}

template <class K>
const void* step_k()
{
    return reinterpret_cast<const void*>(&step_force_kernel<K>);
}

}  // namespace

const void* step_kernel_ptr(Prec p)
{
    switch (p) {
    case Prec::HYBRID: return step_k<PolicyHybrid<1>>();
    case Prec::HYBRID_SPJ: return step_k<PolicyHybrid<1, true>>();
    default: return nullptr;
    }
}

size_t step_smem_bytes(Prec p)
{
    return step_kernel_ptr(p) ? StepSmem<PolicyHybrid<1>>::BYTES : 0;
}

}  // namespace nb
