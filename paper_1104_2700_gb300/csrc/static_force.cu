// nb_force_static: the force evaluation (Eqs. acc, jrk, pot, double-single
// pair arithmetic) for callers that cannot allocate device memory.
//
// The regular entry points keep their buffers in a context that
// nb_set_particles sizes with cudaMalloc.  Some callers cannot do that:
// code that runs where the allocator is not available or not allowed,
// such as a host framework that owns all device memory and forbids other
// allocations, or a process that has reserved the whole GPU for itself.
// This entry point takes the caller's device arrays and uses, as its only
// working memory, one file-scope device array of fixed size
// (NB_STATIC_SCRATCH_BYTES): the j layout the force kernel streams, the
// partial sums of i-groups split across warps, their arrival counters and a
// status word.  It calls no cudaMalloc, cudaFree or allocating library
// routine.
#include <cstdio>
#include <mutex>

#include "nb_device.cuh"
#include "nb_launch.h"
#include "nbody.h"
#include "predict.cuh"

namespace {

// The working memory.  Every GPU that loads this library holds it until the
// process exits.  In host code the name is only a stand-in for the symbol:
// its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char nb_static_scratch[NB_STATIC_SCRATCH_BYTES];

constexpr int STATIC_CTAS_PER_SM = 4;  // fixes the number of warps, hence the scratch size
constexpr int MAX_DEVICES = 64;
constexpr size_t CONTROL_BYTES = 256;  // status word, layout bounds

struct DeviceSetup {
    bool ready = false;
    unsigned char* base = nullptr;  // device address of nb_static_scratch
    int grid = 0;                   // force CTAs
};
DeviceSetup g_setup[MAX_DEVICES];
std::mutex g_mutex;

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

struct Plan {
    size_t counters, layout, scratch, total;
    int64_t n_pad, counter_stride, counter_words;
};

Plan plan_for(int64_t n, int grid)
{
    Plan p;
    const int warps = grid * nb::FORCE_WARPS;
    p.n_pad = (n + nb::TJ - 1) / nb::TJ * nb::TJ;
    p.counter_stride = nb::force_counter_stride(n, warps);
    p.counter_words = nb::force_counter_entries(n, warps);
    p.counters = CONTROL_BYTES;
    p.layout = align256(p.counters + p.counter_words * sizeof(uint32_t));
    p.scratch = align256(p.layout + 4 * p.n_pad * 16);
    p.total = p.scratch + nb::force_scratch_doubles(1, n, warps) * sizeof(double);
    return p;
}

__device__ __noinline__ void split_fp64(double x, uint32_t bound, float& hi, float& lo)
{
    nb::grid_split(x, nb::grid_quantum(bound), hi, lo);
}

// grid_split of x on the grid of `bound`, the same bits, on the FP32 and integer
// pipes: |x| is cut exactly into its leading 24 bits and the other 29 (rest),
// rounded to the grid from both, and the difference summed from exact parts.
// Zeros are common (a cold start); a grid or an x whose parts leave FP32's
// normal range takes the FP64 form.
__device__ __forceinline__ void split(double x, uint32_t bound, float& hi, float& lo)
{
    const uint32_t hw = static_cast<uint32_t>(__double2hiint(x));
    const uint32_t lw = static_cast<uint32_t>(__double2loint(x));
    if (((hw & 0x7fffffffu) | lw) == 0u) {
        hi = lo = 0.f;
        return;
    }
    const uint32_t e = (hw >> 20) & 0x7ffu, eb = (bound >> 23) & 0xffu;
    // |x| outside [2^-60, 2^61), or the grid's quantum outside [2^-121, 2^105]
    if (e - (1023u - 60u) > 120u || eb - 27u > 226u) {
        split_fp64(x, bound, hi, lo);
        return;
    }
    float q, iq;
    nb::grid_quantum_f(bound, q, iq);
    const float xh =
        __uint_as_float(((e - 1023u + 127u) << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29));
    const uint32_t rest = lw & 0x1fffffffu;
    const float unit = __uint_as_float((e - 1075u + 127u) << 23);  // of rest
    const float t = xh * iq;
    float k = rintf(t);
    if (t - k == 0.5f && rest) k += 1.f;  // not a tie
    const float h = k * q;
    float s, err;
    nb::two_sum(__fsub_rn(xh, h), __uint2float_rn(rest >> 5) * (32.f * unit), s, err);
    const float l = __fadd_rn(s, __fadd_rn(err, __uint2float_rn(rest & 31u) * unit));
    hi = (hw >> 31) ? -h : h;
    lo = (hw >> 31) ? -l : l;
}

// Predicted particles (device, n x 3 doubles) -> the double-single j layout
// (grid-aligned splits on the grids of `bound`), with zero-mass ghosts far
// away up to n_pad.  Four groups of 64 threads per tile, one per component and
// one for the masses, as the predictor kernels, and the splits on the FP32
// pipes: with FP64 splits the call took 82.8 us at n = 8192, 500 active, and
// 86.9 with all of a particle in one thread.
__global__ void __launch_bounds__(4 * nb::TJ)
    static_layout_kernel(int64_t n, const double* m, const double* r, const double* v, double G,
                         const uint32_t* bound, float4* L, int64_t n_pad)
{
    __shared__ __align__(16) float rec[4][nb::TJ * 4];
    const int c = threadIdx.x / nb::TJ, slot = threadIdx.x % nb::TJ;
    const int64_t i = (int64_t)blockIdx.x * nb::TJ + slot;
    if (c < 3) {
        float xh = static_cast<float>(nb::GHOST_POS), xl = 0.f, vh = 0.f, vl = 0.f;
        if (i < n) {
            split(r[3 * i + c], bound[0], xh, xl);
            split(v[3 * i + c], bound[1], vh, vl);
        }
        rec[0][4 * slot + c] = xh;
        rec[1][4 * slot + c] = xl;
        rec[2][4 * slot + c] = vh;
        rec[3][4 * slot + c] = vl;
    } else {
        // (in FP64: m alone may lie outside the range of a float)
        const double gm = i < n ? G * m[i] : 0.0;
        const float hi = __double2float_rn(gm);
        rec[0][4 * slot + 3] = hi;
        rec[1][4 * slot + 3] = __double2float_rn(gm - static_cast<double>(hi));
        rec[2][4 * slot + 3] = 0.f;
        rec[3][4 * slot + 3] = 0.f;
    }
    __syncthreads();
    L[c * n_pad + i] = reinterpret_cast<const float4*>(rec[c])[slot];
}

// One-time set-up for the current device: the symbol's device address and
// the force kernel's launch shape.
nb_status setup_device(int dev, DeviceSetup*& out)
{
    if (dev < 0 || dev >= MAX_DEVICES) return NB_EINVAL;
    std::lock_guard<std::mutex> lock(g_mutex);
    DeviceSetup& s = g_setup[dev];
    if (!s.ready) {
        void* addr = nullptr;
        if (cudaGetSymbolAddress(&addr, nb_static_scratch) != cudaSuccess) return NB_ECUDA;
        if (nb::force_setup(nb::Prec::DS, 1, 1) != cudaSuccess) return NB_ECUDA;
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return NB_ECUDA;
        int per_sm = nb::force_ctas_per_sm(nb::Prec::DS, 1, 1);
        if (per_sm < 1) return NB_ECUDA;
        if (per_sm > STATIC_CTAS_PER_SM) per_sm = STATIC_CTAS_PER_SM;
        // The scratch of the split-group sums grows with the number of
        // persistent warps; shrink the grid until the largest system allowed
        // fits the array, so the limit on n holds whatever the SM count: by
        // whole CTAs per SM first (350 CTAs on 152 SMs, where 304 fit evenly,
        // cost a block of 500 of 8192 particles 12 us of its 60).
        while (per_sm > 1 &&
               plan_for(NB_STATIC_MAX_N, per_sm * sms).total > NB_STATIC_SCRATCH_BYTES)
            --per_sm;
        int grid = per_sm * sms;
        while (grid > 1 && plan_for(NB_STATIC_MAX_N, grid).total > NB_STATIC_SCRATCH_BYTES)
            grid -= grid / 8 > 0 ? grid / 8 : 1;
        s.base = static_cast<unsigned char*>(addr);
        s.grid = grid;
        s.ready = true;
    }
    out = &s;
    return NB_OK;
}

}  // namespace

extern "C" nb_status nb_force_static(int64_t n, const double* m, const double* r,
                                     const double* v, double eps, double G, int32_t n_act,
                                     const int32_t* idx, double* acc, double* jerk,
                                     double* pot, void* stream)
{
    if (n < 1 || n > NB_STATIC_MAX_N) {
        std::fprintf(stderr, "nb_force_static: n = %lld outside [1, %d]\n",
                     static_cast<long long>(n), NB_STATIC_MAX_N);
        return NB_EINVAL;
    }
    if (n_act < 0 || n_act > n) {
        std::fprintf(stderr, "nb_force_static: n_act = %d outside [0, n]\n", n_act);
        return NB_EINVAL;
    }
    if (!m || !r || !v || (n_act > 0 && (!idx || !acc || !jerk || !pot))) return NB_EINVAL;
    if (!(eps >= 0.0)) return NB_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NB_ECUDA;
    DeviceSetup* s = nullptr;
    nb_status st = setup_device(dev, s);
    if (st != NB_OK) return st;
    const Plan p = plan_for(n, s->grid);
    if (p.total > NB_STATIC_SCRATCH_BYTES) {
        std::fprintf(stderr, "nb_force_static: needs %zu bytes of scratch, has %d\n", p.total,
                     NB_STATIC_SCRATCH_BYTES);
        return NB_EINVAL;
    }
    if (n_act == 0) return NB_OK;
    cudaStream_t cs = static_cast<cudaStream_t>(stream);
    uint32_t* status = reinterpret_cast<uint32_t*>(s->base);
    uint32_t* bound = reinterpret_cast<uint32_t*>(s->base + 8);
    uint32_t* counters = reinterpret_cast<uint32_t*>(s->base + p.counters);
    float4* L = reinterpret_cast<float4*>(s->base + p.layout);
    double* scratch = reinterpret_cast<double*>(s->base + p.scratch);
    // The array keeps whatever the previous call left: the status word, the
    // layout bounds and the arrival counters must start from zero.
    // (one stretch from the start of the array)
    if (cudaMemsetAsync(s->base, 0, p.counters + p.counter_words * sizeof(uint32_t), cs) !=
        cudaSuccess)
        return NB_ECUDA;
    if (nb::bounds_launch(r, v, 3 * n, bound, cs) != cudaSuccess) return NB_ECUDA;
    static_layout_kernel<<<static_cast<unsigned>(p.n_pad / nb::TJ), 4 * nb::TJ, 0, cs>>>(
        n, m, r, v, G, bound, L, p.n_pad);
    if (cudaGetLastError() != cudaSuccess) return NB_ECUDA;
    nb::ForceArgs f;
    f.prec = nb::Prec::DS;
    f.it = 1;
    for (int k = 0; k < 4; ++k) f.jl.arr[k] = L + k * p.n_pad;
    f.n = n;
    f.n_pad = p.n_pad;
    f.idx = idx;
    f.acc = acc;
    f.jerk = jerk;
    f.pot = pot;
    f.scratch = scratch;
    f.counters = counters;
    f.counter_stride = p.counter_stride;
    f.status = status;
    f.eps2 = eps * eps;
    f.grid = s->grid;
    f.n_act_host = n_act;
    f.cta_mode = 1;
    if (nb::force_launch(f, cs) != cudaSuccess) return NB_ECUDA;
    uint32_t host_status = 0;
    if (cudaMemcpyAsync(&host_status, status, sizeof(host_status), cudaMemcpyDeviceToHost, cs) !=
            cudaSuccess ||
        cudaStreamSynchronize(cs) != cudaSuccess)
        return NB_ECUDA;
    if (host_status & nb::ST_BADINDEX) return NB_EINVAL;
    if (host_status & nb::ST_TIMEOUT) return NB_ETIMEOUT;
    return NB_OK;
}
