// Several time steps of the stencil in one launch (kernel body: fwime_prop.cuh).
#include <algorithm>

#include "fwime_prop.cuh"

namespace fwk {

// ------------------------------------------------------------- several steps per launch
// A step of a few shots on a small grid is a launch of 5-8 us whatever its size (45 k points: 6.2 us, 667 k points:
// 8.2 us): about 5 us of host time per launch, and on the device the launch gap, the tail and one dependent chain of
// loads.  k_march runs a whole segment of steps in one cooperative launch of at most one CTA per SM: every warp owns
// a fixed share of the (shot, strip, chunk) items, and a grid-wide barrier separates the steps.  The fields stay in
// L2; reads of them go there (cp.async.cg, ld.cg), never through L1 or the read-only path.
//
// The barrier is a count of arrivals and a generation word; a flag per CTA that all others watch saved a hop but made
// every store of a flag wait for its watchers (9.1 against 4.4 us per step on 45 k points).  The spin is bounded:
// when it runs out the kernel latches ST_TIMEOUT and returns (fwime_sync then reports FWIME_ETIMEOUT).  A
// cooperative launch starts only with all its CTAs resident, so it does not run out because other streams hold SMs.
constexpr unsigned MARCH_SPINS = 4u << 20;   // about half a microsecond each
constexpr int MARCH_SMEM = 226 * 1024;       // 227 KB less the static word of the barrier
__device__ __forceinline__ bool grid_step_barrier(unsigned *bar, int *status)
{
    __shared__ int dead;
    __syncthreads();
    if (threadIdx.x == 0) {
        dead = 0;
        unsigned gen, old, now;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(gen) : "l"(bar + 1) : "memory");
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(bar) : "memory");
        if (old + 1 == gridDim.x) {             // the last one in: the count starts anew, then the others go on
            asm volatile("st.relaxed.gpu.global.u32 [%0], 0;" ::"l"(bar) : "memory");
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(bar + 1), "r"(gen + 1) : "memory");
        } else {
            unsigned spins = 0;
            do {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(bar + 1) : "memory");
            } while (now == gen && ++spins < MARCH_SPINS);
            if (now == gen) {
                atomicOr(status, ST_TIMEOUT);
                dead = 1;
            }
        }
    }
    __syncthreads();
    return dead == 0;
}

// The operands of one time step that change from step to step.
struct StepPtrs {
    const float *cur, *prev;
    float *out, *d2;
    const float *f0, *fc, *src_amp, *inj_val;
};

template <int LOC>
constexpr int march_warps() { return LOC == 2 ? 8 : 16; }       // 255 and 128 registers

template <int LOC, bool D2, bool SRC, bool INJ>
__global__ void __launch_bounds__(march_warps<LOC>() * 32, 1) k_march(const __grid_constant__ MarchArgs m)
{
    extern __shared__ float4 smem4[];
    const PropArgs &a = m.a;
    const int wic = warp_in_cta(), nw = gridDim.x * (blockDim.x >> 5);
    const int gw = blockIdx.x * (blockDim.x >> 5) + wic;
    float *wsm = reinterpret_cast<float *>(smem4) + wic * prop_smem(a.naux_max);
    for (int k = 0; k < m.nsteps; ++k) {
        StepPtrs sp{a.cur, a.prev, a.out, a.d2, a.f0, a.fc, a.src_amp, a.inj_val};
        if (m.R > 0) {                                          // adjoint ring, m descending
            const int mm = m.m0 - k;
            sp.cur = m.ring + ((mm + 1) % m.R) * m.rstride;
            sp.prev = m.ring + ((mm + 2) % m.R) * m.rstride;
            sp.out = m.ring + (mm % m.R) * m.rstride;
        } else if (k & 1) {
            sp.cur = a.out;
            sp.out = const_cast<float *>(a.cur);
            sp.prev = sp.out;
        }
        if (D2) sp.d2 += k * m.d2_step;
        if (LOC > 0) sp.f0 += k * m.f0_step;
        if (LOC == 2) sp.fc += k * m.fc_step;
        if (SRC) sp.src_amp += k;
        if (INJ) sp.inj_val += k * m.inj_step;
        if (a.rec_d) {                                          // receivers of the step's input
            for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m.S * a.nrec; i += gridDim.x * blockDim.x) {
                const int s = i / a.nrec, r = i - s * a.nrec;
                const float val = __ldcg(sp.cur + s * a.P + a.rec_off[r]);
                float *dp = a.rec_d + k * m.rec_step + s * a.rec_dstride + r;
                *dp = a.rec_acc ? *dp + val : val;
            }
        }
        for (int item = gw; item < m.nitem; item += nw) {
            const int shot = item / m.per_shot;
            prop_body<LOC, D2, SRC, INJ, false, true>(a, sp, item - shot * m.per_shot, shot, wsm);
            __syncwarp();                                       // the warp's rings are free again
        }
        if (k + 1 < m.nsteps && !grid_step_barrier(m.bar, m.status)) return;
    }
}

template <int LOC, bool D2, bool SRC, bool INJ>
static cudaError_t launch_march_t(const MarchArgs &m, int nsm, cudaStream_t st)
{
    static const cudaError_t attr =
        cudaFuncSetAttribute(k_march<LOC, D2, SRC, INJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, MARCH_SMEM);
    if (attr != cudaSuccess) return attr;
    const int per_warp = prop_smem(m.a.naux_max) * (int)sizeof(float);
    const int wmax = std::min(m.warps, MARCH_SMEM / per_warp);
    // a small problem in CTAs of four warps: fewer arrivals at the barrier, and still spread over many SMs (45 k points:
    // 3.80 us per step, with one warp per CTA 3.82, with eight 4.13, with sixteen 5.07)
    const int w = std::min(wmax, std::max(4, (m.nitem + nsm - 1) / nsm));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(std::min(nsm, (m.nitem + w - 1) / w));
    cfg.blockDim = dim3(32 * w);
    cfg.dynamicSmemBytes = (size_t)w * per_warp;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_march<LOC, D2, SRC, INJ>, m);
}

// Warps per CTA for `S` shots (one CTA per SM) and rows per warp's item; 0 where a launch per step is the better way,
// or the only one (f1, f2).  Eight warps where that leaves at most 10 rows (16 row costs) each: the step is then mostly
// the barrier and one chain of loads, and fewer warps arrive sooner (667 k points: 7.8 us per step, with sixteen 8.3).
// Up to 58 rows (64 row costs) per warp: beyond, the per-step launch's 16 warps per SM of 168 registers and its free
// order of items make up for the launches (170 x 920 points,
// steps of 8.2 against 10.0 us for 2 shots, 9.4 / 10.6 for 3, 11.3 / 12.6 for 4, 14.8 / 14.7 for 6).
constexpr int MARCH_COST8 = 16, MARCH_COST = 64;
static int march_shape(const PropArgs &a, int S, int nsm, int *zchunk)
{
    if (a.f1 || a.f2) return 0;
    const int rows = a.NZ - 4 - a.z_first;
    long long cost = 0;
    for (const int w : {8, 16}) {
        if (w == 16 && a.fc) break;             // (255 registers)
        *zchunk = chunk_rows(rows, a.nstrip, S, (long long)nsm * w, &cost);
        if (cost <= (w == 8 && !a.fc ? MARCH_COST8 : MARCH_COST)) return w;
    }
    return 0;
}

bool march_pays(const PropArgs &a, int S, int nsm)
{
    int zc = 0;
    return march_shape(a, S, nsm, &zc) > 0;
}

cudaError_t launch_march(const MarchArgs &m0, int nsm, cudaStream_t st)
{
    MarchArgs m = m0;
    PropArgs &a = m.a;
    prop_pairs(a);
    m.warps = march_shape(a, m.S, nsm, &a.zchunk);
    if (m.warps <= 0) return cudaErrorInvalidValue;
    const int rows = a.NZ - 4 - a.z_first;
    a.nchunk = (rows + a.zchunk - 1) / a.zchunk;
    m.per_shot = a.nstrip * a.nchunk;
    m.nitem = m.per_shot * m.S;
    a.naux_max = 2 + (a.f0 != nullptr) + (a.fc ? 2 : 0);
    const int key = (a.fc ? 2 : a.f0 ? 1 : 0) * 8 + (a.d2 ? 4 : 0) + (a.src_off ? 2 : 0) + (a.inj_val ? 1 : 0);
    switch (key) {
    case 0: return launch_march_t<0, false, false, false>(m, nsm, st);
    case 1: return launch_march_t<0, false, false, true>(m, nsm, st);
    case 2: return launch_march_t<0, false, true, false>(m, nsm, st);
    case 4: return launch_march_t<0, true, false, false>(m, nsm, st);
    case 5: return launch_march_t<0, true, false, true>(m, nsm, st);
    case 6: return launch_march_t<0, true, true, false>(m, nsm, st);
    case 8: return launch_march_t<1, false, false, false>(m, nsm, st);
    case 12: return launch_march_t<1, true, false, false>(m, nsm, st);
    case 16: return launch_march_t<2, false, false, false>(m, nsm, st);
    case 20: return launch_march_t<2, true, false, false>(m, nsm, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace fwk
