// Two time steps of the stencil in one launch (arithmetic: fwime_prop.cuh).
#include <algorithm>

#include "fwime_prop.cuh"

namespace fwk {

// The stencil is bound by memory: 12 B per point and step, each field read or written once per launch.  Two steps per
// launch read q^n and q^{n-1} and write q^{n+1} and q^{n+2}: 16 B instead of 24.  A warp marches down its strip as
// k_prop does, computes row y of the first step, keeps those rows in a second register queue and computes row y - 4 of
// the second step from it; four rows above and below its chunk and four columns left and right of its strip are
// computed twice (250 instructions per row and pair on 120 columns; k_prop spends 139 per row and step on 128).
// Same products and sums in the same order as k_prop: the same bits.
//
// What it took: every ring slot a compile-time constant (rings of nine rows, the period of the unrolled queues), a
// warp index that the compiler knows to be uniform, running offsets and one barrier per row (with addresses computed
// per row 91 ms where this takes 51 and k_prop 67: forward, 100 shots on 458 x 1808 points, 399 steps); registers
// for two CTAs of four warps per SM, of which three fit (bounded to 168: 60 ms), four rows in flight (three: 59).
constexpr int PAIR_WARPS = 4, PAIR_MINB = 2;
constexpr int PAIR_STRIP = STRIP - 8;        // columns that a warp writes: the first step's halo costs it two lanes
constexpr int PAIR_RING = 9;                 // rows per ring
constexpr int PAIR_LRING = 3;                // rows per ring of the local sources
constexpr int PAIR_DEPTH = 4;                // rows in flight

// Floats of shared memory per warp: rows of q^n with their x-halos, c, q^{n-1} (then q^{n+1}, with room for the reads
// of the outer lanes' neighbours), local sources of both steps.
__host__ __device__ constexpr int pair_smem(int loc)
{
    return PAIR_RING * (CUR_ROW + 2 * STRIP) + 8 + loc * 2 * PAIR_LRING * STRIP;
}

template <int LOC, bool D2, bool SRC, bool INJ>
__global__ void __launch_bounds__(PAIR_WARPS * 32, PAIR_MINB) k_prop_pair(const __grid_constant__ PairArgs m)
{
    extern __shared__ float4 smem4[];
    const PropArgs &a = m.a;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int shot = blockIdx.y;
    const long long so = (long long)shot * a.P;
    if (a.rec_d && blockIdx.x == 0) {         // receivers of the inputs: row n, and row n - 1 where a pair wrote it
        for (int r = threadIdx.x; r < a.nrec; r += PAIR_WARPS * 32) {
            const long long o = so + a.rec_off[r];
            float *dp = a.rec_d + shot * a.rec_dstride + r;
            const float v1 = a.cur[o];
            *dp = a.rec_acc ? *dp + v1 : v1;
            if (m.rec_prev) {
                const float v0 = a.prev[o];
                dp -= a.nrec;
                *dp = a.rec_acc ? *dp + v0 : v0;
            }
        }
    }
    const int lane = threadIdx.x & 31;
    const int wic = warp_in_cta();
    const int wid = blockIdx.x * PAIR_WARPS + wic;
    if (wid >= a.nstrip * a.nchunk) return;   // warp-uniform
    const int NXP = a.NXP;
    const int strip = wid % a.nstrip, chunk = wid / a.nstrip;
    const int x0 = strip * PAIR_STRIP - 4;
    const int x = x0 + lane * 4;
    const int z0 = 4 + chunk * a.zchunk, z1 = min(z0 + a.zchunk, a.NZ - 4);
    const bool xin = x >= 0 && x < NXP;
    const bool own = xin && lane >= 1 && lane < 31;
    // the lane's places in the rings
    float *curL = reinterpret_cast<float *>(smem4) + wic * pair_smem(LOC) + 4 * lane;
    float *cL = curL + PAIR_RING * CUR_ROW, *midL = cL + PAIR_RING * STRIP + 4, *fL = midL + PAIR_RING * STRIP + 4;
    // the lane's columns: of the q^n row with its halo, of the row's end (two lanes), its own; a column outside reads
    // nothing (zero-filled)
    const int cA = x0 - 4 + 4 * lane, cB = cA + STRIP;
    const int nA = cA >= 0 && cA + 4 <= NXP ? 16 : 0, nB = cB + 4 <= NXP ? 16 : 0, nX = xin ? 16 : 0;
    const bool two = lane < CUR_ROW / 4 - 32;
    // Odd chunks march up: both sides of a boundary between chunks are then read at the same time, and the rows that
    // two chunks read come from memory once (-2 to -4 %).  A sum of two mirrored rows has the same bits either way.
    const int dz = (chunk & 1) ? -1 : 1, NX = dz * NXP;
    const int y0 = dz > 0 ? z0 - 4 : z1 + 3, ye = dz > 0 ? z1 + 4 : z0 - 5;   // rows of the first step
    int oA = y0 * NXP + (nA ? cA : 0), oB = y0 * NXP + (nB ? cB : 0), oX = y0 * NXP + (nX ? x : 0);
    const float *cur = a.cur + so, *prev = a.prev + so;
    // Row k of q^n after row y (and the offsets) into slot s.  Rows outside the grid are not read: what the rows that
    // depend on them make of the slot's old contents is replaced by zero.
    const int yend = dz > 0 ? min(a.NZ, z1 + 8) : max(-1, z0 - 9);
    const auto issue_cur = [&](int y, int k, int s) {
        if ((y + k * dz - yend) * dz >= 0) return;
        const float *src = cur + (long long)k * NX;
        cp16n(curL + s * CUR_ROW, src + oA, nA);
        if (two) cp16n(curL + s * CUR_ROW + STRIP, src + oB, nB);
    };
    const auto issue_aux = [&](int y, int k, int s) {
        if ((y + k * dz - ye) * dz >= 0) return;
        cp16n(cL + s * STRIP, a.c + (long long)k * NX + oX, nX);
        cp16n(midL + s * STRIP, prev + (long long)k * NX + oX, nX);
    };
    const auto issue_f = [&](int y, int k, int s) {
        const int zr = y + k * dz, zr2 = zr - 4 * dz;
        if ((zr - ye) * dz >= 0) return;
        const bool lin = zr >= a.zs_lo && zr < a.zs_hi, lin2 = zr2 >= a.zs_lo && zr2 < a.zs_hi;
        cp16n(fL + s * STRIP, a.f0 + so + (lin ? (long long)k * NX + oX : 0), lin ? nX : 0);
        cp16n(fL + (PAIR_LRING + s) * STRIP, m.f0b + so + (lin2 ? (long long)(k - 4) * NX + oX : 0), lin2 ? nX : 0);
    };

    // queue of q^n: rows y-4 .. y+3 for the first y; queue of q^{n+1}: rows y-8 .. y-1, none yet
    float4 q[9], p[9];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int zr = y0 + (k - 4) * dz;
        q[k] = xin && zr >= 0 && zr < a.NZ ? ldcg4(cur + (k - 4) * NX + oX) : f4zero();
        p[k] = f4zero();
    }
#pragma unroll
    for (int g = 0; g < PAIR_DEPTH; ++g) {
        if (g < 4) issue_cur(y0, g, g);
        issue_cur(y0, g + 4, g + 4);
        issue_aux(y0, g, g);
        if (LOC == 1 && g < PAIR_LRING) issue_f(y0, g, g);
        cp_commit();
    }
    const float4 gxv = xin ? ldg4(a.gx + x) : f4zero();
    int srow = -1, scol = -1;                 // the point source's row, and its column within this lane's four
    float amp = 0.f, amp2 = 0.f;
    if (SRC) {
        const int off = a.src_off[shot];
        srow = off / NXP;
        scol = off - srow * NXP - x;
        if (scol < 0 || scol > 3) srow = -1;
        amp = a.src_amp[(long long)shot * a.src_stride] * a.src_scale;
        amp2 = a.src_amp[(long long)shot * a.src_stride + 1] * a.src_scale;
    }
    float *out1 = a.out + so, *out2 = m.out2 + so - 4LL * NX;
    float *d1 = D2 ? a.d2 + so : nullptr, *d2b = D2 ? m.d2b + so - 4LL * NX : nullptr;

    // Row y of the first step and row y - 4 of the second.  The queues' logical rows k lie in q[(k + R) % 9] and
    // p[(k + R) % 9], the rings' row y in slot R.
#define FWIME_PAIR_ROW(R)                                                                                    \
    {                                                                                                        \
        cp_wait<(LOC ? PAIR_LRING : PAIR_DEPTH) - 1>();                                                      \
        __syncwarp();                                                                                        \
        issue_cur(y, 4 + PAIR_DEPTH, (4 + PAIR_DEPTH + (R)) % 9);                                            \
        issue_aux(y, PAIR_DEPTH, (PAIR_DEPTH + (R)) % 9);                                                    \
        if (!LOC) cp_commit();                                                                               \
        float4 lf0 = f4zero(), lf1 = f4zero();                                                               \
        if (LOC == 1) {                                                                                      \
            lf0 = lds4(fL + ((R) % PAIR_LRING) * STRIP);                                                     \
            lf1 = lds4(fL + (PAIR_LRING + (R) % PAIR_LRING) * STRIP);                                        \
        }                                                                                                    \
        {                                                                                                    \
            q[(8 + (R)) % 9] = lds4(curL + ((R) + 4) % 9 * CUR_ROW + 4);                                     \
            const float4 L = lds4(curL + (R) * CUR_ROW), Rr = lds4(curL + (R) * CUR_ROW + 8);                \
            const float4 pv = lds4(midL + (R) * STRIP), cv = lds4(cL + (R) * STRIP);                         \
            const int sj = SRC && y == srow ? scol : -1;                                                     \
            float4 o, d2;                                                                                    \
            row_math<LOC, D2, SRC>(a, prop_k(a), L, q[(0 + (R)) % 9], q[(1 + (R)) % 9], q[(2 + (R)) % 9],    \
                                   q[(3 + (R)) % 9], q[(4 + (R)) % 9], q[(5 + (R)) % 9], q[(6 + (R)) % 9],   \
                                   q[(7 + (R)) % 9], q[(8 + (R)) % 9], Rr, pv, cv, lf0, f4zero(), f4zero(),  \
                                   f4zero(), f4zero(), __ldg(a.gz + y), gxv, sj, amp, o, d2);                \
            if (INJ && y >= a.inj_lo && y < a.inj_hi && xin) inject_row<D2>(a, a.inj_val, shot, y, x, cv, o, d2); \
            if (y < 4 || y >= a.NZ - 4) o = f4zero();  /* rows that no step updates */                       \
            p[(8 + (R)) % 9] = o;                                                                            \
            *reinterpret_cast<float4 *>(midL + (R) * STRIP) = o;                                             \
            if (own && y >= z0 && y < z1) {                                                                  \
                st4(out1 + oX, o);                                                                           \
                if (D2 && y >= a.zs_lo && y < a.zs_hi) st4(d1 + oX, d2);                                     \
            }                                                                                                \
        }                                                                                                    \
        if (LOC) {                                                                                           \
            __syncwarp();                                                                                    \
            issue_f(y, PAIR_LRING, (R) % PAIR_LRING);                                                        \
            cp_commit();                                                                                     \
        }                                                                                                    \
        const int yw = y - 4 * dz;                                                                           \
        if (yw >= z0 && yw < z1) {                                                                           \
            constexpr int W = ((R) + 5) % 9;                                                                 \
            const float4 L = lds4(midL + W * STRIP - 4), Rr = lds4(midL + W * STRIP + 4);                    \
            const float4 cv = lds4(cL + W * STRIP);                                                          \
            const int sj = SRC && yw == srow ? scol : -1;                                                 \
            float4 o, d2;                                                                                    \
            row_math<LOC, D2, SRC>(a, prop_k(a), L, p[(0 + (R)) % 9], p[(1 + (R)) % 9], p[(2 + (R)) % 9],    \
                                   p[(3 + (R)) % 9], p[(4 + (R)) % 9], p[(5 + (R)) % 9], p[(6 + (R)) % 9],   \
                                   p[(7 + (R)) % 9], p[(8 + (R)) % 9], Rr, q[(0 + (R)) % 9], cv, lf1,        \
                                   f4zero(), f4zero(), f4zero(), f4zero(), __ldg(a.gz + yw), gxv, sj, amp2, o, d2);              \
            if (INJ && yw >= a.inj_lo && yw < a.inj_hi && xin)                                               \
                inject_row<D2>(a, m.inj_val2, shot, yw, x, cv, o, d2);                                       \
            if (own) {                                                                                       \
                st4(out2 + oX, o);                                                                           \
                if (D2 && yw >= a.zs_lo && yw < a.zs_hi) st4(d2b + oX, d2);                                  \
            }                                                                                                \
        }                                                                                                    \
        y += dz;                                                                                             \
        oA += NX;                                                                                            \
        oB += NX;                                                                                            \
        oX += NX;                                                                                            \
        if (y == ye) break;                                                                                  \
    }
    int y = y0;
    for (;;) {
        FWIME_PAIR_ROW(0) FWIME_PAIR_ROW(1) FWIME_PAIR_ROW(2) FWIME_PAIR_ROW(3) FWIME_PAIR_ROW(4)
        FWIME_PAIR_ROW(5) FWIME_PAIR_ROW(6) FWIME_PAIR_ROW(7) FWIME_PAIR_ROW(8)
    }
#undef FWIME_PAIR_ROW
    cp_wait<0>();
}

template <int LOC, bool D2, bool SRC, bool INJ>
static cudaError_t launch_pair_t(const PairArgs &m, int nshot, cudaStream_t st)
{
    // Shared memory for the three CTAs that the registers allow, the rest to L1, whatever the launch before had: right
    // behind k_prop, which takes all of it, pairs took 54.3 ms where they take 51.1 (a launch that follows without a
    // gap keeps the split unless it asks for another).
    constexpr int cta = sizeof(float) * PAIR_WARPS * pair_smem(LOC) + 1024, carve = (3 * cta * 100 + 233471) / 233472 + 1;
    static PerDevice<cudaError_t> attr;
    const cudaError_t e = attr.get([] {
        const auto k = k_prop_pair<LOC, D2, SRC, INJ>;
        const cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        return r != cudaSuccess ? r : cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, carve);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((m.a.nstrip * m.a.nchunk + PAIR_WARPS - 1) / PAIR_WARPS, nshot);
    cfg.blockDim = dim3(PAIR_WARPS * 32);
    cfg.dynamicSmemBytes = sizeof(float) * PAIR_WARPS * pair_smem(LOC);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;                         // as k_prop's launches
    return cudaLaunchKernelEx(&cfg, k_prop_pair<LOC, D2, SRC, INJ>, m);
}

// The steps that occur in long runs: with the point source, one dense local source or injection at the receivers, with
// or without D2t; no free surface (its rows would have to be mirrored between the two steps).
bool pair_runs(const PropArgs &a)
{
    return (a.src_off != nullptr) + (a.f0 != nullptr) + (a.inj_val != nullptr) == 1 && !a.f1 && !a.f2 && !a.fc &&
           a.fs_row == 0 && a.P < (1LL << 31);
}

// From where a step's three fields no longer stay in this chip's L2 (129 MB); below it saves no traffic (us per step,
// one launch per step and with pairs: 350 x 1700 points, 8 shots 15.8 / 16.4, 16 shots 28.9 / 29.6, 24 shots 45.1 /
// 37.6, 32 shots 55.6 / 46.8; 1200 x 5000 points, 1 shot 17.5 / 22.5, 2 shots 41.4 / 31.4, 4 shots 67.2 / 53.0; the
// line lies between the two sizes' 16 and 24 shots and 1 and 2, and batches of fewer than 8 shots on the smaller grid
// were not measured).
bool pair_pays(long long P, int S) { return P * S >= 13000000; }

cudaError_t launch_pair(const PairArgs &m0, int nshot, cudaStream_t st)
{
    PairArgs m = m0;
    PropArgs &a = m.a;
    if (!pair_runs(a)) return cudaErrorInvalidValue;
    prop_pairs(a);
    const int rows = a.NZ - 8;
    a.nstrip = (a.NXP + PAIR_STRIP - 1) / PAIR_STRIP;
    // an item computes eight rows more than it writes; with half a round for a launch's ends, four shots on 1300 rows
    // take 57 us per step in three rounds instead of 61 in one
    a.zchunk = chunk_rows(rows, a.nstrip, nshot, 152LL * PAIR_MINB * PAIR_WARPS, 12, 1, 0);
    a.nchunk = (rows + a.zchunk - 1) / a.zchunk;
    const bool d2 = a.d2 != nullptr;
    if (a.inj_val)
        return d2 ? launch_pair_t<0, true, false, true>(m, nshot, st) : launch_pair_t<0, false, false, true>(m, nshot, st);
    if (a.f0)
        return d2 ? launch_pair_t<1, true, false, false>(m, nshot, st) : launch_pair_t<1, false, false, false>(m, nshot, st);
    return d2 ? launch_pair_t<0, true, true, false>(m, nshot, st) : launch_pair_t<0, false, true, false>(m, nshot, st);
}

}  // namespace fwk
