// Subsurface-offset extension kernels (Barnier et al., Theory section: Born
// modelling extended with horizontal subsurface offsets, Eq. 1, and its
// adjoint, the extended imaging condition, Eqs. 2-5; tomographic operator,
// Eq. 9).
//
//   scatter    e(y)   = sum_h W(y-h, h) D(y-2h)          (sigma = +1)
//   transpose  z(u)   = sum_h W(u+h, h) L(u+2h)          (sigma = -1)
//   image      I(x,h) += sum_{shots,steps} D(x-h) L(x+h)
//   contract   G(x)   += sum_h p~(x,h) sum D(x-h) L(x+h)  (generic kernel only)
//   local      G(x)   += sum D (alpha L + M2) + Ds L
//
// The weights W = b p~ (nh values per point) are shared by every shot and
// every time step, so these kernels run once per segment of K time steps over
// all K x S (step, shot) pairs of a batch, keeping the weights (scatter) or the
// image accumulators (imaging) in registers for the whole segment, while the
// pairs' rows stream through cp.async rings in shared memory.  Weight and image
// traffic is then 1/(K S) of a per-step formulation.  Both default kernels copy
// rows de-interleaved into their even and odd samples: the products of offset h
// pair samples of one parity (y and y - 2h; x - h and x + h), so a lane that
// owns samples of one parity reuses every loaded sample for several offsets.
#include <algorithm>
#include <utility>

#include "fwime_kernels.cuh"

namespace fwk {

__device__ __forceinline__ long long ring_off(const RingRef &r, int n, int j)
{
    const int slot = r.mod > 0 ? (n + r.shift) % r.mod : j + r.shift;
    return (long long)slot * r.slot_stride;
}

// Walks the (step, shot) pairs of a segment in order p = 0, 1, ... (shot fastest) without
// integer division: pointer to the pair's field row in ring r.
struct RingIt {
    const float *base;
    long long slot_stride, P;
    int S, mod, s, slot;
    __device__ __forceinline__ void init(const RingRef &r, int n0, int S_, long long P_, long long rowoff)
    {
        base = r.base + rowoff; slot_stride = r.slot_stride; P = P_; S = S_; mod = r.mod; s = 0;
        slot = r.mod > 0 ? (n0 + r.shift) % r.mod : r.shift;
    }
    __device__ __forceinline__ const float *ptr() const { return base + (long long)slot * slot_stride + (long long)s * P; }
    __device__ __forceinline__ void next()
    {
        if (++s == S) {
            s = 0;
            if (++slot == mod) slot = 0;   // mod == 0 (direct rings) never wraps
        }
    }
};

// ---- asynchronous global -> shared copies (LDGSTS)
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
// 4-byte asynchronous copy (cp.async.ca); src_bytes = 0 zero-fills.  Used to de-interleave a row
// into its even and odd samples while it is copied into shared memory.
__device__ __forceinline__ void cpa4(unsigned dst, const float *src, bool valid)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
// unconditional 4-byte copies dst + C SSTEP <- src + C GSTEP bytes for C in the sequence (immediate
// offsets: one instruction per copy)
template <int SOFF, int GOFF>
__device__ __forceinline__ void cpa4_imm(unsigned dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0+%2], [%1+%3], 4;\n" ::"r"(dst), "l"(src), "n"(SOFF), "n"(GOFF)
                 : "memory");
}
template <int SSTEP, int GSTEP, int... C>
__device__ __forceinline__ void cpa4_run(unsigned dst, const float *src, std::integer_sequence<int, C...>)
{
    (cpa4_imm<SSTEP * C, GSTEP * C>(dst, src), ...);
}

// Row pointer of the (step, shot) pairs of a segment in order (shot fastest), advanced by one
// addition per pair and a multiply only when the time slot changes.
struct PairRow {
    const float *base, *row;
    long long slot_stride, P;
    int S, mod, s, slot;
    // starting at pair p0
    __device__ __forceinline__ void init(const RingRef &r, int n0, int S_, long long P_, long long rowoff, int p0 = 0)
    {
        base = r.base + rowoff; slot_stride = r.slot_stride; P = P_; S = S_; mod = r.mod;
        const int step = p0 / S_;
        s = p0 % S_;
        slot = r.mod > 0 ? (n0 + r.shift + step) % r.mod : r.shift + step;
        row = base + (long long)slot * slot_stride + (long long)s * P_;
    }
    __device__ __forceinline__ void next()
    {
        if (++s == S) {
            s = 0;
            if (++slot == mod) slot = 0;   // mod == 0 (direct rings) never wraps
            row = base + (long long)slot * slot_stride;
        } else {
            row += P;
        }
    }
};

// ------------------------------------------------------------------ scatter

// Vector loads from shared memory: VW = 4 (16-byte, LDS.128) or 2 (8-byte, LDS.64) consecutive floats.
template <int VW, int N>
__device__ __forceinline__ void lds_vec(float (&dst)[N], const float *src)
{
    static_assert(N % VW == 0, "window length must be a multiple of the vector width");
    if (VW == 4) {
#pragma unroll
        for (int k = 0; k < N / 4; ++k) {
            const float4 v = reinterpret_cast<const float4 *>(src)[k];
            dst[4 * k] = v.x; dst[4 * k + 1] = v.y; dst[4 * k + 2] = v.z; dst[4 * k + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < N / 2; ++k) {
            const float2 v = reinterpret_cast<const float2 *>(src)[k];
            dst[2 * k] = v.x; dst[2 * k + 1] = v.y;
        }
    }
}

// ---------------------------------------------------------- scatter, parity-split (default path)
//
// e(y) = sum_h W(y - sigma h, h) D(y - 2 sigma h) reads D only at samples of y's parity.  A lane
// owns A outputs of one parity, y_j = yf + 2j, whose A x NH products need only A + 2 HM samples of
// that parity: rows are copied into shared memory split into their even and odd samples (4-byte
// cp.async), and every sample a lane loads serves up to A multiply-adds with the A x NH weights it
// keeps in registers for the whole segment.  Lanes 0-15 take the even outputs of the warp's 32 A
// columns, lanes 16-31 the odd ones; one shuffle across the two halves reassembles A consecutive
// outputs per lane for vector stores.  Each warp streams its own window through its own cp.async
// ring, synchronised with __syncwarp only.
#ifndef FWIME_SC_WARPS
#define FWIME_SC_WARPS 4
#endif
#ifndef FWIME_SC_STAGES
#define FWIME_SC_STAGES 8
#endif
#ifndef FWIME_SC_MINB
#define FWIME_SC_MINB 3   // at most 168 registers: 3 CTAs per SM for every nh (nh 31 transposed: 229 -> 168, -3.5 %)
#endif
#ifndef FWIME_IMG_MINB
#define FWIME_IMG_MINB 1
#endif
#ifndef FWIME_SC_A21
#define FWIME_SC_A21 4
#endif
#ifndef FWIME_SC_A31
#define FWIME_SC_A31 4
#endif
// packed two-lane FP32 (f32x2) forms of the multiply-adds, per kernel where they measured faster
// (scatter -1 % at nh 21; imaging -5.5 % at nh 21 (Marmousi2-shaped B~ + B~*), +1.4 % at nh 31
// (North-Sea-shaped gradient), -16 % at nh 41 (Salt-shaped gradient): every nh but 31 packs)
#ifndef FWIME_SC_F32X2
#define FWIME_SC_F32X2 1
#endif
#ifndef FWIME_IMG_F32X2
#define FWIME_IMG_F32X2 1
#endif
#ifndef FWIME_IMG_UNPACKED_NH
#define FWIME_IMG_UNPACKED_NH 31   // the nh whose imaging kernel keeps the scalar form (packed: +1.4 % time)
#endif
#ifndef FWIME_SC_PAIRS
#define FWIME_SC_PAIRS 0      // (step, shot) pairs per loop iteration of the scatter (sharing its weights);
                              // 0: two at nh 21 and 31 (measured -4.3 % at nh 31, -0.6 % at nh 21), else one
#endif
#ifndef FWIME_SC_BALANCE
#define FWIME_SC_BALANCE 1    // split the scatter's pairs over several warps per task to fill the last wave
#endif
#ifndef FWIME_SC_PACK_MAX
#define FWIME_SC_PACK_MAX 96   // largest nh * A whose weights are packed (more spills)
#endif
constexpr int SC_WARPS = FWIME_SC_WARPS;     // warps per CTA (independent pipelines)
constexpr int SC_STAGES = FWIME_SC_STAGES;   // cp.async ring depth per warp

template <int NH, int A>
struct ScatterShape {
    static constexpr int HM = (NH - 1) / 2;
    static constexpr int WOUT = 32 * A;                      // outputs per warp
    static constexpr int SPAN = WOUT + 4 * HM;               // window [yw - 2 HM, yw + WOUT + 2 HM)
    static constexpr int HALF = SPAN / 2;                    // samples of one parity
    static constexpr int OFF = (HALF + 31) / 32 * 32 + 16;   // odd samples, 16 banks after the even ones
    static constexpr int STG = 2 * OFF;                      // floats per stage
    static constexpr int NCP = (SPAN + 31) / 32;             // 4-byte copies per lane and pair
    static constexpr int VW = A % 4 == 0 ? 4 : 2;
    static constexpr int NWIN = A + 2 * HM;                  // samples a lane reads
    static constexpr int NWV = (NWIN + VW - 1) / VW * VW;
    static constexpr size_t SMEM = (size_t)SC_WARPS * SC_STAGES * STG * sizeof(float);
    // copies past SPAN land below OFF (even) or 2 OFF (odd); reads stay below HALF + 4 <= OFF
    static_assert(OFF >= HALF + 16 && 15 * A + NWV <= OFF, "parity array overflow");
};

// SPLIT: each (row, column block) task's pairs are divided among nsplit warps
template <int NH, int A, int SIGMA, bool SPLIT>
__global__ void __launch_bounds__(SC_WARPS * 32, FWIME_SC_MINB) k_scatter_ps(const ExtArgs a, int nwx, int nsplit)
{
    using Sh = ScatterShape<NH, A>;
    constexpr int HM = Sh::HM, NS = SC_STAGES;
    extern __shared__ float4 sm4[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *wsm = reinterpret_cast<float *>(sm4) + warp * NS * Sh::STG;
    // Warps are numbered over (row, column block[, part]) so that no warp of a CTA idles at a row's end;
    // with SPLIT each of a task's nsplit parts takes an equal share of its (step, shot) pairs, the split
    // chosen on the host so that the segment-long CTAs fill their last wave (the unsplit variant keeps
    // the whole range, a kernel parameter, out of its registers).  Warps share nothing: no block-wide
    // barrier follows.
    const int gw = blockIdx.x * SC_WARPS + warp;   // 32-bit indexing (64-bit indexing spilled at nh 31)
    if (gw >= nwx * (a.z_hi - a.z_lo) * (SPLIT ? nsplit : 1)) return;
    const int task = SPLIT ? gw / nsplit : gw;
    int pb = 0, pe = a.npair;
    if constexpr (SPLIT) {
        const int part = (int)(gw % nsplit);
        pb = (int)((long long)part * a.npair / nsplit);
        pe = (int)((long long)(part + 1) * a.npair / nsplit);
        if (pb == pe) return;
    }
    const int Z = a.z_lo + task / nwx;
    const int yw = a.x_lo + (task % nwx) * Sh::WOUT;  // multiple of 4
    const int par = lane >> 4, tp = lane & 15;
    const int yf = yw + par + 2 * A * tp;          // this lane's outputs yf + 2j, j < A
    const long long rowoff = (long long)Z * a.NXP;
    const int wal = yw - 2 * HM;                   // even

    float Wr[A][NH];
#pragma unroll
    for (int j = 0; j < A; ++j) {
        const int y = yf + 2 * j;
#pragma unroll
        for (int ih = 0; ih < NH; ++ih) {
            const int xs = y - SIGMA * (ih - HM);
            Wr[j][ih] = (y < a.x_hi && xs >= 0 && xs < a.NXP) ? __ldg(a.W + ih * a.P + rowoff + xs) : 0.f;
        }
    }
    // packed two-lane arithmetic where the weights leave room for their pairs (no spills)
    constexpr bool PACK = FWIME_SC_F32X2 && NH * A <= FWIME_SC_PACK_MAX;
    // Packed form: output j reads dv[j + o] at offset ih, o = HM - SIGMA (ih - HM), and o has the
    // parity of ih.  For even o the pairs of outputs (0, 1) and (2, 3) read the aligned register
    // pairs (dv[o], dv[o + 1]), (dv[o + 2], dv[o + 3]); for odd o the pair (1, 2) reads the aligned
    // (dv[o + 1], dv[o + 2]) and outputs 0 and 3 stay scalar.  Each output sums its even-o and
    // odd-o products separately (two chains, as in the scalar form).
    constexpr int NE = PACK ? (NH + 1) / 2 : 1, NO = PACK && NH / 2 > 0 ? NH / 2 : 1;   // even / odd o (o = ih mod 2)
    f32x2 WE[NE][A / 2], WO[NO];
    float WO0[NO], WO3[NO];
#pragma unroll
    for (int ih = 0; ih < (PACK ? NH : 0); ++ih) {
        if (ih % 2 == 0) {
#pragma unroll
            for (int q = 0; q < A / 2; ++q) WE[ih / 2][q] = pk(Wr[2 * q][ih], Wr[2 * q + 1][ih]);
        } else if (A == 4) {
            WO[ih / 2] = pk(Wr[1][ih], Wr[A - 2][ih]);
            WO0[ih / 2] = Wr[0][ih];
            WO3[ih / 2] = Wr[A - 1][ih];
        } else {
            WO0[ih / 2] = Wr[0][ih];
            WO3[ih / 2] = Wr[A - 1][ih];
        }
    }
    // the lane copies window samples n = lane + 32 c (column wal + n) into its parity's array
    const unsigned sm0 =
        static_cast<unsigned>(__cvta_generic_to_shared(wsm)) + 4u * ((lane & 1) * Sh::OFF + (lane >> 1));
    const int col0 = wal + lane;
    const bool interior = wal >= 0 && wal + 32 * Sh::NCP <= a.NXP;
    PairRow pin, pout;
    pin.init(a.in, a.n0, a.S, a.P, rowoff, pb);
    pout.init(a.outr, a.n0, a.S, a.P, rowoff, pb);
    unsigned st_in = 0;
    int st_c = 0;
    auto issue = [&](int p) {
        if (p < pe) {
            const unsigned d = sm0 + st_in;
            // samples n = lane + 32 c of the window [0, SPAN): the last round copies only its first REM
            // lanes' samples (nothing past the window is read, from memory or from shared memory)
            constexpr int REM = Sh::SPAN - 32 * (Sh::NCP - 1);
            if (interior) {
                cpa4_run<64, 128>(d, pin.row + col0, std::make_integer_sequence<int, Sh::NCP - 1>{});
                if (REM == 32 || lane < REM) cpa4_imm<64 * (Sh::NCP - 1), 128 * (Sh::NCP - 1)>(d, pin.row + col0);
            } else {
#pragma unroll
                for (int c = 0; c < Sh::NCP; ++c) {
                    if (c == Sh::NCP - 1 && REM < 32 && lane >= REM) break;
                    const int col = col0 + 32 * c;
                    const bool ok = col >= 0 && col < a.NXP;
                    cpa4(d + 64u * c, pin.row + (ok ? col : 0), ok);
                }
            }
            pin.next();
        }
        st_in = st_in + 4u * Sh::STG == 4u * NS * Sh::STG ? 0u : st_in + 4u * Sh::STG;
        cpa_commit();
    };
    // PP pairs per iteration share the weights: PP independent sets of accumulator chains per warp
    constexpr int PP = FWIME_SC_PAIRS > 0 ? FWIME_SC_PAIRS : (NH == 21 || NH == 31 ? 2 : 1);
    static_assert(NS >= 2 * PP, "ring too short for the pairs per iteration");
#pragma unroll 1
    for (int q = 0; q < NS - PP; ++q) issue(pb + q);
    const int ys = yw + 2 * A * tp + A * par;      // first of the A consecutive outputs this lane stores
    const float *lsm = wsm + par * Sh::OFF + A * tp;
#pragma unroll 1
    for (int p = pb; p < pe; p += PP) {
        cpa_wait<NS - 2 * PP>();                   // pairs p .. p + PP - 1 have landed (this lane's copies) ...
        __syncwarp();                              // ... and every lane's; all finished the pairs before
#pragma unroll
        for (int u = 0; u < PP; ++u) issue(p + NS - PP + u);   // refills the stages of the previous pairs
        float dv[PP][Sh::NWV];                     // dv[u][k] = D(yf - 2 HM + 2k) of pair p + u
#pragma unroll
        for (int u = 0; u < PP; ++u) {
            lds_vec<Sh::VW>(dv[u], lsm + st_c);
            st_c = st_c + Sh::STG == NS * Sh::STG ? 0 : st_c + Sh::STG;
        }
        float e[PP][A];
        if constexpr (PACK) {
            f32x2 ae[PP][A / 2], ao[PP];
            float ao0[PP], ao3[PP];
#pragma unroll
            for (int u = 0; u < PP; ++u) {
                ao[u] = pk(0.f, 0.f);
                ao0[u] = ao3[u] = 0.f;
#pragma unroll
                for (int q = 0; q < A / 2; ++q) ae[u][q] = pk(0.f, 0.f);
            }
#pragma unroll
            for (int m = 0; m < NH; ++m) {                 // offsets in the order of their samples
                const int ih = SIGMA > 0 ? NH - 1 - m : m;
                const int o = HM - SIGMA * (ih - HM);
#pragma unroll
                for (int u = 0; u < PP; ++u) {             // the pairs' chains interleaved
                    if (ih % 2 == 0) {
#pragma unroll
                        for (int q = 0; q < A / 2; ++q)
                            ae[u][q] = fma2(WE[ih / 2][q], pk(dv[u][o + 2 * q], dv[u][o + 2 * q + 1]), ae[u][q]);
                    } else {
                        if (A == 4) ao[u] = fma2(WO[ih / 2], pk(dv[u][o + 1], dv[u][o + 2]), ao[u]);
                        ao0[u] = fmaf(WO0[ih / 2], dv[u][o], ao0[u]);
                        ao3[u] = fmaf(WO3[ih / 2], dv[u][o + A - 1], ao3[u]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < PP; ++u) {
                float el[A], ol[A];
#pragma unroll
                for (int q = 0; q < A / 2; ++q) upk(ae[u][q], el[2 * q], el[2 * q + 1]);
                ol[0] = ao0[u];
                ol[A - 1] = ao3[u];
                if (A == 4) upk(ao[u], ol[1], ol[A - 2]);
#pragma unroll
                for (int j = 0; j < A; ++j) e[u][j] = el[j] + ol[j];
            }
        } else {
            // two partial sums per output (even / odd offsets): 2 A independent chains per pair.  Offsets
            // are visited in the order of their samples, so the first products wait only for the first load.
            float acc[PP][2][A];
#pragma unroll
            for (int u = 0; u < PP; ++u)
#pragma unroll
                for (int j = 0; j < A; ++j) acc[u][0][j] = acc[u][1][j] = 0.f;
#pragma unroll
            for (int m = 0; m < NH; ++m) {
                const int ih = SIGMA > 0 ? NH - 1 - m : m;
#pragma unroll
                for (int u = 0; u < PP; ++u)
#pragma unroll
                    for (int j = 0; j < A; ++j)            // D(y_j - 2 SIGMA h) = dv[j - SIGMA (ih - HM) + HM]
                        acc[u][m & 1][j] = fmaf(Wr[j][ih], dv[u][j - SIGMA * (ih - HM) + HM], acc[u][m & 1][j]);
            }
#pragma unroll
            for (int u = 0; u < PP; ++u)
#pragma unroll
                for (int j = 0; j < A; ++j) e[u][j] = acc[u][0][j] + acc[u][1][j];
        }
#pragma unroll
        for (int u = 0; u < PP; ++u) {
            if (PP > 1 && p + u >= pe) break;   // warp-uniform
            float v[A];
            if constexpr (A == 4) {
                const float r0 = __shfl_xor_sync(0xffffffffu, par ? e[u][0] : e[u][2], 16);
                const float r1 = __shfl_xor_sync(0xffffffffu, par ? e[u][1] : e[u][3], 16);
                v[0] = par ? r0 : e[u][0]; v[1] = par ? e[u][2] : r0;
                v[2] = par ? r1 : e[u][1]; v[3] = par ? e[u][3] : r1;
            } else {
                const float r0 = __shfl_xor_sync(0xffffffffu, par ? e[u][0] : e[u][1], 16);
                v[0] = par ? r0 : e[u][0]; v[1] = par ? e[u][1] : r0;
            }
            float *o = const_cast<float *>(pout.row) + ys;
            pout.next();
            if (ys + A <= a.x_hi) {
                if constexpr (A == 4) {
                    float4 w4 = make_float4(v[0], v[1], v[2], v[3]);
                    if (a.accumulate) {
                        const float4 old = *reinterpret_cast<const float4 *>(o);
                        w4.x += old.x; w4.y += old.y; w4.z += old.z; w4.w += old.w;
                    }
                    *reinterpret_cast<float4 *>(o) = w4;
                } else {
                    float2 w2 = make_float2(v[0], v[1]);
                    if (a.accumulate) {
                        const float2 old = *reinterpret_cast<const float2 *>(o);
                        w2.x += old.x; w2.y += old.y;
                    }
                    *reinterpret_cast<float2 *>(o) = w2;
                }
            } else {
#pragma unroll
                for (int k = 0; k < A; ++k)
                    if (ys + k < a.x_hi) o[k] = a.accumulate ? o[k] + v[k] : v[k];
            }
        }
    }
    cpa_wait<0>();
}


// Generic-nh fallback (weights re-read per pair): any odd nh up to MAX_NH.
__global__ void __launch_bounds__(EXT_TX) k_scatter_gen(const ExtArgs a)
{
    extern __shared__ float sm[];
    const int nh = a.nh, hm = (nh - 1) / 2;
    const int Z = a.z_lo + blockIdx.y;
    const int y0 = a.x_lo + blockIdx.x * EXT_TX;
    const int y = y0 + threadIdx.x;
    const bool yin = y < a.x_hi;
    const int span = EXT_TX + 4 * hm;
    const int wbase = y0 - 2 * hm;
    const long long rowoff = (long long)Z * a.NXP;
    float *out_base = const_cast<float *>(a.outr.base);
    for (int p = 0; p < a.npair; ++p) {
        const int j = p / a.S, s = p % a.S, n = a.n0 + j;
        const float *src = a.in.base + ring_off(a.in, n, j) + (long long)s * a.P + rowoff;
        __syncthreads();
        for (int i = threadIdx.x; i < span; i += EXT_TX) {
            const int xp = wbase + i;
            sm[i] = (xp >= 0 && xp < a.NXP) ? __ldg(src + xp) : 0.f;
        }
        __syncthreads();
        float acc = 0.f;
        const int c0 = threadIdx.x + 2 * hm;
        for (int ih = 0; ih < nh; ++ih) {
            const int xs = y - a.sigma * (ih - hm);
            const float wv = (yin && xs >= 0 && xs < a.NXP) ? __ldg(a.W + ih * a.P + rowoff + xs) : 0.f;
            acc = fmaf(wv, sm[c0 - 2 * a.sigma * (ih - hm)], acc);
        }
        if (yin) {
            float *o = out_base + ring_off(a.outr, n, j) + (long long)s * a.P + rowoff + y;
            *o = a.accumulate ? *o + acc : acc;
        }
    }
}

template <int NH, int A>
static void launch_scatter_ps(ExtArgs a, cudaStream_t st)
{
    using Sh = ScatterShape<NH, A>;
    a.x_lo -= a.x_lo % 4;          // outputs start on a 16-byte boundary (leading columns get zero weights)
    const int nwx = (a.x_hi - a.x_lo + Sh::WOUT - 1) / Sh::WOUT;        // warps per row
    const long long nw = (long long)nwx * (a.z_hi - a.z_lo);
    constexpr bool CAN_SPLIT = FWIME_SC_BALANCE;
    // once per instantiation, before any launch (and any capture); a function-local static is
    // initialised once even when several host threads launch: the attributes, then the CTAs per SM of
    // the least resident variant
    static const int resident = [] {
        int r[4] = {0, 0, 0, 0};
        const auto setup = [](auto kern, int &res) {
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::SMEM);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&res, kern, SC_WARPS * 32, Sh::SMEM);
        };
        setup(k_scatter_ps<NH, A, 1, false>, r[0]);
        setup(k_scatter_ps<NH, A, -1, false>, r[1]);
        r[2] = r[3] = r[0];
        if constexpr (CAN_SPLIT) {
            setup(k_scatter_ps<NH, A, 1, true>, r[2]);
            setup(k_scatter_ps<NH, A, -1, true>, r[3]);
        }
        return std::max(1, std::min(std::min(r[0], r[1]), std::min(r[2], r[3])));
    }();
    // Split every task's pairs into nsplit parts, nsplit <= 8 and parts of at least 4 ring depths of
    // pairs, picked to fill the last wave of resident CTAs best (the smallest within 1 %).
    int nsplit = 1;
    if (CAN_SPLIT) {
        int dev = 0, nsm = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        const double wave = (double)resident * std::max(nsm, 1);
        auto fill = [&](int k) {   // used fraction of the launch's waves of CTAs
            const double w = std::ceil((double)nw * k / SC_WARPS) / wave;
            return w / std::ceil(w);
        };
        double best = fill(1);
        for (int k = 2; k <= 8 && a.npair / k >= 4 * SC_STAGES; ++k)
            if (fill(k) > best + 0.01) { best = fill(k); nsplit = k; }
    }
    dim3 grid((unsigned)((nw * nsplit + SC_WARPS - 1) / SC_WARPS));
    const int nt = SC_WARPS * 32;
    if (nsplit > 1) {
        if constexpr (CAN_SPLIT) {
            if (a.sigma > 0) k_scatter_ps<NH, A, 1, true><<<grid, nt, Sh::SMEM, st>>>(a, nwx, nsplit);
            else k_scatter_ps<NH, A, -1, true><<<grid, nt, Sh::SMEM, st>>>(a, nwx, nsplit);
        }
    } else if (a.sigma > 0) {
        k_scatter_ps<NH, A, 1, false><<<grid, nt, Sh::SMEM, st>>>(a, nwx, 1);
    } else {
        k_scatter_ps<NH, A, -1, false><<<grid, nt, Sh::SMEM, st>>>(a, nwx, 1);
    }
}

cudaError_t launch_scatter(const ExtArgs &a, cudaStream_t st)
{
    if (a.npair <= 0 || a.x_hi <= a.x_lo || a.z_hi <= a.z_lo) return cudaSuccess;
    switch (a.nh) {
    case 1: launch_scatter_ps<1, 4>(a, st); break;
    case 3: launch_scatter_ps<3, 4>(a, st); break;
    case 5: launch_scatter_ps<5, 4>(a, st); break;
    case 11: launch_scatter_ps<11, 4>(a, st); break;
    case 21: launch_scatter_ps<21, FWIME_SC_A21>(a, st); break;
    case 31: launch_scatter_ps<31, FWIME_SC_A31>(a, st); break;
    case 41: launch_scatter_ps<41, 2>(a, st); break;
    default: {
        dim3 grid((a.x_hi - a.x_lo + EXT_TX - 1) / EXT_TX, a.z_hi - a.z_lo);
        const int hm = (a.nh - 1) / 2;
        k_scatter_gen<<<grid, EXT_TX, (EXT_TX + 4 * hm) * sizeof(float), st>>>(a);
    }
    }
    return cudaGetLastError();
}

}  // namespace fwk
