// One time step of the 2-D acoustic constant-density wave equation, 2nd order
// in time and 8th order in space, with the Cerjan-type sponge fused in
// (Barnier et al., Theory section: the acoustic isotropic constant-density
// two-way operator f of Eq. 1; Marmousi2 section: absorbing boundaries on all
// sides):
//
//   q^{n+1} = g (2 q^n - g q^{n-1} + c (L q^n + s^n)),   g = gz[IZ] gx[IX],  c = v^2 dt^2
//
// The same kernel advances the adjoint wavefield backward in time: with
// mu = c g lambda the exact transpose of the recursion takes the same form
// (mu^n from mu^{n+1}, mu^{n+2}), so forward and adjoint share this code.
//
// Work decomposition (HBM-bound, no tensor cores): one warp owns a strip of
// 128 x-points (32 lanes x float4) and a chunk of rows, marching down z with a
// 9-row register queue, so every row of q^n is read from memory once per
// strip; the +-4 x-neighbours come from the adjacent lanes by warp shuffles
// and, at the strip edges, one extra float4 per row.  q^{n-1}, c and the
// output are touched once, coalesced.  Sources (point, dense local terms) and
// the second time derivative (for Born-type scattering) are fused in.
#pragma once
#include "fwime_kernels.cuh"

namespace fwk {

// the warp's index in its CTA, as a value that is known to be the same in all its lanes
__device__ __forceinline__ int warp_in_cta() { return __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0); }
__device__ __forceinline__ float4 f4zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
// Read-only loads: of what no launch in flight writes (model, tables, receivers).  The wavefields are read by ordinary
// loads through plain pointers: a launch comes in while the one before still writes them, and what is read as read-only
// may be fetched before the wait, or from a cache that holds an older step's rows.
__device__ __forceinline__ float4 ldg4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
// a wavefield's row: from L2, as the copies, and not before what stands before it (plain loads through L1 took 0.7 to
// 1.2 % more of a small grid's step)
__device__ __forceinline__ float4 ldcg4(const float *p)
{
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void st4(float *p, float4 v) { *reinterpret_cast<float4 *>(p) = v; }
__device__ __forceinline__ float cmp(const float4 &v, int j)
{
    return j == 0 ? v.x : (j == 1 ? v.y : (j == 2 ? v.z : v.w));
}
__device__ __forceinline__ float4 shfl_up4(float4 v)
{
    v.x = __shfl_up_sync(0xffffffffu, v.x, 1);
    v.y = __shfl_up_sync(0xffffffffu, v.y, 1);
    v.z = __shfl_up_sync(0xffffffffu, v.z, 1);
    v.w = __shfl_up_sync(0xffffffffu, v.w, 1);
    return v;
}
__device__ __forceinline__ float4 shfl_down4(float4 v)
{
    v.x = __shfl_down_sync(0xffffffffu, v.x, 1);
    v.y = __shfl_down_sync(0xffffffffu, v.y, 1);
    v.z = __shfl_down_sync(0xffffffffu, v.z, 1);
    v.w = __shfl_down_sync(0xffffffffu, v.w, 1);
    return v;
}

// ---- asynchronous global -> shared copies (LDGSTS)
__device__ __forceinline__ void cp16n(float *dst, const float *src, int n)   // n: 16, or 0 to zero-fill
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// Per-warp pipeline: rings of nine rows of q^n (128 points + 4-point halos, for the x-taps and the register queue),
// q^{n-1} and c; with local sources rings of three rows of those, of q^{n-1} and of c.  Nine is the period of the
// unrolled register queue, so every slot is a compile-time constant.  Row z waits for the copy group issued four rows
// (with local sources three) earlier.  With slots and addresses computed per row and lane a row of 128 points took 211
// instructions in 124 registers, now 139 (one local source) in 102 to 116: 350 x 1700 points, 8 shots, 15.8 / 13.9 us
// per step; from about 16 shots on the kernel is bound by memory and the two are equal.
constexpr int RING = 9, LRING = 3;
// Variants k_prop<LOC, D2, SRC>: LOC = 0 no dense local source, 1 exactly one (f0, weight a0), 2 the
// general sum a0 f0 + a1 f1 + a2 f2 + coef fc; D2 writes D2t; SRC adds the point source.  Register
// bounds (minimum resident CTAs) per kind:
#ifndef FWIME_PROP_MIN_BLOCKS
#define FWIME_PROP_MIN_BLOCKS 1   // general local sources (up to five extra rows per stage)
#endif
#ifndef FWIME_PROP_MINB_LOC1
#define FWIME_PROP_MINB_LOC1 3   // one local source: up to 128 registers, 4 CTAs per SM like the plain variants
#endif
#ifndef FWIME_PROP_MINB_PLAIN
#define FWIME_PROP_MINB_PLAIN 3   // up to 128 registers: still 4 CTAs per SM, fewer rematerialised operands
#endif
constexpr int CUR_ROW = STRIP + 8;
// floats of shared memory per warp; naux = 2 + the number of local source rows
__host__ __device__ constexpr int prop_smem(int naux)
{
    return RING * CUR_ROW + (naux > 2 ? LRING : RING) * naux * STRIP;
}

// The arithmetic of one output row of a lane (four consecutive columns): the Laplacian from the
// x-neighbours (L | Q4 | Rr, 12 consecutive samples) and the nine queue rows Q0..Q8 (the output row
// is Q4), then the sponge-damped update and optionally D2t.  In the scalar form every product and
// sum is the same as
//   lap = (ax0 + az0) q + sum_k ax_k (q[x-k] + q[x+k]) + sum_k az_k (q[z-k] + q[z+k])   (k = 1..4)
//   out = g (2 q - g p + c (lap + s)),   d2 = (out - 2 q + p) / dt^2.
#ifndef FWIME_PROP_F32X2
#define FWIME_PROP_F32X2 1
#endif
#ifndef FWIME_PROP_F32X2_PLAIN
#define FWIME_PROP_F32X2_PLAIN 1
#endif
// Packed two-lane FP32 (f32x2, see fwime_kernels.cuh) on columns (j, j + 1): half the floating-point
// issue slots of the scalar form, with its rounding.  The coefficient operands as register pairs:
struct PropK {
    f32x2 axc, kx[5], kz[5], inv, a0, a1, a2;
};
__device__ __forceinline__ PropK prop_k(const PropArgs &a)
{
    PropK K;
    K.axc = bits(a.axc2);
#pragma unroll
    for (int k = 1; k < 5; ++k) {
        K.kx[k] = bits(a.kx2[k]);
        K.kz[k] = bits(a.kz2[k]);
    }
    K.inv = bits(a.inv2);
    K.a0 = bits(a.a02);
    K.a1 = bits(a.a12);
    K.a2 = bits(a.a22);
    return K;
}
// columns (2 h, 2 h + 1) of a float4
__device__ __forceinline__ f32x2 half2(const float4 &v, int h) { return h == 0 ? pk(v.x, v.y) : pk(v.z, v.w); }

template <int LOC, bool D2, bool SRC>
__device__ __forceinline__ void row_math_pk(const PropArgs &a, const PropK &K, const float4 &L, const float4 &Q0, const float4 &Q1,
                                         const float4 &Q2, const float4 &Q3, const float4 &Q4, const float4 &Q5,
                                         const float4 &Q6, const float4 &Q7, const float4 &Q8, const float4 &Rr,
                                         const float4 &pv, const float4 &cv, const float4 &lf0, const float4 &lf1,
                                         const float4 &lf2, const float4 &lcf, const float4 &lfc, float gzz,
                                         const float4 &gxv, int sj, float amp, float4 &o, float4 &d2)
{
    constexpr bool LOCAL = LOC > 0;
    const float rr[12] = {L.x, L.y, L.z, L.w, Q4.x, Q4.y, Q4.z, Q4.w, Rr.x, Rr.y, Rr.z, Rr.w};
    const f32x2 GZ = pk(gzz, gzz), NGZ = pk(-gzz, -gzz);
    float ov[4], dv[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int j = 2 * h;
        const f32x2 C0 = half2(Q4, h);
        f32x2 lap = mul2(K.axc, C0);
        lap = fma2(K.kx[1], add2(pk(rr[j + 3], rr[j + 4]), pk(rr[j + 5], rr[j + 6])), lap);
        lap = fma2(K.kx[2], add2(pk(rr[j + 2], rr[j + 3]), pk(rr[j + 6], rr[j + 7])), lap);
        lap = fma2(K.kx[3], add2(pk(rr[j + 1], rr[j + 2]), pk(rr[j + 7], rr[j + 8])), lap);
        lap = fma2(K.kx[4], add2(pk(rr[j + 0], rr[j + 1]), pk(rr[j + 8], rr[j + 9])), lap);
        lap = fma2(K.kz[1], add2(half2(Q3, h), half2(Q5, h)), lap);
        lap = fma2(K.kz[2], add2(half2(Q2, h), half2(Q6, h)), lap);
        lap = fma2(K.kz[3], add2(half2(Q1, h), half2(Q7, h)), lap);
        lap = fma2(K.kz[4], add2(half2(Q0, h), half2(Q8, h)), lap);
        if (LOCAL || SRC) {
            f32x2 sv = pk(0.f, 0.f);
            if (LOCAL) {
                sv = fma2(K.a0, half2(lf0, h), sv);
                if (LOC == 2) {
                    sv = fma2(K.a1, half2(lf1, h), sv);
                    sv = fma2(K.a2, half2(lf2, h), sv);
                    sv = fma2(half2(lcf, h), half2(lfc, h), sv);
                }
            }
            if (SRC) sv = add2(sv, pk(sj == j ? amp : 0.f, sj == j + 1 ? amp : 0.f));
            lap = add2(lap, sv);
        }
        const f32x2 GX = half2(gxv, h);
        const f32x2 G = mul2(GZ, GX), NG = mul2(NGZ, GX);
        const f32x2 P = half2(pv, h);
        const f32x2 TC = add2(C0, C0);
        const f32x2 O = mul2(G, fma2(half2(cv, h), lap, fma2(NG, P, TC)));
        upk(O, ov[j], ov[j + 1]);
        if (D2) {
            const f32x2 D = mul2(add2(sub2(O, TC), P), K.inv);
            upk(D, dv[j], dv[j + 1]);
        }
    }
    o = make_float4(ov[0], ov[1], ov[2], ov[3]);
    if (D2) d2 = make_float4(dv[0], dv[1], dv[2], dv[3]);
}
template <int LOC, bool D2, bool SRC>
__device__ __forceinline__ void row_math_sc(const PropArgs &a, const float4 &L, const float4 &Q0, const float4 &Q1,
                                         const float4 &Q2, const float4 &Q3, const float4 &Q4, const float4 &Q5,
                                         const float4 &Q6, const float4 &Q7, const float4 &Q8, const float4 &Rr,
                                         const float4 &pv, const float4 &cv, const float4 &lf0, const float4 &lf1,
                                         const float4 &lf2, const float4 &lcf, const float4 &lfc, float gzz,
                                         const float4 &gxv, int sj, float amp, float4 &o, float4 &d2)
{
    constexpr bool LOCAL = LOC > 0;
    const float rr[12] = {L.x, L.y, L.z, L.w, Q4.x, Q4.y, Q4.z, Q4.w, Rr.x, Rr.y, Rr.z, Rr.w};
    const float axc = a.ax[0] + a.az[0];
    float ov[4], dv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float c0v = rr[j + 4];
        float lap = axc * c0v;
        lap = fmaf(a.ax[1], rr[j + 3] + rr[j + 5], lap);
        lap = fmaf(a.ax[2], rr[j + 2] + rr[j + 6], lap);
        lap = fmaf(a.ax[3], rr[j + 1] + rr[j + 7], lap);
        lap = fmaf(a.ax[4], rr[j + 0] + rr[j + 8], lap);
        lap = fmaf(a.az[1], cmp(Q3, j) + cmp(Q5, j), lap);
        lap = fmaf(a.az[2], cmp(Q2, j) + cmp(Q6, j), lap);
        lap = fmaf(a.az[3], cmp(Q1, j) + cmp(Q7, j), lap);
        lap = fmaf(a.az[4], cmp(Q0, j) + cmp(Q8, j), lap);
        if (LOCAL || SRC) {
            float sv = 0.f;
            if (LOCAL) {
                sv = fmaf(a.a0, cmp(lf0, j), sv);
                if (LOC == 2) {
                    sv = fmaf(a.a1, cmp(lf1, j), sv);
                    sv = fmaf(a.a2, cmp(lf2, j), sv);
                    sv = fmaf(cmp(lcf, j), cmp(lfc, j), sv);
                }
            }
            if (SRC) sv += sj == j ? amp : 0.f;
            lap += sv;
        }
        const float g = gzz * cmp(gxv, j);
        const float pj = cmp(pv, j);
        const float tc = c0v + c0v;
        ov[j] = g * fmaf(cmp(cv, j), lap, fmaf(-g, pj, tc));
        dv[j] = (ov[j] - tc + pj) * a.inv_dt2;
    }
    o = make_float4(ov[0], ov[1], ov[2], ov[3]);
    if (D2) d2 = make_float4(dv[0], dv[1], dv[2], dv[3]);
}
// the packed form where it measured faster: the variants with dense local sources always; the
// plain ones (point source, D2t) only under FWIME_PROP_F32X2_PLAIN
template <int LOC, bool D2, bool SRC>
__device__ __forceinline__ void row_math(const PropArgs &a, const PropK &K, const float4 &L, const float4 &Q0, const float4 &Q1,
                                         const float4 &Q2, const float4 &Q3, const float4 &Q4, const float4 &Q5,
                                         const float4 &Q6, const float4 &Q7, const float4 &Q8, const float4 &Rr,
                                         const float4 &pv, const float4 &cv, const float4 &lf0, const float4 &lf1,
                                         const float4 &lf2, const float4 &lcf, const float4 &lfc, float gzz,
                                         const float4 &gxv, int sj, float amp, float4 &o, float4 &d2)
{
    constexpr bool LOCAL = LOC > 0;
    if constexpr (FWIME_PROP_F32X2 && (LOCAL || FWIME_PROP_F32X2_PLAIN))
        row_math_pk<LOC, D2, SRC>(a, K, L, Q0, Q1, Q2, Q3, Q4, Q5, Q6, Q7, Q8, Rr, pv, cv, lf0, lf1, lf2, lcf, lfc, gzz,
                                    gxv, sj, amp, o, d2);
    else
        row_math_sc<LOC, D2, SRC>(a, L, Q0, Q1, Q2, Q3, Q4, Q5, Q6, Q7, Q8, Rr, pv, cv, lf0, lf1, lf2, lcf, lfc, gzz,
                                    gxv, sj, amp, o, d2);
}

// Adds the injections of the receivers chained from r at one output point: o + c v per receiver, each
// product and sum rounded separately (the arithmetic of a separate injection launch after the step).
__device__ __forceinline__ void inject_point(const PropArgs &a, const float *val, int shot, int r, float c, float &o)
{
    for (; r >= 0; r = __ldg(a.inj_next + r))
        o = __fadd_rn(o, __fmul_rn(c, __ldg(val + (long long)shot * a.inj_vstride + r)));
}

// The same for the four points of a lane at (zz, x), before they are stored; D2t gains what the point gains.
template <bool D2>
__device__ __forceinline__ void inject_row(const PropArgs &a, const float *val, int shot, int zz, int x, const float4 &cv,
                                           float4 &o, float4 &d2)
{
    const int4 m4 = *reinterpret_cast<const int4 *>(a.inj_map + (long long)(zz - a.inj_lo) * a.NXP + x);
    if ((m4.x & m4.y & m4.z & m4.w) < 0) return;   // none of the four
    const float4 o0 = o;
    inject_point(a, val, shot, m4.x, cv.x, o.x);
    inject_point(a, val, shot, m4.y, cv.y, o.y);
    inject_point(a, val, shot, m4.z, cv.z, o.z);
    inject_point(a, val, shot, m4.w, cv.w, o.w);
    if (D2) {
        d2.x = fmaf(o.x - o0.x, a.inv_dt2, d2.x);
        d2.y = fmaf(o.y - o0.y, a.inv_dt2, d2.y);
        d2.z = fmaf(o.z - o0.z, a.inv_dt2, d2.z);
        d2.w = fmaf(o.w - o0.w, a.inv_dt2, d2.w);
    }
}

// The time step of one warp's work item (strip, chunk) of shot `shot`; wsm is the warp's shared
// memory (prop_smem(naux_max) floats).  wid is warp-uniform and known to be so (a shuffle's result): the address
// arithmetic is then done once per warp.
template <int LOC, bool D2, bool SRC, bool INJ, bool FS>
__device__ __forceinline__ void prop_body(const PropArgs &a, const int wid, const int shot, float *wsm)
{
    constexpr bool LOCAL = LOC > 0;
    const int lane = threadIdx.x & 31;
    const int strip = wid % a.nstrip, chunk = wid / a.nstrip;
    const int x0 = strip * STRIP;
    const int x = x0 + lane * 4;
    const int z0 = (FS ? a.z_first : 4) + chunk * a.zchunk;
    const int z1 = min(z0 + a.zchunk, a.NZ - 4);
    const bool xin = x < a.NXP;
    const int NXP = a.NXP;
    const long long so = (long long)shot * a.P, row0 = (long long)z0 * NXP;
    const float *cur = a.cur + so + row0;
    const float *prev = a.prev + so + row0, *c = a.c + row0;
    float *out0 = a.out + so + row0, *d20 = D2 ? a.d2 + so + row0 : nullptr;

    // the lane's places in the rings; local sources: [f0?][f1?][f2?][coef, fc?] (LOC 1: exactly one, f0, weight a0)
    const int i_f1 = a.f0 != nullptr, i_f2 = i_f1 + (a.f1 != nullptr), i_cf = i_f2 + (a.f2 != nullptr);
    const int nloc = LOC == 2 ? i_cf + (a.fc != nullptr ? 2 : 0) : LOC;
    constexpr int AR = LOCAL ? LRING : RING;
    float *curL = wsm + 4 * lane, *prevL = curL + RING * CUR_ROW, *cL = prevL + AR * STRIP, *fL = cL + AR * STRIP;
    // The lane's columns: of the q^n row with its halo, of the row's end (two lanes), its own; relative to row z0, and
    // moved down with z.  A column outside reads nothing (zero-filled).
    const int cA = x0 - 4 + 4 * lane, cB = cA + STRIP;
    const int nA = cA >= 0 && cA + 4 <= NXP ? 16 : 0, nB = cB + 4 <= NXP ? 16 : 0, nX = xin ? 16 : 0;
    const bool two = lane < CUR_ROW / 4 - 32;
    int oA = nA ? cA : 0, oB = nB ? cB : 0, oX = nX ? x : 0;
    // row z + k into slot s
    const auto issue_cur = [&](int z, int k, int s) {
        if (z + k > z1 + 3) return;
        const float *src = cur + (long long)k * NXP;
        cp16n(curL + s * CUR_ROW, src + oA, nA);
        if (two) cp16n(curL + s * CUR_ROW + STRIP, src + oB, nB);
    };
    const auto issue_aux = [&](int z, int k, int s) {
        if (z + k >= z1) return;
        cp16n(prevL + s * STRIP, prev + (long long)k * NXP + oX, nX);
        cp16n(cL + s * STRIP, c + (long long)k * NXP + oX, nX);
    };
    const auto issue_f = [&](int z, int k, int s) {
        if (z + k >= z1) return;
        // local sources vanish outside the source rows: zero-filled there, not read
        const bool lin = z + k >= a.zs_lo && z + k < a.zs_hi;
        const int n = lin ? nX : 0;
        const long long o = row0 + (lin ? (long long)k * NXP + oX : 0);
        float *dst = fL + s * nloc * STRIP;
        if (LOC == 1) {
            cp16n(dst, a.f0 + so + o, n);
        } else {
            if (a.f0) cp16n(dst, a.f0 + so + o, n);
            if (a.f1) cp16n(dst + i_f1 * STRIP, a.f1 + so + o, n);
            if (a.f2) cp16n(dst + i_f2 * STRIP, a.f2 + so + o, n);
            if (a.fc) {
                cp16n(dst + i_cf * STRIP, a.coef + o, n);
                cp16n(dst + (i_cf + 1) * STRIP, a.fc + so + o, n);
            }
        }
    };

    // register queue rows z0-4 .. z0+3
    float4 q[9];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float *qp = cur + (long long)(k - 4) * NXP + oX;
        q[k] = xin ? ldcg4(qp) : f4zero();
    }
    // prologue: one group per row of look-ahead (rows z0 .. z0+3 feed the first x-taps)
    constexpr int DEPTH = LOCAL ? LRING : 4;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        issue_cur(z0, g, g);
        if (g < DEPTH) {
            issue_cur(z0, g + 4, g + 4);
            issue_aux(z0, g, g);
            if (LOCAL) issue_f(z0, g, g);
            if (g < DEPTH - 1 || DEPTH == 4) cp_commit();
        }
    }
    if (DEPTH < 4) cp_commit();
    const float4 gxv = xin ? ldg4(a.gx + x) : f4zero();

    int srow = -1, scol = -1;   // the point source's row, and its column within this lane's four
    float amp = 0.f;
    if (SRC) {
        const int off = a.src_off[shot];
        srow = off / NXP;
        scol = off - srow * NXP - x;
        if (scol < 0 || scol > 3) srow = -1;
        amp = a.src_amp[(long long)shot * a.src_stride] * a.src_scale;
    }

    // One output row z; the queue's logical row k (z-4+k) lives in q[(k + R) % 9], so nine consecutive rows rotate
    // the queue through the registers without moving any of them.
#define FWIME_PROP_ROW(R)                                                                                    \
    {                                                                                                        \
        cp_wait<DEPTH - 1>();                                                                                \
        __syncwarp(); /* every lane's copies are there, and every lane is done with the row before */        \
        issue_cur(z, 4 + DEPTH, (4 + DEPTH + (R)) % RING);                                                   \
        if (!LOCAL) issue_aux(z, DEPTH, (DEPTH + (R)) % AR);                                                 \
        if (!LOCAL) cp_commit();                                                                             \
        q[(8 + (R)) % 9] = lds4(curL + ((R) + 4) % RING * CUR_ROW + 4);                                      \
        const float4 L = lds4(curL + (R) * CUR_ROW), Rr = lds4(curL + (R) * CUR_ROW + 8);                    \
        const float4 pv = lds4(prevL + (R) % AR * STRIP), cv = lds4(cL + (R) % AR * STRIP);                  \
        float4 lf0 = f4zero(), lf1 = f4zero(), lf2 = f4zero(), lcf = f4zero(), lfc = f4zero();               \
        if (LOCAL) {                                                                                         \
            const float *arow = fL + ((R) % LRING) * nloc * STRIP;                                           \
            if (LOC == 1) {                                                                                  \
                lf0 = lds4(arow);                                                                            \
            } else {                                                                                         \
                if (a.f0) lf0 = lds4(arow);                                                                  \
                if (a.f1) lf1 = lds4(arow + i_f1 * STRIP);                                                   \
                if (a.f2) lf2 = lds4(arow + i_f2 * STRIP);                                                   \
                if (a.fc) { lcf = lds4(arow + i_cf * STRIP); lfc = lds4(arow + (i_cf + 1) * STRIP); }        \
            }                                                                                                \
            __syncwarp(); /* the slot's next row may come */                                                 \
            issue_aux(z, DEPTH, (R) % AR);                                                                   \
            issue_f(z, DEPTH, (R) % LRING);                                                                  \
            cp_commit();                                                                                     \
        }                                                                                                    \
        const int sj = SRC && z == srow ? scol : -1;                                                         \
        float4 o, d2;                                                                                        \
        row_math<LOC, D2, SRC>(a, prop_k(a), L, q[(0 + (R)) % 9], q[(1 + (R)) % 9], q[(2 + (R)) % 9], q[(3 + (R)) % 9], \
                                 q[(4 + (R)) % 9], q[(5 + (R)) % 9], q[(6 + (R)) % 9], q[(7 + (R)) % 9],      \
                                 q[(8 + (R)) % 9], Rr, pv, cv, lf0, lf1, lf2, lcf, lfc, __ldg(a.gz + z), gxv, sj, amp, o, d2); \
        if (xin) {                                                                                           \
            st4(out0 + oX, o);                                                                               \
            if (D2 && z >= a.zs_lo && z < a.zs_hi) st4(d20 + oX, d2);                                        \
        }                                                                                                    \
        ++z;                                                                                                 \
        oA += NXP;                                                                                           \
        oB += NXP;                                                                                           \
        oX += NXP;                                                                                           \
        if (z >= z1) break;                                                                                  \
    }

    for (int z = z0;;) {
        FWIME_PROP_ROW(0) FWIME_PROP_ROW(1) FWIME_PROP_ROW(2) FWIME_PROP_ROW(3) FWIME_PROP_ROW(4)
        FWIME_PROP_ROW(5) FWIME_PROP_ROW(6) FWIME_PROP_ROW(7) FWIME_PROP_ROW(8)
    }
#undef FWIME_PROP_ROW
    cp_wait<0>();
    float *out = a.out + so;
    if (INJ && xin) {
        // receivers in this warp's rows: each lane adds the injection to the outputs it wrote itself (read
        // back by the writing thread), after the march so the loop above keeps its registers
        const int zlo = max(z0, a.inj_lo), zhi = min(z1, a.inj_hi);
        for (int zz = zlo; zz < zhi; ++zz) {
            const int4 m4 = *reinterpret_cast<const int4 *>(a.inj_map + (long long)(zz - a.inj_lo) * NXP + x);
            if ((m4.x & m4.y & m4.z & m4.w) < 0) continue;   // none of the lane's four points
            const long long idx = (long long)zz * NXP + x;
            const float4 o0 = *reinterpret_cast<const float4 *>(out + idx);
            float4 o = o0;
            const float4 cv = ldg4(a.c + idx);
            inject_point(a, a.inj_val, shot, m4.x, cv.x, o.x);
            inject_point(a, a.inj_val, shot, m4.y, cv.y, o.y);
            inject_point(a, a.inj_val, shot, m4.z, cv.z, o.z);
            inject_point(a, a.inj_val, shot, m4.w, cv.w, o.w);
            st4(out + idx, o);
            if (D2 && zz >= a.zs_lo && zz < a.zs_hi) {
                // the D2t output gains the injection too: d2 + (o - o0) / dt^2
                float *dp = a.d2 + so + idx;
                float4 d = *reinterpret_cast<const float4 *>(dp);
                d.x = fmaf(o.x - o0.x, a.inv_dt2, d.x);
                d.y = fmaf(o.y - o0.y, a.inv_dt2, d.y);
                d.z = fmaf(o.z - o0.z, a.inv_dt2, d.z);
                d.w = fmaf(o.w - o0.w, a.inv_dt2, d.w);
                st4(dp, d);
            }
        }
    }
    if (FS && xin) {
        // Free surface (pressure release on row fs_row, where the march starts): q = 0 and D2t = 0 there, and the four
        // rows above hold the odd mirror of the four below, each written by the lane that owns the row below (which
        // it reads back: its own stores, injection included); rows further up stay zero.  As a launch of its own
        // after every step this took 6.6 us, a fifth of an objective call (16 shots on 302 x 1001 points).
        const int zlo = max(z0, a.fs_row), zhi = min(z1, a.fs_row + 5);
        for (int zz = zlo; zz < zhi; ++zz) {
            const long long idx = (long long)zz * NXP + x;
            if (zz == a.fs_row) {
                st4(out + idx, f4zero());
                if (D2) st4(a.d2 + so + idx, f4zero());
            } else {
                const float4 o = *reinterpret_cast<const float4 *>(out + idx);
                st4(out + (long long)(2 * a.fs_row - zz) * NXP + x, make_float4(-o.x, -o.y, -o.z, -o.w));
            }
        }
    }
}

// FS: free surface (variants of their own: its registers cost the others 6 % of their time).
// INJ: the receivers' injection into the output (the adjoint step; LOC = 0, no point source; with D2 the
// injection reaches the D2t output as well)
template <int LOC, bool D2, bool SRC, bool INJ, bool FS>
__global__ void __launch_bounds__(PROP_WARPS * 32, LOC == 2 ? FWIME_PROP_MIN_BLOCKS
                                                            : (LOC == 1 ? FWIME_PROP_MINB_LOC1 : FWIME_PROP_MINB_PLAIN))
    k_prop(const PropArgs a)
{
    extern __shared__ float4 smem4[];
    // Launched while the previous launch's last CTAs still run (below): its results are there after the wait.  Only
    // this kernel lets its successor in early, and after its own wait, so whatever older launches wrote is there too.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (a.rec_d && blockIdx.x == 0) {         // receivers of the input field (the previous step's output)
        const long long s = blockIdx.y;
        for (int r = threadIdx.x; r < a.nrec; r += PROP_WARPS * 32) {
            const float val = a.cur[s * a.P + a.rec_off[r]];
            float *dp = a.rec_d + s * a.rec_dstride + r;
            *dp = a.rec_acc ? *dp + val : val;
        }
    }
    const int wic = warp_in_cta();
    const int wid = blockIdx.x * PROP_WARPS + wic;
    if (wid >= a.nstrip * a.nchunk) return;   // warp-uniform
    float *wsm = reinterpret_cast<float *>(smem4) + wic * prop_smem(a.naux_max);
    prop_body<LOC, D2, SRC, INJ, FS>(a, wid, blockIdx.y, wsm);
}

template <bool FS, int LOC, bool D2, bool SRC, bool INJ = false>
static void launch_prop_t(const PropArgs &a, dim3 grid, dim3 block, size_t smem, cudaStream_t st)
{
    // once per instantiation and device
    static PerDevice<cudaError_t> attr;
    (void)attr.get([] {
        return cudaFuncSetAttribute(k_prop<LOC, D2, SRC, INJ, FS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    });
    // The next step's CTAs come in as soon as this one's are all under way and wait there, so that a step starts
    // without the launch gap: 2 to 3 us per step (100 shots on 408 x 1816 points 170 / 167 us, 30 shots 61 / 59 us).
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    (void)cudaLaunchKernelEx(&cfg, k_prop<LOC, D2, SRC, INJ, FS>, a);   // the caller reads the last error
}
template <bool FS>
static cudaError_t dispatch_prop(const PropArgs &a0, int nshot, cudaStream_t st)
{
    PropArgs a = a0;
    prop_pairs(a);
    const int nwarps = a.nstrip * a.nchunk;
    dim3 grid((nwarps + PROP_WARPS - 1) / PROP_WARPS, nshot);
    dim3 block(PROP_WARPS * 32);
    const bool local = a.f0 || a.f1 || a.f2 || a.fc;
    const bool d2 = a.d2 != nullptr;
    const bool src = a.src_off != nullptr;
    a.naux_max = 2 + (local ? (a.f0 != nullptr) + (a.f1 != nullptr) + (a.f2 != nullptr) + (a.fc ? 2 : 0) : 0);
    const size_t smem = (size_t)PROP_WARPS * prop_smem(a.naux_max) * sizeof(float);
    const int loc = !local ? 0 : (a.f1 || a.f2 || a.fc || !a.f0) ? 2 : 1;
    const int key = loc * 4 + (d2 ? 2 : 0) + (src ? 1 : 0);
    if (a.inj_val) {                           // the caller injects only into plain steps, with or without D2t
        if (key != 0 && key != 2) return cudaErrorInvalidValue;
        if (d2) launch_prop_t<FS, 0, true, false, true>(a, grid, block, smem, st);
        else launch_prop_t<FS, 0, false, false, true>(a, grid, block, smem, st);
        return cudaGetLastError();
    }
    switch (key) {                             // no operator has a point source and local sources in one step
    case 0: launch_prop_t<FS, 0, false, false>(a, grid, block, smem, st); break;
    case 1: launch_prop_t<FS, 0, false, true>(a, grid, block, smem, st); break;
    case 2: launch_prop_t<FS, 0, true, false>(a, grid, block, smem, st); break;
    case 3: launch_prop_t<FS, 0, true, true>(a, grid, block, smem, st); break;
    case 4: launch_prop_t<FS, 1, false, false>(a, grid, block, smem, st); break;
    case 6: launch_prop_t<FS, 1, true, false>(a, grid, block, smem, st); break;
    case 8: launch_prop_t<FS, 2, false, false>(a, grid, block, smem, st); break;
    case 10: launch_prop_t<FS, 2, true, false>(a, grid, block, smem, st); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace fwk
