// Subsurface-offset scatter and its transpose (Barnier et al., Theory section: Born modelling extended with
// horizontal subsurface offsets, Eq. 1; tomographic operator, Eq. 9).
//
//   scatter    e(y) = sum_h W(y-h, h) D(y-2h)          (sigma = +1)
//   transpose  z(u) = sum_h W(u+h, h) L(u+2h)          (sigma = -1)
//
// The weights W = b p~ (nh values per point) are shared by every shot and every time step, so one launch serves a
// segment of K time steps over all K x S (step, shot) pairs of a batch, with the weights in registers for the
// whole segment while the pairs' rows stream through a cp.async ring in shared memory: weight traffic is 1/(K S)
// of a per-step formulation.
//
// Outputs y and inputs y - 2 sigma h have one parity, so the columns (2 k, 2 k + 1) of a row form one packed pair
// (f32x2) and both parities one problem in the pair index: with g = -sigma h,
//   E2[k] = sum_g W2[k][g] * D2[k + g],
// every multiply-add packed on registers exactly as a 16-byte load delivers them.  A lane owns KA consecutive k and
// LB of the C = S LB offsets ga <= g < ga + C (KA x LB weight pairs in registers); it reads KA + LB pairs of D per
// (step, shot) pair.  The S adjacent lanes that share a block of k split the offsets and exchange their partial
// sums by shuffles so that each ends with KA / S pairs to store.  Rows keep their 128-byte lines in shared memory
// (see k_image.cu: scattered 16-byte destinations cost an L2 request each), with the chunks of a line permuted so
// that the lanes' blocks fall on distinct banks.
//
// Any nh: the offsets are cut into chunks of C (launch_scatter), one launch each, the later ones accumulating.
#include <algorithm>
#include <cmath>

#include "fwime_ext.cuh"

namespace fwk {

// NW warps per CTA; MINB resident CTAs the registers are capped for; G groups of PB pairs in the copy ring
template <int S_, int LB_, int KA_, int NW_, int MINB_, int G_, int PB_>
struct ScatShape {
    static constexpr int S = S_, LB = LB_, KA = KA_, NW = NW_, MINB = MINB_, G = G_, PB = PB_;
    static constexpr int C = S * LB, M = KA / 2;
    static constexpr int NI = 32 / S * NW;                     // lane groups of a CTA
    static constexpr int TX = 32 * NW, YC = 2 * KA * NI;       // threads, output columns of a CTA
    // chunks of 4 columns of a pair's row, from the 32-column line that holds column yb + 2 ga
    static constexpr int ND = (YC / 4 + C / 2 + 7 + 7) / 8 * 8;
    static constexpr size_t SMEM = (size_t)PB * G * ND * 16;
    static constexpr int GALIGN = M == 3 ? 2 : 2 * M;          // ga is a multiple of this
    static_assert(KA % 2 == 0 && M >= 2 && M <= 4 && YC % 32 == 0 && KA % S == 0 && LB % 2 == 0, "block shape");
    static_assert(S == 1 || LB % KA == 0, "the lanes' windows start at whole blocks");
    __device__ __forceinline__ static int swz(int c)
    {
        return M == 2 ? c ^ ((c >> 3) & 1) : M == 4 ? c ^ ((c >> 3) & 3) : c;
    }
    // chunk q < M of the block of chunks M X .. that starts at byte offset blk = 16 swz(M X)
    __device__ __forceinline__ static int sub(int blk, int q) { return M == 3 ? blk + 16 * q : blk ^ 16 * q; }
};

__device__ __forceinline__ f32x2 shfl_xor2(f32x2 v, int m)
{
    float lo, hi;
    upk(v, lo, hi);
    return pk(__shfl_xor_sync(0xffffffffu, lo, m), __shfl_xor_sync(0xffffffffu, hi, m));
}

template <class Sh>
__global__ void __launch_bounds__(Sh::TX, Sh::MINB)
    k_scatter_band(const ExtArgs a, int y_lo, int ga, int g_lo, int g_hi, int accumulate, int nsplit)
{
    constexpr int S = Sh::S, KA = Sh::KA, LB = Sh::LB, M = Sh::M, TX = Sh::TX, YC = Sh::YC, ND = Sh::ND;
    constexpr int NS = Sh::PB * Sh::G, KO = KA / S;                  // ring stages; pairs a lane stores
    extern __shared__ float4 sm4[];
    const char *smb = reinterpret_cast<const char *>(sm4);
    const int t = threadIdx.x, s = t % S, ig = t / S;
    const long long rowoff = (long long)(a.z_lo + blockIdx.y) * a.NXP;
    const int yb = y_lo + YC * blockIdx.x;                      // multiple of 32
    const int dcol = yb + 2 * ga, dsh = (dcol & 31) >> 2;       // first column read, its chunk in its line
    // this CTA's share of the (step, shot) pairs (the split fills the last wave of CTAs)
    const int pb = (int)((long long)blockIdx.z * a.npair / nsplit);
    const int pe = (int)((long long)(blockIdx.z + 1) * a.npair / nsplit);

    // Copy plan: round r of this thread copies chunk t + TX r; its source pointer moves by one plane per pair and
    // by the ring's own step when the time slot changes.  Chunks outside the row are never copied: every stage
    // holds zeros there.
    constexpr int RC = (ND + TX - 1) / TX;
    const int step0 = pb / a.S;
    int s_in = pb - step0 * a.S, sl_in = a.in.mod > 0 ? (a.n0 + a.in.shift + step0) % a.in.mod : a.in.shift + step0;
    const float *src[RC];
    unsigned copies = 0;                                        // bit r: round r has a chunk to copy
    const unsigned dst = static_cast<unsigned>(__cvta_generic_to_shared(sm4)) + 16u * Sh::swz(t);
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        const int id = t + TX * r, col = dcol + 4 * (id - dsh);
        const bool ok = col >= 0 && col < a.NXP && id < ND;
        src[r] = a.in.base + rowoff + (ok ? col : 0) + (long long)sl_in * a.in.slot_stride + (long long)s_in * a.P;
        if (ok) copies |= 1u << r;
        else if (id < ND)
            for (int k = 0; k < NS; ++k) sm4[k * ND + Sh::swz(id)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // from the last shot's plane of a slot to the first of the next one (direct rings, mod = 0, never wrap)
    const auto step = [&](const RingRef &g, int &sl) -> long long {
        long long d = g.slot_stride - (long long)(a.S - 1) * a.P;
        if (++sl == g.mod) {
            sl = 0;
            d -= g.mod * g.slot_stride;
        }
        return d;
    };
    int p_in = pb;
    unsigned so = 0;                                            // byte offset of the stage being filled
    auto issue = [&]() {                                        // the next PB pairs, one copy group
#pragma unroll
        for (int u = 0; u < Sh::PB; ++u) {
            if (p_in < pe) {
#pragma unroll
                for (int r = 0; r < RC; ++r)
                    if (copies >> r & 1) cpa16(dst + so + 16u * TX * r, src[r], true);
                if (++s_in == a.S) {
                    s_in = 0;
                    const long long d = step(a.in, sl_in);
#pragma unroll
                    for (int r = 0; r < RC; ++r) src[r] += d;
                } else {
#pragma unroll
                    for (int r = 0; r < RC; ++r) src[r] += a.P;
                }
            }
            ++p_in;
            so = so + 16u * ND == 16u * NS * ND ? 0u : so + 16u * ND;
        }
        cpa_commit();
    };
#pragma unroll 1
    for (int g = 0; g < Sh::G - 1; ++g) issue();

    // weights: pair (i, j) of the lane is W(y + g, -sigma g), y = yb + 2 (KA ig + i) + {0, 1}, g = ga + LB s + j
    f32x2 w[KA][LB];
#pragma unroll
    for (int j = 0; j < LB; ++j) {
        const int g = ga + LB * s + j;
        const bool gin = g >= g_lo && g <= g_hi;
        const float *wp = a.W + (gin ? a.hm - a.sigma * g : 0) * a.P + rowoff;
#pragma unroll
        for (int i = 0; i < KA; ++i) {
            float v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int y = yb + 2 * (KA * ig + i) + e, x = y + g;
                v[e] = gin && y < a.x_hi && x >= 0 && x < a.NXP ? __ldg(wp + x) : 0.f;
            }
            w[i][j] = pk(v[0], v[1]);
        }
    }

    // byte offsets in a stage of the blocks of the lane's D window
    constexpr int NQ = (KA + LB) / 2, NA = (NQ + M - 1) / M;
    int o_d[NA];
#pragma unroll
    for (int k = 0; k < NA; ++k) o_d[k] = 16 * Sh::swz(M * (ig + k) + LB / 2 * s + dsh);
    // the lane's output columns and their pointer, walked as the sources
    const int y0 = yb + 2 * (KA * ig + KO * s);
    const bool whole = y0 >= a.x_lo && y0 + 2 * KO <= a.x_hi;
    int s_out = pb - step0 * a.S, sl_out = a.outr.mod > 0 ? (a.n0 + a.outr.shift + step0) % a.outr.mod : a.outr.shift + step0;
    float *out = const_cast<float *>(a.outr.base) + rowoff + y0 + (long long)sl_out * a.outr.slot_stride +
                 (long long)s_out * a.P;
    // two pairs at a time: every weight is used twice in a row, and twice the chains are in flight (the second pair
    // of an odd last one reads a stale stage and is not stored)
    auto pairs = [&](int st, int so2, int n) {                  // byte offsets of the group's stages, of the two in it
        f32x2 e[2][KA];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int i = 0; i < KA; ++i) e[u][i] = pk(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            ulonglong2 v[2];
#pragma unroll
            for (int u = 0; u < 2; ++u)
                v[u] = *reinterpret_cast<const ulonglong2 *>(smb + Sh::sub(o_d[q / M] + st, q % M) + so2 + 16 * ND * u);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < KA; ++i) {
                    const int j = 2 * q + h - i;
#pragma unroll
                    for (int u = 0; u < 2; ++u)
                        if (j >= 0 && j < LB) e[u][i] = fma2(w[i][j], h ? v[u].y : v[u].x, e[u][i]);
                }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            // sum over the S lanes of the block; lane s keeps pairs KO s .. KO s + KO - 1
            f32x2 o[KO];
            if constexpr (S == 1) {
#pragma unroll
                for (int i = 0; i < KA; ++i) o[i] = e[u][i];
            } else if constexpr (S == 2) {
#pragma unroll
                for (int i = 0; i < KO; ++i) {
                    const f32x2 give = s ? e[u][i] : e[u][KO + i], keep = s ? e[u][KO + i] : e[u][i];
                    o[i] = add2(keep, shfl_xor2(give, 1));
                }
            } else {
                f32x2 m[2 * KO];
#pragma unroll
                for (int i = 0; i < 2 * KO; ++i) {
                    const f32x2 give = s & 2 ? e[u][i] : e[u][2 * KO + i], keep = s & 2 ? e[u][2 * KO + i] : e[u][i];
                    m[i] = add2(keep, shfl_xor2(give, 2));
                }
#pragma unroll
                for (int i = 0; i < KO; ++i) {
                    const f32x2 give = s & 1 ? m[i] : m[KO + i], keep = s & 1 ? m[KO + i] : m[i];
                    o[i] = add2(keep, shfl_xor2(give, 1));
                }
            }
            if (u >= n) break;                                  // uniform
            if (whole) {
                if constexpr (KO % 2 == 0) {
#pragma unroll
                    for (int i = 0; i < KO / 2; ++i) {
                        ulonglong2 *op = reinterpret_cast<ulonglong2 *>(out + 4 * i);
                        ulonglong2 v = make_ulonglong2(o[2 * i], o[2 * i + 1]);
                        if (accumulate) {
                            const ulonglong2 old = *op;
                            v = make_ulonglong2(add2(old.x, v.x), add2(old.y, v.y));
                        }
                        *op = v;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < KO; ++i) {
                        f32x2 *op = reinterpret_cast<f32x2 *>(out + 2 * i);
                        *op = accumulate ? add2(*op, o[i]) : o[i];
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < KO; ++i) {
                    float v[2];
                    upk(o[i], v[0], v[1]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int y = y0 + 2 * i + h;
                        if (y >= a.x_lo && y < a.x_hi) out[2 * i + h] = accumulate ? out[2 * i + h] + v[h] : v[h];
                    }
                }
            }
            if (++s_out == a.S) {
                s_out = 0;
                out += step(a.outr, sl_out);
            } else {
                out += a.P;
            }
        }
    };
    // PB pairs per barrier; an iteration waits for its group, then refills the stages of the iteration before,
    // which every warp has left
    int st_c = 0;
#pragma unroll 1
    for (int p = pb; p < pe; p += Sh::PB) {
        cpa_wait<Sh::G - 2>();
        if constexpr (Sh::NW == 1) __syncwarp();
        else __syncthreads();
        issue();
#pragma unroll
        for (int u = 0; u < Sh::PB; u += 2)
            if (u == 0 || p + u < pe) pairs(st_c, u * 16 * ND, min(2, pe - p - u));
        st_c = st_c + Sh::PB * 16 * ND == 16 * NS * ND ? 0 : st_c + Sh::PB * 16 * ND;
    }
    cpa_wait<0>();
}

// one launch for the offsets g_lo .. at most g_hi that fit Sh::C; returns the last one covered
template <class Sh>
static int launch_band(const ExtArgs &a, int g_lo, int accumulate, cudaStream_t st)
{
    const int ga = g_lo - ((g_lo % Sh::GALIGN) + Sh::GALIGN) % Sh::GALIGN;
    const int g_hi = std::min(ga + Sh::C - 1, a.hm);
    // once per instantiation and device: the attribute, then the CTAs resident on the device
    static PerDevice<double> resident;
    const double wave = resident.get([] {
        int r = 0, dev = 0, nsm = 0;
        cudaFuncSetAttribute(k_scatter_band<Sh>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::SMEM);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r, k_scatter_band<Sh>, Sh::TX, Sh::SMEM);
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        return (double)std::max(r, 1) * std::max(nsm, 1);
    });
    const int y_lo = a.x_lo - a.x_lo % 32;                      // whole 128-byte lines
    const int nx = (a.x_hi - y_lo + Sh::YC - 1) / Sh::YC, nz = a.z_hi - a.z_lo;
    // Every CTA streams its pairs for the whole launch, so a partly filled last wave idles SMs for long: the pairs
    // are split into nsplit <= 8 parts of at least 32, picked to fill the last wave best (the smallest within 1 %).
    // A grid that does not fill half a wave is split further, into parts of at least 8 pairs, until it does.
    int nsplit = 1;
    const double ctas = (double)nx * nz;
    if (2 * ctas < wave) {
        nsplit = std::max(1, std::min((int)(wave / ctas), a.npair / 8));
    } else {
        const auto fill = [&](int k) { return ctas * k / wave / std::ceil(ctas * k / wave); };
        double best = fill(1);
        for (int k = 2; k <= 8 && a.npair / k >= 32; ++k)
            if (fill(k) > best + 0.01) { best = fill(k); nsplit = k; }
    }
    k_scatter_band<Sh><<<dim3(nx, nz, nsplit), Sh::TX, Sh::SMEM, st>>>(a, y_lo, ga, g_lo, g_hi, accumulate, nsplit);
    return g_hi;
}

// Shapes <S, LB, KA, NW, MINB, G, PB> by chunk size C = S LB, the best of about fifteen measured per size.  One warp
// per CTA throughout: a block-wide barrier per group of pairs costs more than the wider window saves (C = 24:
// four warps 3574 GB/s, two 4219, one 4283).  Algorithmic GB/s of a segment's launch (Marmousi2-shaped, 50 shots)
// against the parity-split kernel before: nh 5 4859 -> 6086, 11 4804 -> 5691, 21 4019 -> 4441, 31 3113 -> 3180,
// 41 1975 -> 2137; another nh had a generic kernel that re-read its weights per pair (101 offsets: 65 -> 443).
// From 24 offsets up the multiply-adds bound it: FFMA2 with three distinct register pairs issues at 60-100 of the
// nominal 128 products per clock and SM in isolation.
#ifndef FWIME_SC_S8
#define FWIME_SC_S8 1, 8, 4, 1, 12, 5, 2
#endif
#ifndef FWIME_SC_S16
#define FWIME_SC_S16 2, 8, 4, 1, 16, 3, 4
#endif
#ifndef FWIME_SC_S24
#define FWIME_SC_S24 2, 12, 4, 1, 12, 4, 2
#endif
#ifndef FWIME_SC_S32
#define FWIME_SC_S32 2, 16, 4, 1, 8, 3, 4
#endif
#ifndef FWIME_SC_S48
#define FWIME_SC_S48 2, 24, 4, 1, 8, 5, 2
#endif

cudaError_t launch_scatter(const ExtArgs &a, cudaStream_t st, int &launched)
{
    launched = 0;
    if (a.npair <= 0 || a.x_hi <= a.x_lo || a.z_hi <= a.z_lo) return cudaSuccess;
    if (!a.W || !a.in.base || !a.outr.base || a.hm != (a.nh - 1) / 2) return cudaErrorInvalidValue;
    int g = -a.hm, acc = a.accumulate;
    while (g <= a.hm) {
        // the offsets left in as few launches as 48 per launch allow, as evenly as the sizes do (a size's start
        // is rounded down to a multiple of 4: what that costs is added to the offsets wanted of it)
        const int slack = ((g % 4) + 4) % 4, left = a.hm - g + 1, n = (left + slack + 47) / 48;
        const int want = (left + n - 1) / n + slack;
        if (want <= 8) g = launch_band<ScatShape<FWIME_SC_S8>>(a, g, acc, st);
        else if (want <= 16) g = launch_band<ScatShape<FWIME_SC_S16>>(a, g, acc, st);
        else if (want <= 24) g = launch_band<ScatShape<FWIME_SC_S24>>(a, g, acc, st);
        else if (want <= 32) g = launch_band<ScatShape<FWIME_SC_S32>>(a, g, acc, st);
        else g = launch_band<ScatShape<FWIME_SC_S48>>(a, g, acc, st);
        ++g;
        ++launched;
        acc = 1;
    }
    return cudaGetLastError();
}

}  // namespace fwk
