// Imaging kernels (Barnier et al., Theory section: the extended imaging condition, Eqs. 2-5; tomographic
// adjoint, Eq. 9).
//
//   image      I(x,h) += sum_{shots,steps} D(x-h) L(x+h)
//   local      G(x)   += sum D (alpha L + M2) + Ds L
//
// One launch reduces a segment's K x S (step, shot) pairs with the image accumulators in registers, so the
// image is read and written once per segment.
#include <algorithm>

#include "fwime_ext.cuh"

namespace fwk {

// ---------------------------------------------------------- extended imaging
//
// With u = x - h and w = x + h the products of one (step, shot) pair are D(u) L(w), w - u = 2 h: u and w have
// one parity, so the even and the odd samples never mix.  Taking the columns (2 k, 2 k + 1) as one packed
// pair (f32x2) makes both parities one problem in the pair index, D2[k] * L2[l], h = l - k: a banded outer
// product summed over the pairs, every multiply-add packed on registers exactly as a 16-byte load delivers
// them (no de-interleaving copies, no broadcast moves).
//
// A lane owns KA consecutive k and LB of the C = S LB offsets ha <= h < ha + C: entries (i, j), i < KA, j < LB, at
// k = k0 + i, h = ha + LB s + j, so it reads KA pairs of D and KA + LB of L.  The S lanes of a group take
// s = 0 .. S-1 and blocks k0 skewed by LB (S - 1 - s), which makes their L windows the same: a 16-byte
// shared load takes 4 cycles for 32 lanes but 2 when adjacent lanes read one address (measured), and shared-memory
// bandwidth is what limits this kernel beside HBM.  Cycles per warp and pair: 2 KA (D) + KA + LB (L).
//
// Any nh: the offsets are cut into chunks of C = 16, 24, 32 or 48 (launch_image_ext), one launch each; a chunk's
// start ha is a shift of the L window and planes outside [h_lo, h_hi] are not stored.
//
// Shared-memory layout: rows are copied in 16-byte chunks that keep their 128-byte line (an asynchronous copy
// whose lanes scatter a line over several shared rows becomes one L2 request per 16 bytes: measured 1.4 sectors
// per request and an L2 tag rate of 73 % as the limit), chunks permuted within the line (swz of their place in the stage) so that the lanes'
// blocks, M = KA / 2 chunks apart, fall on distinct banks: an exclusive or with the line number for M = 2, 4,
// nothing for M = 3.

// NW warps per CTA; MINB (MINBL: with the local terms) resident CTAs the registers are capped for; G groups of PB pairs in the copy ring
template <int S_, int LB_, int KA_, int NW_, int MINB_, int MINBL_, int G_, int PB_>
struct ImgShape {
    static constexpr int S = S_, LB = LB_, KA = KA_, NW = NW_, MINB = MINB_, MINBL = MINBL_, G = G_, PB = PB_;
    static constexpr int C = S * LB, M = KA / 2, RL = LB / KA;
    static constexpr int NI = 32 / S * NW;                     // lane groups of a CTA
    static constexpr int TX = 32 * NW, UC = 2 * KA * NI;       // threads, columns u of a CTA and s
    static constexpr int SKEW = LB * (S - 1);                  // pairs between the blocks of s = 0 and s = S - 1
    static constexpr int HALIGN = M == 3 ? 2 : 2 * M;          // ha is a multiple of this
    // chunks of 4 columns of a pair's rows: D from column ub; L from the 32-column line that holds column
    // ub + 2 (ha + SKEW) (at most 28 columns before it); second adjoint field and scattered D2t (local terms)
    // from the line that holds the first column of the h = 0 plane
    static constexpr int ND = (UC / 4 + SKEW / 2 + 7) / 8 * 8, NL = (UC / 4 + LB / 2 + 7 + 7) / 8 * 8;
    static constexpr int NM = (UC / 4 + 7 + 31) / 32 * 32;    // swz(c + NM) = swz(c) + NM
    template <bool LOCAL> static constexpr int stg() { return ND + NL + (LOCAL ? 2 * NM : 0); }   // chunks
    template <bool LOCAL> static constexpr int smem_chunks() { return PB * G * stg<LOCAL>(); }
    static_assert(KA % 2 == 0 && LB % KA == 0 && M >= 2 && M <= 4 && UC % 32 == 0 && SKEW % HALIGN == 0, "block shape");
    __device__ __forceinline__ static int swz(int c)
    {
        return M == 2 ? c ^ ((c >> 3) & 1) : M == 4 ? c ^ ((c >> 3) & 3) : c;
    }
    // chunk q < M of the block of chunks M X .. that starts at byte offset blk = 16 swz(M X) of a region
    __device__ __forceinline__ static int sub(int blk, int q) { return M == 3 ? blk + 16 * q : blk ^ 16 * q; }
};

// LOCAL: also the local imaging terms (alpha D L + D M2 + Ds L at h = 0) into img_local, which otherwise
// take their own k_image_local launch re-reading D and L
template <class Sh, bool LOCAL>
__global__ void __launch_bounds__(Sh::TX, LOCAL ? Sh::MINBL : Sh::MINB)
    k_image_band(const ImgArgs a, int u_lo, int ha, int h_lo, int h_hi)
{
    constexpr int S = Sh::S, KA = Sh::KA, LB = Sh::LB, M = Sh::M, C = Sh::C, TX = Sh::TX, UC = Sh::UC;
    constexpr int ND = Sh::ND, NL = Sh::NL, NM = Sh::NM;
    constexpr int STG = Sh::template stg<LOCAL>(), NS = Sh::PB * Sh::G;
    extern __shared__ float4 sm4[];
    const int t = threadIdx.x, lane = t & 31;
    const int s = lane % S, ig = t / S;                         // lane group of the CTA
    const long long rowoff = (long long)(a.z_lo + blockIdx.y) * a.NXP;
    const int ub = u_lo + UC * blockIdx.x;                      // multiple of 32
    const int lcol = ub + 2 * (ha + Sh::SKEW), lsh = (lcol & 31) >> 2;   // first column, its chunk in its line
    const int s0 = LOCAL ? -ha / LB : 0;                        // the s that owns h = 0
    const int mcol = ub + 2 * LB * (S - 1 - s0), msh = (mcol & 31) >> 2;
    const unsigned sbase = static_cast<unsigned>(__cvta_generic_to_shared(sm4));

    // Copy plan: round r of this thread copies chunk t + TX r of the list [D | L | M2 | Ds], which is also its place
    // in the stage.  The source pointer moves by one plane per pair, and by the ring's own step when the time
    // slot changes.  Chunks outside the row are never copied: every stage holds zeros there.
    constexpr int NCH = ND + NL + (LOCAL ? 2 * NM : 0), RC = (NCH + TX - 1) / TX;
    static_assert(TX % 32 == 0 && RC <= 32, "swz(id + TX r) = swz(id) + TX r");
    const float *src[RC];
    unsigned copies = 0;                                        // bit r: round r has a chunk to copy
    const unsigned dst = sbase + 16u * Sh::swz(t);
#pragma unroll
    for (int r = 0; r < RC; ++r) {
        const int id = t + TX * r;
        const RingRef &g = id < ND ? a.D : id < ND + NL ? a.L : id < ND + NL + NM ? a.M2 : a.Ds;
        const int col = id < ND ? ub + 4 * id : id < ND + NL ? lcol + 4 * (id - ND - lsh)
                        : mcol + 4 * (id - ND - NL - (id < ND + NL + NM ? 0 : NM) - msh);
        const bool ok = col >= 0 && col < a.NXP && id < NCH;
        const int slot = g.mod > 0 ? (a.n0 + g.shift) % g.mod : g.shift;
        src[r] = g.base + rowoff + (ok ? col : 0) + (long long)slot * g.slot_stride;
        if (ok) copies |= 1u << r;
        else if (id < NCH)
            for (int k = 0; k < NS; ++k) sm4[k * STG + Sh::swz(id)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const auto slot0 = [&](const RingRef &g) { return g.mod > 0 ? (a.n0 + g.shift) % g.mod : -1; };
    int sl_d = slot0(a.D), sl_l = slot0(a.L), sl_m = LOCAL ? slot0(a.M2) : 0, sl_s = LOCAL ? slot0(a.Ds) : 0;
    // from the last shot's plane of a slot to the first of the next one (direct rings, mod = 0, never wrap)
    const auto step = [&](const RingRef &g, int &sl) -> long long {
        long long d = g.slot_stride - (long long)(a.S - 1) * a.P;
        if (g.mod > 0 && ++sl == g.mod) {
            sl = 0;
            d -= g.mod * g.slot_stride;
        }
        return d;
    };
    int p_in = 0, s_in = 0;
    unsigned so = 0;                                            // byte offset of the stage being filled
    auto issue = [&]() {                                        // the next PB pairs, one copy group
#pragma unroll
        for (int u = 0; u < Sh::PB; ++u) {
            if (p_in < a.npair) {
#pragma unroll
                for (int r = 0; r < RC; ++r)
                    if (copies >> r & 1) cpa16(dst + so + 16u * TX * r, src[r], true);
                if (++s_in == a.S) {
                    s_in = 0;
                    const long long dd = step(a.D, sl_d), dl = step(a.L, sl_l);
                    const long long dm = LOCAL ? step(a.M2, sl_m) : 0, ds = LOCAL ? step(a.Ds, sl_s) : 0;
#pragma unroll
                    for (int r = 0; r < RC; ++r) {
                        const int id = t + TX * r;
                        src[r] += id < ND ? dd : id < ND + NL ? dl : id < ND + NL + NM ? dm : ds;
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < RC; ++r) src[r] += a.P;
                }
            }
            ++p_in;
            so = so + 16u * STG == 16u * NS * STG ? 0u : so + 16u * STG;
        }
        cpa_commit();
    };

    f32x2 acc[KA][LB];
#pragma unroll
    for (int i = 0; i < KA; ++i)
#pragma unroll
        for (int j = 0; j < LB; ++j) acc[i][j] = pk(0.f, 0.f);
    // local terms: thread t owns the column pairs t, t + TX of the UC columns from mcol (h = 0: x = u = w)
    constexpr int NLP = LOCAL ? (UC / 2 + TX - 1) / TX : 0;
    f32x2 loc[NLP > 0 ? NLP : 1];
    int o_ld[NLP > 0 ? NLP : 1], o_ll[NLP > 0 ? NLP : 1], o_lm[NLP > 0 ? NLP : 1];   // byte offsets in a stage
#pragma unroll
    for (int r = 0; r < NLP; ++r) {
        const int gp = min(t + TX * r, UC / 2 - 1), col0 = mcol + 2 * gp;
        loc[r] = pk(0.f, 0.f);
        o_ld[r] = 16 * Sh::swz((col0 - ub) >> 2) + 8 * (gp & 1);
        o_ll[r] = 16 * Sh::swz(ND + ((col0 - lcol) >> 2) + lsh) + 8 * (gp & 1);
        o_lm[r] = 16 * Sh::swz(ND + NL + (gp >> 1) + msh) + 8 * (gp & 1);
    }
    // byte offsets in a stage of the lane's D block and of the blocks of its L window
    constexpr int NQ = (KA + LB) / 2, NA = (NQ + M - 1) / M;
    const char *smb = reinterpret_cast<const char *>(sm4);
    const int o_d = 16 * Sh::swz(M * (ig + Sh::RL * (S - 1 - s)));
    int o_l[NA];
#pragma unroll
    for (int k = 0; k < NA; ++k) o_l[k] = 16 * Sh::swz(ND + M * (ig + k) + lsh);
    auto pair = [&](int st, int so2) {                          // byte offset of the group's stages, of the pair's in it
        f32x2 d[KA];
#pragma unroll
        for (int q = 0; q < M; ++q) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(smb + Sh::sub(o_d + st, q) + so2);
            d[2 * q] = v.x;
            d[2 * q + 1] = v.y;
        }
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(smb + Sh::sub(o_l[q / M] + st, q % M) + so2);
            const f32x2 l[2] = {v.x, v.y};
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int i = 0; i < KA; ++i) {
                    const int j = 2 * q + e - i;
                    if (j >= 0 && j < LB) acc[i][j] = fma2(d[i], l[e], acc[i][j]);
                }
        }
#pragma unroll
        for (int r = 0; r < NLP; ++r) {
            const auto ld = [&](int off) { return *reinterpret_cast<const f32x2 *>(smb + off + st + so2); };
            loc[r] = fma2(ld(o_lm[r] + 16 * NM), ld(o_ll[r]), fma2(ld(o_ld[r]), ld(o_lm[r]), loc[r]));
        }
    };
    // PB pairs per barrier; an iteration waits for its group, then refills the stages of the iteration before,
    // which every warp has left
#pragma unroll 1
    for (int g = 0; g < Sh::G - 1; ++g) issue();
    int st_c = 0;
#pragma unroll 1
    for (int p = 0; p < a.npair; p += Sh::PB) {
        cpa_wait<Sh::G - 2>();
        if constexpr (Sh::NW == 1) __syncwarp();
        else __syncthreads();
        issue();
#pragma unroll
        for (int u = 0; u < Sh::PB; ++u)
            if (u == 0 || p + u < a.npair) pair(st_c, u * 16 * STG);
        st_c = st_c + Sh::PB * 16 * STG == 16 * NS * STG ? 0 : st_c + Sh::PB * 16 * STG;
    }
    cpa_wait<0>();
    // Image update through shared memory, HP planes at a time: plane h of the CTA's columns u is the
    // contiguous row segment x = u + h.  (Straight from the accumulators a warp would touch one 8-byte pair per
    // block of k: a quarter of each 32-byte sector.)
    float *sm = reinterpret_cast<float *>(sm4);
    constexpr int AVAIL = 4 * Sh::template smem_chunks<LOCAL>() - (LOCAL ? UC : 0);
    constexpr int HP = AVAIL / UC < C ? AVAIL / UC : C;
    static_assert(HP >= 1, "epilogue tile");
    float *ltile = sm + HP * UC;
#pragma unroll 1
    for (int r0 = 0; r0 < C; r0 += HP) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < KA; ++i)
#pragma unroll
            for (int j = 0; j < LB; ++j) {
                const int rel = LB * s + j - r0;                // plane h = ha + LB s + j of this pass
                if (rel >= 0 && rel < HP)
                    *reinterpret_cast<f32x2 *>(sm + rel * UC + 2 * (KA * ig + i)) = acc[i][j];
            }
        if (LOCAL && r0 == 0) {
#pragma unroll
            for (int r = 0; r < NLP; ++r)
                if (t + TX * r < UC / 2) *reinterpret_cast<f32x2 *>(ltile + 2 * (t + TX * r)) = loc[r];
        }
        __syncthreads();
        for (int id = t; id < HP * UC; id += TX) {
            const int rr = id / UC, ul = id % UC, h = ha + r0 + rr;
            if (r0 + rr >= C || h < h_lo || h > h_hi) continue;
            const int x = ub + 2 * LB * (S - 1 - (r0 + rr) / LB) + ul + h;
            if (x < a.x_lo || x >= a.x_hi) continue;
            const float v = sm[id];
            a.img[(long long)(h + a.hm) * a.P + rowoff + x] += v;
            if (LOCAL && h == 0) a.img_local[rowoff + x] += fmaf(a.alpha, v, ltile[ul]);
        }
    }
}

template <class Sh, bool LOCAL>
static void launch_band_t(const ImgArgs &a, int ha, int h_lo, int h_hi, cudaStream_t st)
{
    constexpr size_t smem = Sh::template smem_chunks<LOCAL>() * 16;
    // once per instantiation and device
    static PerDevice<cudaError_t> attr;
    (void)attr.get([] {
        return cudaFuncSetAttribute(k_image_band<Sh, LOCAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    // u = x - h of the physical columns: lane s of the CTA at ub covers [ub + 2 LB (S-1-s), .. + UC)
    int u_lo = a.x_lo - ha - Sh::LB * (2 * Sh::S - 1) + 1;
    u_lo -= ((u_lo % 32) + 32) % 32;                            // whole 128-byte lines
    const int u_hi = a.x_hi - ha - Sh::SKEW;
    dim3 grid((u_hi - u_lo + Sh::UC - 1) / Sh::UC, a.z_hi - a.z_lo);
    k_image_band<Sh, LOCAL><<<grid, Sh::TX, smem, st>>>(a, u_lo, ha, h_lo, h_hi);
}

// one launch for the offsets h_lo .. at most h_hi that fit Sh::C; returns the last one covered
template <class Sh>
static int launch_band(const ImgArgs &a, int h_lo, cudaStream_t st)
{
    const int ha = h_lo - ((h_lo % Sh::HALIGN) + Sh::HALIGN) % Sh::HALIGN;
    const int h_hi = std::min(ha + Sh::C - 1, a.hm);
    if (a.img_local && h_lo <= 0 && h_hi >= 0) launch_band_t<Sh, true>(a, ha, h_lo, h_hi, st);
    else launch_band_t<Sh, false>(a, ha, h_lo, h_hi, st);
    return h_hi;
}

// Shapes <S, LB, KA, NW, MINB, MINBL, G, PB> by chunk size C = S LB, the best of about twenty measured per size.
// Small lane blocks at 128 registers (16 warps per SM) beat larger ones with fewer shared loads per product: at
// C = 32 a 4 x 16 block at 168 registers read 2.8 TB/s against 4.1, since the kernel waits on fixed latencies, not
// on one unit (FMA pipe 46 %, shared memory 57 %, DRAM 53 %, issue slots 55 %).  Two warps per CTA beat four (the
// barrier couples them: C = 24 4735 -> 4970 GB/s) and one (more window per column).  Algorithmic GB/s of a
// segment's launch against the parity-split kernel before (Marmousi2-shaped nh 21, North-Sea-shaped nh 31 with the
// local terms, Salt-shaped nh 41 with them): 3548 -> 4970, 2554 -> 5815, 1335 -> 1893 (56 pairs per launch; 3715
// with 256).  Another nh had a generic kernel (101 offsets: 176 -> 419 GB/s).
#ifndef FWIME_IMG_S16
#define FWIME_IMG_S16 4, 4, 4, 2, 8, 8, 5, 2
#endif
#ifndef FWIME_IMG_S24
#define FWIME_IMG_S24 4, 6, 6, 2, 8, 6, 4, 2
#endif
#ifndef FWIME_IMG_S32
#define FWIME_IMG_S32 4, 8, 4, 2, 8, 6, 5, 2
#endif
#ifndef FWIME_IMG_S48
#define FWIME_IMG_S48 4, 12, 4, 2, 6, 6, 4, 2
#endif

static cudaError_t launch_image_ext(const ImgArgs &a, cudaStream_t st, int &launched)
{
    int h = -a.hm;
    while (h <= a.hm) {
        // the offsets left in as few launches as 48 per launch allow, as evenly as the sizes do (a size's start
        // is rounded down to its alignment: what that costs is added to the offsets wanted of it)
        const int left = a.hm - h + 1, n = (left + 1 + 47) / 48, want = (left + n - 1) / n;
        const auto slack = [&](int al) { return ((h % al) + al) % al; };
        if (want + slack(4) <= 16) h = launch_band<ImgShape<FWIME_IMG_S16>>(a, h, st);
        else if (want + slack(4) <= 24) h = launch_band<ImgShape<FWIME_IMG_S24>>(a, h, st);
        else if (want + slack(4) <= 32) h = launch_band<ImgShape<FWIME_IMG_S32>>(a, h, st);
        else h = launch_band<ImgShape<FWIME_IMG_S48>>(a, h, st);
        ++h;
        ++launched;
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------- local imaging
//
// G += sum over the pairs of D (alpha L + M2) + Ds L at h = 0: a pure stream.  A thread owns 4 consecutive
// columns (16-byte loads) of one row, columns starting at x_lo rounded down to a multiple of 4 (only
// [x_lo, x_hi) is accumulated); threads are numbered over (row, column group) so that none idles at a row's end.
// The loads of U pairs are issued together (16 per thread): with four conditional pairs in flight and a row's
// tail idle the kernel read 3827 GB/s, now 6195 (North-Sea-shaped B*, 60 shots).
constexpr int LOC_TX = 128;
template <bool FULL>   // FULL: M2 and Ds present
__global__ void __launch_bounds__(LOC_TX) k_image_local(const ImgArgs a, int xa, int ncol4, int n)
{
    constexpr int U = FULL ? 4 : 8, NF = FULL ? 4 : 2;
    const int id = blockIdx.x * LOC_TX + threadIdx.x;
    if (id >= n) return;
    const int zr = id / ncol4, X = xa + 4 * (id - zr * ncol4);
    const long long off = (long long)(a.z_lo + zr) * a.NXP + X;
    const RingRef *const rings4[4] = {&a.D, &a.L, &a.M2, &a.Ds};
    const RingRef *rings_[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) rings_[f] = rings4[f];
    const RingRef *const (&rings)[NF] = rings_;
    PairRows<NF> it;
    it.init(rings, a.n0, off);
    float acc[4][4] = {};
    auto add = [&](const float4 (&v)[NF], int u) {
        const float dv[4] = {v[0].x, v[0].y, v[0].z, v[0].w}, lv[4] = {v[1].x, v[1].y, v[1].z, v[1].w};
        const float4 m2 = v[FULL ? 2 : 0], ds = v[FULL ? 3 : 0];
        const float mv[4] = {m2.x, m2.y, m2.z, m2.w}, sv[4] = {ds.x, ds.y, ds.z, ds.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float tt = a.alpha * lv[c];
            if (FULL) tt += mv[c];
            float r = dv[c] * tt;
            if (FULL) r = fmaf(sv[c], lv[c], r);
            acc[c][u] += r;
        }
    };
    int p = 0;
#pragma unroll 1
    for (; p + U <= a.npair; p += U) {
        float4 v[U][NF];
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int f = 0; f < NF; ++f) v[u][f] = __ldg(reinterpret_cast<const float4 *>(it.row[f]));
            it.next(rings, a.S, a.P, off);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) add(v[u], u % 4);
    }
#pragma unroll 1
    for (; p < a.npair; ++p) {
        float4 v[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) v[f] = __ldg(reinterpret_cast<const float4 *>(it.row[f]));
        it.next(rings, a.S, a.P, off);
        add(v, 0);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c)
        if (X + c >= a.x_lo && X + c < a.x_hi) a.img[off + c] += (acc[c][0] + acc[c][1]) + (acc[c][2] + acc[c][3]);
}

cudaError_t launch_image(const ImgArgs &a, int mode, cudaStream_t st, int &launched)
{
    launched = 0;
    if (a.npair <= 0 || a.x_hi <= a.x_lo || a.z_hi <= a.z_lo) return cudaSuccess;
    if (!a.img || !a.D.base || !a.L.base || (a.img_local && (!a.M2.base || !a.Ds.base))) return cudaErrorInvalidValue;
    if (mode == IMG_EXT) return launch_image_ext(a, st, launched);
    const int xa = a.x_lo - a.x_lo % 4;   // 16-byte aligned: rows are NXP (a multiple of 32) floats apart
    const int ncol4 = (a.x_hi - xa + 3) / 4;
    const long long n = (long long)ncol4 * (a.z_hi - a.z_lo);
    if (n > 0x7fffffff - LOC_TX || (a.M2.base == nullptr) != (a.Ds.base == nullptr)) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)((n + LOC_TX - 1) / LOC_TX);
    launched = 1;
    if (a.M2.base) k_image_local<true><<<grid, LOC_TX, 0, st>>>(a, xa, ncol4, (int)n);
    else k_image_local<false><<<grid, LOC_TX, 0, st>>>(a, xa, ncol4, (int)n);
    return cudaGetLastError();
}

}  // namespace fwk
