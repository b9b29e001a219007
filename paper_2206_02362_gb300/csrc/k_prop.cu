// Stencil launches without a free surface, grouped forward steps, receiver points (kernel: fwime_prop.cuh).
#include <algorithm>

#include "fwime_prop.cuh"

namespace fwk {

cudaError_t launch_prop_surface(const PropArgs &a, int nshot, cudaStream_t st);   // k_prop_fs.cu

// ------------------------------------------------------------- grouped forward
// One launch advances one time step of every member of a group of shot batches on grids of
// different sizes (and different record lengths): CTA b belongs to the member whose cta_begin is
// the largest <= b.  Members are sorted by decreasing nt, so the members still running at a step
// are a prefix and the grid covers exactly their CTAs.
__global__ void __launch_bounds__(PROP_WARPS * 32, 4) k_prop_group(const GroupMember *__restrict__ m, int nactive, int step)
{
    extern __shared__ float4 smem4[];
    __shared__ PropArgs sa;
    int lo = 0, hi = nactive - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (m[mid].cta_begin <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    if (threadIdx.x == 0) {
        sa = m[lo].a[step & 1];
        sa.src_amp += step;
    }
    __syncthreads();
    const int local = (int)blockIdx.x - m[lo].cta_begin;
    const int cps = m[lo].ctas_per_shot;
    const int shot = local / cps;
    const int wic = warp_in_cta();
    const int wid = (local - shot * cps) * PROP_WARPS + wic;
    if (wid >= sa.nstrip * sa.nchunk) return;   // warp-uniform
    float *wsm = reinterpret_cast<float *>(smem4) + wic * prop_smem(2);
    prop_body<0, false, true, false, false>(sa, wid, shot, wsm);
}

// after step n the new field q^{n+1} of a member is in buffer B for even n, A for odd n
__global__ void k_points_group(const GroupRec *__restrict__ g, int nactive, int step)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int lo = 0, hi = nactive - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g[mid].rec_begin <= i) lo = mid; else hi = mid - 1;
    }
    const GroupRec &r = g[lo];
    const int local = i - r.rec_begin;
    if (local >= r.nshot * r.nrec) return;
    const int s = local / r.nrec, k = local - s * r.nrec;
    const float *f = (step & 1) ? r.fA : r.fB;
    r.d[(long long)s * r.nt * r.nrec + (long long)(step + 1) * r.nrec + k] = f[(long long)s * r.P + r.rec_off[k]];
}

cudaError_t launch_prop_group(const GroupMember *m, int nactive, int ctas, const GroupRec *g, int nrec_threads,
                              int step, cudaStream_t st, bool record)
{
    const size_t smem = (size_t)PROP_WARPS * prop_smem(2) * sizeof(float);
    static PerDevice<cudaError_t> attr;
    const cudaError_t e = attr.get(
        [&] { return cudaFuncSetAttribute(k_prop_group, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); });
    if (e != cudaSuccess) return e;
    if (!record) {
        k_prop_group<<<ctas, PROP_WARPS * 32, smem, st>>>(m, nactive, step);
    } else {
        k_points_group<<<(nrec_threads + 127) / 128, 128, 0, st>>>(g, nactive, step);
    }
    return cudaGetLastError();
}

// Resident CTAs per SM of the plain (no local source) variant with the smem it launches with.
cudaError_t prop_occupancy(int *blocks_per_sm)
{
    const size_t smem = (size_t)PROP_WARPS * prop_smem(2) * sizeof(float);
    const cudaError_t e = cudaFuncSetAttribute(k_prop<0, false, false, false, false>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_prop<0, false, false, false, false>, PROP_WARPS * 32,
                                                         smem);
}

// Rows per warp's item: the items (strip, chunk of rows) of S shots go to `warps` resident warps in rounds of equal
// length; the split of the rows with the least (rounds + start / 2) x (rows + overhead) wins: overhead is about what an
// item's start costs, start / 2 the part of a round that a launch's ramp and drain take, crowd / 2 what it costs that
// the items fill more than half of the places, so that the next launch's CTAs cannot wait there.
// Marmousi2-shaped, us per launch with the former aim of 4864 warps and with this: 32 shots 69 / 60, 50 shots 100 / 87,
// 100 shots 178 / 169.  One shot, ms per 1500 steps on 560 x 1260 points: 7.56 in 418 CTAs of 3 rows per warp, 7.15 in
// 253 of 5; per 1000 steps on 160 x 260 points: 2.71 of 2 rows, 2.55 of 1.
int chunk_rows(int rows, int nstrip, int S, long long warps, int overhead, int start, int crowd)
{
    long long best = -1;
    int best_zc = rows;
    for (int c = 1; c <= rows; ++c) {
        const int zc = (rows + c - 1) / c;
        const long long items = (long long)nstrip * S * ((rows + zc - 1) / zc);
        const long long cost = (2 * ((items + warps - 1) / warps) + start) * (zc + overhead) +
                               (2 * items > warps ? crowd : 0);
        if (best < 0 || cost <= best) { best = cost; best_zc = zc; }   // ties: the more, shorter items
    }
    return std::max(best_zc, 1);
}

cudaError_t launch_prop(const PropArgs &a, int nshot, cudaStream_t st)
{
    return a.fs_row > 0 ? launch_prop_surface(a, nshot, st) : dispatch_prop<false>(a, nshot, st);
}

// ----------------------------------------------------------------- points
// Receiver recording d[n][r] = q^n(rec_r), of the samples that no stencil launch records.
__global__ void k_points(const PointsArgs a)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const int s = blockIdx.y;
    if (r >= a.nrec) return;
    const long long off = (long long)s * a.P + a.rec_off[r];
    float val = a.f1[off];
    if (a.f2) val += a.f2[off];
    float *dp = a.d + (long long)s * a.dstride + r;
    *dp = a.accumulate ? *dp + val : val;
}

cudaError_t launch_points(const PointsArgs &a, int nshot, cudaStream_t st)
{
    dim3 grid((a.nrec + 127) / 128, nshot);
    k_points<<<grid, 128, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace fwk
