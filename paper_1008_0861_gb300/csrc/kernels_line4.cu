// Instantiations of the warp-per-line kernel and of the explicit step (FP32
// with FP32 or FP16 face coefficients, FP64), one variant per limiter family.
#include "explicit_kernel.cuh"

namespace aniso {

// A grid alone that leaves an SM at most 8 warps (of the 32 the 64-register
// form allows) waits for its loads: three rounds in flight in the 128-register
// form.  FP32 us an update, one round / three: 128^2 4.68 / 4.27, 512^2
// 5.34 / 4.63, 768^2 8.21 / 7.55, 1024^2 10.4 / 10.2, 1536^2 (10 warps) 16.9 / 17.1
bool line4_deep(int nblocks, int nthreads) { return (long)nblocks * nthreads <= 152L * 32 * 8; }

cudaError_t launch_line4(int prec, int coef_fp16, const Line2Args &a, int nblocks, int nthreads, size_t smem,
                         cudaStream_t s)
{
    const bool vl = a.limiter == LIM_VANLEER;
    // (with run-time rounds it spills, which shows where several streams fill the
    // GPU: 4 handles of 1216^2 on 4 streams, 20 steps: 1495 us one round, 2030 three)
    const bool deep = !a.jobs && line4_deep(nblocks, nthreads) && (!a.shared || a.rounds);
    if (a.fresh) {
        if (!vl || a.jobs || a.one.chi_alpha != 0.0 || coef_fp16 || (prec == PREC_FP32 && !deep)) return cudaErrorInvalidValue;
        if (prec == PREC_FP64)
            return launch_line_kernel(line4_kernel<double, double, true, false, false, false, false, 1, false, 0, true>, a, nblocks,
                        nthreads, smem, s);
        return launch_line_kernel(line4_kernel<float, float, true, false, false, false, false, 3, false, 0, true>, a, nblocks,
                    nthreads, smem, s);
    }
    if (!a.jobs && a.one.mu == 0.0 && a.one.chi_alpha == 0.0) {  // purely implicit update (4-step halves)
        if (prec == PREC_FP64)
            return launch_line_kernel(line4_kernel<double, double, false, false, false, true>, a, nblocks, nthreads, smem, s);
        if (coef_fp16)
            return launch_line_kernel(line4_kernel<float, __half, false, false, false, true>, a, nblocks, nthreads, smem, s);
        return launch_line_kernel(line4_kernel<float, float, false, false, false, true>, a, nblocks, nthreads, smem, s);
    }
    if (!a.jobs && a.one.chi_alpha != 0.0) {  // temperature-dependent diffusivity (single grids)
        if (coef_fp16) return cudaErrorInvalidValue;
        if (prec == PREC_FP64)
            return vl ? launch_line_kernel(line4_kernel<double, double, true, false, true>, a, nblocks, nthreads, smem, s)
                      : launch_line_kernel(line4_kernel<double, double, false, false, true>, a, nblocks, nthreads, smem, s);
        if (vl && deep && a.rounds) return launch_line4_rounds(0, true, a, nblocks, nthreads, smem, s);
        if (vl && deep)
            return launch_line_kernel(line4_kernel<float, float, true, false, true, false, false, 3>, a, nblocks, nthreads, smem, s);
        return vl ? launch_line_kernel(line4_kernel<float, float, true, false, true>, a, nblocks, nthreads, smem, s)
                  : launch_line_kernel(line4_kernel<float, float, false, false, true>, a, nblocks, nthreads, smem, s);
    }
    if (a.tmem && prec == PREC_FP32) {  // gamma in tensor memory
        if (a.rounds) return launch_line4_rounds_tm(coef_fp16, a, nblocks, nthreads, smem, s);
        if (coef_fp16)
            return vl ? launch_line_kernel(line4_kernel<float, __half, true, false, false, false, true>, a, nblocks, nthreads, smem, s)
                      : launch_line_kernel(line4_kernel<float, __half, false, false, false, false, true>, a, nblocks, nthreads, smem, s);
        return vl ? launch_line_kernel(line4_kernel<float, float, true, false, false, false, true>, a, nblocks, nthreads, smem, s)
                  : launch_line_kernel(line4_kernel<float, float, false, false, false, false, true>, a, nblocks, nthreads, smem, s);
    }
    if (prec == PREC_FP64)
        return vl ? launch_line_kernel(line4_kernel<double, double, true>, a, nblocks, nthreads, smem, s)
                  : launch_line_kernel(line4_kernel<double, double, false>, a, nblocks, nthreads, smem, s);
    if (prec == PREC_FP32 && a.rounds) return launch_line4_rounds(coef_fp16, deep, a, nblocks, nthreads, smem, s);
    if (vl && deep)
        return coef_fp16 ? launch_line_kernel(line4_kernel<float, __half, true, false, false, false, false, 3>, a, nblocks, nthreads, smem, s)
                         : launch_line_kernel(line4_kernel<float, float, true, false, false, false, false, 3>, a, nblocks, nthreads, smem, s);
    if (coef_fp16)
        return vl ? launch_line_kernel(line4_kernel<float, __half, true>, a, nblocks, nthreads, smem, s)
                  : launch_line_kernel(line4_kernel<float, __half, false>, a, nblocks, nthreads, smem, s);
    return vl ? launch_line_kernel(line4_kernel<float, float, true>, a, nblocks, nthreads, smem, s)
              : launch_line_kernel(line4_kernel<float, float, false>, a, nblocks, nthreads, smem, s);
}

template <typename K> static int occ4(K kern, int nthreads, size_t smem)
{
    int blocks = 0;
    if (allow_smem(kern, smem) != cudaSuccess) return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kern, nthreads, smem) != cudaSuccess) return -1;
    return blocks;
}

int line4_rounds(int prec, int limiter, int n, int team)
{
    if (prec != PREC_FP32 || limiter != LIM_VANLEER || n % 4 != 0) return 0;
    const int m = n / 4, V = (m + team - 1) / team;
    return V >= 4 && V <= 8 ? V : 0;
}

int line4_tm_cols(int n, int team)
{
    const int m = n / 4, U = m / team, V = U + (m % team ? 1 : 0);
    return 8 * V <= 32 ? 32 : 64;
}

// Chunks per lane for one FP64 grid's update on its own.  The FP64 unit of an
// SM quarter takes a warp instruction every 64 clocks however many lanes it
// serves, so an update takes as long as the FP64 instructions of the warps
// that share a quarter: about 43 a cell and 15 a level of the reduced system
// a lane, 40 besides.  Longer segments give fewer, longer warps; the team with
// the least for the most loaded of the 4 x 152 quarters wins, from the general
// rule's team (4 chunks a lane) upwards and that one at equal cost.  50^2:
// 28.6 us an update with 4 chunks a lane, 11.9 with 1; 128^2: 19.0 and 12.5;
// from 256 cells a line on both rules agree.
int line4_seg_fp64(int n, int nlines)
{
    const int m = (n + 1) / 2;
    int P = 1, top = 1, best = 4;
    while (P * 2 <= m / 4 && P < 32) P *= 2;
    while (top * 2 <= m && top < 32) top *= 2;
    long best_cost = -1;
    for (; P <= top; P *= 2) {
        const long warps = ((long)nlines * P + 31) / 32, rounds = (warps + 607) / 608;
        long levels = 0;
        while ((1 << levels) < P) ++levels;
        const long cost = rounds * (2L * 43 * ((m + P - 1) / P) + 15 * levels + 40);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = m / P;  // pow2floor(m / (m / P)) == P
        }
    }
    return best;
}

// Chunks per lane for a ragged FP32 update (0: the default 4), alone and in
// batches alike: short segments while every line can have a warp of its own
// (59 x 38, two lanes of 8 chunks a line: 11.9 us an update, 8.1 on the general
// kernel it ran on before).
int line4_seg_ragged(int nlines) { return nlines <= 608 ? 1 : 0; }

// Warps a block for one FP32 grid's update on its own.  Lines of 512 cells and
// more (one a warp) leave a four-warp block four lines wide, so its transposed
// store writes half sectors; eight warps write whole ones.  That is taken where
// eight-warp blocks fill most SMs and run in one wave (768^2: 7.55 -> 7.26 us an
// update, 1024^2: 10.2 -> 9.4; 512^2, 64 blocks: 4.63 -> 5.37; 1280^2, a second
// wave: 13.9 -> 20.4), and on the legacy default stream only: beside other streams'
// work they lose (8 handles of 768^2 on 8 streams, 20 steps: 895 -> 920 us).
int line4_warps_alone(int n, int nlines)
{
    int team, lpb, nt;
    size_t smem;
    if (!line4_config(PREC_FP32, (n + 3) & ~3, true, 8, 0, &team, &lpb, &nt, &smem) || lpb != 8 || nt != 256) return 0;
    const long blocks = ((long)nlines + 7) / 8, resident = (long)((SMEM_LIMIT - 1024) / (smem + 1024));
    return blocks >= 96 && blocks <= 152 * (resident < 4 ? resident : 4) ? 8 : 0;
}

// Whether a launch of nblocks blocks that need *smem bytes of dynamic shared
// memory each may be chained, with *smem raised where that takes more.  A chained
// launch's blocks are placed while their predecessor drains, on whichever SMs are
// free first, and with room for more than its share of the blocks one SM gets
// several of them and another none, which then lasts for the whole launch.  So
// each block asks for as much as keeps an SM to its share.  us, unchained / with
// the natural size / with this one: FP64 352 x 512, 20 steps 1218 / 2762 / 1184; FP32
// 777 x 1001, 20 steps 533 / 754 / 518; FP32 512^2 4-step 358 / 465 / 329; FP32 1024^2
// an update 9.6 / 9.7 / 9.0; 3-D FP32 136 x 192 x 60, 3 steps 160 / 201 / 141.
// That shuts other streams' blocks out of the SM (8 handles of 512^2 FP32 on 8
// streams, 20 steps: 447 us unchained, 978 with it).  It is done on the legacy
// default stream alone, whose work is not shared with other blocking streams; on a
// stream of the caller's only launches of at most 76 blocks are chained, which fit
// the chip beside the launch before, with their natural size (16 handles of 300^2,
// 40 steps: 764 us unchained, 551 so, 1468 with the raised one).
bool line4_chain(bool default_stream, int nblocks, size_t *smem)
{
    const bool few = nblocks <= 76;
    if (!default_stream) return few;
    const int share = (nblocks + 151) / 152;
    const size_t sm = (size_t)228 * 1024, least = sm / (share + 1) - 1024 + 16;
    if (share <= 4 && *smem < least) *smem = least;
    return few || (int)(sm / (*smem + 1024)) <= share;
}

// The kernel keeps 16-byte chunk c of a line at c ^ ((c >> s) & 7) inside
// its group of 8 chunks (the last, incomplete group unswizzled).  The
// coalesced phases have the 8 lanes of a quarter warp touch one whole group,
// conflict-free under any such permutation.  The segment phases have lane t
// walk chunks ce(t) - k from its segment's last down (U + 1 chunks for the first
// m mod P lanes, U for the rest) and back up, so a quarter warp's chunks lie a
// segment length apart and their bank groups (chunk mod 8) repeat unless the
// shift spreads them.  Each candidate (log2 U, none, 1..6) is scored by the wavefronts of
// those walks, the largest number of a quarter's lanes on one bank group,
// summed over the steps k and the quarters; the first lowest wins.
int line4_swizzle(int prec, int n, int team)
{
    const int N = prec == PREC_FP64 ? 2 : 4;
    const int m = (n + N - 1) / N, P = team;
    if (P < 8 || m < 8) return 0;  // a quarter warp spans several lines
    const int U = m / P, rr = m % P, V = U + (rr ? 1 : 0);
    const int mfull = m & ~7;
    int logU = 0;
    while ((2 << logU) <= U) ++logU;
    int best = 0;
    long best_w = -1;
    for (int code = 0; code <= 7; ++code) {
        const int sh = code >= 2 ? code - 1 : logU, msk = code == 1 ? 0 : 7;
        long w = 0;
        for (int k = 0; k < V; ++k)
            for (int q0 = 0; q0 < P; q0 += 8) {
                int cnt[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                for (int t = q0; t < q0 + 8; ++t) {
                    const int Ut = U + (t < rr ? 1 : 0);
                    if (k >= Ut) continue;
                    const int c = t * U + (t < rr ? t : rr) + Ut - 1 - k;
                    ++cnt[(c < mfull ? c ^ ((c >> sh) & msk) : c) & 7];
                }
                int mx = 0;
                for (int g = 0; g < 8; ++g) mx = cnt[g] > mx ? cnt[g] : mx;
                w += mx;
            }
        if (best_w < 0 || w < best_w) {
            best_w = w;
            best = code;
        }
    }
    return best;
}

int line4_blocks_per_sm(int prec, int coef_fp16, int limiter, int nthreads, size_t smem, bool tmem, int tm_cols)
{
    const bool vl = limiter == LIM_VANLEER;
    if (tmem && prec == PREC_FP32) {
        // CUDA's occupancy calculator answers 1 for a kernel that allocates
        // tensor memory, while 5-7 such blocks were measured resident.  The
        // shared-memory form has the same registers and static shared memory:
        // its answer at this dynamic size, capped by the TMEM columns (at
        // most 448 of an SM's 512 were found in use at once: seven 64-column
        // blocks where eight fit otherwise).
        const int cap = 448 / (tm_cols > 0 ? tm_cols : 64);
        const int occ = line4_blocks_per_sm(prec, coef_fp16, limiter, nthreads, smem, false);
        return occ < cap ? occ : cap;
    }
    if (prec == PREC_FP64)
        return vl ? occ4(line4_kernel<double, double, true>, nthreads, smem)
                  : occ4(line4_kernel<double, double, false>, nthreads, smem);
    if (coef_fp16)
        return vl ? occ4(line4_kernel<float, __half, true>, nthreads, smem)
                  : occ4(line4_kernel<float, __half, false>, nthreads, smem);
    return vl ? occ4(line4_kernel<float, float, true>, nthreads, smem)
              : occ4(line4_kernel<float, float, false>, nthreads, smem);
}

template <typename K> static cudaError_t run_explicit(K kern, const ExpArgs &a, cudaStream_t s)
{
    const int rows_total = (a.ny + a.rows - 1) / a.rows;
    const dim3 block(32, 8), grid((a.nx + 31) / 32, (rows_total + 7) / 8);
    kern<<<grid, block, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_explicit(int prec, int coef_fp16, const ExpArgs &a, cudaStream_t s)
{
    const bool vl = a.limiter == LIM_VANLEER;
    if (prec == PREC_FP64)
        return vl ? run_explicit(explicit_kernel<double, double, true>, a, s)
                  : run_explicit(explicit_kernel<double, double, false>, a, s);
    if (coef_fp16)
        return vl ? run_explicit(explicit_kernel<float, __half, true>, a, s)
                  : run_explicit(explicit_kernel<float, __half, false>, a, s);
    return vl ? run_explicit(explicit_kernel<float, float, true>, a, s)
              : run_explicit(explicit_kernel<float, float, false>, a, s);
}

}  // namespace aniso
