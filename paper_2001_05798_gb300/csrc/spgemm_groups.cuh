// spgemm_groups.cuh -- the row products of the setup's SpGEMM (setup.cu) by
// groups of lanes.  On its own, without other headers, so that the kernel also
// compiles for the host, where a test runs its warps in lockstep.
#pragma once

namespace gw {

__device__ __forceinline__ unsigned sg_hash(int c) { return (unsigned)c * 2654435761u; }

// A group of G lanes per row, in one pass over the products: the row's distinct
// columns in an open-addressing table in shared memory (key, and the position
// at which the column first came up), their sums by position.  The group walks
// L's row in order and its lanes take the entries of Rm's row k, which have
// distinct columns, so every output entry receives its terms in ascending k; the
// columns are rank-sorted at the end and the row goes to a temporary of CAP
// entries a row, packed once the row pointers are known (crp null); where that
// temporary would be too large, a first run only counts (oci null) and a second,
// with the row pointers crp, writes each row in its place.  A row of more than
// CAP distinct columns goes to the warp kernels' row list (the second run leaves
// it out).
// What bounds the product is the chain of dependent loads per entry of L and
// FP64 issue (a warp instruction holds the SM's FP64 units for 16 cycles however
// few lanes work): with a warp a row, 4 of 32 lanes worked on A_1 P_1 and 8 on
// R_0 (A P)_0, in two passes.  So G follows the mean row length of Rm, G entries
// of L are loaded at once and SGG_PF of their rows before the first is added.
// At 160^3 (us): A_0 P_0 1592 -> 1350 (against a thread a row with the row in
// shared memory), R_0 (A P)_0 4740 -> 1350, A_1 P_1 2890 -> 840, R_1 (A P)_1
// 1660 -> 450; at 45^3 the four together 700 -> 330.
constexpr int SGG_BS = 128, SGG_PF = 4;

template <int CAP>
constexpr size_t sgg_group_bytes()
{
    return (size_t)CAP * 8 + 2 * CAP * 4 + CAP * 4 + 2 * CAP;  // sums, keys, columns, positions
}
template <int G, int CAP>
constexpr size_t sgg_smem()
{
    return (SGG_BS / G) * (sgg_group_bytes<CAP>() + sizeof(int));
}

// position of column c in the row's table (inserted if new; >= CAP: no room).
// The table has free places at every call (k_sgg), so the search ends at one of
// them; it is bounded by the table all the same
template <int CAP>
__device__ __forceinline__ int sgg_find(volatile int *keys, volatile unsigned char *pos, int *count, int *cols,
                                        double *acc, int c)
{
    unsigned h = sg_hash(c) >> 8 & (unsigned)(2 * CAP - 1);
    for (int probe = 0; probe < 2 * CAP; ++probe) {
        const int k = keys[h];
        if (k == c) return pos[h];
        if (k == -1 && atomicCAS((int *)&keys[h], -1, c) == -1) {
            const int p = atomicAdd(count, 1);
            if (p < CAP) {
                pos[h] = (unsigned char)p;
                cols[p] = c;
                acc[p] = 0.0;
            }
            return p;
        }
        h = (h + 1) & (unsigned)(2 * CAP - 1);
    }
    return CAP;
}

template <int G, int CAP>
__global__ void __launch_bounds__(SGG_BS) k_sgg(int nr, const int *__restrict__ lrp, const int *__restrict__ lci,
                                                const double *__restrict__ lv, const int *__restrict__ rrp,
                                                const int *__restrict__ rci, const double *__restrict__ rv,
                                                const int *__restrict__ crp, int *__restrict__ cnt,
                                                int *__restrict__ oci, double *__restrict__ ov,
                                                int *__restrict__ long_rows, int *__restrict__ nlong)
{
    // the step that passes CAP columns inserts at most G more keys and is the
    // row's last (over stays set while other rows of the warp go on), so a table
    // holds CAP + G <= 3/2 CAP of its 2 CAP keys
    static_assert(G >= SGG_PF && 2 * G <= CAP && CAP <= 256, "group and table sizes");
    extern __shared__ double sgg_mem[];
    constexpr int NG = SGG_BS / G;
    const int g = threadIdx.x / G, lane = threadIdx.x & (G - 1);
    const unsigned all = 0xffffffffu;
    const unsigned mine = G == 32 ? all : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1));
    double *acc = sgg_mem + (size_t)g * CAP;
    int *keys = (int *)(sgg_mem + (size_t)NG * CAP) + (size_t)g * 2 * CAP;
    int *cols = (int *)(sgg_mem + (size_t)NG * CAP) + (size_t)NG * 2 * CAP + (size_t)g * CAP;
    int *count = (int *)(sgg_mem + (size_t)NG * CAP) + (size_t)NG * 3 * CAP + g;
    unsigned char *pos = (unsigned char *)((int *)(sgg_mem + (size_t)NG * CAP) + (size_t)NG * 3 * CAP + NG) +
                         (size_t)g * 2 * CAP;
    for (int t = lane; t < 2 * CAP / 4; t += G) reinterpret_cast<int4 *>(keys)[t] = make_int4(-1, -1, -1, -1);
    // whole warps stay together (shuffles and barriers of the warp)
    const long long step = (long long)gridDim.x * NG;
    for (long long w0 = (long long)blockIdx.x * NG + (threadIdx.x / 32) * (32 / G); w0 < nr; w0 += step) {
        const long long row = w0 + (threadIdx.x & 31) / G;
        const bool live = row < nr && !(crp && crp[row + 1] - crp[row] > CAP);
        const int e0 = live ? lrp[row] : 0, e1 = live ? lrp[row + 1] : 0;
        if (lane == 0) *count = 0;
        __syncwarp();
        bool over = false;
        for (int eb = e0; __any_sync(all, eb < e1 && !over); eb += G) {
            int rs = 0, rl = 0;
            double a = 0.0;
            if (eb + lane < e1 && !over) {
                const int k = lci[eb + lane];
                a = lv[eb + lane];
                rs = rrp[k];
                rl = rrp[k + 1] - rs;
            }
            for (int t0 = 0; t0 < G && __any_sync(all, eb + t0 < e1 && !over); t0 += SGG_PF) {
                int c[SGG_PF], n[SGG_PF], s[SGG_PF];
                double v[SGG_PF];
#pragma unroll
                for (int t = 0; t < SGG_PF; ++t) {
                    s[t] = __shfl_sync(all, rs, t0 + t, G);
                    n[t] = __shfl_sync(all, rl, t0 + t, G);
                    c[t] = 0;
                    v[t] = 0.0;
                    if (lane < n[t]) {
                        c[t] = rci[s[t] + lane];
                        v[t] = rv[s[t] + lane];
                    }
                }
                // one product per lane: the lanes find their places, meet, and add
                // (added where its search ended, a sum would take an FP64 instruction
                // per distinct end of the search)
                auto add = [&](bool on, int col, double prod) {
                    const int p = on && !over ? sgg_find<CAP>(keys, pos, count, cols, acc, col) : CAP;
                    __syncwarp();
                    if (p < CAP) acc[p] = __dadd_rn(acc[p], prod);
                    over = (__ballot_sync(all, over || (on && p >= CAP)) & mine) != 0;
                };
#pragma unroll
                for (int t = 0; t < SGG_PF; ++t) {
                    const double at = __shfl_sync(all, a, t0 + t, G);
                    add(lane < n[t], c[t], __dmul_rn(at, v[t]));
                    for (int f = lane + G; __any_sync(all, f < n[t]); f += G) {
                        const bool on = f < n[t];
                        add(on, on ? rci[s[t] + f] : 0, __dmul_rn(at, on ? rv[s[t] + f] : 0.0));
                    }
                }
            }
        }
        __syncwarp();
        if (live) {
            const int u = *count;
            if (over) {
                if (lane == 0) {
                    long_rows[atomicAdd(nlong, 1)] = (int)row;
                    cnt[row] = 0;
                }
            } else {
                if (lane == 0 && !crp) cnt[row] = u;
                const size_t base = crp ? (size_t)crp[row] : (size_t)row * CAP;
                for (int p = lane; p < u && oci; p += G) {
                    const int c = cols[p];
                    int rank = 0;
                    for (int q = 0; q < u; ++q) rank += cols[q] < c;
                    oci[base + rank] = c;
                    ov[base + rank] = acc[p];
                }
            }
        }
        __syncwarp();
        for (int t = lane; t < 2 * CAP / 4; t += G) reinterpret_cast<int4 *>(keys)[t] = make_int4(-1, -1, -1, -1);
    }
}

}  // namespace gw
