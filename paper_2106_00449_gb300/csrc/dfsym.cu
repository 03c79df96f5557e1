// Symmetric double-float RPY pair kernel: the accurate residual product of the FP32-mixed
// mobility solve with every unordered pair of different bodies evaluated once for both of
// its blobs (M_ij = M_ji, even in d = r_j - r_i).  The pair's distance, reciprocal square
// root and coefficients A, B (about half its double-float operations) are shared; only the
// two products with lambda_j and lambda_i remain per side.
//
// Layout as in the symmetric FP32 kernel (sym.cu): tiles of 512 blobs; a block takes target
// tile I against a range of sources, those of the tile itself ordered.  For later tiles J > I
// each warp holds 128 targets (four per lane); W sources (32, or 16 when the range is
// shorter) are swept in W steps in which lane l takes source (l + step) mod W, and the
// source-side sums (double-float) move one lane per step by shuffles, back at their source's
// lane after W steps; for W = 16 the two lanes of a source are then added.  At the end of
// each sub-chunk the four warps' source-side sums meet in shared memory (double-buffered, one
// barrier per sub-chunk) and warp 0 adds them in warp order into the tile pair's FP64 slot
// (deterministic).
// Target-side sums go to one FP64 slot per item.  Same-body pairs are skipped (the same-body
// block is added exactly in FP64 elsewhere).  Pairs are evaluated exactly as the ordered
// double-float kernel evaluates them (overlapping branch below 2a included).
#include <algorithm>

#include "common.cuh"
#include "df.cuh"

namespace gdc {

constexpr int DFS_TILE = GDC_SYM_TILE;
// dynamic shared memory: the source tile (four planes of one float4 per source: the lanes'
// rotated reads hit consecutive 16-byte words), then two buffers of the four
// warps' source sums of one 32-source sub-chunk (3 doubles per source each)
constexpr int DFS_SMEM = DFS_TILE * 4 * 16 + 2 * 4 * 3 * 32 * 8;

struct DfPair {   // the shared part of one pair: d = r_j - r_i, A, B
    df dx, dy, dz, A, B;
};

__device__ __forceinline__ DfPair df_pair(df xs, df ys, df zs, df xt, df yt, df zt, const RpyConstDF& k) {
    DfPair p;
    p.dx = df_sub(xs, xt);
    p.dy = df_sub(ys, yt);
    p.dz = df_sub(zs, zt);
    const df r2 = df_dot3(p.dx, p.dy, p.dz, p.dx, p.dy, p.dz);
    const df ri = df_rsqrt(r2);
    if (r2.h > k.four_a2.h || (r2.h == k.four_a2.h && r2.l >= k.four_a2.l)) {
        const df ri2 = df_mul(ri, ri);
        // A = (1 + 2a^2/(3 r^2)) / r, B = (1 - 2a^2/r^2) / r^3; r >= 2a, so both brackets are
        // one plus a term below one
        const df w = df_mul_open(k.c2, ri2);
        p.A = df_mul(ri, df_one_plus(df_mul_open(k.c23, ri2)));
        p.B = df_mul(df_mul(ri2, ri), df_one_plus(df{-w.h, -w.l}));
    } else {   // overlapping blobs of different bodies (r > 0 for distinct blobs)
        const df r = df_mul(r2, ri);
        p.A = df_mul(k.cA, df_sub(df{1.f, 0.f}, df_mul(k.c9, r)));
        p.B = df_mul(k.cB, ri);
    }
    return p;
}

// u += A lambda + B (d . lambda) d.  A product is closed (its low part brought below half an ulp
// of the high part) only where it is multiplied again; sums take it open and close once per
// component: 119 operations a side, against 158 with every product and sum closed, and fewer
// roundings of the low parts.  The kernel is bound by FP32 issue: 65,520 blobs 30.6 -> 24.2 ms,
// relative error of the product against FP64 2.0e-14 both; 2,560 blobs 98 -> 78 us, 1.9e-14 ->
// 8.6e-15.
__device__ __forceinline__ df df_accumulate(df u, df A, df l, df s, df d) {
    return df_close(df_add_open(u, df_add_open(df_mul_open(A, l), df_mul_open(s, d))));
}
__device__ __forceinline__ void df_side(const DfPair& p, df lx, df ly, df lz, df& ux, df& uy, df& uz) {
    const df s = df_mul(p.B, df_dot3(p.dx, p.dy, p.dz, lx, ly, lz));
    ux = df_accumulate(ux, p.A, lx, s, p.dx);
    uy = df_accumulate(uy, p.A, ly, s, p.dy);
    uz = df_accumulate(uz, p.A, lz, s, p.dz);
}

__device__ __forceinline__ df shfl_df(df v, int src) {
    return df{__shfl_sync(0xffffffffu, v.h, src), __shfl_sync(0xffffffffu, v.l, src)};
}

// MINB: resident blocks per SM the register allocator is asked to allow, 3 (162 registers) or
// 4 (128, the rule below GDC_TUNE_PAIRS); above, the autotuner times both.
// FULL: every range is whole tiles, as in the symmetric FP32 kernel.
template <int MINB, bool FULL>
__global__ void __launch_bounds__(128, MINB) k_rpy_df_sym(const PairItem* __restrict__ items,
                                                       const long long* __restrict__ susp_blob_off,
                                                       const long long* __restrict__ jbase,
                                                       const double4_32a* __restrict__ spos,
                                                       const double4_32a* __restrict__ slam,
                                                       double4_32a* __restrict__ part_i, double4_32a* __restrict__ part_j,
                                                       int NBL, RpyConstDF k) {
    extern __shared__ __align__(16) unsigned char dfs_smem[];
    float4* sh = reinterpret_cast<float4*>(dfs_smem);                       // [plane][source]
    double* ws = reinterpret_cast<double*>(dfs_smem + DFS_TILE * 4 * 16);  // [buffer][warp][3][32]
    const PairItem it = items[blockIdx.x];
    const long long b0 = susp_blob_off[it.s];
    const int ns = (int)(susp_blob_off[it.s + 1] - b0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tbase = it.I * DFS_TILE;
    // targets tbase + threadIdx.x + 128 m; a target past the end sits on the last blob with
    // lambda = 0 and body -1 (it adds nothing and its sums are not written)
    df xt[4], yt[4], zt[4], lxt[4], lyt[4], lzt[4], ux[4], uy[4], uz[4];
    float bt[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int t = tbase + threadIdx.x + 128 * m;
        const long long g = b0 + min(t, ns - 1);
        const double4_32a p = spos[g], l = slam[g];
        const bool in = t < ns;
        xt[m] = df_from(p.x);
        yt[m] = df_from(p.y);
        zt[m] = df_from(p.z);
        lxt[m] = df_from(in ? l.x : 0.0);
        lyt[m] = df_from(in ? l.y : 0.0);
        lzt[m] = df_from(in ? l.z : 0.0);
        bt[m] = in ? (float)p.w : -1.f;
        ux[m] = uy[m] = uz[m] = df{0.f, 0.f};
    }
    int W = 32;   // sources per sweep
    if (!FULL && it.j1 - it.j0 <= 16) W = 16;
    int buf = 0;
    const int J1 = (it.j1 + DFS_TILE - 1) / DFS_TILE;
    for (int J = it.j0 / DFS_TILE; J < J1; ++J) {   // the part of the range in source tile J
        const int j0 = FULL ? J * DFS_TILE : max(it.j0, J * DFS_TILE);
        const int n = FULL ? min(DFS_TILE, ns - j0) : min((J + 1) * DFS_TILE, it.j1) - j0;
        const int nr = (n + W - 1) & ~(W - 1);
        __syncthreads();   // the previous tile's sources and sums are no longer read
        for (int e = threadIdx.x; e < nr; e += 128) {
            if (e < n) {
                const double4_32a ps = spos[b0 + j0 + e], ls = slam[b0 + j0 + e];
                const df x = df_from(ps.x), y = df_from(ps.y), z = df_from(ps.z);
                const df lx = df_from(ls.x), ly = df_from(ls.y), lz = df_from(ls.z);
                sh[e] = make_float4(x.h, y.h, z.h, (float)ps.w);
                sh[DFS_TILE + e] = make_float4(x.l, y.l, z.l, 0.f);
                sh[2 * DFS_TILE + e] = make_float4(lx.h, ly.h, lz.h, 0.f);
                sh[3 * DFS_TILE + e] = make_float4(lx.l, ly.l, lz.l, 0.f);
            } else {   // padding: body -2 matches no target, lambda 0
                sh[e] = make_float4(0.f, 0.f, 0.f, -2.f);
                sh[DFS_TILE + e] = sh[2 * DFS_TILE + e] = sh[3 * DFS_TILE + e] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        __syncthreads();
        if (J == it.I) {
            // diagonal tile: every ordered pair of different bodies, target side only
            for (int j = 0; j < n; ++j) {
                const float4 s0 = sh[j], s1 = sh[DFS_TILE + j], s2 = sh[2 * DFS_TILE + j], s3 = sh[3 * DFS_TILE + j];
                const df lx{s2.x, s3.x}, ly{s2.y, s3.y}, lz{s2.z, s3.z};
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (s0.w == bt[m] || bt[m] < 0.f) continue;   // same body, or no target
                    const DfPair p = df_pair(df{s0.x, s1.x}, df{s0.y, s1.y}, df{s0.z, s1.z}, xt[m], yt[m], zt[m], k);
                    df_side(p, lx, ly, lz, ux[m], uy[m], uz[m]);
                }
            }
        } else {
            const long long slot = jbase[it.s] + (long long)J * (J - 1) / 2 + it.I;
            for (int jc = 0; jc < nr; jc += W) {
                df jx{0.f, 0.f}, jy{0.f, 0.f}, jz{0.f, 0.f};   // sums of the source this lane holds
                for (int st = 0; st < W; ++st) {
                    const int j = jc + ((lane + st) & (W - 1));
                    const float4 s0 = sh[j], s1 = sh[DFS_TILE + j], s2 = sh[2 * DFS_TILE + j], s3 = sh[3 * DFS_TILE + j];
                    const df xs{s0.x, s1.x}, ys{s0.y, s1.y}, zs{s0.z, s1.z};
                    const df lx{s2.x, s3.x}, ly{s2.y, s3.y}, lz{s2.z, s3.z};
                    const bool pad = s0.w < -1.5f;   // past the end of the suspension
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        if (pad || s0.w == bt[m] || bt[m] < 0.f) continue;   // padding, same body, no target
                        const DfPair p = df_pair(xs, ys, zs, xt[m], yt[m], zt[m], k);
                        df_side(p, lx, ly, lz, ux[m], uy[m], uz[m]);          // target side: M lambda_j
                        df_side(p, lxt[m], lyt[m], lzt[m], jx, jy, jz);       // source side: M lambda_i
                    }
                    const int from = (lane + 1) & 31;   // the source of lane l + 1 is lane l's next
                    jx = shfl_df(jx, from);
                    jy = shfl_df(jy, from);
                    jz = shfl_df(jz, from);
                }
                // after W steps the sums of source jc + (lane mod W) are back at lane; the buffer
                // this sweep writes was last read by warp 0 before the previous barrier
                double v[3] = {df_to(jx), df_to(jy), df_to(jz)};
                if (!FULL && W == 16)
#pragma unroll
                    for (int c = 0; c < 3; ++c) v[c] += __shfl_xor_sync(0xffffffffu, v[c], 16);
                double* wb = ws + buf * (4 * 3 * 32);
                buf ^= 1;
#pragma unroll
                for (int c = 0; c < 3; ++c) wb[(warp * 3 + c) * 32 + lane] = v[c];
                __syncthreads();
                if (warp == 0 && lane < W && jc + lane < n) {   // the four warps' sums, in warp order
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        v[c] = ((wb[(0 * 3 + c) * 32 + lane] + wb[(1 * 3 + c) * 32 + lane]) +
                                wb[(2 * 3 + c) * 32 + lane]) + wb[(3 * 3 + c) * 32 + lane];
                    part_j[slot * DFS_TILE + (j0 - J * DFS_TILE) + jc + lane] = make_double4_32a(v[0], v[1], v[2], 0.0);
                }
            }
        }
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int t = tbase + threadIdx.x + 128 * m;
        if (t < ns)
            part_i[(long long)it.k * NBL + b0 + t] = make_double4_32a(df_to(ux[m]), df_to(uy[m]), df_to(uz[m]), 0.0);
    }
}

template <int MINB, bool FULL>
static cudaError_t dfsym_attribute() {
    return cudaFuncSetAttribute(k_rpy_df_sym<MINB, FULL>, cudaFuncAttributeMaxDynamicSharedMemorySize, DFS_SMEM);
}

gdc_status dfsym_init_attributes(gdc_ctx* c) {
    for (cudaError_t e : {dfsym_attribute<3, true>(), dfsym_attribute<4, true>(), dfsym_attribute<3, false>(),
                          dfsym_attribute<4, false>()})
        if (e != cudaSuccess) return cuda_check(c, e, "symmetric double-float kernel attributes");
    return GDC_OK;
}

// The symmetric double-float pair kernel alone (same-body blocks excluded).
void launch_rpy_df_sym_pairs(gdc_ctx* c) {
#define GDC_DFS_LAUNCH(MB, FULL)                                                                                \
    k_rpy_df_sym<MB, FULL><<<c->dfs_n_items, 128, DFS_SMEM, c->stream>>>(                                       \
        c->dfs_items, c->susp_blob_off, c->sym_jbase, c->spos64, c->slam64, c->dfs_part_i, c->dfs_part_j, c->NBL, \
        df_constants(c->p.a))
    ++c->n_launch;
    const bool full = c->dfs_width >= DFS_TILE;
    if (c->dfs_minb == 3) {
        if (full) GDC_DFS_LAUNCH(3, true); else GDC_DFS_LAUNCH(3, false);
    } else {
        if (full) GDC_DFS_LAUNCH(4, true); else GDC_DFS_LAUNCH(4, false);
    }
#undef GDC_DFS_LAUNCH
}

// Work list: the longest ranges (16 to 1,024 sources; longer in suspensions above 65,536
// blobs, so that a row has at most 64 target-side slots) that give 24 items per SM.  us per
// launch by that rule, and as items of two whole tiles (with every product and sum of df_side
// closed): 2,560 blobs 98 / 2,067, 7,800 blobs 543 / 2,159, 20,202 blobs 3,144 / 3,813, 48
// suspensions of 63,702 blobs 1,196 / 2,624, 65,520 blobs 30,660 / 30,640.  With df_side as it
// is now: 78, 427, 2,450, 905 and 24,170, relative error against FP64 6e-15 to 2e-14.
void build_dfs_list(gdc_ctx* c) {
    long long nmax = 1;
    for (int s = 0; s < c->S; ++s) nmax = std::max(nmax, c->h_blob_off[s + 1] - c->h_blob_off[s]);
    long long w = 1024;
    while (w < (nmax + 63) / 64) w *= 2;
    while (w > 16 && pair_list_items(c, DFS_TILE, w) < 24LL * c->num_sms) w >>= 1;
    build_pair_list(c, DFS_TILE, w, c->h_dfs_items, c->h_dfs_row_nk, c->dfs_kmax);
    c->dfs_width = (int)w;
    c->dfs_n_items = (int)c->h_dfs_items.size();
}

}  // namespace gdc
