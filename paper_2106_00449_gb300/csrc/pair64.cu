// Symmetric FP64 RPY product: every unordered pair of blobs evaluated once for both of its
// blobs (M_ij = M_ji, even in d = r_j - r_i).
//
// What bounds it: the FP64 pipe.  GB300 issues 2 FP64 lanes per clock per SM (a warp
// instruction takes 16 clocks), so loads, shuffles and integer work are free beside it and
// the count of FP64 instructions is everything.  A pair costs 16 of them (difference 3, r^2 3,
// reciprocal square root 5, coefficients 5) plus 10 per side (d . lambda 3, scale 1,
// accumulate 6): 36 per unordered pair against 2 x 33 for the ordered form that this kernel
// replaced.  The comparison with (2a)^2 is made on the bit patterns (integer pipe; both are
// positive), and the reciprocal square root is rsqrt_series (common.cuh).
//
// Work split.  A suspension is cut into tiles of TS = 128 TPL blobs (TPL targets per lane).  An
// item is a target tile I against a range [j0, j1) of sources, j0 >= I TS; ranges of one row
// of tiles do not overlap.  Sources of tile I itself are taken ordered (target side only),
// sources of later tiles symmetrically: W sources (32, or a smaller power of two when the
// range is shorter) are swept in W steps in which lane l reads source (l + step) mod W, and
// the source-side sums travel with their source, one lane per step by shuffles.  The four
// warps' sums of a source meet in shared memory, are added in warp order and go to the one
// slot of (I, J): every slot is written once, all sums run in a fixed order (deterministic).
// Because the pipe is so slow one target per lane already hides every latency, and short
// ranges spread a small suspension over all SMs: 1,560 blobs take 1,287 items of 8 sources.
// Above GDC_P64_WIDE blobs TPL = 4 keeps the slot arrays at n^2/1024 entries.
//
// Measured against the ordered kernel that it replaced (128 or 256 or 512 targets per block
// against source chunks of at least 512): one product of 9,126 blobs 4.81 -> 2.85 ms (83% of
// the pipe's 2.38 ms for 36 instructions per pair); 13 products of 1,560 blobs in a Brownian
// velocity 14.2 -> 3.7 ms, 28 blocks before; a gDC step of 48 blobs 4.46 -> 2.04 ms, where the
// ordered kernel ran on one block.
#include <algorithm>
#include <cstring>

#include "common.cuh"

namespace gdc {

constexpr int P64_STAGE = 128;   // sources staged in shared memory at a time

struct Rpy64K {
    double c23, c2, cA, c9, cB;
    long long four_a2_bits;
};

// RPY coefficients A, B (units of 1/(8 pi eta)) of a pair at squared distance r2
__device__ __forceinline__ void rpy64_coeff(double r2, const Rpy64K& k, double& A, double& B) {
    const double ri = rsqrt_series(r2);
    if (__double_as_longlong(r2) >= k.four_a2_bits) {
        const double ri2 = ri * ri, ri3 = ri2 * ri;
        A = fma(k.c23, ri3, ri);
        B = ri3 * fma(-k.c2, ri2, 1.0);
    } else if (r2 > 1e-290) {   // overlapping blobs
        A = k.cA * fma(-k.c9, r2 * ri, 1.0);
        B = k.cB * ri;
    } else {                    // the self pair (or coincident blobs: B d d^T vanishes with r)
        A = k.cA;
        B = 0.0;
    }
}

template <int TPL>
__global__ void __launch_bounds__(128, TPL == 1 ? 5 : 3) k_rpy64_sym(
    const PairItem* __restrict__ items, const int* __restrict__ active, const long long* __restrict__ susp_blob_off,
    const long long* __restrict__ jbase, const double4_32a* __restrict__ spos, const double* __restrict__ x,
    const int* __restrict__ map, double4_32a* __restrict__ part_i, double4_32a* __restrict__ part_j, int NBL, Rpy64K k) {
    constexpr int TS = 128 * TPL;
    __shared__ double src[6][P64_STAGE];
    __shared__ double red[2][4][3][32];
    const PairItem it = items[blockIdx.x];
    const long long b0 = susp_blob_off[it.s];
    const int ns = (int)(susp_blob_off[it.s + 1] - b0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tbase = it.I * TS;
    if (active && !active[it.s]) {
        // a suspension whose Krylov loop has stopped: its product is not used; leave zeros
        const double4_32a z = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        for (int t = threadIdx.x; t < TS && tbase + t < ns; t += 128) part_i[(long long)it.k * NBL + b0 + tbase + t] = z;
        for (int j = max(it.j0, tbase + TS) + (int)threadIdx.x; j < it.j1; j += 128) {
            const int J = j / TS;
            part_j[(jbase[it.s] + (long long)J * (J - 1) / 2 + it.I) * TS + j - J * TS] = z;
        }
        return;
    }
    // targets tbase + threadIdx.x + 128 m; one past the end sits on the last blob with lambda =
    // 0 (it adds nothing to a source and its own sums are not written)
    double xt[TPL], yt[TPL], zt[TPL], lxt[TPL], lyt[TPL], lzt[TPL], ux[TPL], uy[TPL], uz[TPL];
#pragma unroll
    for (int m = 0; m < TPL; ++m) {
        const int t = tbase + (int)threadIdx.x + 128 * m;
        const long long g = b0 + min(t, ns - 1);
        const double4_32a p = spos[g];
        const long long o = map ? (long long)map[g] : 3 * g;
        xt[m] = p.x;
        yt[m] = p.y;
        zt[m] = p.z;
        lxt[m] = t < ns ? x[o] : 0.0;
        lyt[m] = t < ns ? x[o + 1] : 0.0;
        lzt[m] = t < ns ? x[o + 2] : 0.0;
        ux[m] = uy[m] = uz[m] = 0.0;
    }
    const int range = it.j1 - it.j0;
    int W = 32;   // sources per sweep: a power of two, at least the range when that is short
    while (W > 1 && (W >> 1) >= range) W >>= 1;
    int buf = 0;
    for (int c0 = it.j0; c0 < it.j1; c0 += P64_STAGE) {
        const int n = min(P64_STAGE, it.j1 - c0);
        const int nr = (n + W - 1) & ~(W - 1);
        __syncthreads();   // the previous sources are no longer read
        if ((int)threadIdx.x < nr) {
            const bool in = (int)threadIdx.x < n;   // past the range: the last blob of it with lambda = 0
            const long long g = b0 + c0 + min((int)threadIdx.x, n - 1);
            const double4_32a p = spos[g];
            const long long o = map ? (long long)map[g] : 3 * g;
            src[0][threadIdx.x] = p.x;
            src[1][threadIdx.x] = p.y;
            src[2][threadIdx.x] = p.z;
            src[3][threadIdx.x] = in ? x[o] : 0.0;
            src[4][threadIdx.x] = in ? x[o + 1] : 0.0;
            src[5][threadIdx.x] = in ? x[o + 2] : 0.0;
        }
        __syncthreads();
        for (int jc = 0; jc < n; jc += W) {
            const int J = (c0 + jc) / TS;
            if (J == it.I) {
                // the tile itself: every ordered pair, target side only
                for (int j = jc; j < min(jc + W, n); ++j) {
                    const double xs = src[0][j], ys = src[1][j], zs = src[2][j];
                    const double lx = src[3][j], ly = src[4][j], lz = src[5][j];
#pragma unroll
                    for (int m = 0; m < TPL; ++m) {
                        if (tbase + 32 * warp + 128 * m >= ns) continue;   // no target in this warp
                        const double dx = xs - xt[m], dy = ys - yt[m], dz = zs - zt[m];
                        double A, B;
                        rpy64_coeff(fma(dx, dx, fma(dy, dy, dz * dz)), k, A, B);
                        const double s = B * fma(dx, lx, fma(dy, ly, dz * lz));
                        ux[m] = fma(A, lx, fma(s, dx, ux[m]));
                        uy[m] = fma(A, ly, fma(s, dy, uy[m]));
                        uz[m] = fma(A, lz, fma(s, dz, uz[m]));
                    }
                }
                continue;
            }
            double jx = 0.0, jy = 0.0, jz = 0.0;   // sums of the source this lane holds
            for (int st = 0; st < W; ++st) {
                const int j = jc + ((lane + st) & (W - 1));
                const double xs = src[0][j], ys = src[1][j], zs = src[2][j];
                const double lx = src[3][j], ly = src[4][j], lz = src[5][j];
#pragma unroll
                for (int m = 0; m < TPL; ++m) {
                    if (tbase + 32 * warp + 128 * m >= ns) continue;
                    const double dx = xs - xt[m], dy = ys - yt[m], dz = zs - zt[m];
                    double A, B;
                    rpy64_coeff(fma(dx, dx, fma(dy, dy, dz * dz)), k, A, B);
                    const double s = B * fma(dx, lx, fma(dy, ly, dz * lz));          // M lambda_j
                    ux[m] = fma(A, lx, fma(s, dx, ux[m]));
                    uy[m] = fma(A, ly, fma(s, dy, uy[m]));
                    uz[m] = fma(A, lz, fma(s, dz, uz[m]));
                    const double w = B * fma(dx, lxt[m], fma(dy, lyt[m], dz * lzt[m]));   // M lambda_i
                    jx = fma(A, lxt[m], fma(w, dx, jx));
                    jy = fma(A, lyt[m], fma(w, dy, jy));
                    jz = fma(A, lzt[m], fma(w, dz, jz));
                }
                const int from = (lane + 1) & 31;   // the source of lane l + 1 is lane l's next
                jx = __shfl_sync(0xffffffffu, jx, from);
                jy = __shfl_sync(0xffffffffu, jy, from);
                jz = __shfl_sync(0xffffffffu, jz, from);
            }
            // W < 32: the 32/W lanes with the same remainder mod W hold parts of one source
            for (int o = W; o < 32; o <<= 1) {
                jx += __shfl_xor_sync(0xffffffffu, jx, o);
                jy += __shfl_xor_sync(0xffffffffu, jy, o);
                jz += __shfl_xor_sync(0xffffffffu, jz, o);
            }
            // the buffer this sweep writes was last read before the previous sweep's barrier
            red[buf][warp][0][lane] = jx;
            red[buf][warp][1][lane] = jy;
            red[buf][warp][2][lane] = jz;
            __syncthreads();
            if (warp == 0 && lane < W && jc + lane < n) {   // in warp order
                double v[3];
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    v[c] = ((red[buf][0][c][lane] + red[buf][1][c][lane]) + red[buf][2][c][lane]) + red[buf][3][c][lane];
                const long long slot = jbase[it.s] + (long long)J * (J - 1) / 2 + it.I;
                part_j[slot * TS + (c0 + jc + lane) - J * TS] = make_double4_32a(v[0], v[1], v[2], 0.0);
            }
            buf ^= 1;
        }
    }
#pragma unroll
    for (int m = 0; m < TPL; ++m) {
        const int t = tbase + (int)threadIdx.x + 128 * m;
        if (t < ns) part_i[(long long)it.k * NBL + b0 + t] = make_double4_32a(ux[m], uy[m], uz[m], 0.0);
    }
}

// u_i = c0 (target-side slots of the blob's tile row + source-side slots of the tiles before
// it) [- K V], for this kernel and the symmetric double-float one (dfsym.cu; its same-body
// blocks are added afterwards).  EPI threads per blob, each taking every EPI-th slot, joined in
// a fixed order: the slots are latency-bound L2 reads, and the short ranges of small
// suspensions leave up to 200 of them per blob.  16 threads up to GDC_P64_EPI_WIDE blobs, 4
// above, where the FP64 shuffle sums would cost more than the chain.
template <int EPI>
__global__ void __launch_bounds__(128) k_p64_epilogue(
    int NBL, int TS, const double4_32a* __restrict__ part_i, const double4_32a* __restrict__ part_j,
    const int* __restrict__ blob_susp, const long long* __restrict__ susp_blob_off, const int* __restrict__ row_nk,
    const long long* __restrict__ tile_base, const long long* __restrict__ jbase, double c0, const double* __restrict__ x,
    double* __restrict__ y, int gm_layout, const int* __restrict__ blob_gm, const int* __restrict__ body_gm,
    const int* __restrict__ blob_body, const double* __restrict__ r, const double* __restrict__ Yc) {
    const int sub = threadIdx.x % EPI;
    const int i = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) / EPI);
    double ux = 0.0, uy = 0.0, uz = 0.0;
    if (i < NBL) {
        const int s = blob_susp[i];
        const int loc = (int)(i - susp_blob_off[s]);
        const int J = loc / TS, e = loc - J * TS;
        const int n = row_nk[tile_base[s] + J];
#pragma unroll 4
        for (int q = sub; q < n; q += EPI) {
            const double4_32a v = part_i[(long long)q * NBL + i];
            ux += v.x;
            uy += v.y;
            uz += v.z;
        }
        const long long s0 = jbase[s] + (long long)J * (J - 1) / 2;
#pragma unroll 4
        for (int I = sub; I < J; I += EPI) {
            const double4_32a v = part_j[(s0 + I) * TS + e];
            ux += v.x;
            uy += v.y;
            uz += v.z;
        }
    }
#pragma unroll
    for (int o = 1; o < EPI; o <<= 1) {
        ux += __shfl_xor_sync(0xffffffffu, ux, o);
        uy += __shfl_xor_sync(0xffffffffu, uy, o);
        uz += __shfl_xor_sync(0xffffffffu, uz, o);
    }
    if (i >= NBL || sub != 0) return;
    ux *= c0;
    uy *= c0;
    uz *= c0;
    if (!gm_layout) {
        y[3LL * i] = ux;
        y[3LL * i + 1] = uy;
        y[3LL * i + 2] = uz;
        return;
    }
    // saddle operator: M lambda - K V, K V = U_p + Omega_p x (r_i - Y_p)  (Eq. rigid_body_cond)
    const int p = blob_body[i];
    const double* V = x + body_gm[p];
    const double dx = r[3LL * i] - Yc[3 * p], dy = r[3LL * i + 1] - Yc[3 * p + 1], dz = r[3LL * i + 2] - Yc[3 * p + 2];
    const long long o = blob_gm[i];
    y[o] = ux - (V[0] + (V[4] * dz - V[5] * dy));
    y[o + 1] = uy - (V[1] + (V[5] * dx - V[3] * dz));
    y[o + 2] = uz - (V[2] + (V[3] * dy - V[4] * dx));
}

// Work list: tiles of 128 blobs, or 512 when a suspension is larger than GDC_P64_WIDE; source
// ranges as long as possible while a launch still has 8 items per SM (7 resident with one target
// per lane, at 71 registers; 3 with four, at 142), so that an SM's share differs from the mean by
// about an eighth; longest first.
void build_p64_list(gdc_ctx* c) {
    long long nmax = 0;
    for (int s = 0; s < c->S; ++s) nmax = std::max(nmax, c->h_blob_off[s + 1] - c->h_blob_off[s]);
    const int TS = c->p64_tile = nmax > GDC_P64_WIDE ? 512 : 128;
    c->h_p64_tile_base.assign(c->S + 1, 0);
    c->h_p64_jbase.assign(c->S + 1, 0);
    for (int s = 0; s < c->S; ++s) {
        const long long n = c->h_blob_off[s + 1] - c->h_blob_off[s], T = (n + TS - 1) / TS;
        c->h_p64_tile_base[s + 1] = c->h_p64_tile_base[s] + T;
        c->h_p64_jbase[s + 1] = c->h_p64_jbase[s] + T * (T - 1) / 2;
    }
    const long long want = 8LL * c->num_sms;
    long long w = 2 * TS;
    while (w > 4 && pair_list_items(c, TS, w) < want) w >>= 1;
    // very large suspensions: at most 128 target-side slots per row, ranges of whole tiles
    if (w == 2 * TS) w = std::max<long long>(w, ((nmax + 127) / 128 + TS - 1) / TS * TS);
    build_pair_list(c, TS, w, c->h_p64_items, c->h_p64_row_nk, c->p64_kmax);
}

void launch_rpy64_sym(gdc_ctx* c, const double* x, int gm_layout) {
    const double a = c->p.a, four_a2 = 4.0 * a * a;
    Rpy64K k{2.0 * a * a / 3.0, 2.0 * a * a, 4.0 / (3.0 * a), 9.0 / (32.0 * a), 1.0 / (8.0 * a * a), 0};
    static_assert(sizeof(four_a2) == sizeof(k.four_a2_bits), "bit pattern of a double");
    memcpy(&k.four_a2_bits, &four_a2, sizeof(four_a2));
    const int* map = gm_layout ? c->blob_gm : nullptr;
    const unsigned n = (unsigned)c->h_p64_items.size();
    ++c->n_launch;
    if (c->p64_tile == 128)
        k_rpy64_sym<1><<<n, 128, 0, c->stream>>>(c->p64_items, c->mv_active, c->susp_blob_off, c->p64_jbase, c->spos64, x,
                                                 map, c->p64_part_i, c->p64_part_j, c->NBL, k);
    else
        k_rpy64_sym<4><<<n, 128, 0, c->stream>>>(c->p64_items, c->mv_active, c->susp_blob_off, c->p64_jbase, c->spos64, x,
                                                 map, c->p64_part_i, c->p64_part_j, c->NBL, k);
}

void launch_p64_epilogue(gdc_ctx* c, int prec, const double* x, double* y, int gm_layout) {
    const bool df = prec == GDC_PREC_DF64;   // the double-float kernel's slots
#define GDC_P64_EPI(EPI)                                                                                          \
    k_p64_epilogue<EPI><<<ceil_div((long long)EPI * c->NBL, 128), 128, 0, c->stream>>>(                           \
        c->NBL, df ? GDC_SYM_TILE : c->p64_tile, df ? c->dfs_part_i : c->p64_part_i,                              \
        df ? c->dfs_part_j : c->p64_part_j, c->blob_susp, c->susp_blob_off, df ? c->dfs_row_nk : c->p64_row_nk,    \
        df ? c->sym_tile_base : c->p64_tile_base, df ? c->sym_jbase : c->p64_jbase,                               \
        1.0 / (8.0 * 3.141592653589793 * c->p.eta), x, y, gm_layout, c->blob_gm, c->body_gm, c->blob_body, c->r, c->Yc)
    ++c->n_launch;
    if (c->NBL <= GDC_P64_EPI_WIDE)
        GDC_P64_EPI(16);
    else
        GDC_P64_EPI(4);
#undef GDC_P64_EPI
}

}  // namespace gdc
