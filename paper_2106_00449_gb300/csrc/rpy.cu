// On-the-fly tiled N-body kernels: the RPY product u = M lambda (Sec. 4.1, Eq. ddof_mob) in
// FP32 and FP64, and the soft blob repulsion (Eq. soft_sphere_potential form).  Sources are staged in
// shared memory tile by tile; each thread owns TPT targets.  Work is split into
// (target tile x source chunk) items so that a launch fills every SM several times
// over; chunk partial sums are added in FP64, in chunk order, by the epilogue.
//
// RPY with c0 = 1/(8 pi eta), d = r_j - r_i, r = |d| (the d d^T term is even in d):
//   r >= 2a : u_i += c0 [ (1/r + 2a^2/(3 r^3)) lambda_j + (1/r^3)(1 - 2a^2/r^2) (d.lambda_j) d ]
//   r <  2a : u_i += c0 [ (4/(3a))(1 - 9r/(32a)) lambda_j + (1/(8 a^2 r)) (d.lambda_j) d ]
//   r == 0  : u_i += c0 (4/(3a)) lambda_j                     (self term 1/(6 pi eta a))
#include <algorithm>
#include <numeric>

#include "common.cuh"
#include "pair_common.cuh"
#include "df.cuh"
#include "forces.cuh"

namespace gdc {

#ifndef GDC_MV_TILE
#define GDC_MV_TILE 256
#endif
constexpr int MV_TILE = GDC_MV_TILE;   // sources staged in shared memory per tile

// ---- source packing ---------------------------------------------------------

// FP32 sources in the layout the pair kernel's shared-memory tiles use, three float4 per
// blob: (x,x,y,y) (z,z,lx,lx) (ly,ly,lz,lz) -- each value twice, one per packed lane.  The
// positions are written when a configuration is loaded (k_blob_pos), lambda here or by the
// per-body kernel that produced it.
__global__ void k_pack_lam32(int NBL, const int* __restrict__ map, const double* __restrict__ x,
                             float4* __restrict__ sdup) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NBL) return;
    const long long o = map ? (long long)map[i] : 3LL * i;
    const float lx = (float)x[o], ly = (float)x[o + 1], lz = (float)x[o + 2];
    reinterpret_cast<float2*>(sdup + 3LL * i + 1)[1] = make_float2(lx, lx);
    sdup[3LL * i + 2] = make_float4(ly, ly, lz, lz);
}

__global__ void k_pack_lam64(int NBL, const int* __restrict__ map, const double* __restrict__ x,
                             double4_32a* __restrict__ slam) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NBL) return;
    const long long o = map ? (long long)map[i] : 3LL * i;
    slam[i] = make_double4_32a(x[o], x[o + 1], x[o + 2], 0.0);
}

void launch_pack_lambda(gdc_ctx* c, int prec, const double* x, int gm_layout) {
    const int* map = gm_layout ? c->blob_gm : nullptr;
    if (prec == GDC_FP32_MIXED)
        ++c->n_launch, k_pack_lam32<<<ceil_div(c->NBL, 256), 256, 0, c->stream>>>(c->NBL, map, x, c->sdup);
    else if (prec == GDC_PREC_DF64)
        ++c->n_launch, k_pack_lam64<<<ceil_div(c->NBL, 256), 256, 0, c->stream>>>(c->NBL, map, x, c->slam64);
}

// ---- FP32 RPY pair kernel -----------------------------------------------------

// Each thread owns 2P targets, evaluated two at a time with packed instructions.  Every
// pair of the suspension is evaluated with the far-field form of the RPY tensor at the
// clamped distance max(r, 2a) (branch free); the self pair and the pairs closer than 2a,
// for which that is not the RPY tensor, are corrected in FP64 by the epilogue from a list of
// such pairs built once per configuration.  Shared memory holds each source as
// (x,x,y,y) (z,z,lx,lx) (ly,ly,lz,lz), so one 16-byte load feeds a packed operand.  Sums run
// over 32-source sub-chunks, then per tile, then across tiles with compensation.
//
// Source tiles are staged by the bulk-copy (TMA) engine: the packed source array already
// holds the duplicated layout, so a tile is one contiguous cp.async.bulk into shared
// memory, completed on an mbarrier.  Two buffers: the copy of tile t+1 runs while tile t
// is evaluated.  Waits are bounded; on a timeout the kernel flags status[1] and returns.

// MINB: resident blocks per SM the register allocator is asked to allow, 4 (112 / 124
// registers for P = 1 / 2) or 6 (76 / 80, the latter with a few spilled bytes); the
// autotuner times both.
template <int P, int MINB>
__global__ void __launch_bounds__(128, MINB) k_rpy32(const MvItem* __restrict__ items, const int* __restrict__ active,
                                               const long long* __restrict__ susp_blob_off,
                                               const float4* __restrict__ spos, const float4* __restrict__ sdup,
                                               float4* __restrict__ part, int NBL, RpyConst32 k,
                                               int* __restrict__ status, int first_polls) {
    __shared__ __align__(128) float4 shbuf[2][3 * MV_TILE];
    __shared__ __align__(8) unsigned long long mbar[2];
    const MvItem it = items[blockIdx.x];
    const long long b0 = susp_blob_off[it.s];
    const int ns = (int)(susp_blob_off[it.s + 1] - b0);
    if (active && !active[it.s]) {
        // a suspension whose Krylov loop has stopped: its product is not used; leave zeros
        for (int t = threadIdx.x; t < 256 * P && it.t0 + t < ns; t += 128)
            part[(long long)it.k * NBL + b0 + it.t0 + t] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const float2 c23 = make_float2(k.c23, k.c23), mc2 = make_float2(-k.c2, -k.c2), one = make_float2(1.f, 1.f);
    const float four_a2 = k.four_a2;
    const int ntile = (it.j1 - it.j0 + MV_TILE - 1) / MV_TILE;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_addr(&mbar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_addr(&mbar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0 && ntile > 0)
        bulk_tile_load(shbuf[0], sdup + 3 * (b0 + it.j0), 48u * (unsigned)min(MV_TILE, it.j1 - it.j0), &mbar[0]);

    float2 xt[P], yt[P], zt[P], ax[P], ay[P], az[P], cx[P], cy[P], cz[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float4 pa = spos[b0 + min(it.t0 + (int)threadIdx.x + (2 * p) * 128, ns - 1)];
        const float4 pb = spos[b0 + min(it.t0 + (int)threadIdx.x + (2 * p + 1) * 128, ns - 1)];
        xt[p] = make_float2(pa.x, pb.x);
        yt[p] = make_float2(pa.y, pb.y);
        zt[p] = make_float2(pa.z, pb.z);
        ax[p] = ay[p] = az[p] = make_float2(0.f, 0.f);
        cx[p] = cy[p] = cz[p] = make_float2(0.f, 0.f);
    }
    for (int t = 0; t < ntile; ++t) {
        const int j0 = it.j0 + t * MV_TILE;
        const int n = min(MV_TILE, it.j1 - j0);
        const float4* sh = shbuf[t & 1];
        if (threadIdx.x == 0 && t + 1 < ntile) {
            // buffer (t+1)&1 was last read in iteration t-1, which ended with a barrier
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            const int j1n = j0 + MV_TILE;
            bulk_tile_load(shbuf[(t + 1) & 1], sdup + 3 * (b0 + j1n), 48u * (unsigned)min(MV_TILE, it.j1 - j1n),
                           &mbar[(t + 1) & 1]);
        }
        const bool ok = mbar_wait(&mbar[t & 1], (unsigned)((t >> 1) & 1), first_polls);
        float2 tx[P], ty[P], tz[P];
#pragma unroll
        for (int p = 0; p < P; ++p) tx[p] = ty[p] = tz[p] = make_float2(0.f, 0.f);
        for (int jc = 0; jc < n; jc += 32) {
            const int je = min(jc + 32, n);
            float2 qx[P], qy[P], qz[P];
#pragma unroll
            for (int p = 0; p < P; ++p) qx[p] = qy[p] = qz[p] = make_float2(0.f, 0.f);
#pragma unroll 4
            for (int j = jc; j < je; ++j) {
                const float4 s0 = sh[3 * j], s1 = sh[3 * j + 1], s2 = sh[3 * j + 2];
                const float2 xs = make_float2(s0.x, s0.y), ys = make_float2(s0.z, s0.w), zs = make_float2(s1.x, s1.y);
                const float2 lx = make_float2(s1.z, s1.w), ly = make_float2(s2.x, s2.y), lz = make_float2(s2.z, s2.w);
#pragma unroll
                for (int p = 0; p < P; ++p) {
                    const float2 dx = sub2(xs, xt[p]), dy = sub2(ys, yt[p]), dz = sub2(zs, zt[p]);
                    const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
                    const float2 ri = make_float2(rsqrtf(fmaxf(r2.x, four_a2)), rsqrtf(fmaxf(r2.y, four_a2)));
                    const float2 ri2 = mul2(ri, ri);
                    const float2 ri3 = mul2(ri2, ri);
                    const float2 A = fma2(c23, ri3, ri);
                    const float2 B = mul2(ri3, fma2(mc2, ri2, one));
                    const float2 s = mul2(B, fma2(dx, lx, fma2(dy, ly, mul2(dz, lz))));
                    qx[p] = fma2(A, lx, fma2(s, dx, qx[p]));
                    qy[p] = fma2(A, ly, fma2(s, dy, qy[p]));
                    qz[p] = fma2(A, lz, fma2(s, dz, qz[p]));
                }
            }
#pragma unroll
            for (int p = 0; p < P; ++p) {
                tx[p] = add2(tx[p], qx[p]);
                ty[p] = add2(ty[p], qy[p]);
                tz[p] = add2(tz[p], qz[p]);
            }
        }
        // compensated (Kahan) addition of the tile sums
#pragma unroll
        for (int p = 0; p < P; ++p) {
            float2 y, u;
            y = sub2(tx[p], cx[p]); u = add2(ax[p], y); cx[p] = sub2(sub2(u, ax[p]), y); ax[p] = u;
            y = sub2(ty[p], cy[p]); u = add2(ay[p], y); cy[p] = sub2(sub2(u, ay[p]), y); ay[p] = u;
            y = sub2(tz[p], cz[p]); u = add2(az[p], y); cz[p] = sub2(sub2(u, az[p]), y); az[p] = u;
        }
        // every thread is done with this buffer before it is refilled; a timed-out copy stops the block
        // after its copies in flight have landed: tile t's (whose wait gave up) and tile t+1's
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) {
                atomicExch(status + 1, 1);
                mbar_wait(&mbar[t & 1], (unsigned)((t >> 1) & 1));
                if (t + 1 < ntile) mbar_wait(&mbar[(t + 1) & 1], (unsigned)(((t + 1) >> 1) & 1));
            }
            return;
        }
    }
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const float2 rx = sub2(ax[p], cx[p]), ry = sub2(ay[p], cy[p]), rz = sub2(az[p], cz[p]);
        const int ta = it.t0 + threadIdx.x + (2 * p) * 128, tb = ta + 128;
        if (ta < ns) part[(long long)it.k * NBL + b0 + ta] = make_float4(rx.x, ry.x, rz.x, 0.f);
        if (tb < ns) part[(long long)it.k * NBL + b0 + tb] = make_float4(rx.y, ry.y, rz.y, 0.f);
    }
}

// ---- double-float (df64) RPY pair kernel for accurate residuals ----------------------
//
// GB300 runs FP64 at a small fraction of its FP32 rate, so the accurate product that
// the mixed-precision mobility solve checks its residual with evaluates the pairs of
// different bodies in double-float arithmetic on the FP32 pipes: a value is an
// unevaluated sum hi + lo of two floats (about 48 significant bits).  The error-free
// transformations are Knuth's two-sum, Dekker's fast two-sum and the FMA-based exact
// product.  Same-body pairs are skipped (added exactly in FP64 by k_intra_body).

template <int TPT>
__global__ void __launch_bounds__(128) k_rpy_df(const MvItem* __restrict__ items, const long long* __restrict__ susp_blob_off,
                                                const double4_32a* __restrict__ spos, const double4_32a* __restrict__ slam,
                                                double4_32a* __restrict__ part, int NBL, RpyConstDF k) {
    __shared__ float4 sh[4 * MV_TILE];
    const MvItem it = items[blockIdx.x];
    const long long b0 = susp_blob_off[it.s];
    const int ns = (int)(susp_blob_off[it.s + 1] - b0);
    df xt[TPT], yt[TPT], zt[TPT], ux[TPT], uy[TPT], uz[TPT];
    float bt[TPT];
#pragma unroll
    for (int t = 0; t < TPT; ++t) {
        const double4_32a p = spos[b0 + min(it.t0 + (int)threadIdx.x + t * 128, ns - 1)];
        xt[t] = df_from(p.x);
        yt[t] = df_from(p.y);
        zt[t] = df_from(p.z);
        bt[t] = (float)p.w;
        ux[t] = uy[t] = uz[t] = df{0.f, 0.f};
    }
    const df one{1.f, 0.f};
    for (int j0 = it.j0; j0 < it.j1; j0 += MV_TILE) {
        const int n = min(MV_TILE, it.j1 - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < n; e += 128) {
            const double4_32a ps = spos[b0 + j0 + e];
            const double4_32a ls = slam[b0 + j0 + e];
            const df x = df_from(ps.x), y = df_from(ps.y), z = df_from(ps.z);
            const df lx = df_from(ls.x), ly = df_from(ls.y), lz = df_from(ls.z);
            sh[4 * e] = make_float4(x.h, y.h, z.h, (float)ps.w);
            sh[4 * e + 1] = make_float4(x.l, y.l, z.l, 0.f);
            sh[4 * e + 2] = make_float4(lx.h, ly.h, lz.h, 0.f);
            sh[4 * e + 3] = make_float4(lx.l, ly.l, lz.l, 0.f);
        }
        __syncthreads();
        for (int j = 0; j < n; ++j) {
            const float4 s0 = sh[4 * j], s1 = sh[4 * j + 1], s2 = sh[4 * j + 2], s3 = sh[4 * j + 3];
            const df lx{s2.x, s3.x}, ly{s2.y, s3.y}, lz{s2.z, s3.z};
#pragma unroll
            for (int t = 0; t < TPT; ++t) {
                if (s0.w == bt[t]) continue;   // same body: exact FP64 block elsewhere
                const df dx = df_sub(df{s0.x, s1.x}, xt[t]);
                const df dy = df_sub(df{s0.y, s1.y}, yt[t]);
                const df dz = df_sub(df{s0.z, s1.z}, zt[t]);
                const df r2 = df_add(df_add(df_mul(dx, dx), df_mul(dy, dy)), df_mul(dz, dz));
                const df ri = df_rsqrt(r2);
                df A, B;
                // r^2 >= 4a^2 compared in double-float (both normalised: high parts first)
                if (r2.h > k.four_a2.h || (r2.h == k.four_a2.h && r2.l >= k.four_a2.l)) {
                    const df ri2 = df_mul(ri, ri);
                    const df ri3 = df_mul(ri2, ri);
                    A = df_add(ri, df_mul(k.c23, ri3));
                    B = df_mul(ri3, df_sub(one, df_mul(k.c2, ri2)));
                } else {   // overlapping blobs of different bodies (r > 0 for distinct blobs)
                    const df r = df_mul(r2, ri);
                    A = df_mul(k.cA, df_sub(one, df_mul(k.c9, r)));
                    B = df_mul(k.cB, ri);
                }
                const df dl = df_add(df_add(df_mul(dx, lx), df_mul(dy, ly)), df_mul(dz, lz));
                const df s = df_mul(B, dl);
                ux[t] = df_add(ux[t], df_add(df_mul(A, lx), df_mul(s, dx)));
                uy[t] = df_add(uy[t], df_add(df_mul(A, ly), df_mul(s, dy)));
                uz[t] = df_add(uz[t], df_add(df_mul(A, lz), df_mul(s, dz)));
            }
        }
    }
#pragma unroll
    for (int t = 0; t < TPT; ++t) {
        const int ti = it.t0 + threadIdx.x + t * 128;
        if (ti < ns) part[(long long)it.k * NBL + b0 + ti] = make_double4_32a(df_to(ux[t]), df_to(uy[t]), df_to(uz[t]), 0.0);
    }
}

// x, gm_layout: the vector launch_pack_lambda was given (the FP64 kernel reads it unpacked)
void launch_rpy(gdc_ctx* c, int prec, const double* x, int gm_layout) {
    const int pe = prof_begin(c, prec == GDC_FP32_MIXED ? 0 : (prec == GDC_PREC_DF64 ? 3 : 1));
    if (prec == GDC_FP32_MIXED) {
        const double a = c->p.a;
        const RpyConst32 k = rpy_const32(a);
        // two targets per packed lane pair: tpt 4 -> P = 2, otherwise P = 1
#define GDC_RPY32_LAUNCH(PP, MB)                                                                             \
    k_rpy32<PP, MB><<<c->mv_n_items, 128, 0, c->stream>>>(c->mv_items, c->mv_active, c->susp_blob_off, c->spos, \
                                                          c->sdup, (float4*)c->mv_part, c->NBL, k, c->dev_status, \
                                                          first_wait_polls())
        if (c->use_sym) {
            launch_rpy32_sym(c);
        } else {
            ++c->n_launch;
            if (c->mv_tpt == 4) {
                if (c->mv_minb == 4)
                    GDC_RPY32_LAUNCH(2, 4);
                else
                    GDC_RPY32_LAUNCH(2, 6);
            } else {
                if (c->mv_minb == 4)
                    GDC_RPY32_LAUNCH(1, 4);
                else
                    GDC_RPY32_LAUNCH(1, 6);
            }
        }
#undef GDC_RPY32_LAUNCH
    } else if (prec == GDC_PREC_DF64 && c->dfs_minb) {
        launch_rpy_df_sym_pairs(c);   // its epilogue runs in launch_rpy_epilogue
    } else if (prec == GDC_PREC_DF64) {
        const RpyConstDF k = df_constants(c->p.a);
        if (c->mv_tpt == 4)
            ++c->n_launch, k_rpy_df<4><<<c->mv_n_items, 128, 0, c->stream>>>(c->mv_items, c->susp_blob_off, c->spos64,
                                                                             c->slam64, (double4_32a*)c->mv_part, c->NBL, k);
        else
            ++c->n_launch, k_rpy_df<2><<<c->mv_n_items, 128, 0, c->stream>>>(c->mv_items, c->susp_blob_off, c->spos64,
                                                                             c->slam64, (double4_32a*)c->mv_part, c->NBL, k);
    } else {
        launch_rpy64_sym(c, x, gm_layout);   // its epilogue runs in launch_rpy_epilogue
    }
    prof_end(c, pe);
}

// ---- epilogue: chunk sums in FP64, scale, and the -K V part of the saddle operator ----

template <typename P>
__device__ inline void load_part(const P* part, long long idx, double& x, double& y, double& z) {
    const P v = part[idx];
    x = (double)v.x;
    y = (double)v.y;
    z = (double)v.z;
}

// Exact minus clamped pair coefficients (units of 1/(8 pi eta)) for a pair at distance r < 2a:
// the FP32 pair kernel evaluates every pair, the self pair and overlapping pairs included,
// with the far-field form at r clamped to 2a (A = 7/(12a), B = 1/(16a^3) there); the
// overlapping branch of the RPY tensor has A = 4/(3a) (1 - 9r/(32a)), B = 1/(8a^2 r).
// FP32 suffices: the correction joins a product whose pair terms are FP32.
__device__ inline void near_delta(float a, float r, float& dA, float& dB) {
    dA = 4.f / (3.f * a) * (1.f - 9.f * r / (32.f * a)) - 7.f / (12.f * a);
    dB = (r > 0.f ? 1.f / (8.f * a * a * r) : 0.f) - 1.f / (16.f * a * a * a);
}

// Adds to (ux, uy, uz), in units of 1/(8 pi eta), the exact minus clamped terms of blob i's
// pairs with blobs of other bodies closer than 2a: from the list when it holds them all, else
// by a search of the suspension's blobs [so, se) (FP64 distances; blob_body given: skip
// same-body blobs, else only j = i).  x holds lambda, 3 per blob, or in the saddle layout
// through gm (blob -> offset) when gm is given.  Entries sub, sub + nsub, ... are taken.
__device__ inline void near_pair_correction(long long i, long long so, long long se, const int* __restrict__ near_cnt,
                                            const int* __restrict__ near_idx, const int* __restrict__ blob_body,
                                            const double* __restrict__ r, const double* __restrict__ x,
                                            const int* __restrict__ gm, double a, int sub, int nsub, double& ux,
                                            double& uy, double& uz) {
    const int m = near_cnt[i];
    const double four_a2 = 4.0 * a * a;
    const long long cnt = m <= GDC_NEAR_CAP ? m : se - so;
    for (long long q = sub; q < cnt; q += nsub) {
        const long long j = m <= GDC_NEAR_CAP ? (long long)near_idx[i * GDC_NEAR_CAP + q] : so + q;
        if (j == i || (blob_body && blob_body[j] == blob_body[i])) continue;
        const double dx = r[3 * j] - r[3 * i], dy = r[3 * j + 1] - r[3 * i + 1], dz = r[3 * j + 2] - r[3 * i + 2];
        const double r2 = dx * dx + dy * dy + dz * dz;
        if (!(r2 < four_a2)) continue;   // at or beyond 2a the clamped form is the RPY tensor
        float dA, dB;
        near_delta((float)a, sqrtf((float)r2), dA, dB);
        const long long oj = gm ? (long long)gm[j] : 3LL * j;
        const double lx = x[oj], ly = x[oj + 1], lz = x[oj + 2];
        const double s = (double)dB * (dx * lx + dy * ly + dz * lz);
        ux += (double)dA * lx + s * dx;
        uy += (double)dA * ly + s * dy;
        uz += (double)dA * lz + s * dz;
    }
}

// A sum in FP32 with compensation (FP64 adds are slow on GB300): sum - comp is the value.
struct Kahan {
    float sum = 0.f, comp = 0.f;
    __device__ __forceinline__ void add(float v) {
        const float y = __fsub_rn(v, comp);
        const float t = __fadd_rn(sum, y);
        comp = __fsub_rn(__fsub_rn(t, sum), y);
        sum = t;
    }
    // the sum over a group of EPI neighbouring lanes, on every lane: exact two-sums of the
    // leading parts, their errors joined with the compensations
    template <int EPI>
    __device__ __forceinline__ void group() {
#pragma unroll
        for (int o = 1; o < EPI; o <<= 1) {
            const float s2 = __shfl_xor_sync(0xffffffffu, sum, o), c2 = __shfl_xor_sync(0xffffffffu, comp, o);
            const float t = __fadd_rn(sum, s2), bb = __fsub_rn(t, sum);
            const float err = __fadd_rn(__fsub_rn(sum, __fsub_rn(t, bb)), __fsub_rn(s2, bb));
            comp = __fsub_rn(__fadd_rn(comp, c2), err);
            sum = t;
        }
    }
    __device__ __forceinline__ double value() const { return (double)sum - (double)comp; }
};

// Subtracts from (sx, sy, sz) the terms the FP32 pair kernel added for blob i's own body
// [j0, j1) (self pair included), recomputed from the same FP32 operands with the same
// operations, so that the FP32 rounding of those near-field terms cancels; the intra-body
// kernel then adds the same-body block of the body's template.  Blobs j0 + sub, j0 + sub +
// nsub, ... are taken.
__device__ inline void same_body_subtract(const float4 pt, long long j0, long long j1, const float4* __restrict__ sdup,
                                          const RpyConst32& k, int sub, int nsub, Kahan& sx, Kahan& sy, Kahan& sz) {
    for (long long j = j0 + sub; j < j1; j += nsub) {
        const float4 s0 = sdup[3 * j], s1 = sdup[3 * j + 1], s2 = sdup[3 * j + 2];
        const float dx = __fsub_rn(s0.x, pt.x), dy = __fsub_rn(s0.z, pt.y), dz = __fsub_rn(s1.x, pt.z);
        const float lx = s1.z, ly = s2.x, lz = s2.z;
        const float r2 = __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmul_rn(dz, dz)));
        const float ri = rsqrtf(fmaxf(r2, k.four_a2));
        const float ri2 = __fmul_rn(ri, ri), ri3 = __fmul_rn(ri2, ri);
        const float A = __fmaf_rn(k.c23, ri3, ri);
        const float B = __fmul_rn(ri3, __fmaf_rn(-k.c2, ri2, 1.f));
        const float sj = __fmul_rn(B, __fmaf_rn(dx, lx, __fmaf_rn(dy, ly, __fmul_rn(dz, lz))));
        sx.add(-__fmaf_rn(A, lx, __fmul_rn(sj, dx)));
        sy.add(-__fmaf_rn(A, ly, __fmul_rn(sj, dy)));
        sz.add(-__fmaf_rn(A, lz, __fmul_rn(sj, dz)));
    }
}

// u_i = c0 (sum of the chunk partial sums [+ near-pair corrections]) [- K V]
//
// near_cnt != 0 (FP32 products): corrects the pairs of other bodies closer than 2a and takes
// out the pair kernel's same-body terms (the intra-body kernel adds the template's block).
//
// EPI neighbouring threads share a blob: they take every EPI-th slot, same-body blob and near
// pair, joined by shuffles in a fixed order.  More threads shorten the chain of dependent loads,
// but the FP64 tail (2 lanes per clock per SM) is paid per warp.  us per launch with 1 / 2 / 4
// / 8 threads: 2,560 blobs 13.3 / 10.6 / 8.8 / 8.1, 20,202 blobs 17.8 / 13.6 / 14.5 / 18.0,
// 65,520 blobs 37.8 / 29.1 / 40.2 / 58.0, 161,000 blobs in 160 suspensions 67.8 / 78.1 / 100 /
// 154: 8 threads up to 8,192 blobs, 2 up to 98,304, 1 above.
template <typename P, int EPI>
__global__ void __launch_bounds__(256) k_rpy_epilogue(int NBL, const P* __restrict__ part, const int* __restrict__ blob_susp,
                               const int* __restrict__ nk, double c0, const double* __restrict__ x,
                               double* __restrict__ y, int gm_layout, const int* __restrict__ blob_gm,
                               const int* __restrict__ body_gm, const int* __restrict__ blob_body,
                               const double* __restrict__ r, const double* __restrict__ Yc,
                               const int* __restrict__ near_cnt, const int* __restrict__ near_idx, double a,
                               const long long* __restrict__ susp_blob_off, const long long* __restrict__ body_blob_off,
                               const float4* __restrict__ spos, const float4* __restrict__ sdup, RpyConst32 k32,
                               const float4* __restrict__ sym_part_j, const int* __restrict__ sym_row_nk,
                               const long long* __restrict__ sym_tile_base, const long long* __restrict__ sym_jbase) {
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int sub = (int)(tid % EPI);
    const bool in = tid / EPI < NBL;
    const int i = in ? (int)(tid / EPI) : NBL - 1;   // whole warps reach the shuffles
    double ux = 0.0, uy = 0.0, uz = 0.0;
    Kahan sx, sy, sz;
    if (sym_part_j) {
        // symmetric kernel: the target-side slots of the blob's tile row, then the source-side
        // slots (I, J) of every tile I before the blob's tile J, in order.  FP32 partials are
        // added with compensation in FP32, then converted once.
        const int s = blob_susp[i];
        const long long loc = i - susp_blob_off[s];
        const int J = (int)(loc / GDC_SYM_TILE), e = (int)(loc % GDC_SYM_TILE);
        const int n = sym_row_nk[sym_tile_base[s] + J];
        const float4* pi = reinterpret_cast<const float4*>(part);
#pragma unroll 4
        for (int k = sub; k < n; k += EPI) {
            const float4 v = pi[(long long)k * NBL + i];
            sx.add(v.x);
            sy.add(v.y);
            sz.add(v.z);
        }
        const long long s0 = sym_jbase[s] + (long long)J * (J - 1) / 2;
#pragma unroll 4
        for (int I = sub; I < J; I += EPI) {
            const float4 v = sym_part_j[(s0 + I) * GDC_SYM_TILE + e];
            sx.add(v.x);
            sy.add(v.y);
            sz.add(v.z);
        }
    } else {
        const int n = nk[blob_susp[i]];
        for (int k = sub; k < n; k += EPI) {
            double a0, b, cc;
            load_part(part, (long long)k * NBL + i, a0, b, cc);
            ux += a0;
            uy += b;
            uz += cc;
        }
    }
    bool join64 = true;   // FP64 parts to join
    if (near_cnt) {
        const int p = blob_body[i];
        same_body_subtract(spos[i], body_blob_off[p], body_blob_off[p + 1], sdup, k32, sub, EPI, sx, sy, sz);
        sx.group<EPI>();
        sy.group<EPI>();
        sz.group<EPI>();
        const long long so = susp_blob_off[blob_susp[i]], se = susp_blob_off[blob_susp[i] + 1];
        near_pair_correction(i, so, se, near_cnt, near_idx, blob_body, r, x, gm_layout ? blob_gm : nullptr, a, sub, EPI,
                             ux, uy, uz);
        join64 = !sym_part_j || __any_sync(0xffffffffu, near_cnt[i] != 0);
    }
    if (EPI > 1 && join64) {
#pragma unroll
        for (int o = 1; o < EPI; o <<= 1) {
            ux += __shfl_xor_sync(0xffffffffu, ux, o);
            uy += __shfl_xor_sync(0xffffffffu, uy, o);
            uz += __shfl_xor_sync(0xffffffffu, uz, o);
        }
    }
    if (!in || sub != 0) return;
    if (near_cnt) {
        ux += sx.value();
        uy += sy.value();
        uz += sz.value();
    }
    ux *= c0;
    uy *= c0;
    uz *= c0;
    if (!gm_layout) {
        y[3 * i] = ux;
        y[3 * i + 1] = uy;
        y[3 * i + 2] = uz;
        return;
    }
    // saddle operator: M lambda - K V, K V = U_p + Omega_p x (r_i - Y_p)  (Eq. rigid_body_cond)
    const int p = blob_body[i];
    const double* V = x + body_gm[p];
    const double dx = r[3 * i] - Yc[3 * p], dy = r[3 * i + 1] - Yc[3 * p + 1], dz = r[3 * i + 2] - Yc[3 * p + 2];
    const double kx = V[0] + (V[4] * dz - V[5] * dy);
    const double ky = V[1] + (V[5] * dx - V[3] * dz);
    const double kz = V[2] + (V[3] * dy - V[4] * dx);
    const long long o = blob_gm[i];
    y[o] = ux - kx;
    y[o + 1] = uy - ky;
    y[o + 2] = uz - kz;
}

// Blob rows of the saddle operator with the FCM mobility: y_i = (M_FCM lambda)_i - (K V)_i,
// K V = U_p + Omega_p x (r_i - Y_p) (Eq. rigid_body_cond), u = M_FCM lambda given 3 per blob.
__global__ void k_fcm_saddle_rows(int NBL, const double* __restrict__ u, const double* __restrict__ x,
                                  double* __restrict__ y, const int* __restrict__ blob_gm, const int* __restrict__ body_gm,
                                  const int* __restrict__ blob_body, const double* __restrict__ r,
                                  const double* __restrict__ Yc) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NBL) return;
    const int p = blob_body[i];
    const double* V = x + body_gm[p];
    const double dx = r[3 * i] - Yc[3 * p], dy = r[3 * i + 1] - Yc[3 * p + 1], dz = r[3 * i + 2] - Yc[3 * p + 2];
    const long long o = blob_gm[i];
    y[o] = u[3LL * i] - (V[0] + (V[4] * dz - V[5] * dy));
    y[o + 1] = u[3LL * i + 1] - (V[1] + (V[5] * dx - V[3] * dz));
    y[o + 2] = u[3LL * i + 2] - (V[2] + (V[3] * dy - V[4] * dx));
}

void launch_fcm_saddle_rows(gdc_ctx* c, const double* x, double* y) {
    ++c->n_launch, k_fcm_saddle_rows<<<ceil_div(c->NBL, 256), 256, 0, c->stream>>>(
        c->NBL, c->fcm_u, x, y, c->blob_gm, c->body_gm, c->blob_body, c->r, c->Yc);
}

template <typename P, int EPI>
static void launch_epilogue_t(gdc_ctx* c, const P* part, bool sym, double c0, const double* x, double* y, int gm_layout,
                              bool near) {
    ++c->n_launch, k_rpy_epilogue<P, EPI><<<ceil_div((long long)EPI * c->NBL, 256), 256, 0, c->stream>>>(
        c->NBL, part, c->blob_susp, c->mv_nk, c0, x, y, gm_layout, c->blob_gm, c->body_gm, c->blob_body, c->r, c->Yc,
        near ? c->near_cnt : nullptr, c->near_idx, c->p.a, c->susp_blob_off, c->body_blob_off, c->spos, c->sdup,
        rpy_const32(c->p.a), sym ? c->sym_part_j : nullptr, c->sym_row_nk, c->sym_tile_base, c->sym_jbase);
}

static void launch_epilogue(gdc_ctx* c, int prec, double c0, const double* x, double* y, int gm_layout,
                            bool near) {
    const bool sym = prec == GDC_FP32_MIXED && near && c->use_sym;   // RPY products only, not forces
    if (prec == GDC_FP32_MIXED) {
        const float4* part = sym ? c->sym_part_i : (const float4*)c->mv_part;
        if (c->NBL <= 8192)
            launch_epilogue_t<float4, 8>(c, part, sym, c0, x, y, gm_layout, near);
        else if (c->NBL <= 98304)
            launch_epilogue_t<float4, 2>(c, part, sym, c0, x, y, gm_layout, near);
        else
            launch_epilogue_t<float4, 1>(c, part, sym, c0, x, y, gm_layout, near);
    } else {
        launch_epilogue_t<double4_32a, 2>(c, (const double4_32a*)c->mv_part, false, c0, x, y, gm_layout, false);
    }
}

void launch_rpy_epilogue(gdc_ctx* c, int prec, const double* x, double* y, int gm_layout, bool same_body) {
    if (prec == GDC_FP64 || (prec == GDC_PREC_DF64 && c->dfs_minb))
        launch_p64_epilogue(c, prec, x, y, gm_layout);
    else
        launch_epilogue(c, prec, 1.0 / (8.0 * 3.141592653589793 * c->p.eta), x, y, gm_layout, prec == GDC_FP32_MIXED);
    // same-body blocks from the template: the df64 pair kernel leaves those pairs out and the
    // FP32 epilogue has taken the FP32 pair kernel's same-body terms out again (so without
    // them an FP32 product is exactly the blocks between different bodies)
    if (prec == GDC_PREC_DF64 || (prec == GDC_FP32_MIXED && same_body))
        launch_intra_body(c, x, y, gm_layout, prec == GDC_FP32_MIXED);
}

// ---- pairs closer than 2a ------------------------------------------------------------

// For every blob i, the blobs j of other bodies of its suspension whose FP32 r_ij^2, computed
// exactly as the FP32 pair kernel computes it, is below 4a^2 -- the pairs the pair kernel
// clamps: the pairs whose term the epilogue corrects (same-body pairs are replaced whole).  One block per (256 targets, source chunk) of one
// suspension, two targets per thread in packed arithmetic; a found pair takes the next slot
// of its target's list (near_cnt starts at zero), and k_near_sort then orders every list so
// that the corrections are summed in a fixed order.
// items = nullptr: one suspension, blocks in rows of `chunks` chunks of `src` sources.
__global__ void __launch_bounds__(128) k_near_build(const int4* __restrict__ items, int chunks, int src,
                                                   const long long* __restrict__ susp_blob_off,
                                                   const float4* __restrict__ spos, float four_a2,
                                                   int* __restrict__ near_cnt, int* __restrict__ near_idx) {
    __shared__ float4 sh[2 * 256];
    int4 it;   // (suspension, first target, first source, end source)
    if (items) {
        it = items[blockIdx.x];
    } else {
        const int n = (int)susp_blob_off[1], j0 = (int)(blockIdx.x % chunks) * src;
        it = make_int4(0, (int)(blockIdx.x / chunks) * 256, j0, min(n, j0 + src));
    }
    const long long b0 = susp_blob_off[it.x];
    const int ns = (int)(susp_blob_off[it.x + 1] - b0);
    const int ta = it.y + (int)threadIdx.x, tb = ta + 128;
    const float4 pa = spos[b0 + min(ta, ns - 1)], pb = spos[b0 + min(tb, ns - 1)];
    const float2 xt = make_float2(pa.x, pb.x), yt = make_float2(pa.y, pb.y), zt = make_float2(pa.z, pb.z);
    for (int j0 = it.z; j0 < it.w; j0 += 256) {
        const int n = min(256, it.w - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < n; e += 128) {
            const float4 q = spos[b0 + j0 + e];
            sh[2 * e] = make_float4(q.x, q.x, q.y, q.y);
            sh[2 * e + 1] = make_float4(q.z, q.z, q.w, q.w);   // w: body index bits
        }
        __syncthreads();
#pragma unroll 4
        for (int j = 0; j < n; ++j) {
            const float4 s0 = sh[2 * j], s1 = sh[2 * j + 1];
            const float2 dx = sub2(make_float2(s0.x, s0.y), xt), dy = sub2(make_float2(s0.z, s0.w), yt),
                         dz = sub2(make_float2(s1.x, s1.y), zt);
            const float2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            if (r2.x < four_a2 || r2.y < four_a2) {   // rare
                const int jg = j0 + j;
                const int bj = __float_as_int(s1.z);
                if (r2.x < four_a2 && bj != __float_as_int(pa.w) && ta < ns) {
                    const int slot = atomicAdd(near_cnt + b0 + ta, 1);
                    if (slot < GDC_NEAR_CAP) near_idx[(b0 + ta) * GDC_NEAR_CAP + slot] = (int)(b0 + jg);
                }
                if (r2.y < four_a2 && bj != __float_as_int(pb.w) && tb < ns) {
                    const int slot = atomicAdd(near_cnt + b0 + tb, 1);
                    if (slot < GDC_NEAR_CAP) near_idx[(b0 + tb) * GDC_NEAR_CAP + slot] = (int)(b0 + jg);
                }
            }
        }
    }
}

// Orders each blob's near-pair list (insertion sort; lists are short).  A count above
// GDC_NEAR_CAP leaves the list incomplete: the epilogue then searches the suspension.
__global__ void k_near_sort(int n, const int* __restrict__ near_cnt, int* __restrict__ near_idx) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int m = near_cnt[i];
    if (m < 2 || m > GDC_NEAR_CAP) return;
    int* l = near_idx + i * GDC_NEAR_CAP;
    for (int a = 1; a < m; ++a) {
        const int v = l[a];
        int b = a - 1;
        while (b >= 0 && l[b] > v) {
            l[b + 1] = l[b];
            --b;
        }
        l[b + 1] = v;
    }
}

void launch_near_build(gdc_ctx* c) {
    if (c->p.mobility == GDC_MOB_FCM) return;   // the lists serve the RPY products only
    if (forces_use_cells(c)) {
        launch_near_cell(c);   // the same lists from a cell list, O(N_b)
    } else {
        cudaMemsetAsync(c->near_cnt, 0, sizeof(int) * c->NBL, c->stream);
        ++c->n_launch, k_near_build<<<c->n_near_items, 128, 0, c->stream>>>(c->near_items, 0, 0, c->susp_blob_off, c->spos,
                                                                            (float)(4.0 * c->p.a * c->p.a), c->near_cnt,
                                                                            c->near_idx);
    }
    ++c->n_launch, k_near_sort<<<ceil_div(c->NBL, 256), 256, 0, c->stream>>>(c->NBL, c->near_cnt, c->near_idx);
}

// ---- pair forces between blobs of different bodies, every pair in tiles -------------

// f_i = sum_j F(|r_i - r_j|) (r_i - r_j)/|r_i - r_j| over blobs j of other bodies with F
// the pair force of forces.cuh; pairs beyond its cutoff are skipped.
template <int TPT>
__global__ void __launch_bounds__(128) k_forces32(const MvItem* __restrict__ items, const long long* __restrict__ susp_blob_off,
                                                  const float4* __restrict__ spos, float4* __restrict__ part, int NBL,
                                                  ForceK<float> k) {
    __shared__ float4 sp[MV_TILE];
    const MvItem it = items[blockIdx.x];
    const long long b0 = susp_blob_off[it.s];
    const int ns = (int)(susp_blob_off[it.s + 1] - b0);
    const int ti0 = it.t0 + threadIdx.x;
    float xt[TPT], yt[TPT], zt[TPT], fx[TPT], fy[TPT], fz[TPT];
    int bt[TPT];
    for (int t = 0; t < TPT; ++t) {
        fx[t] = fy[t] = fz[t] = 0.f;
        const float4 p = spos[b0 + min(ti0 + t * 128, ns - 1)];
        xt[t] = p.x;
        yt[t] = p.y;
        zt[t] = p.z;
        bt[t] = __float_as_int(p.w);
    }
    for (int j0 = it.j0; j0 < it.j1; j0 += MV_TILE) {
        const int n = min(MV_TILE, it.j1 - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < n; e += 128) sp[e] = spos[b0 + j0 + e];
        __syncthreads();
        for (int j = 0; j < n; ++j) {
            const float4 ps = sp[j];
            const int bj = __float_as_int(ps.w);
#pragma unroll
            for (int t = 0; t < TPT; ++t) {
                const float dx = xt[t] - ps.x, dy = yt[t] - ps.y, dz = zt[t] - ps.z;
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (bj != bt[t] && r2 < k.rc2 && r2 > 0.f) {
                    const float r = sqrtf(r2);
                    const float s = pair_force(r, k) / r;
                    fx[t] = fmaf(s, dx, fx[t]);
                    fy[t] = fmaf(s, dy, fy[t]);
                    fz[t] = fmaf(s, dz, fz[t]);
                }
            }
        }
    }
    for (int t = 0; t < TPT; ++t) {
        const int ti = ti0 + t * 128;
        if (ti < ns) part[(long long)it.k * NBL + b0 + ti] = make_float4(fx[t], fy[t], fz[t], 0.f);
    }
}

template <int TPT>
__global__ void __launch_bounds__(128) k_forces64(const MvItem* __restrict__ items, const long long* __restrict__ susp_blob_off,
                                                  const double4_32a* __restrict__ spos, double4_32a* __restrict__ part, int NBL,
                                                  ForceK<double> k) {
    __shared__ double4_32a sp[MV_TILE];
    const MvItem it = items[blockIdx.x];
    const long long b0 = susp_blob_off[it.s];
    const int ns = (int)(susp_blob_off[it.s + 1] - b0);
    const int ti0 = it.t0 + threadIdx.x;
    double xt[TPT], yt[TPT], zt[TPT], fx[TPT], fy[TPT], fz[TPT];
    long long bt[TPT];
    for (int t = 0; t < TPT; ++t) {
        fx[t] = fy[t] = fz[t] = 0.0;
        const double4_32a p = spos[b0 + min(ti0 + t * 128, ns - 1)];
        xt[t] = p.x;
        yt[t] = p.y;
        zt[t] = p.z;
        bt[t] = (long long)p.w;
    }
    for (int j0 = it.j0; j0 < it.j1; j0 += MV_TILE) {
        const int n = min(MV_TILE, it.j1 - j0);
        __syncthreads();
        for (int e = threadIdx.x; e < n; e += 128) sp[e] = spos[b0 + j0 + e];
        __syncthreads();
        for (int j = 0; j < n; ++j) {
            const double4_32a ps = sp[j];
            const long long bj = (long long)ps.w;
#pragma unroll
            for (int t = 0; t < TPT; ++t) {
                const double dx = xt[t] - ps.x, dy = yt[t] - ps.y, dz = zt[t] - ps.z;
                const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
                if (bj != bt[t] && r2 < k.rc2 && r2 > 0.0) {
                    const double r = sqrt(r2);
                    const double s = pair_force(r, k) / r;
                    fx[t] = fma(s, dx, fx[t]);
                    fy[t] = fma(s, dy, fy[t]);
                    fz[t] = fma(s, dz, fz[t]);
                }
            }
        }
    }
    for (int t = 0; t < TPT; ++t) {
        const int ti = ti0 + t * 128;
        if (ti < ns) part[(long long)it.k * NBL + b0 + ti] = make_double4_32a(fx[t], fy[t], fz[t], 0.0);
    }
}

#define GDC_FORCES_LAUNCH(TPT)                                                                         \
    do {                                                                                               \
        if (prec == GDC_FP32_MIXED)                                                                    \
            ++c->n_launch, k_forces32<TPT><<<c->mv_n_items, 128, 0, c->stream>>>(c->mv_items, c->susp_blob_off, c->spos, \
                (float4*)c->mv_part, c->NBL, force_constants<float>(c->p));                                \
        else                                                                                           \
            ++c->n_launch, k_forces64<TPT><<<c->mv_n_items, 128, 0, c->stream>>>(c->mv_items, c->susp_blob_off,          \
                c->spos64, (double4_32a*)c->mv_part, c->NBL, force_constants<double>(c->p));                   \
    } while (0)

void launch_forces_pair(gdc_ctx* c, int prec, double* fblob) {
    const int pe = prof_begin(c, 2);
    if (c->mv_tpt == 1)
        GDC_FORCES_LAUNCH(1);
    else if (c->mv_tpt == 4)
        GDC_FORCES_LAUNCH(4);
    else
        GDC_FORCES_LAUNCH(2);
    prof_end(c, pe);
    launch_epilogue(c, prec, 1.0, nullptr, fblob, 0, false);
}

// ---- work list ------------------------------------------------------------------------

void build_mv_items(gdc_ctx* c, int tpt, double waves) {
    c->mv_tpt = tpt;
    c->mv_waves = waves;
    const int tile_targets = 128 * tpt;
    double P = 0.0;
    std::vector<long long> ns(c->S);
    for (int s = 0; s < c->S; ++s) {
        ns[s] = c->h_blob_off[s + 1] - c->h_blob_off[s];
        P += (double)ns[s] * (double)ns[s];
    }
    c->pair_evals_per_matvec = P;
    const double target_items = (double)c->num_sms * 4.0 * waves;  // `waves` launches of 4 blocks per SM
    c->h_mv_items.clear();
    c->h_mv_nk.assign(c->S, 1);
    int kmax = 1;
    for (int s = 0; s < c->S; ++s) {
        const long long n = ns[s];
        const int nt = ceil_div(n, tile_targets);
        int nk = (int)std::lround(target_items * (double)n * (double)n / std::max(P, 1.0) / std::max(nt, 1));
        nk = std::max(1, std::min(nk, std::max(1, ceil_div(n, 32))));
        nk = std::min(nk, 64);
        long long csz = (n + nk - 1) / nk;
        csz = ((csz + 31) / 32) * 32;
        nk = (int)std::max<long long>(1, (n + csz - 1) / csz);
        c->h_mv_nk[s] = nk;
        kmax = std::max(kmax, nk);
        for (int t = 0; t < nt; ++t)
            for (int k = 0; k < nk; ++k) {
                MvItem it{};
                it.s = s;
                it.t0 = t * tile_targets;
                it.j0 = (int)(k * csz);
                it.j1 = (int)std::min<long long>(n, (k + 1) * csz);
                it.k = k;
                if (it.j1 > it.j0) c->h_mv_items.push_back(it);
            }
    }
    // largest items first, so the tail of the launch is made of small ones
    std::stable_sort(c->h_mv_items.begin(), c->h_mv_items.end(), [&](const MvItem& x, const MvItem& y) {
        const long long cx = (long long)std::min<long long>(tile_targets, ns[x.s] - x.t0) * (x.j1 - x.j0);
        const long long cy = (long long)std::min<long long>(tile_targets, ns[y.s] - y.t0) * (y.j1 - y.j0);
        return cx > cy;
    });
    c->mv_n_items = (int)c->h_mv_items.size();
    c->mv_kmax = kmax;
}

}  // namespace gdc

namespace gdc {

// Candidate tilings of the pair kernels: targets per thread x work items per launch.
static const int kTpt[2] = {2, 4};
static const double kWaves[3] = {4.0, 8.0, 16.0};
static const int kSymMinBlocks[3] = {2, 3, 4};   // resident blocks per SM of the symmetric kernel
static const int kMvMinBlocks[2] = {4, 6};       // resident blocks per SM of the ordered kernel
static const int kDfsMinBlocks[2] = {3, 4};      // resident blocks per SM of the symmetric double-float kernel

// Sources per item of the symmetric FP32 kernel: the longest range (a power of two, 32 to
// 2,048) that gives at least 6 full items per SM and is at most 1/48 of the largest suspension, or
// gives at least 16 full items per SM whatever its length.  Short ranges spread few pairs over the
// chip and leave more partial sums to add; long ones end in a ragged last wave, which 16 items
// per SM make short.  Full items, the sources of all rows over the width: thousands of tiny
// suspensions have as many items but hardly any work to hide a long one behind (one of 2,040
// blobs and 4,000 of 12: 407 us with 2,048 sources, 278 with 32).  us per product (positions, near lists, pair kernel, epilogue) at 3 resident
// blocks per SM, by this rule (its width) and at 32 / 128 / 512 / 1,024 / 2,048 sources:
//   one suspension of 2,556 blobs 121 (32): 124 / 134 / 164 / 217 / 295
//   8,400 blobs 190 (64): 204 / 189 / 205 / 269 / 398
//   20,202 blobs 422 (256): 519 / 412 / 425 / 463 / 552
//   65,520 blobs 2,538 (1,024): 3,392 / 2,624 / 2,553 / 2,539 / 2,623
//   24 of 2,700 blobs 304 (64): 308 / 296 / 320 / 336 / 414
//   24 of 9,000 blobs 1,346 (512): 1,661 / 1,400 / 1,346 / 1,343 / 1,393
//   310 of 2,700 blobs 1,853 (1,024): 2,164 / 1,933 / 1,868 / 1,853 / 1,853
//   512 of 8 to 128 bodies, 746,060 blobs, 1,331 (512): 1,534 / 1,384 / 1,331 / 1,333 / 1,335
static int sym_default_width(const gdc_ctx* c) {
    long long nmax = 1;
    for (int s = 0; s < c->S; ++s) nmax = std::max(nmax, c->h_blob_off[s + 1] - c->h_blob_off[s]);
    const long long sources = pair_list_items(c, GDC_SYM_TILE, 1);   // over all rows of tiles
    int w = 2048;
    for (; w > 32; w /= 2) {
        const long long items = sources / w;
        if (items >= 16LL * c->num_sms || (w <= nmax / 48 && items >= 6LL * c->num_sms)) break;
    }
    return w;
}

// The tuner times half, once and twice that width from GDC_TUNE_PAIRS ordered pairs per product
// on; below, the rule stands (timings of a few microseconds would pick differently from one
// context to the next, and the product's rounding with them).
static bool tuned(const gdc_ctx* c) { return c->p.autotune && c->pair_evals_per_matvec >= GDC_TUNE_PAIRS; }

void plan_mv_capacity(gdc_ctx* c) {
    int cap_items = 0, cap_k = 1;
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 3; ++b) {
            build_mv_items(c, kTpt[a], kWaves[b]);
            cap_items = std::max(cap_items, c->mv_n_items);
            cap_k = std::max(cap_k, c->mv_kmax);
        }
    c->mv_cap_items = cap_items;
    c->mv_cap_kmax = cap_k;
    build_mv_items(c, 2, 8.0);
    const int w0 = sym_default_width(c);
    int scap = 0, sk = 1;
    for (int w : {w0 / 2, w0, 2 * w0}) {
        if (w < 32 || (w != w0 && !tuned(c))) continue;
        build_sym_items(c, w);
        scap = std::max(scap, c->sym_n_items);
        sk = std::max(sk, c->sym_kmax);
    }
    c->sym_cap_items = scap;
    c->sym_cap_kmax = sk;
    c->sym_n_tiles = c->h_sym_tile_base.back();
    c->sym_n_jslots = c->h_sym_jbase.back();
    build_sym_items(c, w0);
    build_dfs_list(c);
    build_p64_list(c);
}

static gdc_status upload_items(gdc_ctx* c) {
    cudaError_t e = cudaMemcpyAsync(c->mv_items, c->h_mv_items.data(), sizeof(MvItem) * c->h_mv_items.size(),
                                    cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->mv_nk, c->h_mv_nk.data(), sizeof(int) * c->S, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return cuda_check(c, e, "work-list upload");
}

// At the loaded configuration (lambda = the current W buffer), three FP32 RPY products (pair
// kernel and epilogue: more items leave more partial sums to add) per candidate, and the
// fastest is kept: the symmetric kernel's item width and resident blocks per SM, or with
// pair_kernel = 1 the ordered kernel's tiling (the ordered kernel took 1.2 to 1.9 times as
// long at every size measured); then one launch of each double-float residual kernel.
gdc_status autotune_pair_kernel(gdc_ctx* c) {
    if (!tuned(c)) return default_pair_kernel(c);
    cudaEvent_t e0, e1;
    gdc_status st = cuda_check(c, cudaEventCreate(&e0), "event");
    if (st != GDC_OK) return st;
    if ((st = cuda_check(c, cudaEventCreate(&e1), "event")) != GDC_OK) return st;
    launch_normals(c, 0, 0, c->W);
    launch_pack_lambda(c, GDC_FP32_MIXED, c->W, 0);
    const bool ordered = c->p.pair_kernel == 1;
    float best = 1e30f;
    auto product = [&] {
        launch_rpy(c, GDC_FP32_MIXED, c->W, 0);
        launch_rpy_epilogue(c, GDC_FP32_MIXED, c->W, c->lz_u, 0, false);
    };
    auto time3 = [&](float& ms) -> gdc_status {
        product();  // warm-up
        cudaEventRecord(e0, c->stream);
        for (int r = 0; r < 3; ++r) product();
        cudaEventRecord(e1, c->stream);
        gdc_status s2 = cuda_check(c, cudaEventSynchronize(e1), "autotune");
        if (s2 == GDC_OK) cudaEventElapsedTime(&ms, e0, e1);
        return s2;
    };
    c->use_sym = !ordered;
    if (ordered) {
        int bt = 2, bminb = 6;
        double bw = 8.0;
        for (int a = 0; a < 2 && st == GDC_OK; ++a)
            for (int b = 0; b < 3 && st == GDC_OK; ++b) {
                build_mv_items(c, kTpt[a], kWaves[b]);
                if ((st = upload_items(c)) != GDC_OK) break;
                for (int mb : kMvMinBlocks) {
                    c->mv_minb = mb;
                    float ms = 0.f;
                    if ((st = time3(ms)) != GDC_OK) break;
                    if (ms < best) {
                        best = ms;
                        bt = kTpt[a];
                        bw = kWaves[b];
                        bminb = mb;
                    }
                }
            }
        build_mv_items(c, bt, bw);
        c->mv_minb = bminb;
    } else {
        const int w0 = sym_default_width(c);
        int bwid = w0, bminb = 3;
        for (int w : {w0 / 2, w0, 2 * w0}) {
            if (w < 32 || st != GDC_OK) continue;
            build_sym_items(c, w);
            if ((st = sym_upload(c)) != GDC_OK) break;
            for (int mb : kSymMinBlocks) {
                c->sym_minb = mb;
                float ms = 0.f;
                if ((st = time3(ms)) != GDC_OK) break;
                if (ms < best) {
                    best = ms;
                    bwid = w;
                    bminb = mb;
                }
            }
        }
        build_sym_items(c, bwid);
        c->sym_minb = bminb;
    }
    if (st == GDC_OK) {
        c->autotune_ms = best / 3.0;
        st = upload_items(c);
        if (st == GDC_OK) st = sym_upload(c);
    }
    // the double-float residual kernel, one timed launch each after a warm-up (about 40 ms
    // per product at 65k blobs)
    c->dfs_minb = ordered ? 0 : 4;
    if (c->p.df_kernel) {
        c->dfs_minb = c->p.df_kernel == 1 ? 0 : c->p.df_kernel;
    } else if (!ordered && st == GDC_OK) {
        launch_pack_lambda(c, GDC_PREC_DF64, c->W, 0);
        float dbest = 1e30f;
        int bdf = 4;
        for (int mb : kDfsMinBlocks) {
            c->dfs_minb = mb;
            float ms = 0.f;
            launch_rpy(c, GDC_PREC_DF64, c->W, 0);   // warm-up
            cudaEventRecord(e0, c->stream);
            launch_rpy(c, GDC_PREC_DF64, c->W, 0);
            cudaEventRecord(e1, c->stream);
            if ((st = cuda_check(c, cudaEventSynchronize(e1), "autotune")) != GDC_OK) break;
            cudaEventElapsedTime(&ms, e0, e1);
            if (ms < dbest) {
                dbest = ms;
                bdf = mb;
            }
        }
        c->dfs_minb = bdf;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return st;
}

// Untuned: the kernel params.pair_kernel names (symmetric for 0 and 2) with the default work
// lists, and the double-float kernel of the same kind.
gdc_status default_pair_kernel(gdc_ctx* c) {
    c->use_sym = c->p.pair_kernel != 1;
    c->dfs_minb = c->p.df_kernel ? (c->p.df_kernel == 1 ? 0 : c->p.df_kernel) : (c->use_sym ? 4 : 0);
    gdc_status st = upload_items(c);
    return st != GDC_OK ? st : sym_upload(c);
}

}  // namespace gdc

// ---- allocation-free RPY product (gdc_rpy_apply_noalloc) ------------------------------
//
// For callers that cannot allocate device memory.  All scratch of this variant (packed
// sources, chunk partial sums, the work list) lives in one file-scope device array of
// fixed size, so the call allocates nothing; every GPU that loads the library holds the
// array until the process exits.  It reuses the FP32 pair kernel above on one suspension
// of free blobs, with the same near-pair list and FP64 corrections of the self pair and of
// the pairs closer than 2a.

#include <cooperative_groups.h>

#include <mutex>

#define GDC_NOALLOC_SLOTS (16 * GDC_NOALLOC_MAX_BLOBS)   // partial sums: chunks x blobs of a call
#define GDC_NOALLOC_TILE 256   // targets per work item (two per thread)
#define GDC_NOALLOC_ITEMS 2048 // work items of a call
#define GDC_NOALLOC_EPI 8      // threads per blob of the epilogue

namespace gdc {

namespace cg = cooperative_groups;

struct NoallocScratch {
    float4 spos[GDC_NOALLOC_MAX_BLOBS];
    float4 sdup[3 * GDC_NOALLOC_MAX_BLOBS];
    float4 part[GDC_NOALLOC_SLOTS];
    MvItem items[GDC_NOALLOC_ITEMS];
    int near_cnt[GDC_NOALLOC_MAX_BLOBS];
    int near_idx[GDC_NOALLOC_MAX_BLOBS * GDC_NEAR_CAP];
    long long susp_blob_off[2];
    int status[4];   // set by the pair kernel if a tile copy times out (u is then incomplete)
};

static __device__ __align__(256) NoallocScratch g_noalloc_scratch;

// Start of a call, one cluster of NOALLOC_CL blocks: the blob centroid (sums in a fixed order),
// positions relative to it (FP32), lambda, identity body table, work list, status words.  A
// block keeps its blobs' positions in registers between the two halves.  As a single block for
// the centroid (bound by one SM's FP64 adds) and a second launch for the rest, 3,001 blobs took
// 10.6 + 3.8 us; in one 9.0.
constexpr int NOALLOC_CL = 8;
constexpr int NOALLOC_PER = GDC_NOALLOC_MAX_BLOBS / (NOALLOC_CL * 1024);   // blobs per thread
static_assert(NOALLOC_PER * NOALLOC_CL * 1024 == GDC_NOALLOC_MAX_BLOBS, "the cluster covers every size");

__global__ void __cluster_dims__(NOALLOC_CL, 1, 1) __launch_bounds__(1024)
    k_noalloc_prepare(NoallocScratch* __restrict__ sc, const double* __restrict__ r, const double* __restrict__ lam,
                      int n, int nk, int csz) {
    __shared__ double sh[3 * 1024];
    __shared__ double part[3], cen[3];
    cg::cluster_group cl = cg::this_cluster();
    const int per = (n + NOALLOC_CL - 1) / NOALLOC_CL;
    const int lo = blockIdx.x * per, hi = min(n, lo + per);
    double p[NOALLOC_PER][3], acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int q = 0; q < NOALLOC_PER; ++q) {
        const int i = lo + threadIdx.x + 1024 * q;
#pragma unroll
        for (int d = 0; d < 3; ++d) p[q][d] = i < hi ? r[3 * i + d] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < NOALLOC_PER; ++q)
        if (lo + (int)threadIdx.x + 1024 * q < hi)
#pragma unroll
            for (int d = 0; d < 3; ++d) acc[d] += p[q][d];
    const double v = block_sum3<1024>(acc, sh);
    if (threadIdx.x < 96 && (threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    cl.sync();
    if (threadIdx.x < 3) {
        double t = 0.0;
#pragma unroll
        for (int b = 0; b < NOALLOC_CL; ++b) t += *cl.map_shared_rank(&part[threadIdx.x], b);
        cen[threadIdx.x] = t / n;
    }
    __syncthreads();
    const double c0 = cen[0], c1 = cen[1], c2 = cen[2];
#pragma unroll
    for (int q = 0; q < NOALLOC_PER; ++q) {
        const int i = lo + threadIdx.x + 1024 * q;
        if (i >= hi) continue;
        sc->near_cnt[i] = 0;
        const float x = (float)(p[q][0] - c0), y = (float)(p[q][1] - c1), z = (float)(p[q][2] - c2);
        const float lx = (float)lam[3 * i], ly = (float)lam[3 * i + 1], lz = (float)lam[3 * i + 2];
        sc->spos[i] = make_float4(x, y, z, __int_as_float(i));
        sc->sdup[3 * i] = make_float4(x, x, y, y);
        sc->sdup[3 * i + 1] = make_float4(z, z, lx, lx);
        sc->sdup[3 * i + 2] = make_float4(ly, ly, lz, lz);
    }
    const int ntile = (n + GDC_NOALLOC_TILE - 1) / GDC_NOALLOC_TILE;
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < ntile * nk; b += gridDim.x * blockDim.x) {
        MvItem it{};
        it.s = 0;
        it.t0 = (b / nk) * GDC_NOALLOC_TILE;
        it.k = b % nk;
        it.j0 = it.k * csz;
        it.j1 = min(n, (it.k + 1) * csz);
        sc->items[b] = it;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        sc->susp_blob_off[0] = 0;
        sc->susp_blob_off[1] = n;
    }
    if (blockIdx.x == 0 && threadIdx.x < 4) sc->status[threadIdx.x] = 0;
    cl.sync();   // no block leaves before its sums are read
}

// u_i = c0 (sum of chunk partials + self-pair and near-pair corrections), GDC_NOALLOC_EPI
// neighbouring threads per blob (at most 16,384 blobs: the chain of one thread's dependent loads
// is what a launch waits for)
__global__ void __launch_bounds__(256) k_noalloc_epilogue(const NoallocScratch* __restrict__ sc,
                                                          const double* __restrict__ r, const double* __restrict__ lam,
                                                          int n, int nk, double c0, double a, double* __restrict__ u) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const int sub = tid % GDC_NOALLOC_EPI;
    const bool in = tid / GDC_NOALLOC_EPI < n;
    const int i = in ? tid / GDC_NOALLOC_EPI : n - 1;   // whole warps reach the shuffles
    double x = 0.0, y = 0.0, z = 0.0;
#pragma unroll 4
    for (int k = sub; k < nk; k += GDC_NOALLOC_EPI) {
        const float4 v = sc->part[(long long)k * n + i];
        x += v.x;
        y += v.y;
        z += v.z;
    }
    if (sub == 0) {
        // self pair: exact 4/(3a), clamped far field 7/(12a) (d = 0, so FP32 leaves only the rsqrt rounding)
        const double cs = 4.0 / (3.0 * a) - 7.0 / (12.0 * a);
        x += cs * lam[3 * i];
        y += cs * lam[3 * i + 1];
        z += cs * lam[3 * i + 2];
    }
    near_pair_correction(i, 0, n, sc->near_cnt, sc->near_idx, nullptr, r, lam, nullptr, a, sub, GDC_NOALLOC_EPI, x, y, z);
#pragma unroll
    for (int o = 1; o < GDC_NOALLOC_EPI; o <<= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
    }
    if (!in || sub != 0) return;
    if (sc->status[1] != 0) {   // a tile copy of the pair kernel timed out: u would be incomplete
        u[3 * i] = u[3 * i + 1] = u[3 * i + 2] = __longlong_as_double(0x7ff8000000000000LL);
        return;
    }
    u[3 * i] = c0 * x;
    u[3 * i + 1] = c0 * y;
    u[3 * i + 2] = c0 * z;
}

// Device address of the scratch array and SM count, looked up once per device.
static std::mutex g_noalloc_mu;
static NoallocScratch* g_noalloc_ptr[128] = {};
static int g_noalloc_sms[128] = {};
static thread_local std::string g_noalloc_err;

const char* noalloc_last_error() { return g_noalloc_err.c_str(); }

static gdc_status noalloc_fail(gdc_status s, const std::string& m) {
    g_noalloc_err = m;
    return s;
}

}  // namespace gdc

extern "C" gdc_status gdc_rpy_apply_noalloc(const double* r, const double* lambda, double* u, int n_blobs, double a,
                                            double eta, void* stream) {
    using namespace gdc;
    if (!r || !lambda || !u) return noalloc_fail(GDC_ERR_INVALID_ARG, "gdc_rpy_apply_noalloc: NULL pointer");
    if (n_blobs < 1 || n_blobs > GDC_NOALLOC_MAX_BLOBS)
        return noalloc_fail(GDC_ERR_INVALID_ARG, "gdc_rpy_apply_noalloc: n_blobs must be in [1, " +
                                                     std::to_string(GDC_NOALLOC_MAX_BLOBS) + "], got " +
                                                     std::to_string(n_blobs));
    if (!(a > 0.0) || !(eta > 0.0)) return noalloc_fail(GDC_ERR_INVALID_ARG, "gdc_rpy_apply_noalloc: a and eta must be > 0");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 128)
        return noalloc_fail(GDC_ERR_CUDA, std::string("gdc_rpy_apply_noalloc: no usable device: ") + cudaGetErrorString(e));
    NoallocScratch* sc;
    int sms;
    {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_noalloc_ptr[dev]) {   // first call on this device: look up the array's device address
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess)
                return noalloc_fail(GDC_ERR_CUDA, std::string("gdc_rpy_apply_noalloc: cudaGetSymbolAddress failed: ") +
                                                      cudaGetErrorString(e));
            int v = 0;
            if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 152;
            g_noalloc_sms[dev] = v;
            g_noalloc_ptr[dev] = (NoallocScratch*)p;
        }
        sc = g_noalloc_ptr[dev];
        sms = g_noalloc_sms[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    const int ntile = (n_blobs + GDC_NOALLOC_TILE - 1) / GDC_NOALLOC_TILE;
    // source chunks: 6 blocks per SM (the pair kernel's resident blocks), at least 32 sources
    // each, within the scratch for partial sums and items (64 tiles at most, so 32 chunks fit)
    int nk = std::max(1, (6 * sms + ntile - 1) / ntile);
    nk = std::min(nk, std::min(GDC_NOALLOC_SLOTS / n_blobs, GDC_NOALLOC_ITEMS / ntile));
    nk = std::min(nk, std::max(1, (n_blobs + 31) / 32));
    int csz = (n_blobs + nk - 1) / nk;
    csz = (csz + 31) / 32 * 32;
    nk = (n_blobs + csz - 1) / csz;
    k_noalloc_prepare<<<NOALLOC_CL, 1024, 0, st>>>(sc, r, lambda, n_blobs, nk, csz);
    RpyConst32 k{(float)(2.0 * a * a / 3.0), (float)(2.0 * a * a), (float)(4.0 * a * a), (float)(4.0 / (3.0 * a)),
                 (float)(9.0 / (32.0 * a)), (float)(1.0 / (8.0 * a * a))};
    int near_src = GDC_NEAR_SRC_MIN;   // as in a context's list
    while ((long long)ntile * ((n_blobs + near_src - 1) / near_src) > 64LL * sms) near_src *= 2;
    const int near_chunks = (n_blobs + near_src - 1) / near_src;
    k_near_build<<<ntile * near_chunks, 128, 0, st>>>(nullptr, near_chunks, near_src, sc->susp_blob_off, sc->spos,
                                                      (float)(4.0 * a * a), sc->near_cnt, sc->near_idx);
    k_near_sort<<<(n_blobs + 255) / 256, 256, 0, st>>>(n_blobs, sc->near_cnt, sc->near_idx);
    k_rpy32<1, 6><<<ntile * nk, 128, 0, st>>>(sc->items, nullptr, sc->susp_blob_off, sc->spos, sc->sdup, sc->part,
                                             n_blobs, k, sc->status, first_wait_polls());
    k_noalloc_epilogue<<<(GDC_NOALLOC_EPI * n_blobs + 255) / 256, 256, 0, st>>>(sc, r, lambda, n_blobs, nk,
                                                              1.0 / (8.0 * 3.141592653589793 * eta), a, u);
    e = cudaGetLastError();
    if (e != cudaSuccess)
        return noalloc_fail(GDC_ERR_CUDA, std::string("gdc_rpy_apply_noalloc: launch failed: ") + cudaGetErrorString(e));
    return GDC_OK;
}
