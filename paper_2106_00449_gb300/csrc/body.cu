// Per-body kernels: the K^T map (Eq. force_torque_balance_compact), step-2 least squares (Eq. sol_unconst with the
// closed-form K^T K of Sec. 5), the block-diagonal preconditioner P of Sec. 2.2, and
// the per-template FP64 setup of P (Cholesky of the template's RPY block).
//
// Rigidity makes every intra-body quantity a rotation of a body-frame template
// quantity: with R-hat = diag(R, ..., R) on blobs and R-tilde = diag(R, R) on
// [force; torque], K_p = R-hat K_t R-tilde^T and M_pp = R-hat M_t R-hat^T (RPY is
// rotation covariant and intra-body distances are fixed).  So M_t^-1, G_t = M_t^-1 K_t,
// N_t = (K_t^T M_t^-1 K_t)^+ and (K_t^T K_t)^+ are computed once per template in the
// body frame and applied to rotated vectors.  "^+" is the pseudo-inverse: a collinear
// body (rod) has no axial spin (its K has that null vector), which is then set to 0.
#include <algorithm>

#include "common.cuh"
#include "wall_pair.cuh"

namespace gdc {

// ---- K^T: [sum lambda_i; sum (r_i - Y_p) x lambda_i] per body, eight lanes per body ----
//
// Bound by the FP64 pipe, which charges a warp instruction the same whichever lanes need it:
// a warp per body spends 30 adds on the six shuffle sums of each body, eight lanes per body 18
// on those of four (2,987 bodies: 18.5 us a warp each).

constexpr int KT_LANES = 8;

// the sum of each of six values over the KT_LANES lanes of a body, on every lane
__device__ __forceinline__ void body_sum6(double* g) {
#pragma unroll
    for (int o = 1; o < KT_LANES; o <<= 1)
#pragma unroll
        for (int k = 0; k < 6; ++k) g[k] += __shfl_xor_sync(0xffffffffu, g[k], o);
}

__device__ __forceinline__ void kt_add(double* g, double d0, double d1, double d2, double l0, double l1, double l2) {
    g[0] += l0;
    g[1] += l1;
    g[2] += l2;
    g[3] += d1 * l2 - d2 * l1;
    g[4] += d2 * l0 - d0 * l2;
    g[5] += d0 * l1 - d1 * l0;
}

__global__ void __launch_bounds__(128) k_body_KT(int NB, const long long* __restrict__ body_blob_off,
                                                 const int* __restrict__ blob_gm, const int* __restrict__ body_gm,
                                                 const double* __restrict__ x, int x_gm, double* __restrict__ y, int y_gm,
                                                 double scale, const double* __restrict__ r, const double* __restrict__ Yc) {
    const int sub = threadIdx.x % KT_LANES;
    const int p0 = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) / KT_LANES);
    const int p = min(p0, NB - 1);   // whole warps reach the shuffles
    const double Y0 = Yc[3 * p], Y1 = Yc[3 * p + 1], Y2 = Yc[3 * p + 2];
    double g[6] = {0, 0, 0, 0, 0, 0};
    for (long long i = body_blob_off[p] + sub; i < body_blob_off[p + 1]; i += KT_LANES) {
        const long long o = x_gm ? (long long)blob_gm[i] : 3 * i;
        kt_add(g, r[3 * i] - Y0, r[3 * i + 1] - Y1, r[3 * i + 2] - Y2, x[o], x[o + 1], x[o + 2]);
    }
    body_sum6(g);
    if (p0 < NB && sub < 6) {
        const double v = sub == 0 ? g[0] : sub == 1 ? g[1] : sub == 2 ? g[2] : sub == 3 ? g[3] : sub == 4 ? g[4] : g[5];
        y[(y_gm ? (long long)body_gm[p] : 6LL * p) + sub] = scale * v;
    }
}

void launch_body_KT(gdc_ctx* c, const double* x, int x_gm, double* y, int y_gm, double scale) {
    ++c->n_launch, k_body_KT<<<ceil_div((long long)KT_LANES * c->NB, 128), 128, 0, c->stream>>>(
        c->NB, c->body_blob_off, c->blob_gm, c->body_gm, x, x_gm, y, y_gm, scale, c->r, c->Yc);
}

// ---- step 2: calV_p = (K^T K)_p^+ K_p^T vbrev ----------------------------------------

__device__ inline void rotT(const double* R, const double* v, double* o) {  // o = R^T v
    o[0] = R[0] * v[0] + R[3] * v[1] + R[6] * v[2];
    o[1] = R[1] * v[0] + R[4] * v[1] + R[7] * v[2];
    o[2] = R[2] * v[0] + R[5] * v[1] + R[8] * v[2];
}

__device__ inline void rot(const double* R, const double* v, double* o) {  // o = R v
    o[0] = R[0] * v[0] + R[1] * v[1] + R[2] * v[2];
    o[1] = R[3] * v[0] + R[4] * v[1] + R[5] * v[2];
    o[2] = R[6] * v[0] + R[7] * v[1] + R[8] * v[2];
}

// eight lanes per body; lane a < 6 forms row a of the 6 x 6 product
__global__ void __launch_bounds__(128) k_lsq(int NB, const long long* __restrict__ body_blob_off,
                                             const int* __restrict__ body_tmpl, const double* __restrict__ KtKp,
                                             const double* __restrict__ vb, const double* __restrict__ r,
                                             const double* __restrict__ Yc, const double* __restrict__ Rb,
                                             double* __restrict__ calV) {
    const int sub = threadIdx.x % KT_LANES, lane = threadIdx.x & 31;
    const int p0 = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) / KT_LANES);
    const int p = min(p0, NB - 1);
    const double Y0 = Yc[3 * p], Y1 = Yc[3 * p + 1], Y2 = Yc[3 * p + 2];
    double g[6] = {0, 0, 0, 0, 0, 0};
    for (long long i = body_blob_off[p] + sub; i < body_blob_off[p + 1]; i += KT_LANES)
        kt_add(g, r[3 * i] - Y0, r[3 * i + 1] - Y1, r[3 * i + 2] - Y2, vb[3 * i], vb[3 * i + 1], vb[3 * i + 2]);
    body_sum6(g);
    const double* R = Rb + 9 * p;
    double gb[6];
    rotT(R, g, gb);
    rotT(R, g + 3, gb + 3);
    const int a = min(sub, 5);
    const double* A = KtKp + 36 * body_tmpl[p] + 6 * a;
    double v = 0.0;
#pragma unroll
    for (int b = 0; b < 6; ++b) v = fma(A[b], gb[b], v);
    // rotate back: component a of R v (translation, rotation)
    const int first = (lane & ~(KT_LANES - 1)) + (a >= 3 ? 3 : 0);
    double o = 0.0;
#pragma unroll
    for (int b = 0; b < 3; ++b) o = fma(R[3 * (a % 3) + b], __shfl_sync(0xffffffffu, v, first + b), o);
    if (p0 < NB && sub < 6) calV[6 * p + sub] = o;
}

void launch_lsq(gdc_ctx* c, const double* vbrev, double* calV) {
    ++c->n_launch, k_lsq<<<ceil_div((long long)KT_LANES * c->NB, 128), 128, 0, c->stream>>>(
        c->NB, c->body_blob_off, c->body_tmpl, c->tmpl_KtKp, vbrev, c->r, c->Yc, c->Rb, calV);
}

// ---- per-body products, bodies of one template grouped per block -------------------------
//
// The block preconditioner, the same-body block of a product and the factor products of the
// preconditioned Lanczos operator all apply a (3n)^2 matrix of the body's template to rotated
// blob vectors.  A block takes up to GB bodies of one template (tb_items): each matrix element
// is read once for all of them.  Rows are dealt to threads and, when a block has more threads
// than rows, the columns of a row to KS threads whose partial sums meet in shared memory (a
// 30-row product walks 4 columns per thread instead of 30).
//
// Bound by the L2 latency of the matrix elements (eight in flight per thread) and, in the rest,
// by the FP64 pipe: its cost is per warp instruction, so the rotations, the sums K^T and the
// 6 x 6 products run flat over (body, blob) or (body, row) items of the whole block and leave no
// lanes idle.  One 128-thread block per body spent 200 FP64 warp instructions per body in the
// preconditioner (68% of the pipe), mostly on one lane's 6 x 6 product and 30 shuffle adds.
//
// GB, the bodies per block, in FP32: 8 from 40 bodies per SM on, 4 from 512 bodies on, 1 below and,
// for all templates of a context, with one above 85 blobs (a thread per row then ends).  us per launch with GB = 1 / 4 / 8 (preconditioner; same-body
// block with K^T; factor products): 777 bodies 16.6 / 14.2 / 18.5; 15.1 / 12.3 / 16.3; 23.8 /
// 27.5 / 24.8.  2,520 bodies 39.9 / 21.1 / 22.8; 40.2 / 18.1 / 20.7; 50.2 / 40.0 / 32.6.  12,082
// bodies 140 / 70 / 60; 129 / 57 / 66; 154 / 95 / 77.  One block per body took 40.0, 36.0
// (two launches) and 34.8 at 2,520 bodies.  (With GB = 4 in two chains a row; in four, see gp_parts,
// the first two take 15.7 and 12.7 at 777 bodies, 23.1 and 19.3 at 2,520.)  In FP64 one body per block is as fast or faster up
// to 3,000 bodies (same-body block 57.6 / 54.1 / 65.1, factor 34.9 / 36.6 / 46.3) and always used.
// Against the earlier kernels, which grouped whatever the template and FP64 products too from 4,864
// bodies on, neither rule loses (us per call, before and now): the FP64 preconditioner of 6,000
// bodies 280 / 147, of 36,121 723 / 510; with a 162-blob body among 12,081 of 12 blobs a solve 196,600
// / 164,900 and a Brownian velocity 204,800 / 199,300, among 35,839 in 512 suspensions 9,950 / 8,370
// and 8,430 / 5,960.

constexpr int GP_TH = 256;

// The columns k0..k1 of row i that a product takes: all, or a triangle's.
enum { GP_FULL = 0, GP_FROM_DIAG = 1, GP_TO_DIAG = 2 };

// Threads per row of an n3-row product and the doubles of shared memory its partial sums take.
__host__ __device__ inline int gp_split(int n3) {
    const int R = (n3 + 31) & ~31;
    return R >= GP_TH ? 1 : GP_TH / R;
}

// FP32 rows of more than 64 columns of a body's own block or its inverse keep at least four
// chains, joined in FP64, where up to a few thousand bodies share the work (GB < 8): two of them,
// or two joined in FP32, lose up to a third of the accuracy (relative error of an FP32 product of
// single bodies, two chains and four: 340 blobs 4.2e-7 and 3.2e-7, 85 blobs 2.4e-7 and 1.9e-7).
// Shorter rows have more chains anyway, each shorter; GB = 8 stays with two, half the FP64
// additions, and so do the factors, whose sums enter beside the pair kernel's.
// gp_halves: the parts that a thread takes of a whole row in turn, each summed into FP64;
// gp_parts: the chains that a thread of a split row leaves to be joined.
template <int GB, int SHAPE, typename T>
__host__ __device__ inline int gp_halves(int KS) { return SHAPE == GP_FULL && GB < 8 && sizeof(T) == 4 && KS == 1 ? 2 : 1; }
template <int GB, int SHAPE, typename T>
__host__ __device__ inline int gp_parts(int KS) { return SHAPE == GP_FULL && GB < 8 && sizeof(T) == 4 && KS == 2 ? 2 : 1; }

// out[u n3 + i] = sum_k M[k n3 + i] in[k GB + u] over the columns SHAPE leaves row i, u < GB (in
// padded with zeros): two chains of type T over each thread's columns, the threads' sums added in
// FP64.  part: gp_parts KS GB n3 values of T (unused for KS = 1).  Ends with a barrier.
template <int GB, int SHAPE, typename T>
__device__ __forceinline__ void group_product(const T* __restrict__ M, int n3, const T* in_, T* part, double* out) {
    // 16-byte aligned by the callers' layouts for GB >= 4, so a column's entries are vector loads
    const T* in = GB >= 4 ? (const T*)__builtin_assume_aligned(in_, 16) : in_;
    const int R = (n3 + 31) & ~31, KS = gp_split(n3);
    const int halves = gp_halves<GB, SHAPE, T>(KS), NP = gp_parts<GB, SHAPE, T>(KS);
    const int ks = KS == 1 ? 0 : (int)threadIdx.x / R;
    const int chunk = (n3 + KS * halves - 1) / (KS * halves);
    for (int row = KS == 1 ? (int)threadIdx.x : (int)threadIdx.x % R; row < n3 && ks < KS; row += GP_TH) {
        for (int h = 0; h < halves; ++h) {
            int k0 = (ks + h) * chunk, k1 = min(n3, k0 + chunk);
            if (SHAPE == GP_FROM_DIAG) k0 = max(k0, row);
            if (SHAPE == GP_TO_DIAG) k1 = min(k1, row + 1);
            T a[GB], b[GB];
#pragma unroll
            for (int u = 0; u < GB; ++u) a[u] = b[u] = T(0);
            int k = k0;
            const T* Mr = M + row;
            for (; k + 7 < k1; k += 8) {   // eight elements in flight: the matrix comes from L2
                T f[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) f[q] = Mr[(long long)(k + q) * n3];
#pragma unroll
                for (int q = 0; q < 8; q += 2)
#pragma unroll
                    for (int u = 0; u < GB; ++u) {
                        a[u] = fma(f[q], in[(k + q) * GB + u], a[u]);
                        b[u] = fma(f[q + 1], in[(k + q + 1) * GB + u], b[u]);
                    }
            }
#pragma unroll 2
            for (; k + 1 < k1; k += 2) {
                const T f = Mr[(long long)k * n3], g = Mr[(long long)(k + 1) * n3];
#pragma unroll
                for (int u = 0; u < GB; ++u) {
                    a[u] = fma(f, in[k * GB + u], a[u]);
                    b[u] = fma(g, in[(k + 1) * GB + u], b[u]);
                }
            }
            if (k < k1) {
                const T f = M[(long long)k * n3 + row];
#pragma unroll
                for (int u = 0; u < GB; ++u) a[u] = fma(f, in[k * GB + u], a[u]);
            }
#pragma unroll
            for (int u = 0; u < GB; ++u) {
                if (KS == 1) {
                    const double s = (double)a[u] + (double)b[u];
                    out[u * n3 + row] = h == 0 ? s : out[u * n3 + row] + s;
                } else if (NP == 2) {
                    part[(2 * ks * GB + u) * n3 + row] = a[u];
                    part[((2 * ks + 1) * GB + u) * n3 + row] = b[u];
                } else {
                    part[(ks * GB + u) * n3 + row] = a[u] + b[u];
                }
            }
        }
    }
    __syncthreads();
    if (KS > 1) {
        for (int e = threadIdx.x; e < GB * n3; e += GP_TH) {
            double s = (double)part[e];
            for (int q = 1; q < NP * KS; ++q) s += (double)part[q * GB * n3 + e];
            out[e] = s;
        }
        __syncthreads();
    }
}

// Bytes of group_product's arrays: in (T), part (T), out (double)
template <int GB, int SHAPE, typename T>
static size_t gp_bytes(int n3) {
    const int KS = gp_split(n3);
    return (size_t)GB * n3 * (sizeof(double) + sizeof(T) * (1 + (KS > 1 ? KS * gp_parts<GB, SHAPE, T>(KS) : 0)));
}

// K^T of the group's body-frame vectors v (double, [u][n3]) with blob offsets b: four threads per
// (body, component), added by shuffles; thread with sub = 0 hands the sum to store(u, c, value).
template <typename F>
__device__ __forceinline__ void group_KT(int cnt, int n, const double* b, const double* v, F store) {
    const int n3 = 3 * n, total = cnt * 24;
    for (int it = threadIdx.x; it < ((total + 31) & ~31); it += GP_TH) {
        const bool in = it < total;
        const int q = in ? it >> 2 : 0, sub = it & 3, u = q / 6, c = q - 6 * u;
        const double* a = v + u * n3;
        double s0 = 0.0, s1 = 0.0;
        if (in) {
            if (c < 3) {
                for (int i = sub; i < n; i += 4) s0 += a[3 * i + c];
            } else {
                const int w = (c - 2) % 3, z = (c - 1) % 3;   // the axes after c - 3, cyclic
                for (int i = sub; i < n; i += 4) {
                    s0 = fma(b[3 * i + w], a[3 * i + z], s0);
                    s1 = fma(b[3 * i + z], a[3 * i + w], s1);
                }
            }
        }
        double s = s0 - s1;
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (in && sub == 0) store(u, c, s);
    }
}

struct GroupArgs {   // tables the grouped kernels share
    const int4* items;     // (template, first entry of bodies, count)
    const int* bodies;
    const long long* body_blob_off;
    const int *body_tmpl, *tmpl_n, *tmpl_off;
    const long long* mat_off;   // of a template's matrices; above a wall of each body's
    const int *blob_gm, *body_gm;
    const double* Rb;
    const double* tmpl_xyz;
};

// (template or, above a wall, body; first entry of bodies; count) of the block: GB = 1 takes the
// body of the block's index
template <bool LAB, int GB>
__device__ __forceinline__ int4 group_item(const GroupArgs& ga) {
    if (GB > 1) return ga.items[blockIdx.x];
    return make_int4(LAB ? (int)blockIdx.x : ga.body_tmpl[blockIdx.x], 0, 1, 0);
}

// the lambda part of blob i in the FP32 pair kernels' source layout (its positions are written
// when a configuration is loaded)
__device__ __forceinline__ void pack_lambda32(float4* sdup, long long i, const double* w) {
    const float lx = (float)w[0], ly = (float)w[1], lz = (float)w[2];
    reinterpret_cast<float2*>(sdup + 3 * i + 1)[1] = make_float2(lx, lx);
    sdup[3 * i + 2] = make_float4(ly, ly, lz, lz);
}

// ---- block-diagonal preconditioner ----------------------------------------------------
//
// Solves [M_pp -K_p; -K_p^T 0][lam; V] = [r_lam; r_V] exactly:
//   a = M^-1 r_lam,  V = -N (r_V + K^T a),  lam = a + G V   (N = (K^T M^-1 K)^+, G = M^-1 K)
// in the body frame of the template.
//
// LAB = false: the template's FP64 blocks in the body frame, applied to rotated vectors.
// LAB = true (blobs above a wall): each body's own blocks in the lab frame (set up by
// k_wall_blocks at every configuration), blob offsets d_i = r_i - Y_p, no rotation, one body
// per block.
// T = float: the M^-1 product in FP32 (the template block rounded to FP32, partial sums added
// in FP64; the rest of the block solve stays FP64), for the inner cycles of the FP32-mixed
// mobility solve, whose operator already carries FP32 rounding: the preconditioner only has to
// be a fixed approximation.
// sdup: lambda also goes there in the FP32 pair kernels' layout (the product that follows).
template <bool LAB, int GB, typename T>
__global__ void __launch_bounds__(GP_TH) k_precond(GroupArgs ga, const T* __restrict__ Minv, const double* __restrict__ Gt,
                                                   const double* __restrict__ Nt, const double* __restrict__ rin,
                                                   double* __restrict__ zout, const double* __restrict__ r,
                                                   const double* __restrict__ Yc, float4* __restrict__ sdup) {
    extern __shared__ __align__(16) double sh[];
    const int4 it = group_item<LAB, GB>(ga);
    const int t = it.x, cnt = it.z;
    auto body = [&](int u) { return GB == 1 ? (int)blockIdx.x : ga.bodies[it.y + u]; };
    const int n = LAB ? (int)(ga.body_blob_off[t + 1] - ga.body_blob_off[t]) : ga.tmpl_n[t], n3 = 3 * n;
    double* av = sh;                       // [GB][n3]
    double* misc = av + GB * n3;           // [GB][24]: r_V, K^T a, V
    double* bl = misc + GB * 24;           // LAB: blob offsets (n3)
    T* in = reinterpret_cast<T*>(bl + (LAB ? n3 : 0));   // [n3][GB]
    T* part = in + GB * n3;
    for (int e = threadIdx.x; e < GB * n; e += GP_TH) {
        const int u = e / n, b = e - u * n;
        double w[3] = {0.0, 0.0, 0.0};
        if (u < cnt) {
            const int p = body(u);
            const long long i = ga.body_blob_off[p] + b, o = ga.blob_gm[i];
            const double v[3] = {rin[o], rin[o + 1], rin[o + 2]};
            if (LAB) {
                for (int a = 0; a < 3; ++a) {
                    w[a] = v[a];
                    bl[3 * b + a] = r[3 * i + a] - Yc[3 * p + a];
                }
            } else {
                rotT(ga.Rb + 9 * p, v, w);
            }
        }
        for (int a = 0; a < 3; ++a) in[(3 * b + a) * GB + u] = (T)w[a];
    }
    for (int e = threadIdx.x; e < 2 * cnt; e += GP_TH) {
        const int u = e >> 1, h = e & 1, p = body(u);
        const long long o = ga.body_gm[p] + 3 * h;
        const double v[3] = {rin[o], rin[o + 1], rin[o + 2]};
        double w[3] = {v[0], v[1], v[2]};
        if (!LAB) rotT(ga.Rb + 9 * p, v, w);
        for (int a = 0; a < 3; ++a) misc[24 * u + 3 * h + a] = w[a];
    }
    __syncthreads();
    group_product<GB, GP_FULL, T>(Minv + ga.mat_off[t], n3, in, part, av);   // symmetric: coalesced over rows
    const double* b = LAB ? bl : ga.tmpl_xyz + 3LL * ga.tmpl_off[t];
    group_KT(cnt, n, b, av, [&](int u, int c, double s) { misc[24 * u + 8 + c] = s; });
    __syncthreads();
    for (int e = threadIdx.x; e < 6 * cnt; e += GP_TH) {
        const int u = e / 6, a = e - 6 * u;
        const double* N = Nt + 36LL * t + 6 * a;
        const double* m = misc + 24 * u;
        double acc = 0.0;
#pragma unroll
        for (int k = 0; k < 6; ++k) acc = fma(N[k], m[k] + m[8 + k], acc);
        misc[24 * u + 16 + a] = -acc;
    }
    __syncthreads();
    // G is 3n x 6, blocks back to back (templates, or LAB bodies in blob order)
    const double* Gp = Gt + 18LL * (LAB ? ga.body_blob_off[t] : (long long)ga.tmpl_off[t]);
    for (int e = threadIdx.x; e < cnt * n; e += GP_TH) {
        const int u = e / n, q = e - u * n, p = body(u);
        double lb[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int row = 3 * q + a;
            double acc = av[u * n3 + row];
#pragma unroll
            for (int k = 0; k < 6; ++k) acc = fma(Gp[6 * row + k], misc[24 * u + 16 + k], acc);
            lb[a] = acc;
        }
        double w[3] = {lb[0], lb[1], lb[2]};
        if (!LAB) rot(ga.Rb + 9 * p, lb, w);
        const long long i = ga.body_blob_off[p] + q, o = ga.blob_gm[i];
        zout[o] = w[0];
        zout[o + 1] = w[1];
        zout[o + 2] = w[2];
        if (sdup) pack_lambda32(sdup, i, w);
    }
    for (int e = threadIdx.x; e < 2 * cnt; e += GP_TH) {
        const int u = e >> 1, h = e & 1, p = body(u);
        const double* v = misc + 24 * u + 16 + 3 * h;
        double w[3] = {v[0], v[1], v[2]};
        if (!LAB) rot(ga.Rb + 9 * p, v, w);
        const long long o = ga.body_gm[p] + 3 * h;
        for (int a = 0; a < 3; ++a) zout[o + a] = w[a];
    }
}

// ---- same-body block of the RPY product ------------------------------------------------
//
// y_p += M_pp lambda_p with M_pp = R M_t R^T (M_t: the template's RPY block, built at init in
// FP64).  T = double: the double-float residual product, whose pair kernel leaves same-body
// pairs out; T = float: the FP32 products, whose other terms carry FP32 rounding (M_t and the
// rotated lambda rounded to FP32, the rotations in FP64).  x and y use the saddle layout (gm =
// 1) or 3 doubles per blob (gm = 0); in the saddle layout the body rows -K^T lambda of the
// operator are formed here as well, from the rotated lambda and the template's offsets (one
// launch instead of two, lambda read once).  GB = 4 is held to 48 registers, five blocks per SM:
// with 63 the 816 blocks of 48 suspensions took a wave and a third (their solve 5.44 ms, 5.33 so).
template <int GB, typename T>
__global__ void __launch_bounds__(GP_TH, GB == 4 ? 5 : 0) k_intra_body(GroupArgs ga, const T* __restrict__ Mt, const double* __restrict__ x,
                                                      double* __restrict__ y, int gm) {
    extern __shared__ __align__(16) double sh[];
    const int4 it = group_item<false, GB>(ga);
    const int t = it.x, cnt = it.z, n = ga.tmpl_n[t], n3 = 3 * n;
    auto body = [&](int u) { return GB == 1 ? (int)blockIdx.x : ga.bodies[it.y + u]; };
    double* av = sh;                 // [GB][n3]
    double* rho = av + GB * n3;      // [GB][n3]: the rotated lambda
    double* kt = rho + GB * n3;      // [GB][6]
    T* in = reinterpret_cast<T*>(kt + GB * 6);
    T* part = in + GB * n3;
    for (int e = threadIdx.x; e < GB * n; e += GP_TH) {
        const int u = e / n, b = e - u * n;
        double w[3] = {0.0, 0.0, 0.0};
        if (u < cnt) {
            const int p = body(u);
            const long long i = ga.body_blob_off[p] + b, o = gm ? (long long)ga.blob_gm[i] : 3 * i;
            const double v[3] = {x[o], x[o + 1], x[o + 2]};
            rotT(ga.Rb + 9 * p, v, w);
        }
        for (int a = 0; a < 3; ++a) {
            rho[u * n3 + 3 * b + a] = w[a];
            in[(3 * b + a) * GB + u] = (T)w[a];
        }
    }
    __syncthreads();
    group_product<GB, GP_FULL, T>(Mt + ga.mat_off[t], n3, in, part, av);
    for (int e = threadIdx.x; e < cnt * n; e += GP_TH) {
        const int u = e / n, b = e - u * n, p = body(u);
        double w[3];
        rot(ga.Rb + 9 * p, av + u * n3 + 3 * b, w);
        const long long i = ga.body_blob_off[p] + b, o = gm ? (long long)ga.blob_gm[i] : 3 * i;
        y[o] += w[0];
        y[o + 1] += w[1];
        y[o + 2] += w[2];
    }
    if (!gm) return;
    group_KT(cnt, n, ga.tmpl_xyz + 3LL * ga.tmpl_off[t], rho, [&](int u, int c, double s) { kt[6 * u + c] = s; });
    __syncthreads();
    for (int e = threadIdx.x; e < 2 * cnt; e += GP_TH) {
        const int u = e >> 1, h = e & 1, p = body(u);
        double w[3];
        rot(ga.Rb + 9 * p, kt + 6 * u + 3 * h, w);
        const long long o = ga.body_gm[p] + 3 * h;
        for (int a = 0; a < 3; ++a) y[o + a] = -w[a];
    }
}

__global__ void k_round_f32(long long n, const double* __restrict__ a, float* __restrict__ b) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

// ---- factors of the body blocks: block-preconditioned Lanczos (Sec. 4.1, Chow & Saad) ----
//
// With L_t the Cholesky factor of the template block (M_t = L_t L_t^T), L_p = R-hat_p L_t
// factors body p's block of M (M_pp = R-hat_p M_t R-hat_p^T), and the Lanczos operator of
// Chow & Saad is A = L^-1 M L^-T with L = diag_p(L_p):
//   TRI_LINV_T: out_p = L_p^-T x_p = R-hat_p (L_t^-T x_p)
//   TRI_LINV:   out_p = L_p^-1 x_p (+ add_p) = L_t^-1 (R-hat_p^T x_p) (+ add_p)
//   TRI_L:      out_p = L_p x_p = R-hat_p (L_t x_p)
// F is the template's factor stored so that out_i = sum_k F[k n3 + i] in_k (coalesced over
// the rows i); the triangular structure limits k to [i, n3) (TRI_LINV_T) or [0, i].
// x, add and out hold 3 doubles per blob.
// LAB (blobs above a wall): body p's own factor of its lab-frame block (L_p from
// k_wall_blocks, at blk_off[p]), no rotation, one body per block.  T: the type of the factor
// and of the sums (float for the FP32 products of the FP32-mixed Lanczos, whose other terms
// carry FP32 rounding; the rotations and the added vector stay FP64).  sdup as in k_precond.
template <int MODE, bool LAB, int GB, typename T>
__global__ void __launch_bounds__(GP_TH) k_body_tri(GroupArgs ga, const T* __restrict__ F, const double* __restrict__ x,
                                                    const double* __restrict__ add, double* __restrict__ out,
                                                    float4* __restrict__ sdup) {
    extern __shared__ __align__(16) double sh[];
    const int4 it = group_item<LAB, GB>(ga);
    const int t = it.x, cnt = it.z;
    auto body = [&](int u) { return GB == 1 ? (int)blockIdx.x : ga.bodies[it.y + u]; };
    const int n = LAB ? (int)(ga.body_blob_off[t + 1] - ga.body_blob_off[t]) : ga.tmpl_n[t], n3 = 3 * n;
    double* res = sh;                                 // [GB][n3]
    T* in = reinterpret_cast<T*>(res + GB * n3);      // [n3][GB]
    T* part = in + GB * n3;
    for (int e = threadIdx.x; e < GB * n; e += GP_TH) {
        const int u = e / n, b = e - u * n;
        double w[3] = {0.0, 0.0, 0.0};
        if (u < cnt) {
            const int p = body(u);
            const long long o = 3 * (ga.body_blob_off[p] + b);
            const double v[3] = {x[o], x[o + 1], x[o + 2]};
            if (MODE == TRI_LINV && !LAB) {
                rotT(ga.Rb + 9 * p, v, w);
            } else {
                for (int a = 0; a < 3; ++a) w[a] = v[a];
            }
        }
        for (int a = 0; a < 3; ++a) in[(3 * b + a) * GB + u] = (T)w[a];
    }
    __syncthreads();
    group_product<GB, MODE == TRI_LINV_T ? GP_FROM_DIAG : GP_TO_DIAG, T>(F + ga.mat_off[t], n3, in, part, res);
    for (int e = threadIdx.x; e < cnt * n; e += GP_TH) {
        const int u = e / n, b = e - u * n, p = body(u);
        const double* v = res + u * n3 + 3 * b;
        double w[3] = {v[0], v[1], v[2]};
        if (MODE != TRI_LINV && !LAB) rot(ga.Rb + 9 * p, v, w);
        const long long i = ga.body_blob_off[p] + b, o = 3 * i;
        if (add)
            for (int a = 0; a < 3; ++a) w[a] += add[o + a];
        for (int a = 0; a < 3; ++a) out[o + a] = w[a];
        if (sdup) pack_lambda32(sdup, i, w);
    }
}

// ---- launches of the grouped kernels ---------------------------------------------------

static GroupArgs group_args(const gdc_ctx* c) {
    return GroupArgs{c->tb_items,  c->tb_bodies, c->body_blob_off, c->body_tmpl, c->tmpl_n, c->tmpl_off,
                     c->p.wall ? c->blk_off : c->minv_off, c->blob_gm, c->body_gm, c->Rb, c->tmpl_xyz};
}

// Shared memory of a block: the largest over the templates.  At most 41 KB (eight bodies of 85 blobs),
// so no launch needs the attribute that 48 KB and more take.
template <int GB, int SHAPE, typename T>
static size_t group_smem(const gdc_ctx* c, int more_per_row, int more) {
    size_t s = 0;
    for (int n : c->h_tmpl_n) s = std::max(s, gp_bytes<GB, SHAPE, T>(3 * n) + (size_t)(more_per_row * 3 * n + more) * sizeof(double));
    return s;
}

template <bool LAB, int GB, typename T>
static void precond_launch(gdc_ctx* c, const T* Minv, const double* r, double* z, float4* sdup) {
    const size_t smem = group_smem<GB, GP_FULL, T>(c, LAB ? 1 : 0, 24 * GB);
    ++c->n_launch, k_precond<LAB, GB, T><<<GB == 1 ? c->NB : c->tb_n_items, GP_TH, smem, c->stream>>>(
        group_args(c), Minv, LAB ? c->blk_G : c->tmpl_G, LAB ? c->blk_N : c->tmpl_N, r, z, c->r, c->Yc, sdup);
}

void launch_precond(gdc_ctx* c, const double* r, double* z, bool fp32, bool pack) {
    float4* sdup = pack ? c->sdup : nullptr;
    if (c->p.wall)
        precond_launch<true, 1, double>(c, c->blk_Minv, r, z, sdup);
    else if (fp32 && c->tb_group == 8)
        precond_launch<false, 8, float>(c, c->tmpl_Minv32, r, z, sdup);
    else if (fp32 && c->tb_group == 4)
        precond_launch<false, 4, float>(c, c->tmpl_Minv32, r, z, sdup);
    else if (fp32)
        precond_launch<false, 1, float>(c, c->tmpl_Minv32, r, z, sdup);
    else
        precond_launch<false, 1, double>(c, c->tmpl_Minv, r, z, sdup);
}

template <int GB, typename T>
static void intra_launch(gdc_ctx* c, const T* M, const double* x, double* y, int gm) {
    const size_t smem = group_smem<GB, GP_FULL, T>(c, GB, 6 * GB);
    GroupArgs ga = group_args(c);
    ga.mat_off = c->minv_off;
    ++c->n_launch, k_intra_body<GB, T><<<GB == 1 ? c->NB : c->tb_n_items, GP_TH, smem, c->stream>>>(ga, M, x, y, gm);
}

void launch_intra_body(gdc_ctx* c, const double* x, double* y, int gm, bool fp32) {
    if (!fp32)
        intra_launch<1, double>(c, c->tmpl_M, x, y, gm);
    else if (c->tb_group == 8)
        intra_launch<8, float>(c, c->tmpl_M32, x, y, gm);
    else if (c->tb_group == 4)
        intra_launch<4, float>(c, c->tmpl_M32, x, y, gm);
    else
        intra_launch<1, float>(c, c->tmpl_M32, x, y, gm);
}

template <int MODE, bool LAB, int GB, typename T>
static void tri_launch(gdc_ctx* c, const T* F, const double* x, const double* add, double* out, float4* sdup) {
    const size_t smem = group_smem<GB, GP_TO_DIAG, T>(c, 0, 0);
    ++c->n_launch, k_body_tri<MODE, LAB, GB, T><<<GB == 1 ? c->NB : c->tb_n_items, GP_TH, smem, c->stream>>>(
        group_args(c), F, x, add, out, sdup);
}

template <int MODE>
static void tri_group(gdc_ctx* c, const float* F, const double* x, const double* add, double* out, float4* sdup) {
    if (c->tb_group == 8)
        tri_launch<MODE, false, 8, float>(c, F, x, add, out, sdup);
    else if (c->tb_group == 4)
        tri_launch<MODE, false, 4, float>(c, F, x, add, out, sdup);
    else
        tri_launch<MODE, false, 1, float>(c, F, x, add, out, sdup);
}

void launch_body_tri(gdc_ctx* c, int mode, const double* x, const double* add, double* out, bool fp32, bool pack) {
    float4* sdup = pack ? c->sdup : nullptr;
    const bool lab = c->p.wall != 0;
    if (mode == TRI_LINV_T) {
        if (lab) tri_launch<TRI_LINV_T, true, 1, double>(c, c->blk_X, x, add, out, sdup);
        else if (fp32) tri_group<TRI_LINV_T>(c, c->tmpl_X32, x, add, out, sdup);
        else tri_launch<TRI_LINV_T, false, 1, double>(c, c->tmpl_X, x, add, out, sdup);
    } else if (mode == TRI_LINV) {
        if (lab) tri_launch<TRI_LINV, true, 1, double>(c, c->blk_XT, x, add, out, sdup);
        else if (fp32) tri_group<TRI_LINV>(c, c->tmpl_XT32, x, add, out, sdup);
        else tri_launch<TRI_LINV, false, 1, double>(c, c->tmpl_XT, x, add, out, sdup);
    } else {
        if (lab) tri_launch<TRI_L, true, 1, double>(c, c->blk_LT, x, add, out, sdup);
        else tri_launch<TRI_L, false, 1, double>(c, c->tmpl_LT, x, add, out, sdup);
    }
}

// ---- per-template setup (once, at init) -------------------------------------------------

// Cyclic Jacobi eigendecomposition of a symmetric 6x6 (Golub & Van Loan, Sec. 8.5), then the
// pseudo-inverse with eigenvalues below rel_tol * max set to zero.  Single thread.
__device__ void pinv6(const double* A_in, double* P, double rel_tol) {
    double A[36], V[36];
    for (int k = 0; k < 36; ++k) {
        A[k] = A_in[k];
        V[k] = (k % 7 == 0) ? 1.0 : 0.0;
    }
    for (int sweep = 0; sweep < 60; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int i = 0; i < 6; ++i)
            for (int j = 0; j < 6; ++j) {
                tot += A[6 * i + j] * A[6 * i + j];
                if (i != j) off += A[6 * i + j] * A[6 * i + j];
            }
        if (off <= 1e-30 * tot) break;
        for (int pp = 0; pp < 5; ++pp)
            for (int qq = pp + 1; qq < 6; ++qq) {
                const double apq = A[6 * pp + qq];
                if (apq == 0.0) continue;
                const double tau = (A[6 * qq + qq] - A[6 * pp + pp]) / (2.0 * apq);
                const double tt = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
                const double cs = 1.0 / sqrt(1.0 + tt * tt), sn = tt * cs;
                // A <- J^T A J, J = identity with [c s; -s c] in rows/cols (pp, qq)
                for (int k = 0; k < 6; ++k) {
                    const double akp = A[6 * k + pp], akq = A[6 * k + qq];
                    A[6 * k + pp] = cs * akp - sn * akq;
                    A[6 * k + qq] = sn * akp + cs * akq;
                }
                for (int k = 0; k < 6; ++k) {
                    const double apk = A[6 * pp + k], aqk = A[6 * qq + k];
                    A[6 * pp + k] = cs * apk - sn * aqk;
                    A[6 * qq + k] = sn * apk + cs * aqk;
                }
                for (int k = 0; k < 6; ++k) {
                    const double vkp = V[6 * k + pp], vkq = V[6 * k + qq];
                    V[6 * k + pp] = cs * vkp - sn * vkq;
                    V[6 * k + qq] = sn * vkp + cs * vkq;
                }
            }
    }
    double lmax = 0.0;
    for (int i = 0; i < 6; ++i) lmax = fmax(lmax, fabs(A[7 * i]));
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) {
            double acc = 0.0;
            for (int k = 0; k < 6; ++k) {
                const double lam = A[7 * k];
                if (lam > rel_tol * lmax) acc += V[6 * i + k] * V[6 * j + k] / lam;
            }
            P[6 * i + j] = acc;
        }
}

// One block per template.  work: 2 (3n)^2 doubles of scratch per template at minv_off.
__global__ void k_template_setup(const int* __restrict__ tmpl_n, const int* __restrict__ tmpl_off,
                                 const long long* __restrict__ minv_off, const double* __restrict__ xyz,
                                 double a, double eta, double* __restrict__ Minv, double* __restrict__ Gt,
                                 double* __restrict__ Nt, double* __restrict__ KtKp, double* __restrict__ work,
                                 double* __restrict__ Mt, const double* __restrict__ Mext, int* __restrict__ status,
                                 double* __restrict__ LT, double* __restrict__ Xo, double* __restrict__ XT) {
    const int t = blockIdx.x;
    const int n = tmpl_n[t];
    const int n3 = 3 * n;
    const double* b = xyz + 3LL * tmpl_off[t];
    double* Mi = Minv + minv_off[t];
    double* L = work + 2 * minv_off[t];
    double* X = L + (long long)n3 * n3;
    const double c0 = 1.0 / (8.0 * 3.141592653589793 * eta);
    // 1. the template's mobility block M_t, row-major in L: given (Mext: the FCM block of the
    //    template alone in the periodic cube), or the RPY block (Sec. 4.1)
    for (long long e = threadIdx.x; Mext && e < (long long)n3 * n3; e += blockDim.x) {
        L[e] = Mext[minv_off[t] + e];
        Mt[minv_off[t] + e] = L[e];
    }
    for (long long e = threadIdx.x; !Mext && e < (long long)n3 * n3; e += blockDim.x) {
        const int row = (int)(e / n3), col = (int)(e % n3);
        const int i = row / 3, al = row % 3, j = col / 3, be = col % 3;
        const double d0 = b[3 * j] - b[3 * i], d1 = b[3 * j + 1] - b[3 * i + 1], d2 = b[3 * j + 2] - b[3 * i + 2];
        const double dd[3] = {d0, d1, d2};
        const double r2 = d0 * d0 + d1 * d1 + d2 * d2;
        double A, B;
        if (r2 == 0.0) {
            A = 4.0 / (3.0 * a);
            B = 0.0;
        } else if (r2 < 4.0 * a * a) {
            const double r = sqrt(r2);
            A = 4.0 / (3.0 * a) * (1.0 - 9.0 * r / (32.0 * a));
            B = 1.0 / (8.0 * a * a * r);
        } else {
            const double r = sqrt(r2);
            A = 1.0 / r + 2.0 * a * a / (3.0 * r * r2);
            B = (1.0 - 2.0 * a * a / r2) / (r * r2);
        }
        L[e] = c0 * ((al == be ? A : 0.0) + B * dd[al] * dd[be]);
        Mt[minv_off[t] + e] = L[e];
    }
    __syncthreads();
    // 2. Cholesky M = L L^T (right-looking; lower triangle of L overwritten)
    for (int k = 0; k < n3; ++k) {
        if (threadIdx.x == 0) {
            const double dkk = L[(long long)k * n3 + k];
            if (!(dkk > 0.0)) atomicExch(status, 1);
            L[(long long)k * n3 + k] = sqrt(fmax(dkk, 1e-300));
        }
        __syncthreads();
        const double lkk = L[(long long)k * n3 + k];
        for (int i = k + 1 + threadIdx.x; i < n3; i += blockDim.x) L[(long long)i * n3 + k] /= lkk;
        __syncthreads();
        const int m = n3 - k - 1;
        for (long long e = threadIdx.x; e < (long long)m * m; e += blockDim.x) {
            const int i = k + 1 + (int)(e / m), j = k + 1 + (int)(e % m);
            if (j <= i) L[(long long)i * n3 + j] -= L[(long long)i * n3 + k] * L[(long long)j * n3 + k];
        }
        __syncthreads();
    }
    // 3. X = L^-1 column by column (forward substitution), then M^-1 = X^T X
    for (int col = threadIdx.x; col < n3; col += blockDim.x) {
        for (int i = 0; i < n3; ++i) X[(long long)i * n3 + col] = 0.0;
        for (int i = col; i < n3; ++i) {
            double acc = (i == col) ? 1.0 : 0.0;
            for (int k = col; k < i; ++k) acc -= L[(long long)i * n3 + k] * X[(long long)k * n3 + col];
            X[(long long)i * n3 + col] = acc / L[(long long)i * n3 + i];
        }
    }
    __syncthreads();
    for (long long e = threadIdx.x; e < (long long)n3 * n3; e += blockDim.x) {
        const int i = (int)(e / n3), j = (int)(e % n3);
        double acc = 0.0;
        for (int k = max(i, j); k < n3; ++k) acc += X[(long long)k * n3 + i] * X[(long long)k * n3 + j];
        Mi[e] = acc;
        // the factors for the preconditioned Lanczos operator (L lower; its upper part still
        // holds M and is not part of the factor; X = L^-1 is lower with zeros above)
        const long long o = minv_off[t] + e;
        LT[o] = j >= i ? L[(long long)j * n3 + i] : 0.0;
        Xo[o] = X[e];
        XT[o] = X[(long long)j * n3 + i];
    }
    __syncthreads();
    // 4. G = M^-1 K_t (3n x 6): K_t columns are unit translations and rotations e_b x b_i
    double* G = Gt + 18LL * tmpl_off[t];
    for (long long e = threadIdx.x; e < 6LL * n3; e += blockDim.x) {
        const int row = (int)(e / 6), col = (int)(e % 6);
        double acc = 0.0;
        for (int i = 0; i < n; ++i) {
            double kc[3];
            if (col < 3) {
                kc[0] = col == 0;
                kc[1] = col == 1;
                kc[2] = col == 2;
            } else {
                const int bb = col - 3;  // e_bb x b_i
                const double e3[3] = {(double)(bb == 0), (double)(bb == 1), (double)(bb == 2)};
                kc[0] = e3[1] * b[3 * i + 2] - e3[2] * b[3 * i + 1];
                kc[1] = e3[2] * b[3 * i] - e3[0] * b[3 * i + 2];
                kc[2] = e3[0] * b[3 * i + 1] - e3[1] * b[3 * i];
            }
            for (int al = 0; al < 3; ++al) acc += Mi[(long long)row * n3 + 3 * i + al] * kc[al];
        }
        G[e] = acc;
    }
    __syncthreads();
    // 5. N_t = (K_t^T G)^+ and (K_t^T K_t)^+  (closed form of Sec. 5 for the latter)
    if (threadIdx.x == 0) {
        double A6[36], KK[36];
        for (int k = 0; k < 36; ++k) {
            A6[k] = 0.0;
            KK[k] = 0.0;
        }
        for (int i = 0; i < n; ++i) {
            const double bx = b[3 * i], by = b[3 * i + 1], bz = b[3 * i + 2];
            // K_i = [I, [x b]]: columns e_x, e_y, e_z and e_k x b_i
            double Kc[6][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}, {0, -bz, by}, {bz, 0, -bx}, {-by, bx, 0}};
            for (int u = 0; u < 6; ++u)
                for (int v = 0; v < 6; ++v) {
                    double s1 = 0.0, s2 = 0.0;
                    for (int al = 0; al < 3; ++al) {
                        s1 += Kc[u][al] * G[6LL * (3 * i + al) + v];
                        s2 += Kc[u][al] * Kc[v][al];
                    }
                    A6[6 * u + v] += s1;
                    KK[6 * u + v] += s2;
                }
        }
        for (int u = 0; u < 6; ++u)  // symmetrise rounding
            for (int v = u + 1; v < 6; ++v) {
                const double m = 0.5 * (A6[6 * u + v] + A6[6 * v + u]);
                A6[6 * u + v] = A6[6 * v + u] = m;
            }
        pinv6(A6, Nt + 36 * t, 1e-10);
        pinv6(KK, KtKp + 36 * t, 1e-10);
    }
}

void launch_template_setup(gdc_ctx* c, const double* Mext) {
    ++c->n_launch, k_template_setup<<<c->T, 256, 0, c->stream>>>(c->tmpl_n, c->tmpl_off, c->minv_off, c->tmpl_xyz, c->p.a, c->p.eta,
                                                  c->tmpl_Minv, c->tmpl_G, c->tmpl_N, c->tmpl_KtKp, c->tmpl_work,
                                                  c->tmpl_M, Mext, c->dev_status, c->tmpl_LT, c->tmpl_X, c->tmpl_XT);
    const long long nm = c->h_minv_off[c->T];
    const int gr = (int)std::min<long long>(ceil_div(nm, 256), 1024);
    ++c->n_launch, k_round_f32<<<gr, 256, 0, c->stream>>>(nm, c->tmpl_M, c->tmpl_M32);
    ++c->n_launch, k_round_f32<<<gr, 256, 0, c->stream>>>(nm, c->tmpl_X, c->tmpl_X32);
    ++c->n_launch, k_round_f32<<<gr, 256, 0, c->stream>>>(nm, c->tmpl_Minv, c->tmpl_Minv32);
    ++c->n_launch, k_round_f32<<<gr, 256, 0, c->stream>>>(nm, c->tmpl_XT, c->tmpl_XT32);
}

// ---- per-body blocks above a wall (Sec. 4.1, Sec. 6.2) ---------------------------------
//
// A wall makes a body's block of M depend on its height and orientation, so the blocks of
// the preconditioner (the exact per-body saddle solve) and the factors of the
// preconditioned Lanczos operator are set up for every body at every configuration.  One
// block per body: M_pp = unbounded RPY + wall correction (wall_pair.cuh) from the blob
// offsets d_i = r_i - Y_p and the heights, in FP64; its Cholesky factor L, X = L^-1,
// M_pp^-1 = X^T X, G = M_pp^-1 K_p (K_p from d), N = (K_p^T G)^+, and LT = L^T, X, XT = X^T
// stored for k_body_tri<LAB>.  A blob at or below z = a (overlapping the wall, where the
// correction is not a mobility) sets status[2]; a block that is not positive definite sets
// status[0] = 1.
//
// Bound by the FP64 pipe and by the serial chain of pivots (a suspension above a wall holds
// few bodies, so one block per body leaves the chip mostly idle and the latency of one
// body counts).  The lower triangle lives in shared memory when it fits (bodies of up to 55
// blobs), and factor and inverse come out of one elimination in place, one barrier per
// column: at column k, row i > k is reduced by f_i = a_ik / d_k times the pivot row, whose
// entries left of the diagonal already hold the inverse of the unit factor and right of it
// the remaining matrix (column k by symmetry); entry (i, k) becomes -f_i.  Rows are dealt to
// warps, columns to lanes; the warp that finishes the next pivot forms its reciprocal root
// while the others still update.  M is assembled once per blob pair i >= j (one set of
// coefficients for the nine entries).  The 6 x 6 inverse is a Gauss-Jordan elimination on
// one warp, with the serial Jacobi pseudo-inverse only when the spectrum may reach below the
// pseudo-inverse's cut (a collinear body).  36 bodies of 15 blobs: 138 us, against
// 782 us with the matrices in global memory, an entry-wise assembly, separate Cholesky and
// inverse and a serial Jacobi.

// P = A^-1 for symmetric positive definite A (row-major 6 x 6) on one warp, by Gauss-Jordan
// elimination without pivoting, lane r < 6 holding row r of [A | P].  Returns (on every lane)
// whether all eigenvalues are sure to lie above rel_tol times the largest, so that P is also
// the pseudo-inverse pinv6 forms: |A|_F bounds the largest, 1/|P|_F the smallest.
__device__ bool spd_inverse6(const double* A, double* P, double rel_tol) {
    const int lane = threadIdx.x & 31, row = lane < 6 ? lane : 0;
    double a[6], b[6];
    double na = 0.0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        a[c] = A[6 * row + c];
        b[c] = c == row ? 1.0 : 0.0;
        na = fma(a[c], a[c], na);
    }
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const double piv = __shfl_sync(0xffffffffu, a[k], k);
        ok = ok && piv > 0.0;
        const double inv = 1.0 / piv;
        const double f = a[k] * inv;
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            const double ak = __shfl_sync(0xffffffffu, a[c], k), bk = __shfl_sync(0xffffffffu, b[c], k);
            a[c] = row == k ? ak * inv : fma(-f, ak, a[c]);
            b[c] = row == k ? bk * inv : fma(-f, bk, b[c]);
        }
    }
    double nb = 0.0;
#pragma unroll
    for (int c = 0; c < 6; ++c) nb = fma(b[c], b[c], nb);
    if (lane >= 6) na = nb = 0.0;
    na = warp_sum(na);
    nb = warp_sum(nb);
    if (lane < 6)
#pragma unroll
        for (int c = 0; c < 6; ++c) P[6 * lane + c] = b[c];
    __syncwarp();
    return ok && sqrt(na) * sqrt(nb) * rel_tol < 1.0;   // false for NaN
}

// doubles of shared memory beside the triangle: d, two columns, pivots' reciprocal roots,
// G (6 per row) and the 6 x 6 matrix
__host__ __device__ inline int wall_block_doubles(int n3) { return 10 * n3 + 36 + 2; }

template <bool SMEM>   // the triangle in shared memory (row stride n3 | 1), else in global memory
__global__ void __launch_bounds__(256) k_wall_blocks(const long long* __restrict__ body_blob_off,
                                                     const long long* __restrict__ blk_off, const double* __restrict__ r,
                                                     const double* __restrict__ Yc, double a, double eta, double* work,
                                                     double* __restrict__ Minv, double* __restrict__ Gb,
                                                     double* __restrict__ Nb, double* __restrict__ LT,
                                                     double* __restrict__ Xo, double* __restrict__ XT,
                                                     int* __restrict__ status) {
    extern __shared__ double dsh[];
    const int p = blockIdx.x;
    const long long i0 = body_blob_off[p];
    const int n = (int)(body_blob_off[p + 1] - i0), n3 = 3 * n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const long long mo = blk_off[p];
    double* d = dsh;               // blob offsets
    double* col = d + n3;          // [2][n3]: column k of the remaining matrix, double-buffered
    double* rs = col + 2 * n3;     // 1 / L_kk
    double* G = rs + n3;           // [row][6]
    double* A6 = G + 6 * n3;       // 36
    double* M = SMEM ? A6 + 38 : work + 2 * mo;
    const int ld = SMEM ? (n3 | 1) : n3;
    const double zc = Yc[3 * p + 2];
    for (int e = threadIdx.x; e < n3; e += blockDim.x) d[e] = r[3 * i0 + e] - Yc[3 * p + e % 3];
    for (int b = threadIdx.x; b < n; b += blockDim.x)
        if (!(r[3 * (i0 + b) + 2] > a)) atomicExch(status + 2, 1);
    __syncthreads();
    const double c0 = 1.0 / (8.0 * 3.141592653589793 * eta);
    // 1. M_pp, blob pairs i >= j: RPY block + wall correction
    for (int e = threadIdx.x; e < n * (n + 1) / 2; e += blockDim.x) {
        int i = (int)((sqrtf(8.f * (float)e + 1.f) - 1.f) * 0.5f);   // e = i (i + 1)/2 + j
        while (i * (i + 1) / 2 > e) --i;
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        const int j = e - i * (i + 1) / 2;
        const double dd[3] = {d[3 * j] - d[3 * i], d[3 * j + 1] - d[3 * i + 1], d[3 * j + 2] - d[3 * i + 2]};
        const double r2 = dd[0] * dd[0] + dd[1] * dd[1] + dd[2] * dd[2];
        double A, B;
        if (i == j || r2 == 0.0) {
            A = 4.0 / (3.0 * a);
            B = 0.0;
        } else {
            const double ri = rsqrt_series(r2);
            if (r2 < 4.0 * a * a) {
                A = 4.0 / (3.0 * a) * (1.0 - 9.0 * r2 * ri / (32.0 * a));
                B = 1.0 / (8.0 * a * a) * ri;
            } else {
                const double ri2 = ri * ri, ri3 = ri2 * ri;
                A = ri + 2.0 * a * a / 3.0 * ri3;
                B = ri3 * (1.0 - 2.0 * a * a * ri2);
            }
        }
        const double R[3] = {-dd[0], -dd[1], d[3 * i + 2] + d[3 * j + 2] + 2.0 * zc};
        const WallCoeff<double> w = wall_coeff<double>(R[0], R[1], R[2], d[3 * j + 2] + zc, a * a);
#pragma unroll
        for (int be = 0; be < 3; ++be) {
            const double P2 = be == 2 ? -2.0 : 2.0;   // twice the mirror's sign
#pragma unroll
            for (int al = 0; al < 3; ++al) {
                double v = B * dd[al] * dd[be] + R[al] * R[be] * (w.be0 + P2 * w.be);
                if (al == be) v += A + w.al0 + P2 * w.al;
                if (al == 2) v += P2 * w.ga * R[be];
                if (be == 2) v += P2 * w.ep * R[al];
                if (al == 2 && be == 2) v += P2 * w.ze;
                M[(long long)(3 * i + al) * ld + 3 * j + be] = c0 * v;
            }
        }
    }
    __syncthreads();
    // 2. L and the inverse of its unit form
    for (int i = threadIdx.x; i < n3; i += blockDim.x) col[i] = M[(long long)i * ld];
    if (threadIdx.x == 0) {
        if (!(M[0] > 0.0)) atomicExch(status, 1);
        rs[0] = rsqrt_series(fmax(M[0], 1e-300));
    }
    for (int k = 0; k < n3; ++k) {
        __syncthreads();   // column k, its pivot's root and every row of the previous step
        const double* ck = col + (k & 1) * n3;
        double* cn = col + ((k + 1) & 1) * n3;
        const double rk = rs[k], inv = rk * rk;
        for (int i = threadIdx.x; i < n3; i += blockDim.x) LT[mo + (long long)k * n3 + i] = i >= k ? ck[i] * rk : 0.0;
        const double* Mk = M + (long long)k * ld;
        for (int first = k + 1 + warp; first < n3; first += 32 * nw) {   // up to 32 rows of this warp at a time
            const int mine = first + nw * lane;
            const double fl = mine < n3 ? ck[mine] * inv : 0.0;
            for (int t = 0; t < 32 && first + nw * t < n3; ++t) {
                const int i = first + nw * t;
                const double f = __shfl_sync(0xffffffffu, fl, t);
                double* Mi = M + (long long)i * ld;
                for (int c = lane; c <= i; c += 32) {
                    double v;
                    if (c == k)
                        v = -f;
                    else
                        v = fma(-f, c < k ? Mk[c] : ck[c], Mi[c]);
                    Mi[c] = v;
                    if (c == k + 1) {
                        cn[i] = v;
                        if (i == k + 1) {
                            if (!(v > 0.0)) atomicExch(status, 1);
                            rs[i] = rsqrt_series(fmax(v, 1e-300));
                        }
                    }
                }
            }
        }
    }
    __syncthreads();
    // 3. X = L^-1 (rows scaled by 1 / L_ii), M^-1 = X^T X and the factor layouts
    for (int i = warp; i < n3; i += nw) {
        const double ri = rs[i];
        double* Mi = M + (long long)i * ld;
        for (int c = lane; c < n3; c += 32) {
            const double v = c < i ? Mi[c] * ri : (c == i ? ri : 0.0);
            if (c <= i) Mi[c] = v;
            Xo[mo + (long long)i * n3 + c] = v;
        }
    }
    __syncthreads();
    for (int i = warp; i < n3; i += nw)
        for (int j = lane; j < n3; j += 32) {
            XT[mo + (long long)i * n3 + j] = j >= i ? M[(long long)j * ld + i] : 0.0;
            if (j > i) continue;
            double s0 = 0.0, s1 = 0.0;
            int k = i;
            for (; k + 1 < n3; k += 2) {
                s0 = fma(M[(long long)k * ld + i], M[(long long)k * ld + j], s0);
                s1 = fma(M[(long long)(k + 1) * ld + i], M[(long long)(k + 1) * ld + j], s1);
            }
            if (k < n3) s0 = fma(M[(long long)k * ld + i], M[(long long)k * ld + j], s0);
            Minv[mo + (long long)i * n3 + j] = Minv[mo + (long long)j * n3 + i] = s0 + s1;
        }
    __syncthreads();
    // 4. G = M^-1 K (3n x 6), K columns: unit translations and e_c x d_i (M^-1 is symmetric:
    // read down its columns, coalesced over rows)
    for (int e = threadIdx.x; e < 6 * n3; e += blockDim.x) {
        const int c = e / n3, row = e - c * n3;
        const double* Mc = Minv + mo + row;
        double s0 = 0.0, s1 = 0.0;
        if (c < 3) {
            for (int i = 0; i < n; ++i) s0 += Mc[(long long)(3 * i + c) * n3];
        } else {   // (e_c x d): component c + 2 is d_(c+1), component c + 1 is -d_(c+2) (cyclic)
            const int u = (c + 1) % 3, v = (c + 2) % 3;
            for (int i = 0; i < n; ++i) {
                s0 = fma(Mc[(long long)(3 * i + v) * n3], d[3 * i + u], s0);
                s1 = fma(Mc[(long long)(3 * i + u) * n3], d[3 * i + v], s1);
            }
        }
        G[6 * row + c] = s0 - s1;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 6 * n3; e += blockDim.x) Gb[18LL * i0 + e] = G[e];
    // 5. N = (K^T G)^+ (symmetrised, pseudo-inverse for collinear bodies)
    if (threadIdx.x < 36) {
        const int u = threadIdx.x / 6, v = threadIdx.x % 6;
        double s0 = 0.0, s1 = 0.0;
        if (u < 3) {
            for (int i = 0; i < n; ++i) s0 += G[6 * (3 * i + u) + v];
        } else {
            const int w = (u + 1) % 3, z = (u + 2) % 3;
            for (int i = 0; i < n; ++i) {
                s0 = fma(d[3 * i + w], G[6 * (3 * i + z) + v], s0);
                s1 = fma(d[3 * i + z], G[6 * (3 * i + w) + v], s1);
            }
        }
        A6[threadIdx.x] = s0 - s1;
    }
    __syncthreads();
    double sym = 0.0;
    if (threadIdx.x < 36) sym = 0.5 * (A6[threadIdx.x] + A6[6 * (threadIdx.x % 6) + threadIdx.x / 6]);
    __syncthreads();
    if (threadIdx.x < 36) A6[threadIdx.x] = sym;
    __syncthreads();
    if (warp == 0 && !spd_inverse6(A6, Nb + 36LL * p, 1e-10) && lane == 0) pinv6(A6, Nb + 36LL * p, 1e-10);
}

// the largest body whose triangle fits the 227 KB of shared memory a block may have
static size_t wall_block_smem(int n3, bool tri) {
    return (size_t)(wall_block_doubles(n3) + (tri ? n3 * (n3 | 1) : 0)) * sizeof(double);
}

void launch_wall_blocks(gdc_ctx* c) {
    const int n3 = 3 * c->max_body_blobs, th = n3 <= 64 ? 128 : 256;
    const bool tri = wall_block_smem(n3, true) <= 227 * 1024;
    const size_t smem = wall_block_smem(n3, tri);
    ++c->n_launch;
    if (tri)
        k_wall_blocks<true><<<c->NB, th, smem, c->stream>>>(c->body_blob_off, c->blk_off, c->r, c->Yc, c->p.a, c->p.eta,
                                                            c->blk_work, c->blk_Minv, c->blk_G, c->blk_N, c->blk_LT,
                                                            c->blk_X, c->blk_XT, c->dev_status);
    else
        k_wall_blocks<false><<<c->NB, th, smem, c->stream>>>(c->body_blob_off, c->blk_off, c->r, c->Yc, c->p.a, c->p.eta,
                                                             c->blk_work, c->blk_Minv, c->blk_G, c->blk_N, c->blk_LT,
                                                             c->blk_X, c->blk_XT, c->dev_status);
}

gdc_status wall_init_attributes(gdc_ctx* c) {
    cudaError_t e = cudaFuncSetAttribute(k_wall_blocks<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e == cudaSuccess)   // 10 values per row of the largest template: 82 KB
        e = cudaFuncSetAttribute(k_wall_blocks<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)wall_block_smem(3 * GDC_MAX_TMPL_BLOBS, false));
    return cuda_check(c, e, "wall block attributes");
}

}  // namespace gdc
