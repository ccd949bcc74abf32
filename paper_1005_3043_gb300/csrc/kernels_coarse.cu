// Transfer and coarse-level kernels: block orthonormalisation of the
// prototypes (eq. 4 with the chirality split), restriction r_c = P^dag r,
// prolongation e = P y, the Galerkin coarse operator D_c = P^dag D P and its
// nearest-neighbour application, and the CGNR (CGLS) coarse solve steps.
#include <atomic>
#include <type_traits>

#include "mg_launch.h"
#include "mg_sync.cuh"

namespace wmg {

constexpr int kThreads = 256;

static inline int reduce_grid(size_t n) {
    size_t b = (n + kThreads - 1) / kThreads;
    if (b > (size_t)kMaxReduceBlocks) b = kMaxReduceBlocks;
    return (int)(b > 0 ? b : 1);
}

// ================================================================ block orthonormalisation
// One CTA per (aggregate X, chirality s).  Column i of the panel is prototype i
// restricted to X and to the spins of s (6*Vb complex).  Gram-Schmidt applied
// twice in index order with all projections of a pass at once (classical form:
// c = Q_<i^dag w, w -= Q_<i c), then normalisation: the unique Q factor with a
// positive real R-diagonal, the same as modified Gram-Schmidt twice up to
// rounding.  The column being orthogonalised sits in shared memory; warp w
// forms the projections on columns w, w + 8, ... with warp shuffles, so a
// pass costs three CTA barriers instead of one block reduction per column.
// Bound by the FP64 pipe (16 operations per entry and pair of columns): the six
// calls of a setup on 16^3x32, 4^4 aggregates, 16 to 20 columns: 50 -> 39 ms with the
// updates fused, 32 at the pipe's rate.
constexpr int kOrthoMaxNv = 64;   // nvec <= 25 (parameter check)

__device__ __forceinline__ double block_sum(double v, double* sh) {
    double a[1] = {v};
    block_reduce<1>(a, (double (*)[32])sh);
    __syncthreads();
    if (threadIdx.x == 0) sh[32] = a[0];
    __syncthreads();
    double r = sh[32];
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(256) k_block_ortho(double2* __restrict__ P, const double2* __restrict__ Vin, int nv,
                                                     Geom g, int* status) {
    extern __shared__ double2 wsh[];            // the column being orthogonalised, 6 * Vb entries
    __shared__ double sh[2 * 32 + 2];
    __shared__ double2 cj[kOrthoMaxNv];        // projections of the current pass
    const int X = blockIdx.x >> 1, s = blockIdx.x & 1;
    const int len = 6 * g.Vb, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t vstride = (size_t)g.Vc * 12 * g.Vb;       // one prototype
    double2* panel = P + ((size_t)X * 2 + s) * nv * len;
    for (int i = 0; i < nv; ++i) {
        const double2* vi = Vin + (size_t)i * vstride + ((size_t)X * 12 + 6 * s) * g.Vb;   // k = 6s..6s+5 contiguous
        double n0 = 0;
        for (int e = threadIdx.x; e < len; e += blockDim.x) {
            const double2 v = vi[e];
            wsh[e] = v;
            n0 += v.x * v.x + v.y * v.y;
        }
        n0 = block_sum(n0, sh);   // its barriers also publish wsh
        for (int pass = 0; pass < 2 && i > 0; ++pass) {
            // c_j = <q_j, w>, j < i: one warp per column, lanes over the entries
            for (int j = warp; j < i; j += nw) {
                const double2* qj = panel + (size_t)j * len;
                cx<double> c(0, 0);
                for (int e = lane; e < len; e += 32) cmadc(c, ld<double>(qj + e), ld<double>(wsh + e));
                c.r = warp_sum(c.r);
                c.i = warp_sum(c.i);
                if (lane == 0) cj[j] = make_double2(c.r, c.i);
            }
            __syncthreads();
            // w -= sum_j c_j q_j
            for (int e = threadIdx.x; e < len; e += blockDim.x) {
                cx<double> w = ld<double>(wsh + e);
#pragma unroll 4
                for (int j = 0; j < i; ++j)   // fused: 4 operations of the FP64 pipe a term, w - c q takes 6
                    cmad(w, cx<double>(-cj[j].x, -cj[j].y), ld<double>(panel + (size_t)j * len + e));
                st<double>(wsh + e, w);
            }
            __syncthreads();
        }
        double n = 0;
        for (int e = threadIdx.x; e < len; e += blockDim.x) n += norm2(ld<double>(wsh + e));
        n = sqrt(block_sum(n, sh));
        if (!(n > 1e-12 * sqrt(n0))) {
            if (threadIdx.x == 0) atomicExch(status, 1);
            n = 1.0;
        }
        const double f = 1.0 / n;
        double2* qi = panel + (size_t)i * len;
        for (int e = threadIdx.x; e < len; e += blockDim.x) st<double>(qi + e, f * ld<double>(wsh + e));
        __syncthreads();   // column i visible to the block before it is re-read
    }
}

void block_orthonormalize(double2* P, const double2* V, int nv, const Geom& g, int* d_status, cudaStream_t st) {
    const size_t sm = sizeof(double2) * 6 * g.Vb;   // <= 32.7 KB: blocks hold at most 341 sites (parameter check)
    note_launch();
    k_block_ortho<<<2 * g.Vc, kThreads, sm, st>>>(P, V, nv, g, d_status);
}

// ================================================================ restriction / prolongation
// r_c[X][s*Nv + i] = <P_(X,s,i), r>: one CTA per (X, s); the chirality-s half of
// r on X (6*Vb contiguous) is staged in shared memory, warp w handles i = w, w+8, ...
// Bound by the bytes of P, so a CTA serves NS sources of a batch (lanes) with one
// read of its panel: 12 sources on 16^3x32 read P three times instead of twelve.
template <typename T, int NS>
__global__ void __launch_bounds__(256) k_restrict(v2<T>* __restrict__ rc, const v2<T>* __restrict__ P,
                                                  const v2<T>* __restrict__ r, int nv, Geom g, int cstride, int coff,
                                                  Lanes ln) {
    extern __shared__ unsigned char smem_raw[];
    v2<T>* rs = reinterpret_cast<v2<T>*>(smem_raw);
    const int n0 = blockIdx.y * NS, ns = NS == 1 ? 1 : min(NS, ln.m - n0);
    int X = blockIdx.x >> 1, s = blockIdx.x & 1;
    int len = 6 * g.Vb;
    const v2<T>* rX = r + n0 * ln.a + ((size_t)X * 12 + 6 * s) * g.Vb;
#pragma unroll
    for (int n = 0; n < NS; ++n)
        if (n < ns)
            for (int e = threadIdx.x; e < len; e += blockDim.x) rs[n * len + e] = rX[n * ln.a + e];
    __syncthreads();
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const v2<T>* panel = P + ((size_t)X * 2 + s) * nv * len;
    for (int i = warp; i < nv; i += nw) {
        const v2<T>* pi = panel + (size_t)i * len;
        cx<T> a[NS];
#pragma unroll
        for (int n = 0; n < NS; ++n) a[n] = cx<T>(0, 0);
        for (int e = lane; e < len; e += 32) {
            const cx<T> p = ldg<T>(pi + e);
#pragma unroll
            for (int n = 0; n < NS; ++n)
                if (n < ns) cmadc(a[n], p, ld<T>(rs + n * len + e));
        }
#pragma unroll
        for (int n = 0; n < NS; ++n) {
            double ar = warp_sum((double)a[n].r), ai = warp_sum((double)a[n].i);
            if (lane == 0 && n < ns) {
                v2<T> o; o.x = (T)ar; o.y = (T)ai;
                rc[((size_t)X * 2 * nv + s * nv + i) * cstride + coff + n0 + n] = o;
            }
        }
    }
}
// e[X][k][l] = sum_i P[X][s(k)][i][k%6][l] y[X][s(k)*Nv + i], NS sources per read of P
template <typename T, int NS>
__global__ void __launch_bounds__(256) k_prolong(v2<T>* __restrict__ e, const v2<T>* __restrict__ P,
                                                 const v2<T>* __restrict__ yc, int nv, Geom g, int cstride, int coff,
                                                 Lanes ln) {
    const int n0 = blockIdx.y * NS, ns = NS == 1 ? 1 : min(NS, ln.m - n0);
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;   // over V*12 as (X, k, l)
    long long total = g.V * 12;
    if (idx >= total) return;
    int l = (int)(idx % g.Vb);
    long long t = idx / g.Vb;
    int k = (int)(t % 12);
    int X = (int)(t / 12);
    int s = k / 6, kk = k - 6 * s;
    int len = 6 * g.Vb;
    const v2<T>* p = P + (((size_t)X * 2 + s) * nv * 6 + kk) * g.Vb + l;
    const v2<T>* y = yc + ((size_t)X * 2 * nv + s * nv) * cstride + coff + n0;
    cx<T> a[NS];
#pragma unroll
    for (int n = 0; n < NS; ++n) a[n] = cx<T>(0, 0);
    for (int i = 0; i < nv; ++i) {
        const cx<T> pi = ldg<T>(p + (size_t)i * len);
#pragma unroll
        for (int n = 0; n < NS; ++n)
            if (n < ns) cmad(a[n], pi, ldg<T>(y + (size_t)i * cstride + n));
    }
#pragma unroll
    for (int n = 0; n < NS; ++n)
        if (n < ns) st<T>(e + (n0 + n) * ln.a + idx, a[n]);
}

// sources per CTA: four, their staged halves within 48 KB of shared memory
constexpr int kTransferSources = 4;
template <typename T>
void restrict_(v2<T>* rc, const v2<T>* P, const v2<T>* r, int nv, const Geom& g, cudaStream_t st, int cstride, int coff,
               const Lanes& ln) {
    constexpr int NS = kTransferSources;
    const size_t sm = sizeof(v2<T>) * 6 * g.Vb;
    note_launch();
    if (ln.m > 1 && NS * sm <= 48 * 1024)
        k_restrict<T, NS><<<dim3(2 * g.Vc, (ln.m + NS - 1) / NS), kThreads, NS * sm, st>>>(rc, P, r, nv, g, cstride, coff, ln);
    else
        k_restrict<T, 1><<<dim3(2 * g.Vc, ln.m), kThreads, sm, st>>>(rc, P, r, nv, g, cstride, coff, ln);
}
template <typename T>
void prolong(v2<T>* e, const v2<T>* P, const v2<T>* yc, int nv, const Geom& g, cudaStream_t st, int cstride, int coff,
             const Lanes& ln) {
    constexpr int NS = kTransferSources;
    const unsigned int grid = (unsigned int)((g.V * 12 + kThreads - 1) / kThreads);
    note_launch();
    if (ln.m > 1)
        k_prolong<T, NS><<<dim3(grid, (ln.m + NS - 1) / NS), kThreads, 0, st>>>(e, P, yc, nv, g, cstride, coff, ln);
    else
        k_prolong<T, 1><<<grid, kThreads, 0, st>>>(e, P, yc, nv, g, cstride, coff, ln);
}

// ================================================================ coarse operator build
// One CTA per (aggregate X, hop h = 2*mu + (0 fwd | 1 bwd)).  For site chunks
// of X it forms W_b(x) = H_h(x) P_b(y) for every coarse column b (H_h the
// hop of eq. 2 from x to y = x +/- mu, P_b column b at y) and accumulates
// conj(P_a(x)) . W_b(x) over the 6 components of chirality s_a.  Hops leaving
// X through its face in direction h go to A[X][1+h]; hops staying inside X go
// to Aself[X][h] (summed later with the diagonal (4+m)).
constexpr int kBuildChunk = 8;
// stride (complex entries) of one (site, column) spinor in the build's shared
// memory: 13, not 12, so the lanes of a warp (sixteen consecutive columns) fall on
// distinct banks in the product loop
constexpr int kWStride = 13;

template <typename TC, int MU, bool FWD>
__device__ __forceinline__ void hop_column(const cx<TC> (&p)[4][3], const v2<TC>* __restrict__ u, int Vb, TC coef,
                                           cx<TC> (&out)[4][3]) {
    // spin projection (same convention as the fine operator)
    cx<TC> h[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (MU == 0) {
            h[0][c] = FWD ? p[0][c] + mul_mi(p[3][c]) : p[0][c] + mul_i(p[3][c]);
            h[1][c] = FWD ? p[1][c] + mul_mi(p[2][c]) : p[1][c] + mul_i(p[2][c]);
        } else if (MU == 1) {
            h[0][c] = FWD ? p[0][c] + p[3][c] : p[0][c] - p[3][c];
            h[1][c] = FWD ? p[1][c] - p[2][c] : p[1][c] + p[2][c];
        } else if (MU == 2) {
            h[0][c] = FWD ? p[0][c] + mul_mi(p[2][c]) : p[0][c] + mul_i(p[2][c]);
            h[1][c] = FWD ? p[1][c] + mul_i(p[3][c]) : p[1][c] + mul_mi(p[3][c]);
        } else {
            h[0][c] = FWD ? p[0][c] - p[2][c] : p[0][c] + p[2][c];
            h[1][c] = FWD ? p[1][c] - p[3][c] : p[1][c] + p[3][c];
        }
    }
    cx<TC> w[2][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        w[0][a] = cx<TC>(0, 0);
        w[1][a] = cx<TC>(0, 0);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (FWD) {
                cx<TC> uab = ld<TC>(u + (3 * a + b) * Vb);
                cmad(w[0][a], uab, h[0][b]);
                cmad(w[1][a], uab, h[1][b]);
            } else {
                cx<TC> uba = ld<TC>(u + (3 * b + a) * Vb);
                cmadc(w[0][a], uba, h[0][b]);
                cmadc(w[1][a], uba, h[1][b]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        cx<TC> w0 = coef * w[0][c], w1 = coef * w[1][c];
        out[0][c] = w0;
        out[1][c] = w1;
        if (MU == 0) { out[2][c] = FWD ? mul_i(w1) : mul_mi(w1); out[3][c] = FWD ? mul_i(w0) : mul_mi(w0); }
        else if (MU == 1) { out[2][c] = FWD ? cx<TC>(-w1.r, -w1.i) : w1; out[3][c] = FWD ? w0 : cx<TC>(-w0.r, -w0.i); }
        else if (MU == 2) { out[2][c] = FWD ? mul_i(w0) : mul_mi(w0); out[3][c] = FWD ? mul_mi(w1) : mul_i(w1); }
        else { out[2][c] = FWD ? cx<TC>(-w0.r, -w0.i) : w0; out[3][c] = FWD ? cx<TC>(-w1.r, -w1.i) : w1; }
    }
}

// Sites of an aggregate in the build's order for direction MU: first those whose hop
// leaves the aggregate (count Vb / B_MU), then the others, each set in lexicographic
// order.  One accumulator set then serves both sums: it is written out where the
// first set ends.
template <int MU, bool FWD> __device__ __forceinline__ int build_site(const Geom& g, int m) {
    const unsigned int ls = g.lstride[MU], Bm = g.B[MU], nface = g.Vb / Bm;
    unsigned int q = m, c = FWD ? Bm - 1 : 0, hi;
    if (q < nface) {
        hi = q / ls;
        q -= hi * ls;
    } else {
        q -= nface;
        hi = q / ls;
        q -= hi * ls;
        c = hi % (Bm - 1) + (FWD ? 0 : 1);
        hi /= Bm - 1;
    }
    return (int)(q + ls * (c + Bm * hi));
}
// strides (complex entries) between the sites of a chunk: two (FP32) or one (FP64)
// above a multiple of 16, so that the lanes of a store (sites fastest) fall on
// distinct banks
template <typename TC> __host__ __device__ constexpr int build_stride(int n) {
    constexpr int off = sizeof(TC) == 4 ? 2 : 1;
    return (n + 15 - off) / 16 * 16 + off;
}

// W_b(x) of the chunk's sites, all columns b: Wsh[xi * ws + b * kWStride + k].  Lanes
// run over the sites first: P and U are read in segments of consecutive sites.
template <typename TC, int MU, bool FWD>
__device__ __forceinline__ void build_stage(const v2<TC>* __restrict__ P, const v2<TC>* __restrict__ U, int nv, const Geom& g,
                                            int X, const int (&xcX)[4], int m0, int cs, v2<TC>* Wsh, v2<TC>* Psh, int ws,
                                            int ps) {
    const int nc = 2 * nv, len = 6 * g.Vb;
    for (int t = threadIdx.x; t < kBuildChunk * nc; t += blockDim.x) {
        const int xi = t % kBuildChunk, b = t / kBuildChunk;
        if (xi >= cs) continue;
        const int l = build_site<MU, FWD>(g, m0 + xi);
        int lc[4];
        local_coords(g, l, lc);
        int Xn, ln;
        bool flip;
        neighbour(g, X, l, lc, xcX, MU, FWD ? 1 : -1, Xn, ln, flip);
        const int sb = b >= nv, ib = b - sb * nv;
        cx<TC> p[4][3];
        const v2<TC>* col = P + (((size_t)Xn * 2 + sb) * nv + ib) * len + ln;
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int c = 0; c < 3; ++c)
                p[sp][c] = ((sp >> 1) == sb) ? ld<TC>(col + ((sp & 1) * 3 + c) * g.Vb) : cx<TC>(0, 0);
        const v2<TC>* u = FWD ? U + ((size_t)MU * g.Vc + X) * 9 * g.Vb + l : U + ((size_t)MU * g.Vc + Xn) * 9 * g.Vb + ln;
        cx<TC> o[4][3];
        hop_column<TC, MU, FWD>(p, u, g.Vb, flip ? TC(0.5) : TC(-0.5), o);
#pragma unroll
        for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int c = 0; c < 3; ++c) st<TC>(Wsh + (size_t)xi * ws + b * kWStride + 3 * sp + c, o[sp][c]);
    }
    // P_a(x): Psh[xi * ps + a * 6 + kk]
    for (int t = threadIdx.x; t < kBuildChunk * nc * 6; t += blockDim.x) {
        const int xi = t % kBuildChunk, r = t / kBuildChunk;
        if (xi < cs) Psh[xi * ps + r] = P[((size_t)X * nc * 6 + r) * g.Vb + build_site<MU, FWD>(g, m0 + xi)];
    }
}

template <typename TC>
__device__ __forceinline__ void build_stage_of(int h, const v2<TC>* __restrict__ P, const v2<TC>* __restrict__ U, int nv,
                                               const Geom& g, int X, const int (&xcX)[4], int m0, int cs, v2<TC>* Wsh,
                                               v2<TC>* Psh, int ws, int ps) {
    switch (h) {
        case 0: build_stage<TC, 0, true>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
        case 1: build_stage<TC, 0, false>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
        case 2: build_stage<TC, 1, true>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
        case 3: build_stage<TC, 1, false>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
        case 4: build_stage<TC, 2, true>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
        case 5: build_stage<TC, 2, false>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
        case 6: build_stage<TC, 3, true>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
        default: build_stage<TC, 3, false>(P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps); break;
    }
}

// FP32: one CTA per (aggregate, direction), products in FP32 with the sums over a
// chunk's sites added up in FP64.  Threads: chirality
// of the row (2) x 8 x 16, each with NT x NT products, rows ta + 8 i, columns
// tb + 16 j (NT = ceil(nv / 8), at most 4 for nv <= 25): an entry of shared memory
// feeds NT products.  (With one product per two entries the shared-memory pipe, not
// the FMA units, was at work: the six builds of a setup on 16^3x32, 4^4 aggregates,
// 16 to 20 columns: 40 -> 22 ms; the products alone take 5, their sums and
// conversions in FP64 another 6.)
template <int NT>
__global__ void __launch_bounds__(256, NT <= 3 ? 2 : 1)
k_coarse_hop(double2* __restrict__ A, double2* __restrict__ Aself, const float2* __restrict__ P, const float2* __restrict__ U,
             int nv, Geom g) {
    using TC = float;
    extern __shared__ unsigned char smem_raw[];
    const int nc = 2 * nv, ws = build_stride<TC>(nc * kWStride), ps = build_stride<TC>(nc * 6);
    v2<TC>* Wsh = reinterpret_cast<v2<TC>*>(smem_raw);
    v2<TC>* Psh = Wsh + (size_t)kBuildChunk * ws;
    const int X = blockIdx.x >> 3, h = blockIdx.x & 7;
    const int sa = threadIdx.x >> 7, ta = (threadIdx.x >> 4) & 7, tb = threadIdx.x & 15;
    int xcX[4], pa[NT], pb[NT];
    coarse_coords(g, X, xcX);
#pragma unroll
    for (int i = 0; i < NT; ++i) {   // rows and columns past the last repeat it and are not stored
        pa[i] = (sa * nv + min(ta + 8 * i, nv - 1)) * 6;
        pb[i] = min(tb + 16 * i, nc - 1) * kWStride + 6 * sa;
    }
    const int nface = g.Vb / (h < 2 ? g.B[0] : h < 4 ? g.B[1] : h < 6 ? g.B[2] : g.B[3]);
    for (int set = 0; set < 2; ++set) {
        const int end = set ? g.Vb : nface;
        cx<double> acc[NT][NT];
#pragma unroll
        for (int i = 0; i < NT; ++i)
#pragma unroll
            for (int j = 0; j < NT; ++j) acc[i][j] = cx<double>(0, 0);
        for (int m0 = set ? nface : 0; m0 < end; m0 += kBuildChunk) {
            const int cs = min(kBuildChunk, end - m0);
            build_stage_of<TC>(h, P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps);
            __syncthreads();
            cx<TC> t[NT][NT];
#pragma unroll
            for (int i = 0; i < NT; ++i)
#pragma unroll
                for (int j = 0; j < NT; ++j) t[i][j] = cx<TC>(0, 0);
            for (int xi = 0; xi < cs; ++xi) {
                const v2<TC>* wx = Wsh + (size_t)xi * ws;
                const v2<TC>* px = Psh + xi * ps;
#pragma unroll
                for (int kk = 0; kk < 6; ++kk) {
                    cx<TC> w[NT], p[NT];
#pragma unroll
                    for (int i = 0; i < NT; ++i) {
                        w[i] = ld<TC>(wx + pb[i] + kk);
                        p[i] = ld<TC>(px + pa[i] + kk);
                    }
#pragma unroll
                    for (int i = 0; i < NT; ++i)
#pragma unroll
                        for (int j = 0; j < NT; ++j) cmadc(t[i][j], p[i], w[j]);
                }
            }
#pragma unroll
            for (int i = 0; i < NT; ++i)
#pragma unroll
                for (int j = 0; j < NT; ++j) acc[i][j] = acc[i][j] + cx<double>((double)t[i][j].r, (double)t[i][j].i);
            __syncthreads();
        }
        // column-major: A[X][1 + h][b][a], Aself[X][h][b][a]
        double2* out = set ? Aself + ((size_t)X * 8 + h) * nc * nc : A + ((size_t)X * 9 + 1 + h) * nc * nc;
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
            for (int i = 0; i < NT; ++i)
                if (ta + 8 * i < nv && tb + 16 * j < nc)
                    st<double>(out + (size_t)(tb + 16 * j) * nc + sa * nv + ta + 8 * i, acc[i][j]);
    }
}
// FP64: bound by the FP64 pipe, two operations a clock and SM, whatever feeds it.  So no
// product is formed that is not stored: the pairs (a, b) are dealt out in order, Q per
// thread, and warps past the last pair have nothing to do (the tiles above form 1.4 times
// the products at nv = 20, 1.8 times at nv = 12).  Builds of one setup at 2 to 20 columns
// on 16^3x32: 799 ms, in tiles about 1130, with two accumulators per pair 930; at 2 to 12
// columns on 12^3x24 54, 100 and 71.
template <int Q>
__global__ void __launch_bounds__(256) k_coarse_hop_pairs(double2* __restrict__ A, double2* __restrict__ Aself,
                                                          const double2* __restrict__ P, const double2* __restrict__ U,
                                                          int nv, Geom g) {
    extern __shared__ unsigned char smem_raw[];
    const int nc = 2 * nv, npair = nc * nc, ws = build_stride<double>(nc * kWStride), ps = build_stride<double>(nc * 6);
    double2* Wsh = reinterpret_cast<double2*>(smem_raw);
    double2* Psh = Wsh + (size_t)kBuildChunk * ws;
    const int X = blockIdx.x >> 3, h = blockIdx.x & 7;
    int xcX[4], pa[Q], pb[Q];
    coarse_coords(g, X, xcX);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int pr = threadIdx.x + q * 256, a = pr < npair ? pr / nc : 0, b = pr < npair ? pr - a * nc : 0;
        pa[q] = a * 6;
        pb[q] = b * kWStride + (a >= nv ? 6 : 0);
    }
    const int nface = g.Vb / (h < 2 ? g.B[0] : h < 4 ? g.B[1] : h < 6 ? g.B[2] : g.B[3]);
    for (int set = 0; set < 2; ++set) {
        const int end = set ? g.Vb : nface;
        cx<double> acc[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) acc[q] = cx<double>(0, 0);
        for (int m0 = set ? nface : 0; m0 < end; m0 += kBuildChunk) {
            const int cs = min(kBuildChunk, end - m0);
            build_stage_of<double>(h, P, U, nv, g, X, xcX, m0, cs, Wsh, Psh, ws, ps);
            __syncthreads();
            cx<double> t[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) t[q] = cx<double>(0, 0);
            for (int xi = 0; xi < cs; ++xi) {
                const double2* wx = Wsh + (size_t)xi * ws;
                const double2* px = Psh + xi * ps;
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if ((int)threadIdx.x + q * 256 < npair)
#pragma unroll
                        for (int kk = 0; kk < 6; ++kk) cmadc(t[q], ld<double>(px + pa[q] + kk), ld<double>(wx + pb[q] + kk));
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) acc[q] = acc[q] + t[q];
            __syncthreads();
        }
        double2* out = set ? Aself + ((size_t)X * 8 + h) * npair : A + ((size_t)X * 9 + 1 + h) * npair;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int a = pa[q] / 6, b = pb[q] / kWStride;   // 6 < kWStride
            if ((int)threadIdx.x + q * 256 < npair) st<double>(out + (size_t)b * nc + a, acc[q]);
        }
    }
}
// A[X][0] = (4+m) I + sum_h Aself[X][h] (fixed order)
__global__ void k_coarse_diag(double2* A, const double2* __restrict__ Aself, int nc, double diag, Geom g) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    long long total = (long long)g.Vc * nc * nc;
    if (idx >= total) return;
    int X = (int)(idx / (nc * nc));
    int r = (int)(idx - (long long)X * nc * nc);    // b*nc + a
    int b = r / nc, a = r - b * nc;
    cx<double> v(a == b ? diag : 0.0, 0.0);
    for (int h = 0; h < 8; ++h) v = v + ld<double>(Aself + ((size_t)X * 8 + h) * nc * nc + r);
    st<double>(A + (size_t)X * 9 * nc * nc + r, v);
}

// T: precision of the products
template <typename T>
static void coarse_build_with(void (*kern)(double2*, double2*, const v2<T>*, const v2<T>*, int, Geom), double2* A, double2* Aself,
                              const v2<T>* P, const v2<T>* U, int nv, double mass, const Geom& g, cudaStream_t st) {
    const int nc = 2 * nv;
    const size_t sm = sizeof(v2<T>) * kBuildChunk * (build_stride<T>(nc * kWStride) + build_stride<T>(nc * 6));
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    note_launch();
    kern<<<g.Vc * 8, kThreads, sm, st>>>(A, Aself, P, U, nv, g);
    long long total = (long long)g.Vc * nc * nc;
    note_launch();
    k_coarse_diag<<<(int)((total + kThreads - 1) / kThreads), kThreads, 0, st>>>(A, Aself, nc, 4.0 + mass, g);
}
void coarse_build_f32(double2* A, double2* Aself, const float2* P, const float2* U, int nv, double mass, const Geom& g,
                      cudaStream_t st) {
    coarse_build_with<float>(nv <= 8 ? k_coarse_hop<1> : nv <= 16 ? k_coarse_hop<2> : nv <= 24 ? k_coarse_hop<3> : k_coarse_hop<4>,
                             A, Aself, P, U, nv, mass, g, st);
}

void coarse_build(double2* A, double2* Aself, const double2* P, const double2* U, int nv, double mass, const Geom& g,
                  cudaStream_t st) {
    coarse_build_with<double>(nv <= 8 ? k_coarse_hop_pairs<1> : nv <= 16 ? k_coarse_hop_pairs<4> : k_coarse_hop_pairs<10>, A,
                              Aself, P, U, nv, mass, g, st);
}

__global__ void k_coarse_shift(double2* A, int nc, double dm, int Vc) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= (long long)Vc * nc) return;
    int X = (int)(idx / nc), a = (int)(idx - (long long)X * nc);
    double2* p = A + (size_t)X * 9 * nc * nc + (size_t)a * nc + a;
    p->x += dm;
}
void coarse_shift_mass(double2* A, int nc, double dm, const Geom& g, cudaStream_t st) {
    long long total = (long long)g.Vc * nc;
    note_launch();
    k_coarse_shift<<<(int)((total + kThreads - 1) / kThreads), kThreads, 0, st>>>(A, nc, dm, g.Vc);
}

// [X][d][a][b] <-> [X][d][b][a]
__global__ void k_transpose_blocks(double2* out, const double2* __restrict__ in, int nc, long long nblk) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= nblk * nc * nc) return;
    long long blk = idx / (nc * nc);
    int r = (int)(idx - blk * nc * nc);
    int i = r / nc, j = r - i * nc;
    out[blk * nc * nc + (size_t)j * nc + i] = in[idx];
}
void coarse_op_transpose(double2* out, const double2* in, int nc, int Vc, cudaStream_t st) {
    long long total = (long long)Vc * 9 * nc * nc;
    note_launch();
    k_transpose_blocks<<<(int)((total + kThreads - 1) / kThreads), kThreads, 0, st>>>(out, in, nc, (long long)Vc * 9);
}

// ================================================================ coarse apply
// y[X][a] = sum_d sum_b A[X][d][b][a] x[X+d][b]; one thread per (X, a), lanes
// read consecutive a (column-major blocks), x[X+d][b] is a warp broadcast.
// dag: sigma3 on x and on y.  FIN: 0 none, 1 ||y||^2 -> slot, 2 CG alpha,
// 3 CG beta (the CG variants are skipped once scal[S_CG_DONE] is set).
template <typename T, bool DAG, int FIN>
__global__ void __launch_bounds__(256) k_coarse_apply(v2<T>* __restrict__ y, const v2<T>* __restrict__ A,
                                                      const v2<T>* __restrict__ x, int nc, Geom g, int slot, Reduce R) {
    if (FIN >= 2 && R.scal[S_CG_DONE] != 0.0) return;
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    int nvh = nc >> 1;
    double red[1] = {0.0};
    if (idx < (long long)g.Vc * nc) {
        int X = (int)(idx / nc), a = (int)(idx - (long long)X * nc);
        cx<T> acc(0, 0);
        for (int d = 0; d < 9; ++d) {
            int Y = coarse_neighbour(g, X, d);
            const v2<T>* Ad = A + ((size_t)X * 9 + d) * nc * nc + a;
            const v2<T>* xY = x + (size_t)Y * nc;
            if (DAG) {
                for (int b = 0; b < nvh; ++b) cmad(acc, ldg<T>(Ad + (size_t)b * nc), ldg<T>(xY + b));
                for (int b = nvh; b < nc; ++b) {
                    cx<T> xb = ldg<T>(xY + b);
                    cmad(acc, ldg<T>(Ad + (size_t)b * nc), cx<T>(-xb.r, -xb.i));
                }
            } else {
                for (int b = 0; b < nc; ++b) cmad(acc, ldg<T>(Ad + (size_t)b * nc), ldg<T>(xY + b));
            }
        }
        if (DAG && a >= nvh) acc = cx<T>(-acc.r, -acc.i);
        st<T>(y + idx, acc);
        red[0] = (double)norm2(acc);
    }
    if (FIN == 1) {
        grid_reduce<1>(red, R.partials, R.ticket, R.partial_bytes, [&](double (&t)[1]) { R.scal[slot] = t[0]; });
    } else if (FIN == 2) {
        grid_reduce<1>(red, R.partials, R.ticket, R.partial_bytes, [&](double (&t)[1]) {
            if (t[0] > 0) R.scal[S_CG_ALPHA] = R.scal[S_CG_GAMMA] / t[0];
            else { R.scal[S_CG_ALPHA] = 0.0; R.scal[S_CG_DONE] = 1.0; }
        });
    } else if (FIN == 3) {
        grid_reduce<1>(red, R.partials, R.ticket, R.partial_bytes, [&](double (&t)[1]) {
            double gam = R.scal[S_CG_GAMMA];
            R.scal[S_CG_BETA] = gam > 0 ? t[0] / gam : 0.0;
            R.scal[S_CG_GAMMA] = t[0];
        });
    }
}

template <typename T>
void coarse_apply(v2<T>* y, const v2<T>* A, const v2<T>* x, int nc, bool dag, int slot, const Geom& g, const Reduce& R,
                  cudaStream_t st) {
    long long total = (long long)g.Vc * nc;
    int grid = (int)((total + kThreads - 1) / kThreads);
    if (slot >= 0) {
        if (dag) { note_launch(); k_coarse_apply<T, true, 1><<<grid, kThreads, 0, st>>>(y, A, x, nc, g, slot, R); }
        else { note_launch(); k_coarse_apply<T, false, 1><<<grid, kThreads, 0, st>>>(y, A, x, nc, g, slot, R); }
    } else {
        if (dag) { note_launch(); k_coarse_apply<T, true, 0><<<grid, kThreads, 0, st>>>(y, A, x, nc, g, slot, R); }
        else { note_launch(); k_coarse_apply<T, false, 0><<<grid, kThreads, 0, st>>>(y, A, x, nc, g, slot, R); }
    }
}

// ================================================================ CGNR (CGLS) on D_c
template <typename T>
__global__ void k_cg_start(v2<T>* __restrict__ y, v2<T>* __restrict__ r, const v2<T>* __restrict__ rc, size_t n,
                           double tol, int maxit, Reduce R) {
    T a = 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        v2<T> v = rc[i];
        r[i] = v;
        v2<T> z; z.x = 0; z.y = 0;
        y[i] = z;
        a += v.x * v.x + v.y * v.y;
    }
    double acc[1] = {(double)a};
    grid_reduce<1>(acc, R.partials, R.ticket, R.partial_bytes, [&](double (&t)[1]) {
        R.scal[S_CG_RC2] = t[0];
        R.scal[S_CG_R2] = t[0];
        R.scal[S_CG_TOL2] = tol * tol;
        R.scal[S_CG_MAXIT] = (double)maxit;
        R.scal[S_CG_ITERS] = 0.0;
        R.scal[S_CG_DONE] = (t[0] > 0 && maxit > 0) ? 0.0 : 1.0;
    });
}
template <typename T>
__global__ void k_cg_copy(v2<T>* __restrict__ p, const v2<T>* __restrict__ s, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) p[i] = s[i];
}
// y += alpha p; r -= alpha q; ||r||^2; iteration count and stopping test
template <typename T>
__global__ void k_cg_update1(v2<T>* __restrict__ y, v2<T>* __restrict__ r, const v2<T>* __restrict__ p,
                             const v2<T>* __restrict__ q, size_t n, Reduce R) {
    if (R.scal[S_CG_DONE] != 0.0) return;
    T al = (T)R.scal[S_CG_ALPHA];
    T a = 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        st<T>(y + i, ld<T>(y + i) + al * ld<T>(p + i));
        cx<T> v = ld<T>(r + i) - al * ld<T>(q + i);
        st<T>(r + i, v);
        a += norm2(v);
    }
    double acc[1] = {(double)a};
    grid_reduce<1>(acc, R.partials, R.ticket, R.partial_bytes, [&](double (&t)[1]) {
        double it = R.scal[S_CG_ITERS] + 1.0;
        R.scal[S_CG_ITERS] = it;
        R.scal[S_CG_R2] = t[0];
        if (t[0] <= R.scal[S_CG_TOL2] * R.scal[S_CG_RC2] || it >= R.scal[S_CG_MAXIT]) R.scal[S_CG_DONE] = 1.0;
    });
}
// p = s + beta p
template <typename T>
__global__ void k_cg_update2(v2<T>* __restrict__ p, const v2<T>* __restrict__ s, size_t n, const double* __restrict__ scal) {
    if (scal[S_CG_DONE] != 0.0) return;
    T be = (T)scal[S_CG_BETA];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        st<T>(p + i, ld<T>(s + i) + be * ld<T>(p + i));
}

template <typename T>
void cg_init(v2<T>* y, v2<T>* r, const v2<T>* rc, size_t n, double tol, int maxit, const Reduce& R, cudaStream_t st) {
    note_launch();
    k_cg_start<T><<<reduce_grid(n), kThreads, 0, st>>>(y, r, rc, n, tol, maxit, R);
}
// s = D_c^dag r, gamma = ||s||^2, p = s
template <typename T>
void cg_first_direction(v2<T>* s, v2<T>* p, const v2<T>* r, const v2<T>* A, int nc, const Geom& g, const Reduce& R,
                        cudaStream_t st) {
    size_t n = (size_t)g.Vc * nc;
    coarse_apply<T>(s, A, r, nc, true, S_CG_GAMMA, g, R, st);
    note_launch();
    k_cg_copy<T><<<reduce_grid(n), kThreads, 0, st>>>(p, s, n);
}
template <typename T>
void cg_step(v2<T>* y, v2<T>* r, v2<T>* s, v2<T>* p, v2<T>* q, const v2<T>* A, int nc, const Geom& g, const Reduce& R,
             cudaStream_t st) {
    size_t n = (size_t)g.Vc * nc;
    int grid = (int)((n + kThreads - 1) / kThreads);
    note_launch();
    k_coarse_apply<T, false, 2><<<grid, kThreads, 0, st>>>(q, A, p, nc, g, -1, R);        // q = D_c p, alpha
    note_launch();
    k_cg_update1<T><<<reduce_grid(n), kThreads, 0, st>>>(y, r, p, q, n, R);               // y, r, stop test
    note_launch();
    k_coarse_apply<T, true, 3><<<grid, kThreads, 0, st>>>(s, A, r, nc, g, -1, R);         // s = D_c^dag r, beta
    note_launch();
    k_cg_update2<T><<<reduce_grid(n), kThreads, 0, st>>>(p, s, n, R.scal);                // p = s + beta p
}

#define INST(T)                                                                                                     \
    template void restrict_<T>(v2<T>*, const v2<T>*, const v2<T>*, int, const Geom&, cudaStream_t, int, int,        \
                               const Lanes&);                                                                       \
    template void prolong<T>(v2<T>*, const v2<T>*, const v2<T>*, int, const Geom&, cudaStream_t, int, int,          \
                             const Lanes&);                                                                         \
    template void coarse_apply<T>(v2<T>*, const v2<T>*, const v2<T>*, int, bool, int, const Geom&, const Reduce&,    \
                                  cudaStream_t);                                                                    \
    template void cg_init<T>(v2<T>*, v2<T>*, const v2<T>*, size_t, double, int, const Reduce&, cudaStream_t);       \
    template void cg_first_direction<T>(v2<T>*, v2<T>*, const v2<T>*, const v2<T>*, int, const Geom&, const Reduce&, \
                                        cudaStream_t);                                                              \
    template void cg_step<T>(v2<T>*, v2<T>*, v2<T>*, v2<T>*, v2<T>*, const v2<T>*, int, const Geom&, const Reduce&,  \
                             cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace wmg

namespace wmg {
// P64[X][s][i][k6][l] -> boundary [i][lex site][spin][colour] (zero on the other chirality)
__global__ void k_prolongator_to_boundary(double2* out, const double2* __restrict__ P, int nv, Geom g) {
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;   // over nv * V * 12 in internal order
    long long total = (long long)nv * g.V * 12;
    if (idx >= total) return;
    int i = (int)(idx / (g.V * 12));
    long long r = idx - (long long)i * g.V * 12;
    int X = (int)(r / (12LL * g.Vb));
    int rem = (int)(r - (long long)X * 12 * g.Vb);
    int k = rem / g.Vb, l = rem - k * g.Vb;
    int s = k / 6, kk = k - 6 * s;
    long long lex = lex_site(g, X, l);
    double2 v = P[((((size_t)X * 2 + s) * nv + i) * 6 + kk) * g.Vb + l];
    out[((size_t)i * g.V + lex) * 12 + 6 * s + kk] = v;
}
void prolongator_to_boundary(double2* out, const double2* P, int nv, const Geom& g, cudaStream_t st) {
    long long total = (long long)nv * g.V * 12;
    note_launch();
    k_prolongator_to_boundary<<<(int)((total + 255) / 256), 256, 0, st>>>(out, P, nv, g);
}
}  // namespace wmg

// ================================================================ persistent CGNR
// The whole coarse solve in one cooperative launch: G co-resident CTAs loop
// over the CGLS iterations, separated by grid barriers.  Every spin-wait is
// bounded: after kBarrierSpinLimit polls the CTA sets *err and returns, and
// CTAs waiting at a barrier return as soon as *err is set.  Reductions:
// each CTA writes its partial sum, and after the barrier every CTA adds all
// partials in the same order, so all CTAs take identical decisions.
namespace wmg {

// How the rows are dealt out (host: cgnr_split).  The rows of every aggregate
// are cut into rsp parts of equal size; unit u = X * rsp + part.  A CTA works on
// upb consecutive units at a time, tpu = 9 * bs * (row groups of a part) threads
// each: thread (unit, d, column part, row group).
// FP32 and FP16 operators (bound by the operator's bytes): whole aggregates (rsp =
// 1), as many as fit the CTA while every SM has one, then column parts.  FP64 (bound by
// the FP64 pipe, two FMAs per clock and SM): every SM has to have an equal share of the
// rows.  With
// whole aggregates an 8^4 lattice (16 aggregates) ran on 4 SMs and 12^3 x 24
// (162 aggregates) on 54; cut into parts, one CTA per SM (its partial sums are
// re-added in FP64 by every CTA, so no more CTAs than SMs).  Measured with the
// FP64 operator's CTAs above: an 8^4 solve (Nv = 8) 321 -> 169 ms, 12^3 x 24
// (Nv = 12) 285 -> 193 ms.
struct CgnrSplit {
    int upb, rsp, bs;
    // the FP32 / FP16 split with its constants known to the compiler (index
    // arithmetic by run-time divisors cost 5-8 % of an iteration)
    template <typename T> __device__ int parts() const { return sizeof(T) == 4 ? 1 : rsp; }
};

// entries between two blocks of a unit's resident rows: two more than they hold, so
// that the directions and column parts of a warp's lanes start on different banks
__host__ __device__ constexpr int res_block(int nc, int rows) { return nc * rows + 2; }

// One CG phase on the units of this CTA, upb at a time: stage the operand on
// their aggregates and the 8 neighbours in shared memory, then apply the coarse
// stencil.  A thread accumulates R consecutive rows a of block A[X][d] (one
// 16-byte load carries rows a, a+1 of column b) with U independent loads in
// flight; shared memory sums the 9 directions and the column parts.
// The operand is formed while staging (STAGE):
//   ST_P: pn = s + beta * p_old   (first iteration: pn = s); own entries -> p_new
//         output q = D_c pn;          partial sums: n0 = ||q||^2
//   ST_R: rn = r_old - alpha * q; own entries -> r_new, y += alpha * p_cur;
//         output s = D_c^dag rn;      partial sums: n0 = ||s||^2, n1 = ||rn||^2
//   ST_PLAIN: operand = in;          output out = D_c(^dag) in, n0 = ||out||^2
// Red-black form (a phase is one half of Dhat, see kernels_schur.cu): HALF_O
// computes t = sum_{d >= 1} H x on the odd sites, the operand x (of the even
// neighbours) formed as above; HALF_E computes y = H[0] x + sum_{d >= 1} H t on the
// even sites, x formed for the site itself (with its own entries' updates) and t
// read.  Only x and y carry sigma3 in the adjoint.
enum { ST_PLAIN = 0, ST_P = 1, ST_R = 2 };
enum { HALF_NONE = 0, HALF_O = 1, HALF_E = 2 };

template <typename T, bool H16 = false> struct RowsPerThread { static constexpr int value = H16 ? 4 : 2; };

template <typename T, int R> struct RowLoad;
template <> struct RowLoad<double, 2> {
    static __device__ __forceinline__ void load(const v2<double>* p, cx<double> (&v)[2]) {
        double2 a = __ldg(p), b = __ldg(p + 1);
        v[0] = cx<double>(a.x, a.y);
        v[1] = cx<double>(b.x, b.y);
    }
};
template <> struct RowLoad<float, 2> {
    static __device__ __forceinline__ void load(const v2<float>* p, cx<float> (&v)[2]) {
        float4 a = __ldg(reinterpret_cast<const float4*>(p));
        v[0] = cx<float>(a.x, a.y);
        v[1] = cx<float>(a.z, a.w);
    }
};
// four consecutive rows of the FP16 operator in one 16-byte load
__device__ __forceinline__ void row_load16(const __half2* p, cx<float> (&v)[4]) {
    uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    const __half2* h = reinterpret_cast<const __half2*>(&u);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float2 f = __half22float2(h[r]);
        v[r] = cx<float>(f.x, f.y);
    }
}

template <typename T> struct PhaseArgs {
    const v2<T>* in;       // ST_PLAIN operand
    const v2<T>* s;        // ST_P: s
    const v2<T>* p_old;    // ST_P: previous direction (ignored when first)
    v2<T>* p_new;          // ST_P: own entries of pn; ST_R: p_cur (read)
    const v2<T>* r_old;    // ST_R
    const v2<T>* q;        // ST_R
    v2<T>* r_new;          // ST_R
    v2<T>* y;              // ST_R
    v2<T>* out;            // result
    T coef;                // beta (ST_P) or alpha (ST_R)
    bool first;            // ST_P, first iteration
    const int* sites;      // red-black: the sites of this half, in the order of the units
    v2<T>* t;              // red-black: t of the odd sites (HALF_O writes, HALF_E reads)
};

template <typename T, bool DAG, int STAGE, bool H16, int HALF>
__device__ void cg_phase(const PhaseArgs<T>& ph, const v2<T>* __restrict__ A, const __half2* __restrict__ A16,
                         const float* __restrict__ s16, int nc, const CgnrSplit& sp, const Geom& g, v2<T>* xs,
                         cx<T>* part, const int* __restrict__ nbr, T& n0, T& n1) {
    constexpr int R = RowsPerThread<T, H16>::value;
    const int rsp = sp.template parts<T>(), bs = sp.bs;
    const int nvh = nc >> 1, nrow = 9 * nc, ngl = nc / R / rsp, rows = sizeof(T) == 4 ? nc : ngl * R, nsum = 9 * bs;
    const int tpu = nsum * ngl, nsite = HALF ? g.Vc / 2 : g.Vc, nunit = nsite * rsp;
    const int ul = threadIdx.x / tpu, rem = threadIdx.x - ul * tpu;
    const int db = rem / ngl, a0 = (rem - db * ngl) * R;   // a0: row within the part
    const int d = db / bs, bp = db - d * bs;
    const int bc = (nc + bs - 1) / bs, b_lo = bp * bc, b_hi = min(nc, b_lo + bc);
    for (int Ub = blockIdx.x * sp.upb; Ub < nunit; Ub += gridDim.x * sp.upb) {
        const int Ue = min(Ub + sp.upb, nunit), Xb = Ub / rsp, nall = ((Ue - 1) / rsp - Xb + 1) * nrow;
        for (int i = threadIdx.x; i < nall; i += blockDim.x) {
            int xi = i / nrow, ri = i - xi * nrow;
            int di = ri / nc, b = ri - di * nc;
            const int X = HALF ? __ldg(ph.sites + Xb + xi) : Xb + xi;
            if (HALF != HALF_O || di > 0) {
                // the CTA that owns row b of X does that entry's vector updates
                const int u = (Xb + xi) * rsp + b / rows;
                const bool own = di == 0 && (sizeof(T) == 4 || (u >= Ub && u < Ue));
                int Y = __ldg(nbr + (size_t)X * 9 + di);
                size_t o = (size_t)Y * nc + b;
                cx<T> v;
                if (HALF == HALF_E && di > 0) {
                    st<T>(xs + i, ld<T>(ph.t + o));
                    continue;
                }
                if (STAGE == ST_PLAIN) {
                    v = ld<T>(ph.in + o);
                } else if (STAGE == ST_P) {
                    v = ld<T>(ph.s + o);
                    if (!ph.first) v = v + ph.coef * ld<T>(ph.p_old + o);
                    if (own) st<T>(ph.p_new + o, v);
                } else {
                    v = ld<T>(ph.r_old + o) - ph.coef * ld<T>(ph.q + o);
                    if (own) {
                        st<T>(ph.r_new + o, v);
                        st<T>(ph.y + o, ld<T>(ph.y + o) + ph.coef * ld<T>(ph.p_new + o));
                        n1 += norm2(v);
                    }
                }
                if (DAG && b >= nvh) v = cx<T>(-v.r, -v.i);
                st<T>(xs + i, v);
            }
        }
        __syncthreads();
        const int U0 = Ub + ul, Xi = U0 / rsp, ar = (U0 - Xi * rsp) * rows + a0;   // ar: row within the block
        if (ul < sp.upb && U0 < nunit && (HALF != HALF_O || d > 0)) {
            const int X = HALF ? __ldg(ph.sites + Xi) : Xi;
            const v2<T>* xd = xs + (Xi - Xb) * nrow + d * nc;
            cx<T>* pd = part + (size_t)(ul * nsum + db) * rows + a0;
            cx<T> acc[R][2];
#pragma unroll
            for (int r = 0; r < R; ++r) { acc[r][0] = cx<T>(0, 0); acc[r][1] = cx<T>(0, 0); }
            constexpr int U = 4;
            if constexpr (H16) {
                const __half2* Ad = A16 + ((size_t)X * 9 + d) * nc * nc + ar;
                for (int b0 = b_lo; b0 < b_hi; b0 += U) {
                    uint4 raw[U];
#pragma unroll
                    for (int j = 0; j < U; ++j)
                        if (b0 + j < b_hi) raw[j] = __ldg(reinterpret_cast<const uint4*>(Ad + (size_t)(b0 + j) * nc));
#pragma unroll
                    for (int j = 0; j < U; ++j)
                        if (b0 + j < b_hi) {
                            cx<T> xb = ld<T>(xd + b0 + j);
                            const __half2* h = reinterpret_cast<const __half2*>(&raw[j]);
#pragma unroll
                            for (int r = 0; r < R; ++r) {
                                float2 f = __half22float2(h[r]);
                                cmad(acc[r][j & 1], cx<T>(f.x, f.y), xb);
                            }
                        }
                }
                const T sc = (T)s16[(size_t)X * 9 + d];
#pragma unroll
                for (int r = 0; r < R; ++r) pd[r] = sc * (acc[r][0] + acc[r][1]);
            } else {
                const v2<T>* Ad = A + ((size_t)X * 9 + d) * nc * nc + ar;
                for (int b0 = b_lo; b0 < b_hi; b0 += U) {
                    cx<T> av[U][R];
#pragma unroll
                    for (int j = 0; j < U; ++j)
                        if (b0 + j < b_hi) RowLoad<T, R>::load(Ad + (size_t)(b0 + j) * nc, av[j]);
#pragma unroll
                    for (int j = 0; j < U; ++j)
                        if (b0 + j < b_hi) {
                            cx<T> xb = ld<T>(xd + b0 + j);
#pragma unroll
                            for (int r = 0; r < R; ++r) cmad(acc[r][j & 1], av[j][r], xb);
                        }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) pd[r] = acc[r][0] + acc[r][1];
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < sp.upb * rows; t += blockDim.x) {
            const int u2 = t / rows, U2 = Ub + u2, Xi2 = U2 / rsp, a2 = (U2 - Xi2 * rsp) * rows + (t - u2 * rows);
            if (U2 < nunit) {
                const int X2 = HALF ? __ldg(ph.sites + Xi2) : Xi2, d0 = HALF == HALF_O ? bs : 0;   // no self block in t
                const cx<T>* ps = part + (size_t)u2 * nsum * rows + (t - u2 * rows);
                // four chains: an FP64 add is some sixty clocks to the next that needs it
                cx<T> c[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) c[q] = ps[(d0 + q) * rows];
                int dd = d0 + 4;
                for (; dd + 4 <= nsum; dd += 4)
#pragma unroll
                    for (int q = 0; q < 4; ++q) c[q] = c[q] + ps[(dd + q) * rows];
                for (; dd < nsum; ++dd) c[0] = c[0] + ps[dd * rows];
                cx<T> sum = (c[0] + c[1]) + (c[2] + c[3]);
                if (HALF == HALF_O) {
                    st<T>(ph.t + (size_t)X2 * nc + a2, sum);
                    continue;
                }
                if (DAG && a2 >= nvh) sum = cx<T>(-sum.r, -sum.i);
                st<T>(ph.out + (size_t)X2 * nc + a2, sum);
                n0 += norm2(sum);
            }
        }
        __syncthreads();
    }
}

// The same phase with what a CTA reads in every iteration kept in its shared memory
// (FP64, one batch of units per CTA): the operator's rows, As[ul][d][b][row] with
// blocks of ablk entries, and where each staged entry comes from, src[i] (-1: not
// needed; bit 31: this CTA's own entry, bit 30: an entry of t).  A barrier empties
// the SM's L1, so from global memory a phase is five L2 round trips in a row (site,
// neighbour, operand, two or more groups of operator loads); here it is one, with
// four entries' operands in flight per thread.  Same products in the same order.
constexpr unsigned int kSrcOwn = 1u << 31, kSrcT = 1u << 30, kSrcNone = 0xffffffffu;

template <bool DAG, int STAGE, int HALF>
__device__ void cg_phase_res(const PhaseArgs<double>& ph, const double2* __restrict__ As, const unsigned int* __restrict__ src,
                             int nc, const CgnrSplit& sp, int nsite, double2* xs, cx<double>* part, double& n0, double& n1) {
    constexpr int R = RowsPerThread<double>::value, F = 4;
    const int rsp = sp.rsp, bs = sp.bs;
    const int nvh = nc >> 1, nrow = 9 * nc, ngl = nc / R / rsp, rows = ngl * R, nsum = 9 * bs;
    const int tpu = nsum * ngl, nunit = nsite * rsp, ablk = res_block(nc, rows);
    const int ul = threadIdx.x / tpu, rem = threadIdx.x - ul * tpu;
    const int db = rem / ngl, a0 = (rem - db * ngl) * R;
    const int d = db / bs, bp = db - d * bs;
    const int bc = (nc + bs - 1) / bs, b_lo = bp * bc, b_hi = min(nc, b_lo + bc);
    const int Ub = blockIdx.x * sp.upb, Ue = min(Ub + sp.upb, nunit), Xb = Ub / rsp, nall = ((Ue - 1) / rsp - Xb + 1) * nrow;
    for (int i0 = threadIdx.x; i0 < nall; i0 += F * blockDim.x) {
        cx<double> v[F], w[F];
        unsigned int o[F];
#pragma unroll
        for (int j = 0; j < F; ++j) {
            const int i = i0 + j * blockDim.x;
            o[j] = i < nall ? src[i] : kSrcNone;
            if (o[j] == kSrcNone) continue;
            const unsigned int e = o[j] & ~(kSrcOwn | kSrcT);
            w[j] = cx<double>(0, 0);
            if (HALF == HALF_E && (o[j] & kSrcT)) {
                v[j] = ld<double>(ph.t + e);
            } else if (STAGE == ST_PLAIN) {
                v[j] = ld<double>(ph.in + e);
            } else if (STAGE == ST_P) {
                v[j] = ld<double>(ph.s + e);
                if (!ph.first) w[j] = ld<double>(ph.p_old + e);
            } else {
                v[j] = ld<double>(ph.r_old + e);
                w[j] = ld<double>(ph.q + e);
            }
        }
#pragma unroll
        for (int j = 0; j < F; ++j) {
            if (o[j] == kSrcNone) continue;
            const int i = i0 + j * blockDim.x;
            if (!(HALF == HALF_E && (o[j] & kSrcT))) {
                const unsigned int e = o[j] & ~(kSrcOwn | kSrcT);
                if (STAGE == ST_P) {
                    if (!ph.first) v[j] = v[j] + ph.coef * w[j];
                    if (o[j] & kSrcOwn) st<double>(ph.p_new + e, v[j]);
                } else if (STAGE == ST_R) {
                    v[j] = v[j] - ph.coef * w[j];
                    if (o[j] & kSrcOwn) {
                        st<double>(ph.r_new + e, v[j]);
                        st<double>(ph.y + e, ld<double>(ph.y + e) + ph.coef * ld<double>(ph.p_new + e));
                        n1 += norm2(v[j]);
                    }
                }
                if (DAG && i % nc >= nvh) v[j] = cx<double>(-v[j].r, -v[j].i);
            }
            st<double>(xs + i, v[j]);
        }
    }
    __syncthreads();
    const int U0 = Ub + ul;
    if (ul < sp.upb && U0 < nunit && (HALF != HALF_O || d > 0)) {
        const double2* xd = xs + (U0 / rsp - Xb) * nrow + d * nc;
        const double2* Ad = As + (size_t)(ul * 9 + d) * ablk + a0;
        cx<double> acc[R][2];
#pragma unroll
        for (int r = 0; r < R; ++r) { acc[r][0] = cx<double>(0, 0); acc[r][1] = cx<double>(0, 0); }
        for (int b0 = b_lo; b0 < b_hi; b0 += 2)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (b0 + j < b_hi) {
                    const cx<double> xb = ld<double>(xd + b0 + j);
#pragma unroll
                    for (int r = 0; r < R; ++r) cmad(acc[r][j], ld<double>(Ad + (b0 + j) * rows + r), xb);
                }
        cx<double>* pd = part + (size_t)(ul * nsum + db) * rows + a0;
#pragma unroll
        for (int r = 0; r < R; ++r) pd[r] = acc[r][0] + acc[r][1];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < (Ue - Ub) * rows; t += blockDim.x) {
        const int u2 = t / rows, U2 = Ub + u2, Xi2 = U2 / rsp, a2 = (U2 - Xi2 * rsp) * rows + (t - u2 * rows);
        const int d0 = HALF == HALF_O ? bs : 0;   // no self block in t
        const cx<double>* ps = part + (size_t)u2 * nsum * rows + (t - u2 * rows);
        cx<double> c[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = ps[(d0 + q) * rows];
        int dd = d0 + 4;
        for (; dd + 4 <= nsum; dd += 4)
#pragma unroll
            for (int q = 0; q < 4; ++q) c[q] = c[q] + ps[(dd + q) * rows];
        for (; dd < nsum; ++dd) c[0] = c[0] + ps[dd * rows];
        cx<double> sum = (c[0] + c[1]) + (c[2] + c[3]);
        const int X2 = HALF ? __ldg(ph.sites + Xi2) : Xi2;
        if (HALF == HALF_O) {
            st<double>(ph.t + (size_t)X2 * nc + a2, sum);
            continue;
        }
        if (DAG && a2 >= nvh) sum = cx<double>(-sum.r, -sum.i);
        st<double>(ph.out + (size_t)X2 * nc + a2, sum);
        n0 += norm2(sum);
    }
}
// fill of As and src for one set of sites (sites: a red-black half's, nullptr: all)
__device__ __forceinline__ void cg_resident(double2* As, unsigned int* src, const double2* __restrict__ A, const int* sites,
                                            int half, int nc, const CgnrSplit& sp, int nsite, const int* __restrict__ nbr) {
    const int rsp = sp.rsp, rows = nc / rsp, nrow = 9 * nc, ablk = res_block(nc, rows);
    const int Ub = blockIdx.x * sp.upb, Ue = min(Ub + sp.upb, nsite * rsp), Xb = Ub / rsp;
    for (int i = threadIdx.x; i < (Ue - Ub) * nrow * rows; i += blockDim.x) {
        const int row = i % rows, j = i / rows, ul = j / nrow, db = j - ul * nrow, d = db / nc, b = db - d * nc;
        const int Xi = (Ub + ul) / rsp, X = sites ? sites[Xi] : Xi;
        As[(size_t)(ul * 9 + d) * ablk + b * rows + row] =
            A[(((size_t)X * 9 + d) * nc + b) * nc + (Ub + ul - Xi * rsp) * rows + row];
    }
    const int nall = ((Ue - 1) / rsp - Xb + 1) * nrow;
    for (int i = threadIdx.x; i < nall; i += blockDim.x) {
        const int xi = i / nrow, ri = i - xi * nrow, d = ri / nc, b = ri - d * nc, u = (Xb + xi) * rsp + b / rows;
        const int X = sites ? sites[Xb + xi] : Xb + xi;
        unsigned int o = (unsigned int)(nbr[(size_t)X * 9 + d] * nc + b);
        if (d == 0 && u >= Ub && u < Ue) o |= kSrcOwn;
        if (half == HALF_E && d > 0) o |= kSrcT;
        src[i] = half == HALF_O && d == 0 ? kSrcNone : o;
    }
}

// CGLS (CG on the normal equations), the textbook recurrences
//   q = D_c p, alpha = gamma/||q||^2, y += alpha p, r -= alpha q,
//   s = D_c^dag r, beta = ||s||^2/gamma, p = s + beta p
// with two grid barriers per iteration: the elementwise updates of p and r are
// done while staging the neighbour operands of the next stencil (p and r
// double-buffered so that no CTA overwrites what another still reads).
// FP64: one CTA per SM, registers for all columns of a thread's loads in flight
template <typename T> struct CgnrMaxThreads { static constexpr int value = 384, blocks = sizeof(T) == 8 ? 1 : 2; };

// EO: CG on the normal equations of Dhat (even entries of the vectors; each stencil
// the two halves with a grid barrier between them); a.rc is then rhat and a.rc_full
// the right-hand side whose norm the tolerance refers to.
// RES: operator and sources in shared memory (cg_phase_res).
template <typename T, bool H16, bool EO, bool RES>
__global__ void __launch_bounds__(CgnrMaxThreads<T>::value, CgnrMaxThreads<T>::blocks) k_cgnr_persistent(CgnrArgs<T> a) {
    extern __shared__ unsigned char smem_raw[];
    const int nc = a.nc;
    const CgnrSplit sp{a.upb, a.rsp, a.bs};
    v2<T>* xs = reinterpret_cast<v2<T>*>(smem_raw);
    const int nstage = 9 * nc * ((sp.upb + 2 * sp.rsp - 2) / sp.rsp);
    cx<T>* part = reinterpret_cast<cx<T>*>(xs + nstage);
    __shared__ T shr[66];
    const unsigned int G = gridDim.x;
    v2<T>* rbuf[2] = {a.r, a.r1};
    v2<T>* pbuf[2] = {a.p, a.p1};
    const int nsite = EO ? a.g.Vc / 2 : a.g.Vc;
    PhaseArgs<T> ph{};
    // RES: rows of the units (EO: of the even, then of the odd sites), then the sources
    const int rows = nc / sp.rsp;   // rows of a unit
    const int nres = sp.upb * 9 * res_block(nc, rows);
    v2<T>* As = reinterpret_cast<v2<T>*>(part + 9 * sp.bs * rows * sp.upb);
    unsigned int* src = reinterpret_cast<unsigned int*>(As + (EO ? 2 : 1) * nres);
    if constexpr (RES) {
        cg_resident(As, src, a.A, EO ? a.ord : nullptr, EO ? HALF_E : HALF_NONE, nc, sp, nsite, a.nbr);
        if (EO) cg_resident(As + nres, src + nstage, a.A, a.ord + nsite, HALF_O, nc, sp, nsite, a.nbr);
        __syncthreads();
    }
    // one stencil out = D x (or its adjoint), D = D_c or Dhat; false when a barrier gave up
    auto stencil = [&](auto dag, auto stage, T& n0, T& n1) -> bool {
        constexpr bool DAG = decltype(dag)::value != 0;
        constexpr int STAGE = decltype(stage)::value;
        ph.t = a.t;
        if constexpr (EO) {
            T u0 = 0, u1 = 0;
            ph.sites = a.ord + nsite;
            if constexpr (RES) cg_phase_res<DAG, STAGE, HALF_O>(ph, As + nres, src + nstage, nc, sp, nsite, xs, part, u0, u1);
            else cg_phase<T, DAG, STAGE, H16, HALF_O>(ph, a.A, a.A16, a.s16, nc, sp, a.g, xs, part, a.nbr, u0, u1);
            if (!grid_sync(a.bar, G, a.err)) return false;
            ph.sites = a.ord;
            if constexpr (RES) cg_phase_res<DAG, STAGE, HALF_E>(ph, As, src, nc, sp, nsite, xs, part, n0, n1);
            else cg_phase<T, DAG, STAGE, H16, HALF_E>(ph, a.A, a.A16, a.s16, nc, sp, a.g, xs, part, a.nbr, n0, n1);
        } else if constexpr (RES) {
            cg_phase_res<DAG, STAGE, HALF_NONE>(ph, As, src, nc, sp, nsite, xs, part, n0, n1);
        } else {
            cg_phase<T, DAG, STAGE, H16, HALF_NONE>(ph, a.A, a.A16, a.s16, nc, sp, a.g, xs, part, a.nbr, n0, n1);
        }
        return true;
    };
    // y = 0, r = rc on the units of this CTA; ||rc||^2
    T loc = 0;
    for (int Ub = blockIdx.x * sp.upb; Ub < nsite * sp.rsp; Ub += G * sp.upb)
        for (int t = threadIdx.x; t < sp.upb * rows; t += blockDim.x) {
            const int u = Ub + t / rows;
            if (u < nsite * sp.rsp) {
                const int Xi = u / sp.rsp, a0 = (u - Xi * sp.rsp) * rows + t % rows;
                const size_t o = (size_t)(EO ? a.ord[Xi] : Xi) * nc + a0;
                v2<T> v = a.rc[o];
                a.r[o] = v;
                v2<T> z; z.x = 0; z.y = 0;
                a.y[o] = z;
                if (EO) {
                    const v2<T> e = a.rc_full[o], d = a.rc_full[(size_t)a.ord[nsite + Xi] * nc + a0];
                    loc += e.x * e.x + e.y * e.y + d.x * d.x + d.y * d.y;
                } else {
                    loc += v.x * v.x + v.y * v.y;
                }
            }
        }
    write_partial<T>(loc, a.partials, 0, shr);
    if (!grid_sync(a.bar, G, a.err)) return;
    const T rc2 = sum_partials<T>(a.partials, 0, G, shr);
    int it = 0;
    T r2 = rc2;
    if (rc2 > T(0) && a.maxit > 0) {
        using Yes = std::integral_constant<int, 1>;
        using No = std::integral_constant<int, 0>;
        T n0 = 0, n1 = 0;
        // s = D_c^dag r, gamma = ||s||^2
        ph.in = a.r;
        ph.out = a.s;
        if (!stencil(Yes{}, std::integral_constant<int, ST_PLAIN>{}, n0, n1)) return;
        write_partial<T>(n0, a.partials, 1, shr);
        if (!grid_sync(a.bar, G, a.err)) return;
        T gamma = sum_partials<T>(a.partials, 1, G, shr);
        T beta = 0;
        for (;;) {
            const int b = it & 1;
            // p = s + beta p; q = D_c p
            ph = PhaseArgs<T>{};
            ph.s = a.s; ph.p_old = pbuf[b ^ 1]; ph.p_new = pbuf[b]; ph.out = a.q;
            ph.coef = beta; ph.first = (it == 0);
            n0 = 0; n1 = 0;
            if (!stencil(No{}, std::integral_constant<int, ST_P>{}, n0, n1)) return;
            write_partial<T>(n0, a.partials, 0, shr);
            if (!grid_sync(a.bar, G, a.err)) return;
            T qq = sum_partials<T>(a.partials, 0, G, shr);
            if (!(qq > T(0))) break;
            T alpha = gamma / qq;
            // y += alpha p; r -= alpha q; s = D_c^dag r
            ph = PhaseArgs<T>{};
            ph.r_old = rbuf[b]; ph.q = a.q; ph.r_new = rbuf[b ^ 1]; ph.y = a.y; ph.p_new = pbuf[b];
            ph.out = a.s; ph.coef = alpha;
            n0 = 0; n1 = 0;
            if (!stencil(Yes{}, std::integral_constant<int, ST_R>{}, n0, n1)) return;
            write_partial2<T>(n0, n1, a.partials, 1, shr);
            if (!grid_sync(a.bar, G, a.err)) return;
            T gnew;
            sum_partials2<T>(a.partials, 1, G, shr, gnew, r2);
            ++it;
            if (r2 <= (T)a.tol2 * rc2 || it >= a.maxit) break;
            beta = gnew / gamma;
            gamma = gnew;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.scal[S_CG_ITERS] = (double)it;
        a.scal[S_CG_R2] = (double)r2;
        a.scal[S_CG_RC2] = (double)rc2;
        a.scal[S_CG_DONE] = 1.0;
        a.scal[S_CG_TOTAL] += (double)it;
    }
}

// Split of the rows (see CgnrSplit) and its shared memory.
template <typename T, bool H16> size_t cgnr_smem(int nc, const CgnrSplit& s) {
    const size_t xmax = (s.upb + 2 * s.rsp - 2) / s.rsp;   // aggregates that upb consecutive units can touch
    return sizeof(v2<T>) * 9 * nc * xmax + sizeof(cx<T>) * 9 * s.bs * (nc / s.rsp) * s.upb;
}
template <typename T, bool H16> int cgnr_block_threads(int nc, const CgnrSplit& s) {
    const int tpu = 9 * s.bs * (nc / RowsPerThread<T, H16>::value / s.rsp);
    return std::max(128, (s.upb * tpu + 31) / 32 * 32);   // at least four warps to stage the operand
}
template <typename T, bool H16> CgnrSplit cgnr_split(int nc, int Vc, int sms) {
    constexpr int most = CgnrMaxThreads<T>::value;
    const int ngrp = nc / RowsPerThread<T, H16>::value;
    if (sizeof(T) == 4) {
        // as many aggregates as fit while every SM has one; small lattices' aggregates in
        // column parts
        const int fit = std::max(1, most / (9 * ngrp)), upb = std::max(1, std::min(fit, Vc / sms));
        return CgnrSplit{upb, 1, std::max(1, std::min(most / (9 * ngrp * upb), nc / 8))};
    }
    // FP64: the parts per aggregate that give the busiest SM the fewest rows, counted in
    // the passes of equal size that its threads take for its units (2 % per part for the
    // operand staged once per CTA that shares an aggregate, 2 % per pass for its barriers).
    // Without the passes 16^3x32 at nv = 16 was cut in two: 10 units a CTA in two passes
    // on 103 SMs, 125 us per iteration; in four parts 14 on 147 SMs, 94 us.
    int rsp = 1, per = 1;
    double best = 1e30;
    for (int r = 1; r <= ngrp; ++r) {
        if (ngrp % r) continue;
        const int share = (Vc * r + sms - 1) / sms, fit = std::max(1, most / (9 * (ngrp / r)));
        const int passes = (share + fit - 1) / fit, units = (share + passes - 1) / passes;
        const double cost = (double)(units * passes) / r * (1.0 + 0.02 * r + 0.02 * passes);
        if (cost < best) { best = cost; rsp = r; per = units; }
    }
    // columns in bs parts while the busiest CTA's units leave threads idle
    const int ngl = ngrp / rsp;
    int bs = 1;
    while (bs < 8 && 2 * bs * 4 <= nc && 9 * ngl * 2 * bs * per <= most) bs *= 2;
    return CgnrSplit{per, rsp, bs};
}

// shared memory of a CTA less the kernel's static arrays
constexpr size_t kResidentSmem = 226 * 1024;

// grid: co-resident CTAs for this split (FP64: one per SM), then the smallest
// balanced grid covering all units
template <typename T, bool H16, bool EO, bool RES>
cudaError_t cgnr_launch_as(const CgnrArgs<T>& args, const CgnrSplit& sp, int batches, size_t sm, cudaStream_t st) {
    const int thr = cgnr_block_threads<T, H16>(args.nc, sp);
    const void* fn = (const void*)k_cgnr_persistent<T, H16, EO, RES>;
    if (sm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    int per = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, thr, sm);
    if (e != cudaSuccess) return e;
    const int gmax = (sizeof(T) == 8 ? std::min(per, 1) : per) * device_sm_count();
    if (gmax <= 0) return cudaErrorCooperativeLaunchTooLarge;
    const int rounds = (batches + gmax - 1) / gmax;                    // pieces per CTA
    CgnrArgs<T> a = args;
    a.upb = sp.upb; a.rsp = sp.rsp; a.bs = sp.bs;
    void* params[] = {&a};
    note_launch();
    return cudaLaunchCooperativeKernel(fn, dim3((batches + rounds - 1) / rounds), dim3(thr), params, sm, st);
}
template <typename T, bool H16, bool EO> cudaError_t cgnr_launch(const CgnrArgs<T>& args, cudaStream_t st) {
    const int nc = args.nc, sms = device_sm_count(), nsite = EO ? args.g.Vc / 2 : args.g.Vc;   // a red-black half
    const CgnrSplit sp = cgnr_split<T, H16>(nc, nsite, sms);
    const size_t sm = cgnr_smem<T, H16>(nc, sp);
    const int batches = (nsite * sp.rsp + sp.upb - 1) / sp.upb;   // CTA-sized pieces of work
    if constexpr (sizeof(T) == 8) {
        // One piece per CTA whose operator fits beside the operand: from global memory
        // 42.7 us per iteration on 8^4 (nv 8, red-black) and 32.6 on 12^3 x 24 (nv 12),
        // from shared memory 37.8 and 29.0.
        const size_t nstage = 9 * (size_t)nc * ((sp.upb + 2 * sp.rsp - 2) / sp.rsp);
        const size_t smr = sm + (EO ? 2 : 1) * (sizeof(v2<T>) * sp.upb * 9 * res_block(nc, nc / sp.rsp) +
                                                sizeof(unsigned int) * nstage);
        if (batches <= sms && smr <= kResidentSmem) return cgnr_launch_as<T, H16, EO, true>(args, sp, batches, smr, st);
    }
    return cgnr_launch_as<T, H16, EO, false>(args, sp, batches, sm, st);
}
template <> cudaError_t cgnr_persistent<float>(const CgnrArgs<float>& a, cudaStream_t st) {
    if (a.A16) {
        if (a.nc % 4 != 0) return cudaErrorInvalidValue;
        return a.ord ? cgnr_launch<float, true, true>(a, st) : cgnr_launch<float, true, false>(a, st);
    }
    return a.ord ? cgnr_launch<float, false, true>(a, st) : cgnr_launch<float, false, false>(a, st);
}
template <> cudaError_t cgnr_persistent<double>(const CgnrArgs<double>& a, cudaStream_t st) {
    return a.ord ? cgnr_launch<double, false, true>(a, st) : cgnr_launch<double, false, false>(a, st);
}

// coarse neighbour table nbr[X][d] (d = 0 self, 1+2mu / 2+2mu: +mu / -mu)
__global__ void k_coarse_nbr(int* nbr, Geom g) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < g.Vc * 9) nbr[i] = coarse_neighbour(g, i / 9, i % 9);
}
void coarse_neighbour_table(int* nbr, const Geom& g, cudaStream_t st) {
    note_launch();
    k_coarse_nbr<<<(g.Vc * 9 + 255) / 256, 256, 0, st>>>(nbr, g);
}

// FP16 copy of the coarse operator with one scale per (X, d) block: A16 = A / s, s = max |Re, Im|
__global__ void k_coarse_pack16(__half2* A16, float* s16, const double2* __restrict__ A, int nc) {
    __shared__ double sh[33];
    const size_t blk = blockIdx.x, nn = (size_t)nc * nc;
    const double2* Ab = A + blk * nn;
    double mx = 0;
    for (size_t i = threadIdx.x; i < nn; i += blockDim.x) mx = fmax(mx, fmax(fabs(Ab[i].x), fabs(Ab[i].y)));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, sh[w]);
        sh[32] = m > 0 ? m : 1.0;
        s16[blk] = (float)sh[32];
    }
    __syncthreads();
    const double inv = 1.0 / (double)(float)sh[32];
    for (size_t i = threadIdx.x; i < nn; i += blockDim.x)
        A16[blk * nn + i] = __floats2half2_rn((float)(Ab[i].x * inv), (float)(Ab[i].y * inv));
}
void coarse_pack16(__half2* A16, float* s16, const double2* A, int nc, int Vc, cudaStream_t st) {
    note_launch();
    k_coarse_pack16<<<Vc * 9, 256, 0, st>>>(A16, s16, A, nc);
}



}  // namespace wmg
