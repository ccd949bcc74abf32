// Red-black form of a coarse operator D_c (nearest neighbour on a lattice of even
// extents): the odd sites are eliminated exactly, and the coarse solver of a
// multigrid solve runs CG on the normal equations of the even-site Schur complement
//   Dhat = A_ee - A_eo A_oo^-1 A_oe,   Dhat^dag = sigma3 Dhat sigma3,
// whose condition number is about half that of D_c, so that CG takes about half
// the iterations at the same number of operator bytes per iteration.  The residual
// of the reconstructed solution vanishes on the odd sites and is the Schur
// residual on the even ones, so the solver's stopping test is unchanged.
//
// H[X][d] holds all of it in the layout of the operator itself: on an even site
// H[X][0] = A[X][0] and H[X][d] = -A[X][d]; on an odd site H[X][0] = A[X][0]^-1 and
// H[X][d] = A[X][0]^-1 A[X][d] (d = 1..8).  One application of Dhat is then two
// half-lattice stencils with the same blocks as D_c,
//   t_o = sum_{d >= 1} H[o][d] x[o + d],   y_e = H[e][0] x_e + sum_{d >= 1} H[e][d] t[e + d].
#include <algorithm>

#include "mg_launch.h"

namespace wmg {

bool schur_supported(const Geom& g) {
    for (int m = 0; m < 4; ++m)
        if (g.Lc[m] % 2) return false;
    return g.Vc >= 2;
}
__device__ __forceinline__ int site_parity(const Geom& g, int X) {
    int xc[4];
    coarse_coords(g, X, xc);
    return (xc[0] + xc[1] + xc[2] + xc[3]) & 1;
}
// ord[i], i < Vc/2: the even sites, then the odd ones, both in lexicographic order.
// Sites 2 j and 2 j + 1 differ in x only (even extent): one of each parity.
__global__ void k_parity_order(int* ord, Geom g) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= g.Vc / 2) return;
    const int p = site_parity(g, 2 * j);
    ord[j] = 2 * j + p;
    ord[g.Vc / 2 + j] = 2 * j + (p ^ 1);
}
void parity_order(int* ord, const Geom& g, cudaStream_t st) {
    note_launch();
    k_parity_order<<<(g.Vc / 2 + 255) / 256, 256, 0, st>>>(ord, g);
}

// One CTA per site; an odd one inverts its diagonal block (Gauss-Jordan in place with
// row pivoting, the block in shared memory) and multiplies it with the hop blocks, all
// in FP64: an operator stored in 32 or 16 bits is then rounded once, as D_c is.  Bound
// by the FP64 pipe, two operations per clock and SM: 1.8 M clocks per site at nc = 48.
// *growth receives, as the bits of a float, the largest over the odd sites of
// max |H[o][d]|, d >= 1, and max |A_oo^-1| max |A_oo|: how much larger than D_c's own the
// errors of the form's stored blocks can be (infinite for a singular block).
constexpr int kSchurThreads = 256;
constexpr float kInfinite = 3.0e38f;   // "no bound": above every accepted growth
__device__ __forceinline__ float finite_or_infinite(float x) { return x < kInfinite ? x : kInfinite; }   // NaN too
__device__ __forceinline__ float abs_bound(double2 v) {
    return finite_or_infinite((float)fabs(v.x) + (float)fabs(v.y));
}
__global__ void __launch_bounds__(kSchurThreads) k_schur(double2* __restrict__ H, const double2* __restrict__ A, int nc,
                                                         Geom g, int* growth) {
    extern __shared__ unsigned char smem_raw[];
    double2* M = reinterpret_cast<double2*>(smem_raw);          // M[i * nc + j]
    double2* col = M + (size_t)nc * nc;
    int* piv = reinterpret_cast<int*>(col + 2 * nc);
    double2* Bs = reinterpret_cast<double2*>(piv + ((nc + 3) & ~3));   // the inverse, [c][a]
    double2* As = Bs + (size_t)nc * nc;                         // a hop block, [b][c]
    __shared__ int s_p;
    __shared__ float s_max[kSchurThreads / 32];
    const int X = blockIdx.x, t = threadIdx.x, nn = nc * nc;
    const double2* Ax = A + (size_t)X * 9 * nn;
    double2* Hx = H + (size_t)X * 9 * nn;
    if (!site_parity(g, X)) {
        for (int i = t; i < 9 * nn; i += kSchurThreads) {
            const double2 v = Ax[i];
            Hx[i] = i < nn ? v : make_double2(-v.x, -v.y);
        }
        return;
    }
    float ma = 0.f, mi = 0.f, mh = 0.f;   // this thread's max |A_oo|, |A_oo^-1|, |H[o][d]|
    for (int i = t; i < nn; i += kSchurThreads) {   // A[b][a] -> M[a][b]
        M[(i % nc) * nc + i / nc] = Ax[i];
        ma = fmaxf(ma, abs_bound(Ax[i]));
    }
    __syncthreads();
    for (int k = 0; k < nc; ++k) {
        if (t < 32) {   // pivot: the largest |M[i][k]|^2, i >= k (the first of equals)
            double best = -1.0;
            int at = k;
            for (int i = k + t; i < nc; i += 32) {
                const double2 v = M[i * nc + k];
                const double q = v.x * v.x + v.y * v.y;
                if (q > best) { best = q; at = i; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                const double q = __shfl_xor_sync(0xffffffffu, best, o);
                const int i = __shfl_xor_sync(0xffffffffu, at, o);
                if (q > best || (q == best && i < at)) { best = q; at = i; }
            }
            if (t == 0) {
                s_p = at;
                piv[k] = at;
                if (!(best > 0.0) || best > 1e300) atomicMax(growth, __float_as_int(kInfinite));
            }
        }
        __syncthreads();
        const int p = s_p;
        for (int j = t; j < nc; j += kSchurThreads) {   // rows k and p change places; row k times 1 / pivot below
            const double2 v = M[k * nc + j];
            M[k * nc + j] = M[p * nc + j];
            if (p != k) M[p * nc + j] = v;
        }
        __syncthreads();
        const double2 d = M[k * nc + k];
        const double q = 1.0 / (d.x * d.x + d.y * d.y);
        const double2 inv = make_double2(d.x * q, -d.y * q);
        for (int i = t; i < nc; i += kSchurThreads) {
            col[i] = M[i * nc + k];
            const double2 v = M[k * nc + i];
            col[nc + i] = i == k ? inv : make_double2(v.x * inv.x - v.y * inv.y, v.x * inv.y + v.y * inv.x);
        }
        __syncthreads();
        for (int e = t; e < nn; e += kSchurThreads) {
            const int i = e / nc, j = e - i * nc;
            const double2 r = col[nc + j];
            if (i == k) {
                M[e] = r;
            } else {
                const double2 c = col[i];
                double2 v = j == k ? make_double2(0.0, 0.0) : M[e];
                v.x -= c.x * r.x - c.y * r.y;
                v.y -= c.x * r.y + c.y * r.x;
                M[e] = v;
            }
        }
        __syncthreads();
    }
    for (int k = nc - 1; k >= 0; --k) {   // undo the row exchanges on the columns
        const int p = piv[k];
        if (p != k)
            for (int i = t; i < nc; i += kSchurThreads) {
                const double2 v = M[i * nc + k];
                M[i * nc + k] = M[i * nc + p];
                M[i * nc + p] = v;
            }
        __syncthreads();
    }
    for (int i = t; i < nn; i += kSchurThreads) {
        const int b = i / nc, a = i - b * nc;
        const double2 v = M[a * nc + b];
        Hx[i] = v;
        Bs[i] = v;
        mi = fmaxf(mi, abs_bound(v));
    }
    for (int dd = 1; dd < 9; ++dd) {
        __syncthreads();
        for (int i = t; i < nn; i += kSchurThreads) As[i] = Ax[(size_t)dd * nn + i];
        __syncthreads();
        // two rows and two columns per thread (nc is even)
        for (int i = t; i < nn / 4; i += kSchurThreads) {
            const int b = 2 * (i / (nc / 2)), a = 2 * (i % (nc / 2));
            cx<double> s00(0, 0), s01(0, 0), s10(0, 0), s11(0, 0);
            for (int c = 0; c < nc; ++c) {
                const cx<double> b0 = ld<double>(Bs + c * nc + a), b1 = ld<double>(Bs + c * nc + a + 1);
                const cx<double> a0 = ld<double>(As + b * nc + c), a1 = ld<double>(As + (b + 1) * nc + c);
                cmad(s00, b0, a0);
                cmad(s01, b1, a0);
                cmad(s10, b0, a1);
                cmad(s11, b1, a1);
            }
            double2* o = Hx + (size_t)dd * nn + (size_t)b * nc + a;
            st<double>(o, s00);
            st<double>(o + 1, s01);
            st<double>(o + nc, s10);
            st<double>(o + nc + 1, s11);
            for (int q = 0; q < 4; ++q) mh = fmaxf(mh, abs_bound(o[(q >> 1) * nc + (q & 1)]));
        }
    }
    // one value per CTA: fmax((max ma) (max mi), max mh)
    auto block_max = [&](float v) {
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        __syncthreads();
        if ((t & 31) == 0) s_max[t >> 5] = v;
        __syncthreads();
        for (int w = 0; w < kSchurThreads / 32; ++w) v = fmaxf(v, s_max[w]);
        return v;
    };
    ma = block_max(ma);
    mi = block_max(mi);
    mh = block_max(mh);
    if (t == 0) atomicMax(growth, __float_as_int(finite_or_infinite(fmaxf(ma * mi, mh))));
}
cudaError_t schur_build(double2* H, const double2* A, int nc, const Geom& g, int* growth, cudaStream_t st) {
    const size_t sm = sizeof(double2) * (3 * (size_t)nc * nc + 2 * nc) + 4 * ((nc + 3) & ~3);
    cudaError_t e = cudaFuncSetAttribute(k_schur, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    note_launch();
    k_schur<<<g.Vc, kSchurThreads, sm, st>>>(H, A, nc, g, growth);
    return cudaGetLastError();
}

// out[X] = base[X] + sign * sum_{d0 <= d < d1} H[X][d] in[X + d] over the sites of one
// parity (base may be null): the pieces around the Schur solve,
//   v_o = A_oo^-1 r_o,  rhat_e = r_e - A_eo v_o,  y_o = v_o - A_oo^-1 A_oe y_e.
// One CTA per site, the rows over the lanes, the columns of the blocks over groups
// of nc threads; bound by the blocks' bytes, read once.
constexpr int kRowGroups = 8, kRowCols = 4;   // threads of a row, panel columns per read of the blocks
template <typename T, int NC>
__global__ void k_schur_rows(v2<T>* out, const v2<T>* base, const v2<T>* __restrict__ H, const v2<T>* in,
                             const int* __restrict__ sites, const int* __restrict__ nbr, int nc, int d0, int d1, T sign,
                             int cols, size_t cstride) {
    extern __shared__ unsigned char smem_raw[];
    v2<T>* xs = reinterpret_cast<v2<T>*>(smem_raw);       // [d][b][NC]
    v2<T>* part = xs + 9 * nc * NC;                       // [group][a][NC]
    const int X = sites[blockIdx.x], K = (d1 - d0) * nc, n0 = blockIdx.y * NC, ncol = min(NC, cols - n0);
    for (int i = threadIdx.x; i < K * NC; i += blockDim.x) {
        const int k = i / NC, n = i - k * NC;
        v2<T> v; v.x = 0; v.y = 0;
        if (n < ncol) v = in[((size_t)__ldg(nbr + (size_t)X * 9 + d0 + k / nc) * nc + k % nc) * cstride + n0 + n];
        xs[i] = v;
    }
    __syncthreads();
    const int a = threadIdx.x % nc, grp = threadIdx.x / nc;
    if (grp < kRowGroups) {
        cx<T> s[NC];
#pragma unroll
        for (int n = 0; n < NC; ++n) s[n] = cx<T>(0, 0);
        const v2<T>* h = H + ((size_t)X * 9 + d0) * nc * nc + a;
#pragma unroll 4
        for (int k = grp; k < K; k += kRowGroups) {
            const cx<T> hk = ldg<T>(h + (size_t)k * nc);
#pragma unroll
            for (int n = 0; n < NC; ++n) cmad(s[n], hk, ld<T>(xs + k * NC + n));
        }
#pragma unroll
        for (int n = 0; n < NC; ++n) st<T>(part + (grp * nc + a) * NC + n, s[n]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nc * ncol; i += blockDim.x) {
        const int r = i / ncol, n = i - r * ncol;
        cx<T> s = ld<T>(part + r * NC + n);
        for (int q = 1; q < kRowGroups; ++q) s = s + ld<T>(part + (q * nc + r) * NC + n);
        const size_t o = ((size_t)X * nc + r) * cstride + n0 + n;
        s = sign * s;
        if (base) s = s + ld<T>(base + o);
        st<T>(out + o, s);
    }
}
template <typename T>
void schur_rows(v2<T>* out, const v2<T>* base, const v2<T>* H, const v2<T>* in, const int* sites, int nsites,
                const int* nbr, int nc, int d0, int d1, double sign, int cols, int cstride, cudaStream_t st) {
    const int thr = (kRowGroups * nc + 31) / 32 * 32;
    const size_t sm = sizeof(v2<T>) * (9 + kRowGroups) * nc;
    note_launch();
    if (cols > 1)
        k_schur_rows<T, kRowCols><<<dim3(nsites, (cols + kRowCols - 1) / kRowCols), thr, kRowCols * sm, st>>>(
            out, base, H, in, sites, nbr, nc, d0, d1, (T)sign, cols, cstride);
    else
        k_schur_rows<T, 1><<<nsites, thr, sm, st>>>(out, base, H, in, sites, nbr, nc, d0, d1, (T)sign, cols, cstride);
}
template void schur_rows<float>(v2<float>*, const v2<float>*, const v2<float>*, const v2<float>*, const int*, int, const int*,
                                int, int, int, double, int, int, cudaStream_t);
template void schur_rows<double>(v2<double>*, const v2<double>*, const v2<double>*, const v2<double>*, const int*, int,
                                 const int*, int, int, int, double, int, int, cudaStream_t);

}  // namespace wmg
