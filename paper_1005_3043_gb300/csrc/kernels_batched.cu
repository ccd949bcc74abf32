// Batched (multi right-hand side) coarse level: CG on the normal equations of
// D_c for a panel of right-hand sides, whole solve in one persistent cooperative
// launch, the stencil a dense contraction on the 5th-generation tensor cores.
//
// Panel layout: xB[X][b][n] complex FP32, n < npad (RHS index fastest).  For one
// aggregate X the stencil is
//   y[X][a][n] = sum_d sum_b A[X][d][a][b] x[X+d][b][n].
// As a real GEMM the rows are the real parts of A followed by the imaginary
// parts (M = 2 nc <= 96 of the MMA's 128), K = b, and a right-hand side is four
// columns: Re x and Im x, each split into FP16 hi + 2^-11 lo (22 bits; lo is kept times
// 2^11, so that it is a normal number wherever hi is):
//   D[a] = Re A x, D[nc + a] = Im A x,
//   Re y = D[a][Re] - D[nc + a][Im],  Im y = D[a][Im] + D[nc + a][Re].
// So neither the operator nor the operand is stored twice (the embedding
// [[Re, -Im], [Im, Re]] doubles the operator's bytes and its MMAs): at 16^3x32
// (Nv = 20) an aggregate's stencil reads 58 KB of operator and takes 27 MMAs of
// 128 x 64 x 16 for 16 right-hand sides.
//
// The operand is kept in global memory as FP16 tiles in the tensor-core layout,
// written once by the CTA that owns the aggregate when it computes the entries
// (scaled by a power of two per right-hand side from the last known norm), so a
// stencil only moves tiles: per direction one bulk copy of A[X][d] and one of the
// tile of x[X+d].
//
// Iteration: the Chronopoulos-Gear arrangement of CG on D_c^dag D_c (as the
// single-source solver): phase A u = D_c s, one exchange of (|u|^2, |s|^2, |r|^2)
// per right-hand side, phase B w = D_c^dag u and, in its epilogue,
//   p = s + beta p, z = w + beta z, q = u + beta q, y += alpha p, r -= alpha q,
//   s -= alpha z,
// two grid barriers per iteration.  Separate kernels for the split, the stencil,
// the reductions and the updates (ten launches per iteration, replayed from a
// graph) took 76 us per iteration on 16^3x32 with 12 sources (Nv = 16), 34 us of it
// in each stencil, and 64 us on 8^3x16 with 21 sources, all latency; this kernel
// takes 29 and 16 us (red-black, four barriers: 38 and 31 us for less than half the
// iterations).
// What is left: about 1.2 us per job (copies, 18 MMAs and the epilogue overlap), 2 to
// 3 us per grid barrier.
#include <cuda_fp16.h>

#include <algorithm>

#include "mg_launch.h"
#include "mg_ptx.cuh"

namespace wmg {

// ---------------------------------------------------------------- operator tiles
// At[X][d][kc][rg][8][8]: core matrices (8 rows x 8 K, 128 bytes) of one K group
// kc adjacent over the row groups rg; row a the real part of row a of A, row
// nc + a the imaginary part.  The nine blocks of an aggregate add up in one
// accumulator, so they share one scale, its inverse in as[X]: a power of two that brings
// the largest of their entries to [2^14, 2^15), or (top) the one that brings it to 2^15.
// An entry keeps its 11 bits down to 2^-28 of the largest, and none overflows.  top: the
// diagonal, all near the largest entry, is then rounded just below a power of two, where
// FP16 is finest (the correction of one source at mass 0.2, 12 x 16^2 x 10 with 2^4
// aggregates, is 4.7e-6 instead of 8.1e-6 off its FP64 value).
__global__ void __launch_bounds__(256) k_coarse_tiles(__half* At, float* as, const double2* __restrict__ A, int nc, bool top) {
    __shared__ float s_max[8];
    const int X = blockIdx.x, n = 9 * nc * nc;
    const double2* Ax = A + (size_t)X * n;
    float mx = 0.f;
    for (int i = threadIdx.x; i < n; i += blockDim.x) mx = fmaxf(mx, (float)fmax(fabs(Ax[i].x), fabs(Ax[i].y)));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = mx;
    __syncthreads();
    for (int w = 0; w < 8; ++w) mx = fmaxf(mx, s_max[w]);
    const bool fits = mx > 1e-30f && mx < 1e30f;
    const float s = !fits ? 1.f : top ? 0x1p-15f * mx : ldexpf(1.f, ilogbf(mx) - 14);
    const double f = 1.0 / (double)s;
    if (threadIdx.x == 0) as[X] = s;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int blk = i / (nc * nc), rem = i - blk * nc * nc, b = rem / nc, a = rem - b * nc;
        const double2 v = Ax[i];   // column-major block: A[b][a] = A_ab
        __half* t = At + ((size_t)X * 9 + blk) * 2 * nc * nc + (size_t)(b >> 3) * (nc >> 2) * 64 + (b & 7);
        const int m = nc + a;
        t[((a >> 3) << 6) + ((a & 7) << 3)] = __double2half(f * v.x);
        t[((m >> 3) << 6) + ((m & 7) << 3)] = __double2half(f * v.y);
    }
}
void coarse_tiles(__half* At, float* as, const double2* A, int nc, int Vc, bool top, cudaStream_t st) {
    note_launch();
    k_coarse_tiles<<<Vc, 256, 0, st>>>(At, as, A, nc, top);
}

// ---------------------------------------------------------------- the persistent kernel
// Warps: 0 copies the operator's tiles and 1 the operand's, a lane per direction; 2
// and 3 issue the MMAs of every second job each (lane 0); 4..11 the epilogue.  One
// thread for all copies and one for all MMAs were the pipeline's rate: 2.5 us per
// job at 16^3x32, 12 sources.
constexpr int kEpiWarps = 8, kEpi = 32 * kEpiWarps, kEpi0 = 128, kBcgThreads = kEpi0 + kEpi;
constexpr int kBcgMaxStages = 16;
constexpr long long kBcgWait = 20000000LL;    // polls of a wait before it gives up
constexpr int kBcgStatic = 1024;              // barriers, flags

// shared memory of a shape: stages of (operator, operand) tiles, then T (the
// products of one job), S2 (entries on their way into the tile), the column
// sums and the per-column scalars
struct BcgSmem {
    int kcp;            // K groups of a stage (nc / 8 rounded up to even, the last one zero)
    uint32_t a_bytes, b_bytes, stage, a_copy, b_copy;
    size_t off_t, off_s2, off_acc, off_col, total;
    int ts, rgs;
    __host__ __device__ BcgSmem(int nc, int nw, int npad, int stages) {
        kcp = ((nc >> 3) + 1) & ~1;
        a_copy = (uint32_t)nc * nc * 4;            // (nc / 8) x (2 nc x 8) halves
        b_copy = (uint32_t)nc * nw * 8;            // (nc / 8) x (4 nw x 8) halves
        a_bytes = (uint32_t)kcp * nc * 32;
        b_bytes = (uint32_t)kcp * nw * 64;
        if (b_bytes < 2048) b_bytes = 2048;        // the 128-row MMA reads up to 1.8 KB past the operator rows
        stage = a_bytes + b_bytes;
        ts = nw + 1;
        rgs = kEpi / nw;
        off_t = (size_t)stages * stage;
        off_s2 = off_t + (size_t)2 * nc * ts * 8;
        off_acc = off_s2 + (size_t)nc * ts * 8;
        off_col = off_acc + (size_t)3 * rgs * npad * 8;
        off_col = (off_col + 15) & ~(size_t)15;
        total = off_col + (size_t)npad * (3 * 8 + 13 * 4);
    }
};

__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// barrier of the epilogue warps; the return value is the OR of p over them
__device__ __forceinline__ bool epi_sync(bool p = false) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"((uint32_t)p), "n"(kEpi)
        : "memory");
    return r != 0;
}
// 8 consecutive FP32 columns of this thread's TMEM lane; tmem_wait_ld before use
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}
// waits for this thread's loads; the registers pass through, so that no use of
// them moves above the wait
__device__ __forceinline__ void tmem_wait_ld8(uint32_t (&a)[8], uint32_t (&b)[8], uint32_t (&c)[8], uint32_t (&d)[8]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(a[0]), "+r"(a[1]), "+r"(a[2]), "+r"(a[3]), "+r"(a[4]), "+r"(a[5]), "+r"(a[6]), "+r"(a[7]),
                   "+r"(b[0]), "+r"(b[1]), "+r"(b[2]), "+r"(b[3]), "+r"(b[4]), "+r"(b[5]), "+r"(b[6]), "+r"(b[7])
                 :
                 : "memory");
    asm volatile(""
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]), "+r"(c[4]), "+r"(c[5]), "+r"(c[6]), "+r"(c[7]),
                   "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3]), "+r"(d[4]), "+r"(d[5]), "+r"(d[6]), "+r"(d[7])
                 :
                 : "memory");
}
// wait for a phase of an mbarrier: false when the CTA's fail flag is up or the
// poll limit is reached (the flag and the launch's error flag are then raised)
__device__ __forceinline__ bool bcg_wait(uint64_t* bar, uint32_t parity, volatile int* fail, int* err) {
    for (long long i = 0; i < kBcgWait; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63) == 63) {
            if (*fail) return false;
            __nanosleep(20);
        }
    }
    *fail = 1;
    atomicExch(err, 1);
    return false;
}
// until *count reaches want (it only grows); false as bcg_wait.  The counts order waits
// on mbarriers, no data: what a thread reads after its wait it acquires there.  Not
// inlined: the loop of the MMA threads stays as short as it was (0.5 us per phase).
__device__ __noinline__ bool wait_count(const unsigned int* count, unsigned int want, volatile int* fail, int* err) {
    for (long long i = 0;; ++i) {
        unsigned int have;
        asm volatile("ld.relaxed.cta.shared::cta.u32 %0, [%1];" : "=r"(have) : "r"(smem_u32(count)) : "memory");
        if ((int)(have - want) >= 0) return true;
        if (*fail) return false;
        if (i > kBcgWait) {
            *fail = 1;
            atomicExch(err, 1);
            return false;
        }
        if (i > 64) __nanosleep(20);
    }
}
// sum in two floats (Knuth's two-sum): the column sums run over many aggregates
// and CTAs, and FP64 adds are two per clock and SM here
struct Sum2 {
    float h, l;
};
__device__ __forceinline__ void add2(Sum2& s, float x) {
    const float t = s.h + x, b = t - s.h;
    s.l += (s.h - (t - b)) + (x - b);
    s.h = t;
}
// power of two near 2^-5 sqrt(rows / s): entries of a column with |x|^2 = s then have
// rms about 2^-5, 2^9 above the FP16 subnormal range, with room for a column
// concentrated on one site that grows some 10^3 times from one scale to the next
__device__ __forceinline__ float col_scale(double s, float rows) {
    const float x = 0x1p-10f * rows / (float)s;
    if (!(x > 1e-38f) || !(x < 1e38f)) return 1.f;
    return __int_as_float((127 + ((((__float_as_int(x) >> 23) & 255) - 127) >> 1)) << 23);
}
__device__ __forceinline__ uint32_t half_pair(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// units of a fixed-point grid sum whose last value was s: 2^36 / s to a power of two
__device__ __forceinline__ float unit_of(float s) {
    if (!(s > 0.f)) return 0x1p42f;
    const int e = ((__float_as_int(s) >> 23) & 255) - 127;
    return __int_as_float((127 + min(36 - e, 120)) << 23);
}

struct BcgCta {
    const BcgArgs& a;
    const BcgSmem L;
    int nc, nvh, nw, nch, j0, j1;
    unsigned char* sm;
    uint64_t *full, *empty, *acc_full, *acc_empty, *gate;
    volatile int *fail, *stop;
    unsigned int *passed, *entered;   // progress of the two MMA threads: items, phases

    __device__ BcgCta(const BcgArgs& args, unsigned char* smem, uint64_t* bars, int* flags)
        : a(args), L(args.nc, args.nw, args.npad, args.stages), sm(smem) {
        nc = a.nc; nvh = nc >> 1; nw = a.nw; nch = a.npad / nw;
        const long long NJ = (long long)(a.ord ? a.g.Vc / 2 : a.g.Vc) * nch;
        j0 = (int)(blockIdx.x * NJ / gridDim.x);
        j1 = (int)((blockIdx.x + 1) * NJ / gridDim.x);
        full = bars; empty = bars + kBcgMaxStages; acc_full = bars + 2 * kBcgMaxStages; acc_empty = acc_full + 2;
        gate = acc_empty + 2;
        fail = flags; stop = flags + 1;
        passed = reinterpret_cast<unsigned int*>(flags) + 2; entered = passed + 2;
    }

    // Phases.  A stencil is one phase over all sites, or, in the red-black form, a phase
    // over the odd sites (their eight neighbours, all even) and one over the even sites
    // (the site itself and its neighbours); a phase has the same jobs in every CTA's
    // share, nd items (directions 9 - nd ..) per job.
    __device__ int dirs(int phase) const { return a.ord && !(phase & 1) ? 8 : 9; }
    __device__ int site(int phase, int job) const {
        const int i = job / nch;
        return a.ord ? __ldg(a.ord + ((phase & 1) ? 0 : a.g.Vc / 2) + i) : i;
    }
    // operand of the phase's stencil: the adjoint's (btu) and D's (bts) take turns
    __device__ const __half* operand(int phase) const {
        const int stencil = a.ord ? phase >> 1 : phase;
        return ((stencil & 1) != (a.first_dag != 0)) ? a.btu : a.bts;
    }

    // ------------------------------------------------------------ copies (two warps)
    // Items (job, direction) in order, item i of the launch in stage i % stages, whose
    // "full" barrier takes one arrival and the bytes of each tile.  Both warps run over
    // all items, up to `stages` directions at a time (so that no lane waits for what
    // another lane of its round has yet to copy).  The operator does not depend on the
    // iteration: its tiles run ahead across the grid barriers, as far as stages are
    // free; the operand's wait for the gate of each phase.
    __device__ void copy_operator(unsigned int* b_items) {
        const int S = a.stages, lane = threadIdx.x & 31;
        const size_t blk = (size_t)2 * nc * nc;
        unsigned int next = 0;      // items armed
        bool ok = true;
        for (int phase = 0; ok; ++phase) {
            const int nd = dirs(phase), R = min(S, nd);
            for (int j = j0; j < j1 && ok; ++j) {
                const int X = site(phase, j);
                for (int l0 = 0; l0 < nd && ok; l0 += R) {
                    const int n = min(R, nd - l0);
                    const unsigned int i = next + lane, k = i / S;
                    const int st = (int)(i - k * S), d = 9 - nd + l0 + lane;
                    // all lanes of a round or none, so that `next` is the number armed
                    ok = __all_sync(0xffffffffu, lane >= n || i < (unsigned int)S || wait_stop(empty + st, (k - 1) & 1u));
                    if (ok) {
                        if (lane < n) {
                            mbar_expect_tx(full + st, L.a_copy);
                            bulk_copy_g2s(sm + (size_t)st * L.stage, a.At + ((size_t)X * 9 + d) * blk, L.a_copy, full + st);
                        }
                        next += n;
                    }
                }
            }
        }
        // drain: the tiles that no operand joined (the arrival that is missing is made
        // here); after a failure, time enough for any copy to land
        asm volatile("barrier.cta.sync 2, 64;" ::: "memory");
        if (*fail) {
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);
            return;
        }
        for (unsigned int i = *b_items + lane; i < next; i += 32) {
            const unsigned int k = i / S;
            const int st = (int)(i - k * S);
            mbar_arrive(full + st);
            mbar_wait(full + st, k & 1u, kBcgWait);
        }
    }
    __device__ void copy_operand(unsigned int* b_items) {
        const int S = a.stages, lane = threadIdx.x & 31;
        const size_t tile = (size_t)4 * nc * nw;
        unsigned int next = 0;
        uint32_t gate_par = 0;
        bool ok = true;
        for (int phase = 0; ok; ++phase, gate_par ^= 1u) {
            if (!__all_sync(0xffffffffu, bcg_wait(gate, gate_par, fail, a.err)) || *stop) break;
            fence_proxy_async_all();    // tiles written by other CTAs before the grid barrier
            const __half* bt = operand(phase);
            const int nd = dirs(phase), R = min(S, nd);
            for (int j = j0; j < j1 && ok; ++j) {
                const int X = site(phase, j), c = j - j / nch * nch;
                for (int l0 = 0; l0 < nd && ok; l0 += R, next += R) {
                    const int n = min(R, nd - l0);
                    bool mine = true;
                    if (lane < n) {
                        const unsigned int i = next + lane, k = i / S;
                        const int st = (int)(i - k * S), Y = __ldg(a.nbr + (size_t)X * 9 + 9 - nd + l0 + lane);
                        mine = i < (unsigned int)S || bcg_wait(empty + st, (k - 1) & 1u, fail, a.err);
                        if (mine) {
                            mbar_expect_tx(full + st, L.b_copy);
                            bulk_copy_g2s(sm + (size_t)st * L.stage + L.a_bytes, bt + ((size_t)Y * nch + c) * tile,
                                          L.b_copy, full + st);
                        }
                    }
                    ok = __all_sync(0xffffffffu, mine);
                    if (n < R) next -= R - n;
                }
            }
        }
        if (lane == 0) *b_items = next;
        asm volatile("barrier.cta.sync 2, 64;" ::: "memory");
    }
    // as bcg_wait; false without an error when the launch has ended
    __device__ bool wait_stop(uint64_t* bar, uint32_t parity) {
        for (long long i = 0; i < kBcgWait; ++i) {
            if (mbar_try_wait(bar, parity)) return true;
            if (*fail || *stop) return false;
            if (i > 64) __nanosleep(20);
        }
        *fail = 1;
        atomicExch(a.err, 1);
        return false;
    }

    __device__ void set_count(unsigned int* count, unsigned int v) {
        asm volatile("st.relaxed.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(count)), "r"(v) : "memory");
    }

    // ------------------------------------------------------------ MMAs (one thread of two warps)
    // A wait by parity tells a phase of a barrier from its neighbours only.  So a thread
    // waits for a stage that the job before also used only after the other thread has
    // passed its waits of that job (`passed`; without it a thread a job ahead took a
    // stage that had yet to be filled for that job for a full one: certain with fewer
    // stages than a job has directions; the copies come in order, so the other thread
    // is past them when the stage's tiles arrive), and the next
    // phase's gate opens only after both have passed this one's (`entered`; a phase of
    // one job has work for one of them).
    __device__ void multiply(uint32_t tmem, int which, uint64_t* drain) {
        const unsigned int S = a.stages, jobs = j1 - j0;
        const int nks = L.kcp >> 1;
        const uint32_t idesc = idesc_f16(128, 4 * nw), lbo_a = (uint32_t)nc * 32, lbo_b = (uint32_t)nw * 64;
        // descriptors of stage 0; the address field counts 16 bytes
        const uint64_t da0 = smem_desc(smem_u32(sm), lbo_a, 128), db0 = smem_desc(smem_u32(sm) + L.a_bytes, lbo_b, 128);
        const uint64_t step_a = lbo_a >> 3, step_b = lbo_b >> 3, step_st = L.stage >> 4;
        const uint32_t acc = tmem + (uint32_t)(which * 4 * nw);
        uint32_t gate_par = 0, acc_par = 1u;   // a fresh barrier passes a wait for parity 1
        unsigned int job = 0, base = 0;        // jobs and items before this phase
        int phase = 0;
        for (bool ok = true; ok; job += jobs, base += jobs * dirs(phase), ++phase) {
            if (!bcg_wait(gate, gate_par, fail, a.err)) break;
            set_count(entered + which, phase + 1);
            if (*stop) break;
            gate_par ^= 1u;
            const int nd = dirs(phase), dw = max((int)S - nd, 0);
            for (unsigned int j = (job ^ which) & 1u; j < jobs && ok; j += 2) {   // this warp's jobs: (job + j) odd or even
                if (!bcg_wait(acc_empty + which, acc_par, fail, a.err)) { ok = false; break; }
                acc_par ^= 1u;
                tc_fence_after();
                const unsigned int i0 = base + j * nd, k0 = i0 / S;
                unsigned int st = i0 - k0 * S;
                uint32_t par = k0 & 1u;
                uint64_t da = da0 + st * step_st, db = db0 + st * step_st;
                // items from dw on use stages that the job before used (item i0 + d - S)
                int d = 0, end = j > 0 ? min(dw, nd) : nd;
                for (;;) {
                    for (; d < end; ++d) {
                        if (!bcg_wait(full + st, par, fail, a.err)) { ok = false; break; }
                        tc_fence_after();
                        mma_f16(acc, da, db, idesc, d > 0 ? 1u : 0u);
                        if (nks > 1) mma_f16(acc, da + step_a, db + step_b, idesc, 1u);
                        if (nks > 2) mma_f16(acc, da + 2 * step_a, db + 2 * step_b, idesc, 1u);
                        mma_commit(empty + st);
                        da += step_st;
                        db += step_st;
                        if (++st == S) {
                            st = 0;
                            par ^= 1u;
                            da = da0;
                            db = db0;
                        }
                    }
                    if (!ok || end == nd) break;
                    if (!wait_count(passed + (which ^ 1), i0, fail, a.err)) { ok = false; break; }
                    end = nd;
                }
                if (ok) {
                    set_count(passed + which, i0 + nd);
                    mma_commit(acc_full + which);
                }
            }
        }
        mma_commit(drain);
        mbar_wait(drain, 0, kBcgWait);
    }

    // ------------------------------------------------------------ epilogue warps
    float2 *T, *S2;
    Sum2* acc;
    int t, n, rg, rgs;
    long long job_count = 0;
    unsigned int arrived = 0, opened = 0;

    // entries staged in S2[row][n] (scaled) -> the four FP16 rows of the tile.  A single
    // right-hand side (a.third): what its hi and lo leave, times 2^22, goes into the hi
    // rows of the unused column 1, so that its operand has the 24 bits of an FP32 number.
    __device__ __forceinline__ void write_tile(__half* bt, int X, int c) {
        if (a.third && c == 0) write_parts<true>(bt, X, c);
        else write_parts<false>(bt, X, c);
    }
    template <bool THIRD> __device__ void write_parts(__half* bt, int X, int c) {
        __half* base = bt + ((size_t)X * nch + c) * 4 * nc * nw;
        for (int i = t; i < (nc >> 3) * nw; i += kEpi) {
            const int kc = i / nw, m = i - kc * nw;
            uint32_t w[4][4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                float2 v[2];
                float hr[2], hi[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    v[q] = S2[(kc * 8 + 2 * e + q) * L.ts + (THIRD && m == 1 ? 0 : m)];
                    v[q].x = fminf(fmaxf(v[q].x, -65504.f), 65504.f);
                    v[q].y = fminf(fmaxf(v[q].y, -65504.f), 65504.f);
                    hr[q] = __half2float(__float2half_rn(v[q].x));
                    hi[q] = __half2float(__float2half_rn(v[q].y));
                    v[q].x = 0x1p11f * (v[q].x - hr[q]);
                    v[q].y = 0x1p11f * (v[q].y - hi[q]);
                    if (THIRD && m == 1) {
                        hr[q] = 0x1p11f * (v[q].x - __half2float(__float2half_rn(v[q].x)));
                        hi[q] = 0x1p11f * (v[q].y - __half2float(__float2half_rn(v[q].y)));
                        v[q] = make_float2(0.f, 0.f);
                    }
                }
                w[0][e] = half_pair(hr[0], hr[1]);
                w[1][e] = half_pair(hi[0], hi[1]);
                w[2][e] = half_pair(v[0].x, v[1].x);
                w[3][e] = half_pair(v[0].y, v[1].y);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int row = j * nw + m;
                *reinterpret_cast<uint4*>(base + ((size_t)(kc * (nw >> 1) + (row >> 3)) << 6) + ((row & 7) << 3)) =
                    make_uint4(w[j][0], w[j][1], w[j][2], w[j][3]);
            }
        }
    }

    // grid barrier of the epilogue warps (all writes before it visible to all reads
    // after it, tile writes to the bulk copies too); opens the gate of the next phase.
    // One thread's release covers the warps' writes (they are ordered before it by the
    // barrier of the warps), its acquire their reads.
    __device__ bool grid_barrier(bool open) {
        fence_proxy_async_all();
        if (epi_sync(*fail != 0)) return false;
        if (t == 0) {
            ++arrived;
            const unsigned int want = arrived * gridDim.x;
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
            long long spins = 0;
            unsigned int got;
            for (;;) {
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(a.bar) : "memory");
                if ((int)(got - want) >= 0) break;
                if (*(volatile int*)a.err) { *fail = 1; break; }
                if (++spins > kBcgWait) { *fail = 1; atomicExch(a.err, 1); break; }
                if (spins > 64) __nanosleep(20);
            }
            fence_proxy_async_all();
            if (open && !*fail) next_phase();
        }
        return !epi_sync(*fail != 0);
    }
    __device__ void next_phase() {   // thread 0
        if (wait_count(entered, opened, fail, a.err) && wait_count(entered + 1, opened, fail, a.err)) {
            ++opened;
            mbar_arrive(gate);
        }
    }
    __device__ void open_gate() {
        if (t == 0) next_phase();
    }

    // products of the next job (column chunk c) into T, in units of the operator's scale
    // (unit); false on failure (uniform over the warps)
    __device__ float unit(int X) const { return __ldg(a.as + X); }
    __device__ bool take(uint32_t tmem, int c) {
        const int buf = (int)(job_count & 1), warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        const int quad = warp & 3, half = (warp - 4) >> 2, m = 32 * quad + lane;
        const bool ok = __all_sync(0xffffffffu, bcg_wait(acc_full + buf, (uint32_t)((job_count >> 1) & 1), fail, a.err));
        tc_fence_after();
        if (ok && 32 * quad < 2 * nc) {
            const uint32_t base = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)(buf * 4 * nw);
            for (int c0 = 8 * half; c0 < nw; c0 += 16) {
                uint32_t rh[8], ih[8], rl[8], il[8];
                tmem_ld8(base + c0, rh);
                tmem_ld8(base + nw + c0, ih);
                tmem_ld8(base + 2 * nw + c0, rl);
                tmem_ld8(base + 3 * nw + c0, il);
                tmem_wait_ld8(rh, ih, rl, il);
                if (a.third && c == 0 && c0 == 0) {
                    rl[0] = __float_as_uint(__uint_as_float(rl[0]) + 0x1p-11f * __uint_as_float(rh[1]));
                    il[0] = __float_as_uint(__uint_as_float(il[0]) + 0x1p-11f * __uint_as_float(ih[1]));
                    rh[1] = ih[1] = 0u;
                }
                if (m < 2 * nc)
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        T[(size_t)m * L.ts + c0 + e] =
                            make_float2(__uint_as_float(rh[e]) + 0x1p-11f * __uint_as_float(rl[e]),
                                        __uint_as_float(ih[e]) + 0x1p-11f * __uint_as_float(il[e]));
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty + buf);
        ++job_count;
        return !epi_sync(!ok);
    }
    __device__ __forceinline__ float2 product(int r, float inv, bool dag) const {
        const float2 x = T[(size_t)r * L.ts + n], w = T[(size_t)(nc + r) * L.ts + n];
        const float f = dag && r >= nvh ? -inv : inv;
        return make_float2(f * (x.x - w.y), f * (x.y + w.x));
    }
    __device__ __forceinline__ void stage(int r, float2 v, float sc, bool dag) {
        const float f = dag && r >= nvh ? -sc : sc;
        S2[r * L.ts + n] = make_float2(f * v.x, f * v.y);
    }
    __device__ __forceinline__ Sum2& col_acc(int val, int col) { return acc[((size_t)val * rgs + rg) * a.npad + col]; }

    // Grid sums of the column sums, in 64-bit fixed point: integer adds give the same
    // sum in any order, so a CTA adds its share with one atomic per value and reads the
    // sums after the grid barrier.  (Every CTA adding up all CTAs' partial sums in a
    // fixed order took 5-7 us per iteration at 152 x 48 values.)  The unit of a value
    // is 2^-36 of its last grid sum, at first of the largest CTA's share (publish_size),
    // so a sum keeps more bits than its FP32 terms have; a value out of range (it grew
    // 2^19 times in one iteration, or is not finite) marks its column, which ends there.
    __device__ void publish(const float* fx, unsigned long long* sums) {
        epi_sync();
        for (int i = t; i < 3 * a.npad; i += kEpi) {
            const int v = i / a.npad, c = i - v * a.npad;
            Sum2 s{0.f, 0.f};
            for (int g = 0; g < rgs; ++g) {
                Sum2& e = acc[((size_t)v * rgs + g) * a.npad + c];
                add2(s, e.h);
                s.l += e.l;
                e = Sum2{0.f, 0.f};
            }
            const float h = s.h * fx[i], l = s.l * fx[i];
            if (!(fabsf(h) < 0x1p55f)) {
                atomicOr(a.bad + c, 1u);
                continue;
            }
            const long long q = __float2ll_rn(h) + __float2ll_rn(l);
            if (q != 0) atomicAdd(sums + i, (unsigned long long)q);
        }
    }
    // The largest CTA's share of a value's column sums into mx (float bits order as
    // integers; fabs: one sign for every NaN).
    __device__ void publish_size(int val, unsigned int* mx, bool clear) {
        epi_sync();
        for (int i = t; i < a.npad; i += kEpi) {
            float s = 0.f;
            for (int g = 0; g < rgs; ++g) {
                Sum2& e = acc[((size_t)val * rgs + g) * a.npad + i];
                s += e.h;
                if (clear) e = Sum2{0.f, 0.f};
            }
            atomicMax(mx + i, __float_as_uint(fabsf(s)));
        }
    }

    __device__ void epilogue(uint32_t tmem) {
        t = threadIdx.x - kEpi0;
        rgs = L.rgs;
        n = t % nw;
        rg = t / nw;
        const bool act = rg < rgs;
        T = reinterpret_cast<float2*>(sm + L.off_t);
        S2 = reinterpret_cast<float2*>(sm + L.off_s2);
        acc = reinterpret_cast<Sum2*>(sm + L.off_acc);
        const int np = a.npad, jobs = j1 - j0;
        double* gam = reinterpret_cast<double*>(sm + L.off_col);   // 1 / gamma, 1 / alpha of the last iteration, |r_0|^2
        double* alo = gam + np;
        double* rho0 = alo + np;
        float* fx = reinterpret_cast<float*>(rho0 + np);           // [3][npad] units of the grid sums (reciprocals)
        float* al = fx + 3 * np;                                   // alpha, beta of this iteration
        float* be = al + np;
        float* iss = be + np;                                      // 1 / scale of the s tile, of the u tile
        float* isu = iss + np;
        float* sc_s = isu + np;                                    // scales for the next s and u tiles
        float* sc_u = sc_s + np;
        float* fr = sc_u + np;                                     // power of two that brings rc to unit size
        float* sc_tu = fr + np;
        int* done = reinterpret_cast<int*>(sc_tu + np);               // 1: this column is frozen
        int* its = done + np;
        const float rows = (float)((double)a.g.Vc * nc);
        for (int i = t; i < 3 * rgs * np; i += kEpi) acc[i] = Sum2{0.f, 0.f};
        epi_sync();

        if (a.mode == BCG_APPLY) {   // y = D_c x (dag: D_c^dag x): tiles of x, one stencil
            for (int j = 0; j < jobs; ++j) {
                const int X = (j0 + j) / nch, c = j0 + j - X * nch;
                if (act)
                    for (int r = rg; r < nc; r += rgs)
                        stage(r, a.rc[((size_t)X * nc + r) * np + c * nw + n], 1.f, a.dag != 0);
                epi_sync();
                write_tile(a.dag ? a.btu : a.bts, X, c);
                epi_sync();
            }
            if (!grid_barrier(true)) return;
            for (int j = 0; j < jobs; ++j) {
                const int X = (j0 + j) / nch, c = j0 + j - X * nch;
                const float f = unit(X);
                if (!take(tmem, c)) return;
                if (act)
                    for (int r = rg; r < nc; r += rgs)
                        a.y[((size_t)X * nc + r) * np + c * nw + n] = product(r, f, a.dag != 0);
                epi_sync();
            }
            if (t == 0) *stop = 1;
            epi_sync();
            open_gate();
            return;
        }

        // entry o of column col of the right-hand side that the tolerance refers to, at the
        // job's site and, red-black, at its odd counterpart
        const bool eo = a.ord != nullptr;
        auto full2 = [&](int j, int r, int col) {
            const int i = (j0 + j) / nch;
            const float2 v = a.rc_full[((size_t)(eo ? __ldg(a.ord + i) : i) * nc + r) * np + col];
            float q = v.x * v.x + v.y * v.y;
            if (eo) {
                const float2 w = a.rc_full[((size_t)__ldg(a.ord + a.g.Vc / 2 + i) * nc + r) * np + col];
                q += w.x * w.x + w.y * w.y;
            }
            return q;
        };
        // the size of that right-hand side per column: the largest CTA's share of its norm
        if (act)
            for (int j = 0; j < jobs; ++j) {
                const int col = (j0 + j) % nch * nw + n;
                float s = 0.f;
                for (int r = rg; r < nc; r += rgs) s += full2(j, r, col);
                add2(col_acc(0, col), s);
            }
        publish_size(0, a.mx, true);
        if (!grid_barrier(false)) return;
        for (int i = t; i < np; i += kEpi) {
            const unsigned int m = __ldcg(a.mx + i);
            const bool zero = m < 0x00800000u, finite = m < 0x7f800000u;   // below the normal range counts as zero
            // rc 2^-e with 2^(2 e) near its largest share: every right-hand side starts near
            // unit size, exactly; a column that is not finite passes on its NaNs
            const int e = ((int)(m >> 23) - 127) >> 1;
            fr[i] = finite ? __int_as_float((127 - e) << 23) : 1.f;
            done[i] = (i >= a.nrhs || zero || !finite || a.maxit <= 0) ? (finite ? 1 : 2) : 0;
            its[i] = 0;
            rho0[i] = 0.0;
            sc_s[i] = sc_u[i] = col_scale(4.0, rows);
            iss[i] = isu[i] = 1.f / sc_s[i];
            fx[i] = fx[np + i] = fx[2 * np + i] = 0x1p42f;
        }
        epi_sync();
        int phase = 0;
        double last = 0.0;   // thread 0: |r|^2 of column 0
        // the odd half of a red-black stencil: t = sum H x, straight into the operand's tiles
        // (the scale of x, so that both halves' operands add up in one accumulator)
        auto odd_half = [&](__half* bt, const float* inv, const float* sc) {
            if (!eo) return true;
            for (int j = 0; j < jobs; ++j) {
                const int X = site(phase, j0 + j), c = (j0 + j) % nch, col = c * nw + n;
                const float f = unit(X);
                if (!take(tmem, c)) return false;
                if (act) {
                    const float p = f * inv[col];
                    for (int r = rg; r < nc; r += rgs) stage(r, product(r, p, false), sc[col], false);
                }
                epi_sync();
                write_tile(bt, X, c);
            }
            ++phase;
            return grid_barrier(true);
        };
        // sites of the other phases
        auto at = [&](int j) { return eo ? __ldg(a.ord + (j0 + j) / nch) : (j0 + j) / nch; };
        // r = rc 2^-e, y = 0; the tile of r for s = D_c^dag r
        for (int j = 0; j < jobs; ++j) {
            const int X = at(j), c = (j0 + j) % nch, col = c * nw + n;
            if (act) {
                float s = 0.f;
                const float f = done[col] ? 0.f : fr[col], sc = sc_u[col];
                const bool nan = done[col] == 2;
                for (int r = rg; r < nc; r += rgs) {
                    const size_t o = ((size_t)X * nc + r) * np + col;
                    float2 v = a.rc[o];
                    const float2 z = nan ? make_float2(0.f * v.x, 0.f * v.y) : make_float2(0.f, 0.f);
                    v = f != 0.f ? make_float2(f * v.x, f * v.y) : make_float2(0.f, 0.f);
                    a.r[o] = v;
                    a.y[o] = z;
                    s += f * f * full2(j, r, col);   // |r_0|^2 of the full system
                    stage(r, v, sc, true);
                }
                add2(col_acc(2, col), s);
            }
            epi_sync();
            write_tile(a.btu, X, c);
            epi_sync();
        }
        if (!grid_barrier(true)) return;
        // s = D_c^dag r, its tile and norm
        if (!odd_half(a.btu, isu, sc_u)) return;
        for (int j = 0; j < jobs; ++j) {
            const int X = at(j), c = (j0 + j) % nch, col = c * nw + n;
            const float f = unit(X);
            if (!take(tmem, c)) return;
            if (act) {
                float s = 0.f;
                const float inv = f * isu[col], sc = sc_s[col];
                for (int r = rg; r < nc; r += rgs) {
                    const float2 v = product(r, inv, true);
                    a.s[((size_t)X * nc + r) * np + col] = v;
                    s += v.x * v.x + v.y * v.y;
                    stage(r, v, sc, false);
                }
                add2(col_acc(1, col), s);
            }
            epi_sync();
            write_tile(a.bts, X, c);
        }
        ++phase;
        publish_size(1, a.mx + np, false);
        for (int it = 0;; ++it) {
            if (!grid_barrier(true)) return;
            // phase A: u = D_c s, its tile and norm
            if (!odd_half(a.bts, iss, sc_s)) return;
            for (int j = 0; j < jobs; ++j) {
                const int X = at(j), c = (j0 + j) % nch, col = c * nw + n;
                const float f = unit(X);
                if (!take(tmem, c)) return;
                if (act) {
                    float s = 0.f;
                    const float inv = f * iss[col], sc = sc_u[col];
                    for (int r = rg; r < nc; r += rgs) {
                        const float2 v = product(r, inv, false);
                        a.u[((size_t)X * nc + r) * np + col] = v;
                        s += v.x * v.x + v.y * v.y;
                        stage(r, v, sc, true);
                    }
                    add2(col_acc(0, col), s);
                }
                epi_sync();
                write_tile(a.btu, X, c);
            }
            ++phase;
            if (it == 0) {
                // units of the first sums: |D^dag r|^2 and |D D^dag r|^2 of a right-hand side of
                // low modes are many orders of magnitude below |r|^2
                publish_size(0, a.mx + 2 * np, false);
                if (!grid_barrier(false)) return;
                for (int i = t; i < np; i += kEpi) {
                    fx[i] = unit_of(__uint_as_float(__ldcg(a.mx + 2 * np + i)));
                    fx[np + i] = unit_of(__uint_as_float(__ldcg(a.mx + np + i)));
                }
            }
            unsigned long long* sums = a.sums + (size_t)(it & 1) * 3 * np;
            publish(fx, sums);
            if (!grid_barrier(true)) return;
            // the scalars of the iteration, while phase B's copies and MMAs run
            if (blockIdx.x == 0)   // the other half's readers are all past this barrier, its writers behind the next
                for (int i = t; i < 3 * np; i += kEpi) a.sums[(size_t)((it + 1) & 1) * 3 * np + i] = 0ull;
            bool running = false;
            for (int i = t; i < np; i += kEpi) {
                isu[i] = 1.f / sc_u[i];
                sc_tu[i] = sc_u[i];   // the scale of the u tile, for the odd half's
                if (!done[i]) {
                    double tot[3];
#pragma unroll
                    for (int v = 0; v < 3; ++v) {
                        const long long q = (long long)__ldcg(sums + v * np + i);
                        tot[v] = (double)q * (double)(1.f / fx[v * np + i]);
                        fx[v * np + i] = unit_of((float)tot[v]);
                    }
                    const double delta = tot[0], gamma = tot[1], rho = tot[2];
                    its[i] = it;
                    if (i == 0) last = rho;
                    double beta = 0.0, den = delta;
                    if (it > 0) {   // gam, alo: reciprocals of the last gamma and alpha
                        beta = gamma * gam[i];
                        den = delta - beta * gamma * alo[i];
                    } else {
                        rho0[i] = rho;
                    }
                    if (__ldcg(a.bad + i) || (it > 0 && rho <= a.tol2 * rho0[i]) || it >= a.maxit || !(gamma > 0) || !(den > 0)) {
                        done[i] = 1;
                        al[i] = be[i] = 0.f;
                    } else {
                        const double alpha = gamma / den;
                        gam[i] = gamma;   // turned into reciprocals after phase B
                        alo[i] = alpha;
                        al[i] = (float)alpha;
                        be[i] = (float)beta;
                        running = true;
                        sc_s[i] = col_scale(gamma, rows);
                        sc_u[i] = col_scale(delta, rows);
                    }
                }
            }
            running = epi_sync(running);
            // phase B: w = D_c^dag u and the updates on the own rows
            const bool first = it == 0;
            if (eo && running) {
                if (!odd_half(a.btu, isu, sc_tu)) return;
            } else if (eo) {   // the odd half that was started; its even half never is
                for (int j = 0; j < jobs; ++j)
                    if (!take(tmem, (j0 + j) % nch)) return;
                break;
            }
            for (int j = 0; j < jobs; ++j) {
                const int X = at(j), c = (j0 + j) % nch, col = c * nw + n;
                const float f = unit(X);
                if (!take(tmem, c)) return;
                if (!running) continue;   // nothing left to do but to take what was started
                if (act) {
                    float sg = 0.f, sr = 0.f;
                    const bool frozen = done[col] != 0;
                    const float inv = f * isu[col], sc = sc_s[col], alpha = al[col], beta = be[col];
#pragma unroll 3
                    for (int r = rg; r < nc; r += rgs) {
                        const size_t o = ((size_t)X * nc + r) * np + col;
                        float2 s = a.s[o];
                        if (!frozen) {
                            const float2 u = a.u[o], w = product(r, inv, true);
                            float2 p = s, z = w, q = u, y = a.y[o], rr = a.r[o];
                            if (!first) {
                                const float2 p0 = a.p[o], z0 = a.z[o], q0 = a.q[o];
                                p.x += beta * p0.x; p.y += beta * p0.y;
                                z.x += beta * z0.x; z.y += beta * z0.y;
                                q.x += beta * q0.x; q.y += beta * q0.y;
                            }
                            y.x += alpha * p.x; y.y += alpha * p.y;
                            rr.x -= alpha * q.x; rr.y -= alpha * q.y;
                            s.x -= alpha * z.x; s.y -= alpha * z.y;
                            a.p[o] = p; a.z[o] = z; a.q[o] = q;
                            a.y[o] = y; a.r[o] = rr; a.s[o] = s;
                            sg += s.x * s.x + s.y * s.y;
                            sr += rr.x * rr.x + rr.y * rr.y;
                        }
                        stage(r, s, sc, false);
                    }
                    if (!frozen) {
                        add2(col_acc(1, col), sg);
                        add2(col_acc(2, col), sr);
                    }
                }
                epi_sync();
                write_tile(a.bts, X, c);
            }
            for (int i = t; i < np; i += kEpi) {
                iss[i] = 1.f / sc_s[i];
                if (!done[i]) {
                    gam[i] = 1.0 / gam[i];
                    alo[i] = 1.0 / alo[i];
                }
            }
            ++phase;
            if (!running) break;
        }
        // the solution in the units of rc
        if (act)
            for (int j = 0; j < jobs; ++j) {
                const int X = at(j), col = (j0 + j) % nch * nw + n;
                if (done[col] == 2) continue;
                const float f = 1.f / fr[col];
                for (int r = rg; r < nc; r += rgs) {
                    const size_t o = ((size_t)X * nc + r) * np + col;
                    const float2 v = a.y[o];
                    a.y[o] = make_float2(f * v.x, f * v.y);
                }
            }
        if (blockIdx.x == 0)
            for (int i = t; i < np; i += kEpi) {
                a.iters[i] = (double)its[i];
                if (i == 0 && a.scal) {   // rho0 and last in the units of rc
                    const double f = 1.0 / ((double)fr[0] * fr[0]);
                    a.scal[S_CG_RC2] = f * rho0[0];
                    a.scal[S_CG_R2] = f * last;
                    a.scal[S_CG_DONE] = 1.0;
                    a.scal[S_CG_ITERS] = (double)its[0];
                    a.scal[S_CG_TOTAL] += (double)its[0];
                }
            }
        if (t == 0) *stop = 1;
        epi_sync();
        open_gate();
    }
};

__global__ void __launch_bounds__(kBcgThreads, 1) k_bcg(BcgArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[2 * kBcgMaxStages + 7];
    __shared__ uint32_t s_taddr;
    __shared__ unsigned int s_items;
    __shared__ int s_flags[6];
    BcgCta c(a, smem, bars, s_flags);
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kBcgMaxStages; ++i) { mbar_init(c.full + i, 2); mbar_init(c.empty + i, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(c.acc_full + i, 1); mbar_init(c.acc_empty + i, kEpiWarps); }
        for (int i = 0; i < 3; ++i) mbar_init(c.gate + i, 1);   // the gate, the MMA threads' drains
        fence_mbar_init();
        for (int i = 0; i < 6; ++i) s_flags[i] = 0;
        s_items = 0;
    }
    // zero the stages: the padding K group stays zero, the copies fill the rest
    for (size_t i = threadIdx.x; i < (size_t)a.stages * c.L.stage / 16; i += kBcgThreads)
        reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
    fence_proxy_async();
    if (warp == 2) {
        tmem_alloc(&s_taddr, a.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_taddr;
    if (warp == 0) {
        c.copy_operator(&s_items);
    } else if (warp == 1) {
        c.copy_operand(&s_items);
    } else if (warp < 4) {
        if ((threadIdx.x & 31) == 0) c.multiply(tmem, warp - 2, c.gate + warp - 1);
    } else {
        c.epilogue(tmem);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 2) tmem_dealloc(tmem, a.tmem_cols);
}

// ---------------------------------------------------------------- shape and launch
// Columns per job: the multiple of 8 that divides npad and gives the busiest SM
// the fewest bytes of tiles (operator per job, operand per column); more jobs
// than SMs on the small lattices, the operator read once for up to 64 columns
// on the large ones.
bool bcg_shape(int nc, int npad, int Vc, int* nw_out, int* stages_out) {
    // the panel widths the interface takes (Nv = 24: up to 224 columns)
    if (nc % 8 || nc > 48 || npad % 8 || npad < 8 || npad > 256 || nc * (64 + npad) > 14512) return false;
    const long long sms = device_sm_count();
    double best = 1e300;
    for (int nw = 8; nw <= 64 && nw <= npad; nw += 8) {
        if (npad % nw) continue;
        const BcgSmem one(nc, nw, npad, 1);
        const long long room = 227 * 1024 - kBcgStatic - (long long)(one.total - one.stage);
        const int stages = (int)std::min<long long>(kBcgMaxStages, room / one.stage);
        if (stages < 3) continue;
        const long long jobs = (long long)Vc * (npad / nw), per = (jobs + sms - 1) / sms;
        // a job of few columns also pays for its barriers: 20 KB of tiles' worth
        const double cost = (double)per * (9.0 * (one.a_copy + one.b_copy) + 20480.0);
        if (cost < best) {
            best = cost;
            *nw_out = nw;
            *stages_out = stages;
        }
    }
    return best < 1e300;
}
size_t bcg_tile_bytes(int nc, int npad, long long Vc) { return (size_t)Vc * 4 * nc * npad * sizeof(__half); }

cudaError_t bcg_launch(const BcgArgs& args, cudaStream_t st) {
    BcgArgs a = args;
    a.mx = a.bar + 4;
    a.sums = reinterpret_cast<unsigned long long*>(a.bar + 4 + 3 * a.npad);
    a.bad = reinterpret_cast<unsigned int*>(a.sums + 6 * (size_t)a.npad);
    if (!bcg_shape(a.nc, a.npad, a.ord ? a.g.Vc / 2 : a.g.Vc, &a.nw, &a.stages)) return cudaErrorInvalidValue;
    a.first_dag = a.mode == BCG_APPLY ? a.dag : 1;   // the CG starts with s = D_c^dag r
    if (!a.rc_full) a.rc_full = a.rc;
    a.third = a.nrhs == 1;
    const int sms = device_sm_count();
    const long long jobs = (long long)(a.ord ? a.g.Vc / 2 : a.g.Vc) * (a.npad / a.nw);
    const int grid = (int)std::min<long long>(jobs, sms);
    // past half an SM, so that one CTA has the SM's tensor memory to itself
    const size_t sm = std::max<size_t>(BcgSmem(a.nc, a.nw, a.npad, a.stages).total, 116 * 1024);
    a.tmem_cols = 32;
    while (a.tmem_cols < 8 * a.nw) a.tmem_cols *= 2;
    cudaError_t e = cudaFuncSetAttribute(k_bcg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(a.bar, 0, bcg_sync_bytes(a.npad), st);
    if (e != cudaSuccess) return e;
    TmemOrder order(st);
    if (order.error() != cudaSuccess) return order.error();
    void* params[] = {&a};
    note_launch();
    e = cudaLaunchCooperativeKernel((const void*)k_bcg, dim3(grid), dim3(kBcgThreads), params, sm, st);
    if (e != cudaSuccess) return e;
    return order.launched();
}

// ---------------------------------------------------------------- SIMT reference of the same contraction
// One thread per (X, a, n); reads the FP64 operator.  Used by the FP64 batched
// path and to cross-check the tensor-core kernel.
template <typename T>
__global__ void k_coarse_apply_batched_simt(v2<T>* __restrict__ y, const double2* __restrict__ A,
                                            const v2<T>* __restrict__ x, int nc, int npad, int dag, Geom g) {
    int X = blockIdx.x, a = blockIdx.y;
    int nvh = nc / 2;
    for (int n = threadIdx.x; n < npad; n += blockDim.x) {
        cx<double> acc(0, 0);
        for (int d = 0; d < 9; ++d) {
            int Y = coarse_neighbour(g, X, d);
            const double2* Ad = A + ((size_t)X * 9 + d) * nc * nc + a;
            for (int b = 0; b < nc; ++b) {
                v2<T> xv = x[((size_t)Y * nc + b) * npad + n];
                cx<double> xb((double)xv.x, (double)xv.y);
                if (dag && b >= nvh) xb = cx<double>(-xb.r, -xb.i);
                cmad(acc, ld<double>(Ad + (size_t)b * nc), xb);
            }
        }
        if (dag && a >= nvh) acc = cx<double>(-acc.r, -acc.i);
        v2<T> o; o.x = (T)acc.r; o.y = (T)acc.i;
        y[((size_t)X * nc + a) * npad + n] = o;
    }
}
template <typename T>
void coarse_apply_batched_simt(v2<T>* y, const double2* A, const v2<T>* x, int nc, int npad, bool dag, const Geom& g,
                               cudaStream_t st) {
    note_launch();
    k_coarse_apply_batched_simt<T><<<dim3(g.Vc, nc), 128, 0, st>>>(y, A, x, nc, npad, dag ? 1 : 0, g);
}
template void coarse_apply_batched_simt<float>(v2<float>*, const double2*, const v2<float>*, int, int, bool,
                                               const Geom&, cudaStream_t);
template void coarse_apply_batched_simt<double>(v2<double>*, const double2*, const v2<double>*, int, int, bool,
                                                const Geom&, cudaStream_t);

}  // namespace wmg

namespace wmg {
static inline int ew_grid2(long long total) {
    long long b = (total + 255) / 256;
    if (b > 8LL * device_sm_count()) b = 8LL * device_sm_count();
    return (int)(b > 0 ? b : 1);
}
// columns n < nrhs of a panel from nrhs stacked coarse vectors in[n][row] (FP64), other columns zero
__global__ void k_panel_pack(float2* __restrict__ out, const double2* __restrict__ in, long long rows, int nrhs, int npad) {
    long long total = rows * npad;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        long long r = i / npad;
        int n = (int)(i - r * npad);
        float2 v = make_float2(0.f, 0.f);
        if (n < nrhs) {
            double2 d = in[(size_t)n * rows + r];
            v = make_float2((float)d.x, (float)d.y);
        }
        out[i] = v;
    }
}
__global__ void k_panel_unpack(double2* __restrict__ out, const float2* __restrict__ in, long long rows, int nrhs, int npad) {
    long long total = rows * nrhs;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        long long n = i / rows, r = i - n * rows;
        float2 v = in[r * npad + n];
        out[i] = make_double2((double)v.x, (double)v.y);
    }
}
template <typename T>
__global__ void k_panel_pack_t(v2<T>* __restrict__ out, const double2* __restrict__ in, long long rows, int nrhs, int npad) {
    long long total = rows * npad;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        long long r = i / npad;
        int n = (int)(i - r * npad);
        v2<T> v; v.x = 0; v.y = 0;
        if (n < nrhs) { double2 d = in[(size_t)n * rows + r]; v.x = (T)d.x; v.y = (T)d.y; }
        out[i] = v;
    }
}
template <typename T>
__global__ void k_panel_unpack_t(double2* __restrict__ out, const v2<T>* __restrict__ in, long long rows, int nrhs, int npad) {
    long long total = rows * nrhs;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        long long n = i / rows, r = i - n * rows;
        v2<T> v = in[r * npad + n];
        out[i] = make_double2((double)v.x, (double)v.y);
    }
}
__global__ void k_panel_column(float2* __restrict__ out, const float2* __restrict__ in, long long n, int npad) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n * npad; i += (long long)gridDim.x * blockDim.x)
        out[i] = i % npad == 0 ? in[i / npad] : make_float2(0.f, 0.f);
}
__global__ void k_column_of_panel(float2* __restrict__ out, const float2* __restrict__ in, long long n, int npad) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = in[i * npad];
}
void panel_column(float2* out, const float2* in, long long n, int npad, cudaStream_t st) {
    note_launch();
    k_panel_column<<<ew_grid2(n * npad), 256, 0, st>>>(out, in, n, npad);
}
void column_of_panel(float2* out, const float2* in, long long n, int npad, cudaStream_t st) {
    note_launch();
    k_column_of_panel<<<ew_grid2(n), 256, 0, st>>>(out, in, n, npad);
}
void panel_pack(float2* out, const double2* in, long long rows, int nrhs, int npad, cudaStream_t st) {
    note_launch();
    k_panel_pack<<<ew_grid2(rows * npad), 256, 0, st>>>(out, in, rows, nrhs, npad);
}
void panel_unpack(double2* out, const float2* in, long long rows, int nrhs, int npad, cudaStream_t st) {
    note_launch();
    k_panel_unpack<<<ew_grid2(rows * nrhs), 256, 0, st>>>(out, in, rows, nrhs, npad);
}
void panel_pack64(double2* out, const double2* in, long long rows, int nrhs, int npad, cudaStream_t st) {
    note_launch();
    k_panel_pack_t<double><<<ew_grid2(rows * npad), 256, 0, st>>>(out, in, rows, nrhs, npad);
}
void panel_unpack64(double2* out, const double2* in, long long rows, int nrhs, int npad, cudaStream_t st) {
    note_launch();
    k_panel_unpack_t<double><<<ew_grid2(rows * nrhs), 256, 0, st>>>(out, in, rows, nrhs, npad);
}
}  // namespace wmg
