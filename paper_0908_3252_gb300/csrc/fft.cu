// fft.cu -- shared-memory FFTs for the Toeplitz (Gram) operator, its kernel
// spectrum, and the row passes of the CG iteration that fuse into them.
//
// T x = H^H H x is a 2-D linear convolution of x with conj(G) (Appendix B).
// Embedded in an M x M circulant (M >= 2N-1; the "circular convolution" of
// section 3.4 holds only after this zero padding) it becomes
//     T x = crop_N( IFFT2( Chat .* FFT2( pad_M(x) ) ) ),
// with Chat = FFT2(c) / M^2 real because c[-y][-x] = conj c[y][x] (the point
// symmetry of G).  The apply runs in three passes over an N x M buffer X:
//   rows:    N row FFTs of the zero-padded rows (N inputs, M outputs),
//   columns: per column FFT (N nonzero inputs) -> * Chat -> IFFT, rows < N,
//   rows:    N row IFFTs, columns < N kept.
// Inside the CG iteration the last row pass (the column pass at M >= 2048) also
// forms q2 = Re<d, T d> and the first line-search step.  The bodies of the passes
// live in fft_device.cuh and fft_half.cuh (shared with the persistent loop of
// cg_loop.cu); this file holds the stand-alone kernels and their launchers.
//
// FFTs are self-sorting Stockham transforms in shared memory.  For
// power-of-two M (what every plan's transforms run on, fft_grid) the transform
// is compile-time:
// one radix-4 butterfly per thread per stage (plus one radix-2 stage for odd
// log2 M), values in registers between a read and a write phase.  Any other
// M = 2^a 3^b 5^c (a caller's spectrum on such a grid, spirec_toeplitz_noalloc)
// runs the runtime mixed-radix path with a ping-pong buffer.
// At M = 256 and 512 the three passes are 256-point register transforms of half a
// warp each (fft_half.cuh); at M = 2048 and 4096 they split every transform
// into warp-sized 1024-point DFTs (k_rows_fwd_split, k_cols_split, k_rows_inv_split).
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "chain.cuh"
#include "fft_device.cuh"
#include "fft_half.cuh"
#include "fft_reg.cuh"
#include "internal.cuh"
#include "phase.cuh"
#include "reduce.cuh"

namespace spirec {

bool make_fft_plan(int M, FftPlan* p)
{
    p->M = M;
    p->nstages = 0;
    int r = M;
    while (r > 1) {
        int rad;
        if (r % 4 == 0) rad = 4;
        else if (r % 2 == 0) rad = 2;
        else if (r % 3 == 0) rad = 3;
        else if (r % 5 == 0) rad = 5;
        else return false;
        if (p->nstages >= kMaxStages) return false;
        p->radix[p->nstages++] = rad;
        r /= rad;
    }
    return true;
}

namespace {

using namespace fftd;

// Threads of a T pass's block, at most.
template <int MC>
__host__ __device__ constexpr int t_threads() { return half_warp_size<MC>() ? 128 : 1024; }

// ------------------------------------------------------------- row pass 1

// Row FFTs of `in` (n_in nonzero entries a row) into X.  At M = 256 and 512 the T
// passes are register transforms (fft_half.cuh) whose tables are loaded before the
// wait for the predecessor: latency bounds these passes (loads, one exchange,
// stores), and the radix-4 stages with a block barrier each added to it.  T at N =
// 256, M = 512 15.6 us with radix-4 stages, now 11.0; at N = 128, M = 256 9.7 and
// 8.6.
template <int MC>
__global__ void __launch_bounds__(t_threads<MC>()) k_rows_fwd(const float2* in, int ld_in, int n_in, int rows, float2* X, FftPlan fp,
                           const float2* __restrict__ tw, int rpc)
{
    extern __shared__ float2 sm[];
    if constexpr (half_warp_size<MC>()) {
        half_tables<MC>(sm, tw);
        chain_enter();
        chain_next();
        __syncthreads();
        const int l = threadIdx.x & 15, h = (threadIdx.x >> 4) & 1;
        const int q = blockIdx.x * rpc + (int)(threadIdx.x / (MC / 16));
        const bool own = q < rows;
        const float2* row = in + (int64_t)q * ld_in;
        float2 x[16];
        half_fwd<MC>(x, [&](int n) { return __ldcg(row + n); }, own ? n_in : 0,
                     sm + kHalfTables + (threadIdx.x >> 4) * kHalfArea, sm, l, h);
        if (own)
#pragma unroll
            for (int k = 0; k < 16; ++k) X[(int64_t)q * MC + half_freq<MC>(l, h, k)] = x[k];
        return;
    }
    chain_enter();
    chain_next();
    float2* a = sm;
    float2* b = sm + rpc * seq_len<MC>(fp.M);
    const int r0 = blockIdx.x * rpc;
    const int nr = min(rpc, rows - r0);
    rows_fwd_group<MC>(in, ld_in, n_in, r0, nr, rpc, X, fp, tw, a, b);
}

// ------------------------------------------------------------- row pass 3

// The grid sum q2 = Re<d, T d> of every thread's acc, and from it the first
// line-search step t1 = -(q1 + num0) / (2 q2 + den0) (0 when the curvature is not
// > 0), by the last block.
__device__ __forceinline__ void finish_q2(float acc, const CgPass& c)
{
    float v[1] = {acc};
    FF bt[1];
    block_partial<1>(v, bt);
    store_parts<1>(bt, c.parts, kMaxParts);
    if (last_block(c.counter)) {
        FF t[1];
        sum_parts_ff<1>(c.parts, kMaxParts, gridDim.x, t);
        if (threadIdx.x == 0) {
            const double q2 = ff_to_double(t[0]);
            c.scal[S_Q2] = q2;
            const double curv = 2.0 * q2 + c.scal[S_DEN0];
            c.scal[S_T1] = curv > 0.0 ? -(c.scal[S_Q1] + c.scal[S_NUM0]) / curv : 0.0;
            *c.counter = 0u;
        }
    }
}

// Row IFFTs of X, first n_out columns to out; CG: also Re<dotx, out> and finish_q2.
template <int MC, bool CG>
__global__ void __launch_bounds__(t_threads<MC>()) k_rows_inv(const float2* X, int rows, float2* out, int n_out, FftPlan fp,
                           const float2* __restrict__ tw, int rpc, const float2* dotx, CgPass c)
{
    extern __shared__ float2 sm[];
    float acc = 0.f;
    if constexpr (half_warp_size<MC>()) {
        half_tables<MC>(sm, tw);
        chain_enter();
        chain_next();
        __syncthreads();
        const int l = threadIdx.x & 15, h = (threadIdx.x >> 4) & 1;
        const int q = blockIdx.x * rpc + (int)(threadIdx.x / (MC / 16));
        const bool own = q < rows;
        const float2* row = X + (int64_t)q * MC;
        float2 x[16], y[8];
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = own ? __ldcg(row + half_freq<MC>(l, h, k)) : make_float2(0.f, 0.f);
        half_inv<MC>(x, y, sm + kHalfTables + (threadIdx.x >> 4) * kHalfArea, sm, l, h);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int m = half_elem<MC>(l, h, i);
            if (own && m < n_out) {
                const int64_t o = (int64_t)q * n_out + m;
                out[o] = y[i];
                if (dotx) acc += redot(__ldcg(dotx + o), y[i]);
            }
        }
    } else {
        chain_enter();
        chain_next();
        float2* a = sm;
        float2* b = sm + rpc * seq_len<MC>(fp.M);
        const int r0 = blockIdx.x * rpc;
        const int nr = min(rpc, rows - r0);
        rows_inv_group<MC>(X, r0, nr, rpc, out, n_out, fp, tw, dotx, a, b, acc);
    }
    if (CG) finish_q2(acc, c);
}

// ------------------------------------------------------------- column pass

// M = 256, 512: kHalfCols columns a block, staged as row pieces of 32 bytes at
// half_col_ld (4 mod 16: the stores of 16 lanes, four rows of four columns, meet
// distinct banks).  Chat is older than the predecessor, so it is read before the wait.
constexpr int kHalfCols = 4;

template <int MC>
__host__ __device__ constexpr int half_col_ld() { return MC / 2 + 4; }

template <int MC>
__global__ void __launch_bounds__(t_threads<MC>()) k_cols_filter(float2* X, int n_in, int n_out, FftPlan fp, const float2* __restrict__ tw,
                              const float* __restrict__ Chat, int cpc)
{
    extern __shared__ float2 sm[];
    const int x0 = blockIdx.x * cpc;
    if constexpr (half_warp_size<MC>()) {
        constexpr int LD = half_col_ld<MC>(), THREADS = kHalfCols * MC / 16, E = kHalfCols * (MC / 2) / THREADS;
        float2* cols = sm + kHalfTables;
        half_tables<MC>(sm, tw);
        const int tid = threadIdx.x, l = tid & 15, h = (tid >> 4) & 1, c = tid / (MC / 16);
        float hs[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) hs[k] = __ldg(Chat + (int64_t)(x0 + c) * MC + half_freq<MC>(l, h, k));
        chain_enter();
        chain_next();
        float2 v[E];
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int e = tid + i * THREADS, y = e / kHalfCols;
            v[i] = y < n_in ? __ldcg(X + (int64_t)y * MC + x0 + e % kHalfCols) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int e = tid + i * THREADS;
            cols[(e % kHalfCols) * LD + e / kHalfCols] = v[i];
        }
        __syncthreads();
        float2* area = cols + kHalfCols * LD + (tid >> 4) * kHalfArea;
        float2* col = cols + c * LD;
        float2 x[16], out[8];
        half_fwd<MC>(x, [&](int n) { return col[n]; }, n_in, area, sm, l, h);
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = make_float2(x[k].x * hs[k], x[k].y * hs[k]);
        half_inv<MC>(x, out, area, sm, l, h);
#pragma unroll
        for (int i = 0; i < 8; ++i) col[half_elem<MC>(l, h, i)] = out[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int e = tid + i * THREADS, y = e / kHalfCols;
            if (y < n_out) X[(int64_t)y * MC + x0 + e % kHalfCols] = cols[(e % kHalfCols) * LD + y];
        }
        return;
    }
    chain_enter();
    chain_next();
    const int ld = seq_len<MC>(fp.M) + 4;
    cols_group<MC>(X, n_in, n_out, x0, min(cpc, fp.M - x0), cpc, fp, tw, Chat, sm, sm + cpc * ld);
}

// ------------------------------------------------- passes at M = 1024 S >= 2048
//
// The transforms of the apply have at most M/2 nonzero inputs and keep at most
// M/2 outputs, so each splits into S warp-sized 1024-point DFTs, one per
// output class r = k mod S:
//   forward: X[S k + r] = DFT1024(z_r)[k],
//            z_r[m] = w_M^(r m) sum_{t < S/2} x[m + 1024 t] w_S^(r t);
//   inverse: u_r = IDFT1024 of class r, out[n] = sum_r w_M^(-r n) u_r[n mod 1024],
//            n and n + 1024 from the same S values.
// The columns of X are in class order, c = 1024 r + k for the frequency S k + r,
// and so is Chat in both indices (split_pos).  X lies in pairs of columns, each
// in tiles of two rows and two columns, one 32-byte sector: element (y, c) at
//      ((c / 2) ldx + 2 (y / 2)) 2 + 2 (c % 2) + y % 2,
// ldx = N rounded up to even (split_ld).  The column pass, the heaviest, moves a
// pair of columns as one contiguous run; the row passes, two rows at a time,
// move whole sectors, each as one 32-byte access.
//
// At 2048^2, M = 4096 (us, the same with 16-byte pieces of a row-major X and two
// or three columns or rows a block, staged by loads): row pass 1 48 (about 60),
// column pass 103 (155), row pass 3 47 (49 with its dot product, which is now a
// few multiply-adds of the column pass); one T apply 254 -> 180.  The column
// pass is bound by its instructions (55% of the issue slots at 16 warps an SM,
// 62 M instructions) and by shared memory; with X by columns and the row passes
// writing and reading 16-byte pieces it takes 93, but they take 102 and 81.

// One warp, the 1024-point DFT (conjugate twiddles when INV) of the sequence
// whose element lane + 32 j is in x[j], as four steps: DFT over the
// registers, twiddles w1024^(lane k1) from t2, transpose through this warp's
// area (32 x 33), DFT over the registers.  Element lane + 32 k2 of the result
// ends in x[bitrev5(k2)].  t2[k1 * 32 + l] = w1024^(k1 l).
template <bool INV>
__device__ __forceinline__ void dft1024_warp(float2 (&x)[32], float2* area, const float2* t2, int lane)
{
    freg::dft32_dif<INV>(x);
#pragma unroll
    for (int k1 = 0; k1 < 32; ++k1) {
        const float2 w = t2[k1 * 32 + lane];
        area[k1 * 33 + lane] = cmul(x[freg::bitrev5(k1)], INV ? conjf2(w) : w);
    }
    __syncwarp();
#pragma unroll
    for (int l = 0; l < 32; ++l) x[l] = area[lane * 33 + l];
    __syncwarp();
    freg::dft32_dif<INV>(x);
}

// x[k] <-> x[bitrev5(k)]: the bit-reversed register order to the natural one
// (compile-time indices: a renaming, no data moves).
__device__ __forceinline__ void unreverse32(float2 (&x)[32])
{
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        const int b = freg::bitrev5(k);
        if (k < b) {
            const float2 t = x[k];
            x[k] = x[b];
            x[b] = t;
        }
    }
}

constexpr int kSplitWarps = 8;
constexpr int kSplitThreads = 32 * kSplitWarps;
constexpr int kSplitCtasPerSm = 2;  // 128 registers a thread, up to 108 KB of shared memory
constexpr int kSplitArea = 32 * 33;

// Shared memory of the split passes: the warps' areas, the 32 x 32 twiddles
// and the fold's twiddles w_{32 S}^e.
struct SplitSmem {
    float2 area[kSplitWarps][kSplitArea];
    float2 t2[1024];
    float2 fold[128];
};

template <int S>
__device__ __forceinline__ void split_tables(SplitSmem& sm, const float2* __restrict__ tw)
{
    constexpr int M = 1024 * S;
    for (int e = threadIdx.x; e < 1024; e += kSplitThreads) sm.t2[e] = __ldg(tw + ((S * (e >> 5) * (e & 31)) & (M - 1)));
    for (int e = threadIdx.x; e < 32 * S; e += kSplitThreads) sm.fold[e] = __ldg(tw + 32 * e);
    __syncthreads();
}

// One 32-byte sector (p 32-byte aligned) as one access.
__device__ __forceinline__ void store_sector(float2* p, float2 a, float2 b, float2 c, float2 d)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(b.x),
                 "f"(b.y), "f"(c.x), "f"(c.y), "f"(d.x), "f"(d.y)
                 : "memory");
}
__device__ __forceinline__ void load_sector(const float2* p, float2 (&v)[4])
{
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x), "=f"(v[3].y)
        : "l"(p)
        : "memory");
}

// Barrier of `threads` threads of the block (whole warps), id 1 .. 15.
__device__ __forceinline__ void team_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The folded input of class r: z_r[m], m = lane + 32 j, from src[0 .. n) in
// shared memory, with
// the factor w_4^r = (-i)^r exact (a swap and sign changes) and w_M^(r m) =
// w_M^(r lane) w_{32 S}^(r j).
template <int S>
__device__ __forceinline__ void load_folded(float2 (&x)[32], const float2* src, int n, int r, int lane,
                                            const float2* fold, float2 wl)
{
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const int m = lane + 32 * j;
        x[j] = m < n ? src[m] : make_float2(0.f, 0.f);
    }
    if constexpr (S == 4) {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const int m = lane + 32 * j + 1024;
            const float2 v = m < n ? src[m] : make_float2(0.f, 0.f);
            const float2 rv = r == 0 ? v : r == 1 ? make_float2(v.y, -v.x) : r == 2 ? make_float2(-v.x, -v.y)
                                                                                    : make_float2(-v.y, v.x);
            x[j] = freg::add(x[j], rv);
        }
    }
    if (r > 0) {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = cmul(x[j], cmul(fold[r * j], wl));
    }
}

// Outputs m and m + 1024 (S = 4) of the inverse transform from the classes'
// values u[r] = u_r[m]: v_r = w_M^(-r m) u_r, y[m] = sum v_r, y[m + 1024] =
// sum i^r v_r.
template <int S>
__device__ __forceinline__ void combine_classes(const float2 (&u)[S], const float2 (&w)[S], float2& y0, float2& y1)
{
    const float2 v1 = cmul(u[1], conjf2(w[1]));
    if constexpr (S == 2) {
        y0 = freg::add(u[0], v1);
        y1 = make_float2(0.f, 0.f);
    } else {
        const float2 v2 = cmul(u[2], conjf2(w[2])), v3 = cmul(u[3], conjf2(w[3]));
        const float2 a = freg::add(u[0], v2), b = freg::sub(u[0], v2), c = freg::add(v1, v3), d = freg::sub(v1, v3);
        y0 = freg::add(a, c);
        y1 = make_float2(b.x - d.y, b.y + d.x);
    }
}

// w[r] = w_M^(r m), r = 1 .. S - 1.
template <int S>
__device__ __forceinline__ void class_twiddles(float2 (&w)[S], int m, const float2* __restrict__ tw)
{
#pragma unroll
    for (int r = 1; r < S; ++r) w[r] = __ldg(tw + r * m);
}

// The split passes' shared memory with what comes next on its way: a column a
// team (4 of 1024 rows at S = 2, 2 of 2048 at S = 4) or 8/S rows.
struct StagedSmem {
    SplitSmem s;
    float2 stage[4096];
};

__device__ __forceinline__ void cp_async16(float2* dst, const float2* src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(float2* dst, const float2* src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// Column pass: FFT * Chat * IFFT of every column of X (N rows), a team of 2S
// warps a pair of columns, S a column, teams looping over the pairs on their
// own.  A team's next pair is copied into its stage as soon as the fold has read
// it, and a column's spectrum is loaded before its first DFT.  CG: also Re<d, T
// d> = sum Chat |FFT2(d)|^2 (Parseval: the row pass then reads no d) and finish_q2.
template <int S, bool CG>
__global__ void __launch_bounds__(kSplitThreads, kSplitCtasPerSm)
k_cols_split(float2* X, int N, int ldx, const float2* __restrict__ tw, const float* __restrict__ Chat, CgPass dot)
{
    chain_enter();
    constexpr int M = 1024 * S, C = kSplitWarps / (2 * S), T = 64 * S;  // pairs a block, threads a team
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StagedSmem& ss = *reinterpret_cast<StagedSmem*>(smem_raw);
    SplitSmem& sm = ss.s;
    split_tables<S>(sm, tw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int team = warp / (2 * S), cc = (warp / S) & 1, r = warp % S, t = threadIdx.x % T;
    const float2 wl = __ldg(tw + r * lane);
    float2* area = sm.area[warp];
    float2* stage = ss.stage + team * (1024 * S);  // column cc at 512 S cc
    // 16-byte chunk e of the pair: rows 2 (e / 2), + 1 of column e % 2
    auto fetch = [&](int pair) {
        const float2* src = X + (int64_t)pair * 2 * ldx;
        for (int e = t; e < ldx; e += T) cp_async16(stage + (e & 1) * (512 * S) + (e & ~1), src + 2 * e);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc = 0.f;
    int pair = blockIdx.x * C + team;
    if (pair < M / 2) fetch(pair);
    for (; pair < M / 2; pair += gridDim.x * C) {
        const int c = 2 * pair + cc;
        float h[32];
        {
            const float* ch = Chat + (int64_t)c * M + 1024 * r + lane;
#pragma unroll
            for (int k2 = 0; k2 < 32; ++k2) h[k2] = __ldg(ch + 32 * k2);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        team_sync(1 + team, T);  // the pair has landed; the team's areas are read
        float2 x[32];
        load_folded<S>(x, stage + cc * (512 * S), N, r, lane, sm.fold, wl);
        team_sync(1 + team, T);  // the stage is read
        if (pair + (int)gridDim.x * C < M / 2) fetch(pair + (int)gridDim.x * C);
        dft1024_warp<false>(x, area, sm.t2, lane);  // frequency S (lane + 32 k2) + r in x[bitrev5(k2)]
        unreverse32(x);
#pragma unroll
        for (int k2 = 0; k2 < 32; ++k2) {
            const float2 y = make_float2(x[k2].x * h[k2], x[k2].y * h[k2]);
            if (CG) acc += redot(x[k2], y);
            x[k2] = y;
        }
        dft1024_warp<true>(x, area, sm.t2, lane);  // u_r[lane + 32 m2] in x[bitrev5(m2)]
#pragma unroll
        for (int m2 = 0; m2 < 32; ++m2) area[lane + 32 * m2] = x[freg::bitrev5(m2)];
        team_sync(1 + team, T);
        // rows m, m + 1 (and + 1024) of both columns: one sector each
        const float2(*u)[kSplitArea] = &sm.area[team * 2 * S];
#pragma unroll 1
        for (int m = 2 * t; m < 1024; m += 2 * T) {
            float2 w0[S], w1[S], y0[4], y1[4];
            class_twiddles<S>(w0, m, tw);
            class_twiddles<S>(w1, m + 1, tw);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float2 a[S], b[S];
#pragma unroll
                for (int i = 0; i < S; ++i) {
                    const float4 v = *reinterpret_cast<const float4*>(&u[k * S + i][m]);
                    a[i] = make_float2(v.x, v.y);
                    b[i] = make_float2(v.z, v.w);
                }
                combine_classes<S>(a, w0, y0[2 * k], y1[2 * k]);
                combine_classes<S>(b, w1, y0[2 * k + 1], y1[2 * k + 1]);
            }
            float2* o = X + (int64_t)pair * 2 * ldx + 2 * m;
            if (m < N) store_sector(o, y0[0], y0[1], y0[2], y0[3]);
            if (S == 4 && m + 1024 < N) store_sector(o + 2048, y1[0], y1[1], y1[2], y1[3]);
        }
    }
    if (CG) finish_q2(acc, dot);
}

// Row pass 1: the row FFTs of `in` (N x N) into X, R = 8/S rows a block at a
// time, the next ones copied into the stage meanwhile.  Warp (q, r) transforms
// class r of row q; the R warps of a class then write its columns, a sector of
// two rows and two columns at a time (rows past N: zeros).
template <int S>
__global__ void __launch_bounds__(kSplitThreads, kSplitCtasPerSm)
k_rows_fwd_split(const float2* __restrict__ in, int N, float2* X, int ldx, const float2* __restrict__ tw)
{
    chain_enter();
    constexpr int R = kSplitWarps / S, T = 32 * S;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StagedSmem& ss = *reinterpret_cast<StagedSmem*>(smem_raw);
    SplitSmem& sm = ss.s;
    split_tables<S>(sm, tw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = warp / S, r = warp - q * S;
    const float2 wl = __ldg(tw + r * lane);
    float2* area = sm.area[warp];
    float2* stage = ss.stage + q * (512 * S);
    const bool al16 = (N & 1) == 0 && ((uintptr_t)in & 15) == 0;  // 16-byte copies of a row
    auto fetch = [&](int row) {
        if (row < N) {
            const float2* src = in + (int64_t)row * N;
            if (al16)
                for (int e = 2 * (32 * r + lane); e < N; e += 2 * T) cp_async16(stage + e, src + e);
            else
                for (int e = 32 * r + lane; e < N; e += T) cp_async8(stage + e, src + e);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int r0 = blockIdx.x * R;
    fetch(r0 + q);
    for (; r0 < N; r0 += gridDim.x * R) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        team_sync(8 + q, T);  // the row has landed
        float2 x[32];
        load_folded<S>(x, stage, r0 + q < N ? N : 0, r, lane, sm.fold, wl);
        team_sync(8 + q, T);  // the stage is read
        fetch(r0 + (int)gridDim.x * R + q);
        dft1024_warp<false>(x, area, sm.t2, lane);
#pragma unroll
        for (int k2 = 0; k2 < 32; ++k2) area[lane + 32 * k2] = x[freg::bitrev5(k2)];
        team_sync(1 + r, 32 * R);
#pragma unroll 4
        for (int k = 2 * (32 * q + lane); k < 1024; k += 64 * R) {
#pragma unroll
            for (int h = 0; h < R; h += 2) {
                const float4 a = *reinterpret_cast<const float4*>(&sm.area[h * S + r][k]);
                const float4 b = *reinterpret_cast<const float4*>(&sm.area[(h + 1) * S + r][k]);
                if (r0 + h < N)
                    store_sector(X + ((int64_t)(512 * r + (k >> 1)) * ldx + r0 + h) * 2, make_float2(a.x, a.y),
                                 make_float2(b.x, b.y), make_float2(a.z, a.w), make_float2(b.z, b.w));
            }
        }
        team_sync(1 + r, 32 * R);  // the class's areas are read
    }
}

// Row pass 3: the row IFFTs of X to out (N x N), R = 8/S rows a block at a time.
// The R warps of a class bring its part of the rows into the areas (every
// sector of a thread in flight at once), warp (q, r) transforms class r of row
// q, and the S warps of a row combine its classes.
template <int S>
__global__ void __launch_bounds__(kSplitThreads, kSplitCtasPerSm)
k_rows_inv_split(const float2* __restrict__ X, int N, int ldx, float2* __restrict__ out, const float2* __restrict__ tw)
{
    chain_enter();
    constexpr int R = kSplitWarps / S;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SplitSmem& sm = *reinterpret_cast<SplitSmem*>(smem_raw);
    split_tables<S>(sm, tw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = warp / S, r = warp - q * S;
    float2* area = sm.area[warp];
    for (int r0 = blockIdx.x * R; r0 < N; r0 += gridDim.x * R) {
        {
            constexpr int V = 512 / (32 * R);  // sectors of a row pair a thread
            float2 v[R / 2 * V][4];
#pragma unroll
            for (int i = 0; i < R / 2 * V; ++i) {
                const int h = 2 * (i / V), k2 = 32 * q + lane + 32 * R * (i % V);
#pragma unroll
                for (int e = 0; e < 4; ++e) v[i][e] = make_float2(0.f, 0.f);
                if (r0 + h < N) load_sector(X + ((int64_t)(512 * r + k2) * ldx + r0 + h) * 2, v[i]);
            }
#pragma unroll
            for (int i = 0; i < R / 2 * V; ++i) {
                const int h = 2 * (i / V), k = 2 * (32 * q + lane + 32 * R * (i % V));
                *reinterpret_cast<float4*>(&sm.area[h * S + r][k]) = make_float4(v[i][0].x, v[i][0].y, v[i][2].x, v[i][2].y);
                *reinterpret_cast<float4*>(&sm.area[(h + 1) * S + r][k]) =
                    make_float4(v[i][1].x, v[i][1].y, v[i][3].x, v[i][3].y);
            }
        }
        team_sync(1 + r, 32 * R);
        float2 x[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = area[lane + 32 * j];
        __syncwarp();
        dft1024_warp<true>(x, area, sm.t2, lane);  // u_r[lane + 32 m2] in x[bitrev5(m2)]
#pragma unroll
        for (int m2 = 0; m2 < 32; ++m2) area[lane + 32 * m2] = x[freg::bitrev5(m2)];
        team_sync(8 + q, 32 * S);
        if (r0 + q < N) {
            float2* o = out + (int64_t)(r0 + q) * N;
#pragma unroll 4
            for (int m = 32 * r + lane; m < 1024; m += 32 * S) {
                float2 w[S], u[S], y0, y1;
                class_twiddles<S>(w, m, tw);
#pragma unroll
                for (int i = 0; i < S; ++i) u[i] = sm.area[q * S + i][m];
                combine_classes<S>(u, w, y0, y1);
                if (m < N) o[m] = y0;
                if (S == 4 && m + 1024 < N) o[m + 1024] = y1;
            }
        }
        __syncthreads();  // the next rows refill the areas
    }
}

// ------------------------------------------------------- kernel spectrum
//
// Chat[kx][ky] = (1 / M^2) sum_{u,v} c_{u,v} exp(-i2pi (kx u + ky v) / M) with
// c_{u,v} = conj G_{u,v}, |u|, |v| < N.  G is point-symmetric, c_{-u,-v} = conj
// c_{u,v}, so the transforms T[u][ky] along v satisfy T[-u] = conj T[u] and
//      M^2 Chat[kx][ky] = 2 Re sum_{u = 0}^{N-1} e_u T[u][ky] exp(-i2pi kx u / M),
// e_0 = 1/2, e_u = 1: N row transforms straight from G's stored half (u >= 0)
// and column transforms of N inputs, instead of M and M over an embedded
// M x M array (embedding, rows and columns at M = 1024, N = 512: 34 -> 25 us).

// Rows u of G's half, conjugated, at v mod M: T[u][ky] to X[u * M + split_pos(ky)].
template <int MC>
__global__ void __launch_bounds__(1024) k_rows_spectrum(const float2* G, int N, float2* X, FftPlan fp,
                                                        const float2* __restrict__ tw, int rpc)
{
    extern __shared__ float2 sm[];
    chain_enter();
    const int M = fp.M, ld = seq_len<MC>(M), W = 2 * N - 1;
    float2* a = sm;
    float2* b = sm + rpc * ld;
    const int u0 = blockIdx.x * rpc, nr = min(rpc, N - u0);
    for (int e = threadIdx.x; e < rpc * M; e += blockDim.x) {
        const int q = e / M, y = e - q * M;
        const int v = y < N ? y : y - M;  // -N < v < N holds a lag
        float2 c = make_float2(0.f, 0.f);
        if (q < nr && v > -N) {
            const float2 g = G[(int64_t)(u0 + q) * W + (v + N - 1)];
            c = make_float2(g.x, -g.y);
        }
        a[q * ld + sidx<MC>(y)] = c;
    }
    __syncthreads();
    float2* res = fft_block<MC, false>(a, b, fp, rpc, ld, tw);
    for (int e = threadIdx.x; e < nr * M; e += blockDim.x) {
        const int q = e / M, m = e - q * M;
        X[(int64_t)(u0 + q) * M + split_pos<MC>(m)] = res[q * ld + sidx<MC>(m)];
    }
}

// Column transforms of X (rows u < N) and the real spectrum: to
// out[kx * M + ky], both by split_pos (Chat), or out[ky * M + kx] (ROWS_KY, the
// caller's grid when it is not a power of two).
template <int MC, bool ROWS_KY>
__global__ void __launch_bounds__(1024) k_cols_spectrum(const float2* X, int N, FftPlan fp, const float2* __restrict__ tw,
                                float* out, int cpc)
{
    extern __shared__ float2 sm[];
    chain_enter();
    const int M = fp.M;
    const int ld = seq_len<MC>(M) + 4;
    float2* a = sm;
    float2* b = sm + cpc * ld;
    const int x0 = blockIdx.x * cpc;
    const int nc = min(cpc, M - x0);
    for (int e = threadIdx.x; e < cpc * M; e += blockDim.x) {
        const int y = e / cpc, cc = e - y * cpc;
        float2 v = make_float2(0.f, 0.f);
        if (cc < nc && y < N) {
            v = X[(int64_t)y * M + x0 + cc];
            if (y == 0) v = make_float2(0.5f * v.x, 0.5f * v.y);
        }
        a[cc * ld + sidx<MC>(y)] = v;
    }
    __syncthreads();
    float2* res = fft_block<MC, false>(a, b, fp, cpc, ld, tw);
    const float inv = 2.0f / ((float)M * (float)M);
    for (int e = threadIdx.x; e < nc * M; e += blockDim.x) {
        const int cc = ROWS_KY ? e / M : e % nc, kx = ROWS_KY ? e - cc * M : e / nc;
        const float v = res[cc * ld + sidx<MC>(kx)].x * inv;
        out[ROWS_KY ? (int64_t)(x0 + cc) * M + kx : (int64_t)split_pos<MC>(kx) * M + x0 + cc] = v;
    }
}

// ------------------------------------------------------------- launch shapes

constexpr int kFftSmemCap = 200 * 1024;

// Rows of X at M >= 2048 (the split passes): N rounded up to even.
int split_ld(int N) { return (N + 1) & ~1; }

struct Shape {
    int per_cta;  // rows or columns per CTA
    int threads;
    size_t smem;
};

// Compile-time path: nseq * M / 4 threads (<= 1024), single buffer; as few rows
// and columns a block as keep two warps busy and 32-byte pieces whole, so that
// small grids spread over the SMs and their stages' barriers span few warps
// (T at N = 64 with 8 rows and 32 columns a block and plain launches 18.5 us, now
// 7.7).  The T passes at M = 256, 512 have shapes of their own (t_row_shape).
// Runtime path: 256 threads, ping-pong buffers.
Shape row_shape(int M, bool pow2)
{
    if (pow2) {
        const int nb = M / 4;
        const int rpc = nb >= 64 ? 1 : 64 / nb;
        return Shape{rpc, rpc * nb, (size_t)rpc * seq_len<1>(M) * sizeof(float2)};
    }
    const int rpc = M >= 1024 ? 1 : 1024 / M;
    return Shape{rpc, 256, 2 * (size_t)rpc * M * sizeof(float2)};
}

Shape col_shape(int M, bool pow2)
{
    if (pow2) {
        const int nb = M / 4;
        int cpc = nb >= 256 ? (nb >= 1024 ? 1 : 1024 / nb) : 4;
        const size_t ld = seq_len<1>(M) + 4;
        while (cpc > 1 && (size_t)cpc * ld * sizeof(float2) > (size_t)kFftSmemCap) cpc /= 2;
        return Shape{cpc, cpc * nb, (size_t)cpc * ld * sizeof(float2)};
    }
    // few columns a block: a small grid has to fill the SMs
    int cpc = 4;
    while (cpc > 1 && 2 * (size_t)cpc * (M + 4) * sizeof(float2) > (size_t)kFftSmemCap) --cpc;
    return Shape{cpc, 256, 2 * (size_t)cpc * (M + 4) * sizeof(float2)};
}

template <int MC>
int set_attrs()
{
    const int bytes = kFftSmemCap;
    SPIREC_CK(cudaFuncSetAttribute(k_rows_fwd<MC>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    SPIREC_CK(cudaFuncSetAttribute(k_rows_inv<MC, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    SPIREC_CK(cudaFuncSetAttribute(k_rows_inv<MC, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    SPIREC_CK(cudaFuncSetAttribute(k_cols_filter<MC>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    SPIREC_CK(cudaFuncSetAttribute(k_rows_spectrum<MC>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    SPIREC_CK(cudaFuncSetAttribute(k_cols_spectrum<MC, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    SPIREC_CK(cudaFuncSetAttribute(k_cols_spectrum<MC, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    return SPIREC_OK;
}

template <int S>
int set_split_attrs()
{
    const int bytes = (int)sizeof(SplitSmem);
    SPIREC_CK(cudaFuncSetAttribute(k_rows_fwd_split<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StagedSmem)));
    SPIREC_CK(cudaFuncSetAttribute(k_cols_split<S, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StagedSmem)));
    SPIREC_CK(cudaFuncSetAttribute(k_cols_split<S, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(StagedSmem)));
    SPIREC_CK(cudaFuncSetAttribute(k_rows_inv_split<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    return SPIREC_OK;
}

// Calls f.template operator()<MC>() with the compile-time size for M, or
// MC = 0 for sizes without a specialisation.
template <typename F>
int with_size(int M, F&& f)
{
    switch (M) {
    case 16: return f.template operator()<16>();
    case 32: return f.template operator()<32>();
    case 64: return f.template operator()<64>();
    case 128: return f.template operator()<128>();
    case 256: return f.template operator()<256>();
    case 512: return f.template operator()<512>();
    case 1024: return f.template operator()<1024>();
    case 2048: return f.template operator()<2048>();
    case 4096: return f.template operator()<4096>();
    default: return f.template operator()<0>();
    }
}

bool is_pow2_specialised(int M) { return M >= 16 && M <= 4096 && (M & (M - 1)) == 0; }

struct AttrAll {
    template <int MC>
    int operator()() { return MC > 0 ? set_attrs<MC>() : SPIREC_OK; }
};

// Grid of a split pass over `items` rows or columns, `per` a block.
int split_grid(int items, int per, int* grid)
{
    int sms = 0;
    if (device_sms(&sms) != SPIREC_OK) return SPIREC_ECUDA;
    const int groups = (items + per - 1) / per, cap = kSplitCtasPerSm * sms;
    *grid = groups < cap ? groups : cap;
    return SPIREC_OK;
}

// The shapes of the T passes: at M = 256, 512 two warps a block of rows (one row a
// warp or two) and kHalfCols columns a block, M / 16 threads a sequence.
template <int MC>
Shape t_row_shape(int M)
{
    if constexpr (half_warp_size<MC>())
        return Shape{1024 / MC, 64, (kHalfTables + 4 * kHalfArea) * sizeof(float2)};
    else
        return row_shape(M, MC > 0);
}

template <int MC>
Shape t_col_shape(int M)
{
    if constexpr (half_warp_size<MC>())
        return Shape{kHalfCols, kHalfCols * MC / 16,
                     (kHalfTables + kHalfCols * (half_col_ld<MC>() + MC / 256 * kHalfArea)) * sizeof(float2)};
    else
        return col_shape(M, MC > 0);
}

struct LaunchRowsFwd {
    spirec_plan p;
    const float2* in;
    template <int MC>
    int operator()()
    {
        const int N = p->N;
        if constexpr (MC >= 2048) {
            constexpr int S = MC / 1024;
            int grid = 0, rc;
            if ((rc = split_grid(N, kSplitWarps / S, &grid)) != SPIREC_OK) return rc;
            chain(k_rows_fwd_split<S>, grid, kSplitThreads, sizeof(StagedSmem), p->stream, in, N, p->X, split_ld(N), p->twiddle);
        } else {
            const Shape s = t_row_shape<MC>(p->MF);
            chain(k_rows_fwd<MC>, (N + s.per_cta - 1) / s.per_cta, s.threads, s.smem, p->stream, 
                in, N, N, N, p->X, p->fft, p->twiddle, s.per_cta);
        }
        SPIREC_CK(cudaGetLastError());
        p->launches += 1;
        return SPIREC_OK;
    }
};

struct LaunchCols {
    spirec_plan p;
    const CgPass* cg;
    template <int MC>
    int operator()()
    {
        const int N = p->N;
        if constexpr (MC >= 2048) {
            constexpr int S = MC / 1024;
            int grid = 0, rc;
            if ((rc = split_grid(MC / 2, kSplitWarps / (2 * S), &grid)) != SPIREC_OK) return rc;
            auto kern = cg ? k_cols_split<S, true> : k_cols_split<S, false>;
            chain(kern, grid, kSplitThreads, sizeof(StagedSmem), p->stream, p->X, N, split_ld(N), p->twiddle, p->Chat,
                                                                        cg ? *cg : CgPass{});
        } else {
            const Shape s = t_col_shape<MC>(p->MF);
            chain(k_cols_filter<MC>, (p->MF + s.per_cta - 1) / s.per_cta, s.threads, s.smem, p->stream, 
                p->X, N, N, p->fft, p->twiddle, p->Chat, s.per_cta);
        }
        SPIREC_CK(cudaGetLastError());
        p->launches += 1;
        return SPIREC_OK;
    }
};

struct LaunchRowsInv {
    spirec_plan p;
    float2* out;
    const float2* x;
    const CgPass* cg;
    template <int MC>
    int operator()()
    {
        const int N = p->N;
        if constexpr (MC >= 2048) {
            constexpr int S = MC / 1024;
            int grid = 0, rc;
            if ((rc = split_grid(N, kSplitWarps / S, &grid)) != SPIREC_OK) return rc;
            chain(k_rows_inv_split<S>, grid, kSplitThreads, sizeof(SplitSmem), p->stream, p->X, N, split_ld(N), out, p->twiddle);
        } else {
            const Shape s = t_row_shape<MC>(p->MF);
            auto kern = cg ? k_rows_inv<MC, true> : k_rows_inv<MC, false>;
            chain(kern, (N + s.per_cta - 1) / s.per_cta, s.threads, s.smem, p->stream, 
                p->X, N, out, N, p->fft, p->twiddle, s.per_cta, cg ? x : nullptr, cg ? *cg : CgPass{});
        }
        SPIREC_CK(cudaGetLastError());
        p->launches += 1;
        return SPIREC_OK;
    }
};

// The spectrum on the grid of fp from G, by way of the N x M rows in cwork, to
// out (rows_ky: in the caller's layout).
struct LaunchSpectrum {
    spirec_plan p;
    const FftPlan* fp;
    const float2* tw;
    bool rows_ky;
    float* out;
    Shape rs, cs;
    template <int MC>
    int operator()()
    {
        const int M = fp->M, N = p->N;
        chain(k_rows_spectrum<MC>, dim3((N + rs.per_cta - 1) / rs.per_cta), dim3(rs.threads), rs.smem, p->stream, p->G, N,
              p->cwork, *fp, tw, rs.per_cta);
        SPIREC_CK(cudaGetLastError());
        const int blocks = (M + cs.per_cta - 1) / cs.per_cta;
        chain(rows_ky ? k_cols_spectrum<MC, true> : k_cols_spectrum<MC, false>, dim3(blocks), dim3(cs.threads), cs.smem, p->stream,
              p->cwork, N, *fp, tw, out, cs.per_cta);
        SPIREC_CK(cudaGetLastError());
        p->launches += 2;
        return SPIREC_OK;
    }
};

// out[ky * M + kx] = Chat[kx][ky] for a power-of-two M (the caller's layout).
template <int MC>
__global__ void __launch_bounds__(256) k_transpose_real(const float* __restrict__ in, int M, float* __restrict__ out)
{
    __shared__ float tile[32][33];
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int ky = x0 + tx, kx = y0 + ty + 8 * k;
        if (ky < M && kx < M) tile[ty + 8 * k][tx] = __ldg(in + (int64_t)split_pos<MC>(kx) * M + split_pos<MC>(ky));
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int ky = x0 + ty + 8 * k, kx = y0 + tx;
        if (ky < M && kx < M) out[(int64_t)ky * M + kx] = tile[tx][ty + 8 * k];
    }
}

struct LaunchSpectrumOut {
    spirec_plan p;
    float* out;
    template <int MC>
    int operator()()
    {
        const unsigned t = (unsigned)((p->M + 31) / 32);
        k_transpose_real<MC><<<dim3(t, t), dim3(32, 8), 0, p->stream>>>(p->Chat, p->M, out);
        SPIREC_CK(cudaGetLastError());
        p->launches += 1;
        return SPIREC_OK;
    }
};

}  // namespace

int fft_setup_attributes(int)
{
    int rc;
    if ((rc = set_attrs<0>()) != SPIREC_OK) return rc;
    if ((rc = set_split_attrs<2>()) != SPIREC_OK) return rc;
    if ((rc = set_split_attrs<4>()) != SPIREC_OK) return rc;
    for (int M = 16; M <= 4096; M *= 2)
        if ((rc = with_size(M, AttrAll{})) != SPIREC_OK) return rc;
    return SPIREC_OK;
}

namespace {
// tw[k] = exp(-2 pi i k / M), formed in FP64 and rounded once
__global__ void k_twiddles(float2* tw, int M)
{
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < M; k += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(-2.0 * (double)k / (double)M, &s, &c);
        tw[k] = make_float2((float)c, (float)s);
    }
}
}  // namespace

int launch_twiddles(float2* tw, int M, cudaStream_t st)
{
    k_twiddles<<<(M + 255) / 256, 256, 0, st>>>(tw, M);
    SPIREC_CK(cudaGetLastError());
    return SPIREC_OK;
}

int launch_toeplitz(spirec_plan p, const float2* x, float2* Tx, const CgPass* cg)
{
    int rc;
    if ((rc = with_size(p->MF, LaunchRowsFwd{p, x})) != SPIREC_OK) return rc;
    if ((rc = with_size(p->MF, LaunchCols{p, cg})) != SPIREC_OK) return rc;
    return with_size(p->MF, LaunchRowsInv{p, Tx, x, cg});
}

// A power of two from 64 on as it is; anything else (the 2^a 3^b 5^c grids a plan picks
// by default among them) is embedded in the next power of two that holds the
// lags: T is the same linear convolution on any grid of at least 2N - 1, and
// the power-of-two passes are the faster ones at every N although the grid
// grows by up to 1.9 times a side.  Measured, M = 2^a 3^b 5^c against the power of two
// (us): one T apply and one CG iteration
//   N = 50,   M = 100 / 128      26.5 / 17.8    40 / 23
//   N = 129,  M = 270 / 512      45.5 / 22.0    63 / 30
//   N = 384,  M = 768 / 1024     55.3 / 38.0    76 / 30
//   N = 520,  M = 1080 / 2048    66.4 / 50.3    92 / 89
//   N = 1030, M = 2160 / 4096   250   / 169    342 / 227
int fft_grid(int N, int M)
{
    if (M >= 64 && is_pow2_specialised(M)) return M;
    int g = 64;  // the persistent loop's smallest
    while (g < 2 * N - 1) g *= 2;
    return g;
}

int launch_spectrum(spirec_plan p)
{
    const int M = p->MF;
    const bool pow2 = is_pow2_specialised(M);
    return with_size(M, LaunchSpectrum{p, &p->fft, p->twiddle, false, p->Chat, row_shape(M, pow2), col_shape(M, pow2)});
}

// Complex values of X.
size_t x_elems(int N, int MF) { return (size_t)(MF >= 2048 ? split_ld(N) : N) * MF; }

// Complex values of cwork: the N x M rows of a spectrum build on either grid.
size_t cwork_elems(int N, int M, int MF) { return (size_t)N * (M > MF ? M : MF); }

int launch_spectrum_out(spirec_plan p, float* out)
{
    if (p->M != p->MF) {
        const int M = p->M;
        const bool pow2 = is_pow2_specialised(M);
        return with_size(M, LaunchSpectrum{p, &p->fft_M, p->twiddle_M, true, out, row_shape(M, pow2), col_shape(M, pow2)});
    }
    return with_size(p->M, LaunchSpectrumOut{p, out});
}

}  // namespace spirec

// ------------------------------------------------ T x without any allocation
//
// spirec_toeplitz_noalloc: the Toeplitz apply above for callers that cannot
// allocate device memory (for example code running inside a memory-pool
// budget that forbids cudaMalloc, or a host process that must not grow the
// GPU footprint after start-up).  The caller passes the input, the kernel
// spectrum and the output; the intermediate N x M rows, the transposed
// spectrum and the twiddle table live in one file-scope device array that
// every GPU loading this library keeps until the process exits.

namespace spirec {
namespace {

constexpr int kNoAllocMaxN = 512;
constexpr int kNoAllocMaxM = 1024;
constexpr size_t kNoAllocRowsBytes = (size_t)kNoAllocMaxN * kNoAllocMaxM * sizeof(float2);
constexpr size_t kNoAllocSpecBytes = (size_t)kNoAllocMaxM * kNoAllocMaxM * sizeof(float);
constexpr size_t kNoAllocTwBytes = (size_t)kNoAllocMaxM * sizeof(float2);
constexpr size_t kNoAllocBytes = kNoAllocRowsBytes + kNoAllocSpecBytes + kNoAllocTwBytes;

// Shared by every call on a device; holds the last call's contents.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;
// device address of the array per device, published once its set-up is done
// (release store, acquire load); the mutex makes the first calls of several
// host threads on one device run the set-up once
std::atomic<void*> g_noalloc_base[kNoAllocMaxDevices];
std::mutex g_noalloc_mu;

// spectrum[ky][kx] (the layout spirec_kernel_spectrum_dev returns) into the
// column-major form the column pass reads, chat[kx][ky] (both at split_pos).
template <int MC>
__global__ void k_noalloc_spectrum(const float* __restrict__ spec, int M, float* __restrict__ chat)
{
    const int64_t MM = (int64_t)M * M;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < MM;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int kx = (int)(e / M), ky = (int)(e % M);
        chat[(int64_t)split_pos<MC>(kx) * M + split_pos<MC>(ky)] = spec[(int64_t)ky * M + kx];
    }
}

struct LaunchNoAlloc {
    const float2* x;
    float2* Tx;
    float2* rows;
    const float* chat;
    const float2* tw;
    FftPlan fp;
    int N;
    cudaStream_t st;
    template <int MC>
    int operator()()
    {
        const int M = fp.M;
        const Shape rs = t_row_shape<MC>(M), cs = t_col_shape<MC>(M);
        const int rblocks = (N + rs.per_cta - 1) / rs.per_cta;
        k_rows_fwd<MC><<<rblocks, rs.threads, rs.smem, st>>>(x, N, N, N, rows, fp, tw, rs.per_cta);
        SPIREC_CK(cudaGetLastError());
        k_cols_filter<MC><<<(M + cs.per_cta - 1) / cs.per_cta, cs.threads, cs.smem, st>>>(rows, N, N, fp, tw,
                                                                                          chat, cs.per_cta);
        SPIREC_CK(cudaGetLastError());
        k_rows_inv<MC, false><<<rblocks, rs.threads, rs.smem, st>>>(rows, N, Tx, N, fp, tw, rs.per_cta, nullptr, CgPass{});
        SPIREC_CK(cudaGetLastError());
        return SPIREC_OK;
    }
};

}  // namespace

}  // namespace spirec

extern "C" int spirec_toeplitz_noalloc(const float* x, const float* spectrum, float* Tx, int32_t N,
                                       int32_t M, void* stream)
{
    using namespace spirec;
    if (!x || !spectrum || !Tx) {
        set_error("null pointer");
        return SPIREC_EINVAL;
    }
    if (N < 2 || N > kNoAllocMaxN || M < 2 * N - 1 || M > kNoAllocMaxM) {
        set_error("spirec_toeplitz_noalloc handles 2 <= N <= %d and 2N-1 <= M <= %d (got N=%d, M=%d)",
                  kNoAllocMaxN, kNoAllocMaxM, N, M);
        return SPIREC_EINVAL;
    }
    FftPlan fp;
    if (!make_fft_plan(M, &fp)) {
        set_error("M=%d must factor into 2, 3 and 5", M);
        return SPIREC_EINVAL;
    }
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= kNoAllocMaxDevices) {
        set_error("device %d out of range", dev);
        return SPIREC_EUNSUPPORTED;
    }
    // first call on this device: the array's device address and the kernels'
    // shared-memory limits (no allocation; must happen outside stream capture)
    void* addr = g_noalloc_base[dev].load(std::memory_order_acquire);
    if (!addr) {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        addr = g_noalloc_base[dev].load(std::memory_order_relaxed);
        if (!addr) {
            e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
            if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress");
            int rc = fft_setup_attributes(M);
            if (rc != SPIREC_OK) return rc;
            g_noalloc_base[dev].store(addr, std::memory_order_release);
        }
    }
    unsigned char* base = static_cast<unsigned char*>(addr);
    float2* rows = reinterpret_cast<float2*>(base);
    float* chat = reinterpret_cast<float*>(base + kNoAllocRowsBytes);
    float2* tw = reinterpret_cast<float2*>(base + kNoAllocRowsBytes + kNoAllocSpecBytes);
    cudaStream_t st = (cudaStream_t)stream;
    const int rc = launch_twiddles(tw, M, st);
    if (rc != SPIREC_OK) return rc;
    if (M == 1024) k_noalloc_spectrum<1024><<<4 * 152, 256, 0, st>>>(spectrum, M, chat);
    else k_noalloc_spectrum<0><<<4 * 152, 256, 0, st>>>(spectrum, M, chat);
    SPIREC_CK(cudaGetLastError());
    return with_size(M, LaunchNoAlloc{(const float2*)x, (float2*)Tx, rows, chat, tw, fp, N, st});
}
