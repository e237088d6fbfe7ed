// cg.cu -- line search and Polak-Ribiere update (section 3.3) on the
// rewritten criterion (section 3.4, Eq. NewCritLS):
//
//   J(f)      = ||s||^2 - 2 Re<f, D> + Re<f, T f> + R(f)
//   grad J(f) = 2 (T f - D) + grad R(f)       (dJ/dRe f + i dJ/dIm f)
// The iteration carries res = T f - D, not T f: it starts as T x0 - D and
// moves by t T d with every step.
//   R(f)      = lambda1 sum_edges phi1(|f_q - f_p|) + lambda0 sum_p phi0(|f_p|)
//
// One iteration k is seven kernels, all on the device, no host round trip:
//   direction d = -g + beta d_old; q1 = Re<d, 2 res>; line-search sums
//             at t = 0                                             (here)
//   rows_fwd  row FFTs of d                                        (fft.cu)
//   cols      column FFT * Chat * IFFT                             (fft.cu)
//   rows_inv  row IFFTs -> T d; q2 = Re<d, T d>; t1                (fft.cu)
//   2 x line-search step j -> t_{j+1} = t_j - h'(t_j) / curvature (here)
//   update    f += t3 d, res += t3 T d, g' = grad J(f), J, beta    (here)
// h(t) = J(f + t d) = J_LS(f) + q1 t + q2 t^2 + R(f + t d); each step
// minimises the half-quadratic majorant of h at t_j:
//   h'(t)  = q1 + 2 q2 t + sum_e lambda b(|z_e + t w_e|) Re(conj(z_e + t w_e) w_e)
//   curv   = 2 q2 + sum_e lambda b(|z_e + t w_e|) |w_e|^2
// with z the differences (or pixels) of f and w those of d.  Vectors are FP32;
// sums go through the float-float reductions of reduce.cuh; the scalars are
// FP64 in device memory.
#include <stdint.h>

#include "cg_device.cuh"
#include "chain.cuh"
#include "fft_device.cuh"
#include "internal.cuh"
#include "reduce.cuh"

namespace spirec {

// One pixel per thread up to kVecBlocksPerSm resident blocks an SM (the
// vector kernels are built to fit that many), grid-stride beyond: a single
// wave, and few block partials for the last block to add.
int vec_blocks(int N)
{
    const int64_t P = (int64_t)N * N;
    int sms = 0;
    if (device_sms(&sms) != SPIREC_OK || sms <= 0) sms = 152;
    int64_t b = (P + kVecThreads - 1) / kVecThreads;
    if (b > (int64_t)kVecBlocksPerSm * sms) b = (int64_t)kVecBlocksPerSm * sms;
    if (b > kMaxParts) b = kMaxParts;
    if (b < 1) b = 1;
    return (int)b;
}

namespace {

using cgd::redot;

// A block's part of an N x N image: `rows` rows (fewer at the end) of a strip of
// 256 columns, a thread a column.  The right neighbour of a value comes from
// the next lane, that of a warp's last lane (`edge`) from memory.
struct Strip {
    int n0, n1;
    bool in, has_r, edge;
    int64_t first;  // the thread's pixel of row n0
    __device__ __forceinline__ Strip(int N, int rows)
    {
        const int m = blockIdx.x * kVecThreads + threadIdx.x;
        n0 = blockIdx.y * rows;
        n1 = min(N, n0 + rows);
        in = m < N && n0 < n1;
        has_r = m + 1 < N;
        edge = (threadIdx.x & 31) == 31 && has_r && n0 < n1;
        first = (int64_t)n0 * N + m;
    }
    // the right neighbour's value: `own` of the next lane, `mem` in the last
    static __device__ __forceinline__ float2 right(float2 own, float2 mem)
    {
        const float2 s = make_float2(__shfl_down_sync(0xffffffffu, own.x, 1), __shfl_down_sync(0xffffffffu, own.y, 1));
        return (threadIdx.x & 31) == 31 ? mem : s;
    }
};

// The new direction d = -g + beta d_old (into d_new) and the first line-search
// sums: q1 = Re<d, 2 res> and, over the right and down edges and the pixels,
//   num0 = sum lambda b(|z|) Re(conj(z) w), den0 = sum lambda b(|z|) |w|^2
// (z of f, w of d).  A block walks `rows` rows down a strip of 256 columns: the
// row below's d and f are formed once and kept, the right neighbour's come
// from the next lane, so a pixel costs its own four loads.
//
// Bound by memory latency: 41 us at 2048^2 (five images of 33.5 MB).  With the row FFTs
// in one kernel, where 16 warps an SM hid neither the loads nor each other, the
// two took 160 us; they take 41 + 48.
template <int KIND>
__global__ void __launch_bounds__(kVecThreads, kVecBlocksPerSm)
k_direction(const float2* g, const float2* d_old, float2* d_new, const float2* f, const float2* res, int N, int rows, Reg reg, float2* parts,
            unsigned* counter, double* scal)
{
    chain_enter();
    const double bd = scal[S_BETA];
    const float beta = (float)bd;
    const bool restart = (__double_as_longlong(bd) << 1) == 0;  // beta = 0 (an FP64 compare would be redone every pixel)
    const Strip st(N, rows);
    const float2 zero = make_float2(0.f, 0.f);
    auto dir = [&](int64_t o) { return fftd::new_direction(__ldcg(g + o), restart ? zero : __ldcg(d_old + o), beta, restart); };
    float v[3] = {0.f, 0.f, 0.f};
    int64_t o = st.first;
    float2 dn = st.in ? dir(o) : zero, fn = st.in ? __ldcg(f + o) : zero;
#pragma unroll 2
    for (int n = st.n0; n < st.n1; ++n, o += N) {
        const bool has_d = n + 1 < N;
        const float2 dd = st.in && has_d ? dir(o + N) : dn, fd = st.in && has_d ? __ldcg(f + o + N) : fn;
        const float2 rs = st.in ? __ldcg(res + o) : zero;
        const float2 dr = st.right(dn, st.edge ? dir(o + 1) : dn), fr = st.right(fn, st.edge ? __ldcg(f + o + 1) : fn);
        if (st.in) {
            d_new[o] = dn;
            v[0] += 2.f * redot(dn, rs);
            cgd::ls_terms<KIND>(fn, dn, fr, dr, fd, dd, st.has_r, has_d, reg, 0.f, v[1], v[2]);
        }
        dn = dd;
        fn = fd;
    }
    FF bt[3];
    block_partial<3>(v, bt);
    store_parts<3>(bt, parts, kMaxParts);
    if (last_block(counter)) {
        FF t[3];
        sum_parts_ff<3>(parts, kMaxParts, gridDim.x * gridDim.y, t);
        if (threadIdx.x == 0) {
            scal[S_Q1] = ff_to_double(t[0]);
            scal[S_NUM0] = ff_to_double(t[1]);
            scal[S_DEN0] = ff_to_double(t[2]);
            *counter = 0u;
        }
    }
}

// Line-search step `step` (1 or 2) at t = t_step; the last block forms
// t_{step+1} (cgd::ls_next).  KIND: phi fixed at compile time.
template <int KIND>
__global__ void __launch_bounds__(kVecThreads, kVecBlocksPerSm)
k_line_search(const float2* f, const float2* d, int N, Reg reg, int step, float2* parts,
              unsigned* counter, double* scal)
{
    chain_enter();
    const double t = scal[S_T1 + step - 1];
    const float tf = (float)t;
    const int P = N * N;
    float v[2] = {0.f, 0.f};
#pragma unroll 2
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x)
        cgd::ls_pixel<KIND>(p, N, f, d, reg, tf, v[0], v[1]);
    FF bt[2];
    block_partial<2>(v, bt);
    store_parts<2>(bt, parts, kMaxParts);
    if (last_block(counter)) {
        FF tot[2];
        sum_parts_ff<2>(parts, kMaxParts, gridDim.x, tot);
        if (threadIdx.x == 0) {
            scal[S_T1 + step] = cgd::ls_next(t, scal[S_Q1], scal[S_Q2], ff_to_double(tot[0]), ff_to_double(tot[1]));
            *counter = 0u;
        }
    }
}

// Gradient and step (cgd::update_pixel); the last block forms J and beta.
template <bool FIRST, int KIND>
__global__ void __launch_bounds__(kVecThreads, kVecBlocksPerSm)
k_update(const float2* f_in, float2* f_out, const float2* d, float2* res, const float2* Td,
         const float2* __restrict__ D, float2* g, int N, Reg reg, float2* parts, unsigned* counter,
         double* scal, double* Jout)
{
    chain_enter();
    const float t = FIRST ? 0.f : (float)scal[S_T3];
    const int P = N * N;
    float a[kUpdVals];
#pragma unroll
    for (int i = 0; i < kUpdVals; ++i) a[i] = 0.f;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x)
        cgd::update_pixel<FIRST, KIND>(p, N, f_in, f_out, d, res, Td, D, g, reg, t, a);
    FF bt[kUpdVals];
    block_partial<kUpdVals>(a, bt);
    store_parts<kUpdVals>(bt, parts, kMaxParts);
    if (last_block(counter)) {
        FF tot[kUpdVals];
        sum_parts_ff<kUpdVals>(parts, kMaxParts, gridDim.x, tot);
        if (threadIdx.x == 0) {
            double s[kUpdVals];
            for (int i = 0; i < kUpdVals; ++i) s[i] = ff_to_double(tot[i]);
            double J, beta;
            cgd::update_finish(s, scal[S_SS], scal[S_GG], FIRST, &J, &beta);
            scal[S_GG] = s[0];
            scal[S_BETA] = beta;
            scal[S_J] = J;
            scal[S_R] = s[3];
            if (Jout) *Jout = J;
            *counter = 0u;
        }
    }
}

float2* slot(spirec_plan p, int s) { return reinterpret_cast<float2*>(p->part) + (size_t)s * kMaxParts; }

// res = res - D (res holds T x0) or res = -D (x0 = 0): the residual the
// iteration starts from.
__global__ void k_res_init(float2* res, const float2* __restrict__ D, int64_t n, int have_tx)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 dv = D[i];
        const float2 t = have_tx ? res[i] : make_float2(0.f, 0.f);
        res[i] = make_float2(t.x - dv.x, t.y - dv.y);
    }
}

}  // namespace

int launch_res_init(spirec_plan p, float2* res, bool have_tx)
{
    k_res_init<<<vec_blocks(p->N), kVecThreads, 0, p->stream>>>(res, p->D, (int64_t)p->N * p->N, have_tx ? 1 : 0);
    SPIREC_CK(cudaGetLastError());
    p->launches += 1;
    return SPIREC_OK;
}

namespace {
template <int KIND>
void line_search_k(spirec_plan p, const float2* f, const float2* d, int step)
{
    chain(k_line_search<KIND>, vec_blocks(p->N), kVecThreads, 0, p->stream, f, d, p->N, p->reg, step, slot(p, P_LS),
                                                                         p->counters + C_LS, p->scal);
}

template <int KIND>
void update_k(spirec_plan p, const float2* f_in, float2* f_out, const float2* d, float2* res, const float2* Td,
              float2* g, int first, double* Jout)
{
    if (first)
        chain(k_update<true, KIND>, vec_blocks(p->N), kVecThreads, 0, p->stream, 
            f_in, f_out, d, res, Td, p->D, g, p->N, p->reg, slot(p, P_UPD), p->counters + C_UPD, p->scal, Jout);
    else
        chain(k_update<false, KIND>, vec_blocks(p->N), kVecThreads, 0, p->stream, 
            f_in, f_out, d, res, Td, p->D, g, p->N, p->reg, slot(p, P_UPD), p->counters + C_UPD, p->scal, Jout);
}
}  // namespace

// phi fixed at compile time in the per-pixel work: one kernel per phi
int launch_line_search(spirec_plan p, const float2* f, const float2* d, int step)
{
    switch (p->reg.kind) {
    case SPIREC_PHI_HUBER: line_search_k<SPIREC_PHI_HUBER>(p, f, d, step); break;
    case SPIREC_PHI_HYPERBOLIC: line_search_k<SPIREC_PHI_HYPERBOLIC>(p, f, d, step); break;
    default: line_search_k<SPIREC_PHI_QUADRATIC>(p, f, d, step); break;
    }
    SPIREC_CK(cudaGetLastError());
    p->launches += 1;
    return SPIREC_OK;
}

int launch_update(spirec_plan p, const float2* f_in, float2* f_out, const float2* d, float2* res,
                  const float2* Td, float2* g, int first, double* Jout)
{
    switch (p->reg.kind) {
    case SPIREC_PHI_HUBER: update_k<SPIREC_PHI_HUBER>(p, f_in, f_out, d, res, Td, g, first, Jout); break;
    case SPIREC_PHI_HYPERBOLIC: update_k<SPIREC_PHI_HYPERBOLIC>(p, f_in, f_out, d, res, Td, g, first, Jout); break;
    default: update_k<SPIREC_PHI_QUADRATIC>(p, f_in, f_out, d, res, Td, g, first, Jout); break;
    }
    SPIREC_CK(cudaGetLastError());
    p->launches += 1;
    return SPIREC_OK;
}

namespace {
// Strips of 256 columns by as many rows as fill the resident blocks once.
dim3 strip_grid(int N, int* rows)
{
    int sms = 0;
    if (device_sms(&sms) != SPIREC_OK || sms <= 0) sms = 152;
    const int strips = (N + kVecThreads - 1) / kVecThreads, slots = kVecBlocksPerSm * sms;
    *rows = (int)(((int64_t)N * strips + slots - 1) / slots);
    if (*rows < 1) *rows = 1;
    return dim3((unsigned)strips, (unsigned)((N + *rows - 1) / *rows));
}

template <int KIND>
void direction_k(spirec_plan p, int k)
{
    int rows = 0;
    const dim3 grid = strip_grid(p->N, &rows);
    chain(k_direction<KIND>, grid, kVecThreads, 0, p->stream, p->g, p->dbuf[(k + 1) & 1], p->dbuf[k & 1], p->f[k & 1], p->res,
                                                           p->N, rows, p->reg, slot(p, P_ROWA), p->counters + C_ROWA,
                                                           p->scal);
}

// d of iteration k, q1 and the t = 0 line-search sums.
int launch_direction(spirec_plan p, int k)
{
    switch (p->reg.kind) {
    case SPIREC_PHI_HUBER: direction_k<SPIREC_PHI_HUBER>(p, k); break;
    case SPIREC_PHI_HYPERBOLIC: direction_k<SPIREC_PHI_HYPERBOLIC>(p, k); break;
    default: direction_k<SPIREC_PHI_QUADRATIC>(p, k); break;
    }
    SPIREC_CK(cudaGetLastError());
    p->launches += 1;
    return SPIREC_OK;
}
}  // namespace

// q2 = Re<d, T d> and the first line-search step
//   t1 = -(q1 + num0) / (2 q2 + den0)   (0 when the curvature is not > 0),
// as the fused row pass 3 of the FFT path computes them.
__global__ void k_q2_t1(const float2* d, const float2* Td, int64_t n, float2* parts, unsigned* counter,
                        double* scal)
{
    chain_enter();
    float v[1] = {0.f};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 a = __ldcg(d + i), b = __ldcg(Td + i);
        v[0] += fmaf(a.x, b.x, a.y * b.y);
    }
    FF bt[1];
    block_partial<1>(v, bt);
    store_parts<1>(bt, parts, kMaxParts);
    if (last_block(counter)) {
        FF t[1];
        sum_parts_ff<1>(parts, kMaxParts, gridDim.x, t);
        if (threadIdx.x == 0) {
            const double q2 = ff_to_double(t[0]);
            scal[S_Q2] = q2;
            const double curv = 2.0 * q2 + scal[S_DEN0];
            scal[S_T1] = curv > 0.0 ? -(scal[S_Q1] + scal[S_NUM0]) / curv : 0.0;
            *counter = 0u;
        }
    }
}

int launch_normal_direct(spirec_plan p, const float2* x, float2* Tx, bool dot_q2_t1)
{
    if (!p->ydir) {
        set_error("direct mode needs spirec_set_mode first");
        return SPIREC_ESTATE;
    }
    int rc;
    if ((rc = launch_forward(p, x, p->ydir)) != SPIREC_OK) return rc;
    if ((rc = launch_adjoint(p, p->ydir, Tx)) != SPIREC_OK) return rc;
    if (dot_q2_t1) {
        chain(k_q2_t1, vec_blocks(p->N), kVecThreads, 0, p->stream, x, Tx, (int64_t)p->N * p->N, slot(p, P_ROWC),
                                                                  p->counters + C_ROWC, p->scal);
        SPIREC_CK(cudaGetLastError());
        p->launches += 1;
    }
    return SPIREC_OK;
}

int cg_iteration(spirec_plan p, int k, double* Jdev)
{
    const float2* fin = p->f[k & 1];
    float2* fout = p->f[(k + 1) & 1];
    float2* dk = p->dbuf[k & 1];
    int rc;
    if ((rc = launch_direction(p, k)) != SPIREC_OK) return rc;
    if (p->mode == SPIREC_MODE_DIRECT) {
        if ((rc = launch_normal_direct(p, dk, p->Td, true)) != SPIREC_OK) return rc;
    } else {
        const CgPass c{slot(p, P_ROWC), p->counters + C_ROWC, p->scal};
        if ((rc = launch_toeplitz(p, dk, p->Td, &c)) != SPIREC_OK) return rc;
    }
    for (int j = 1; j <= 2; ++j)
        if ((rc = launch_line_search(p, fin, dk, j)) != SPIREC_OK) return rc;
    return launch_update(p, fin, fout, dk, p->res, p->Td, p->g, 0, Jdev ? Jdev + k + 1 : nullptr);
}

}  // namespace spirec
