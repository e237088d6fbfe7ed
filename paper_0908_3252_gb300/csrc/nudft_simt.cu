// nudft_simt.cu -- FP32 CUDA-core contractions of the exact NUDFT:
//   G (Eq. AnnMatG), D = H^H s (Eq. AnnMatGD) and y = H x (Eq. ModDirect).
//
// G and D are both "phase GEMMs" of K = L whose operands are generated in
// shared memory from the fixed-point trajectory (phase.cuh) and never stored
// in HBM.  The B operand is a pure phase and its conjugate is the phase of the
// mirrored output column, so the four real products of A' = Ar + i Ai and
// E = Br + i Bi give two output columns (PairGeom, internal.cuh): half the
// multiply-adds of forming every column on its own.  Because the output is
// small (N x (2N-1) at most) and K is huge, the sample axis is split over
// grid.z (split-K); each split writes FP32 partials and a second kernel sums
// them in a fixed order, so results do not depend on scheduling.
#include <stdint.h>

#include "internal.cuh"
#include "phase.cuh"

namespace spirec {

namespace {

constexpr int TM = 64;   // tile rows (i)
constexpr int TN = 64;   // tile cols (c)
constexpr int KC = 32;   // samples per shared-memory stage
constexpr int NT = 256;  // threads

// acc.{x,y} += a.{x,y} * b.{x,y}: one packed FP32 instruction.
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t dup2(float v)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

// Block shapes of k_phase_gemm: ROWS x 64 outputs, four rows and four B columns
// a thread; 128 rows by one block of 16 warps an SM, 64 rows by two of 8.
template <int ROWS>
struct GemmShape {
    static constexpr int THREADS = 4 * ROWS;
    static constexpr int BLOCKS_PER_SM = 128 / ROWS;
    static constexpr int FACTORS = ROWS / 8 + 8 + TN / 8 + 8;  // base and offset phasors of a sample
    // two chunks of the operands and the factor tables (rows padded so that
    // the factors of one sample are in distinct banks)
    struct Smem {
        float2 As[2][KC][ROWS];
        float2 Bs[2][KC][TN];
        float2 tab[2][FACTORS][KC + 1];
    };
};

// A tile of ROWS rows i x 64 B columns j:
//   A'(l,i) = w'_l exp(sa i2pi ka_l (i + oa)) (w' = 1 unweighted),
//   E(l,j)  = exp(sb i2pi kb_l (j + half/2)),
// sums (P_ac, P_ad) += (Ar, Ar) * (Br, Bi) and (P_bc, P_bd) += (Ai, Ai) *
// (Br, Bi), stored as the two output columns c+(j), c-(j).  A tile entry (l, i)
// is base[l][i/8] * off[l][i%8] with base = exp(i2pi k (i0 + 8a + o)) and off =
// exp(i2pi k b).
//
// Pipelined over chunks of 32 samples with one barrier a chunk: while chunk c
// is multiplied, the operands of c + 1 and the factors of c + 2 are formed.
// Half of each scheduler's warps form first and multiply after, the others the
// other way round, so that the FP32 pipe has work from some warp.
//
// Bound by the FP32 pipe (71% busy, issue slots 55%: forming the operands is a
// quarter of the instructions).  D at N = 256, L = 32768: 174 us, 4.3e9
// multiply-adds at 65% of the pipe's rate; 460 us before, when every column was
// formed on its own by scalar multiply-adds between three barriers a chunk.
// With 64 x 64 blocks, three barriers and A stored duplicated the pairing gave
// 245 us, with this pipeline and A duplicated 238 us (shared-memory loads).
template <bool WEIGHTED, int ROWS>
__global__ void __launch_bounds__(GemmShape<ROWS>::THREADS, GemmShape<ROWS>::BLOCKS_PER_SM)
k_phase_gemm(const int64_t* __restrict__ ka, const int64_t* __restrict__ kb,
             const float2* __restrict__ w, int64_t L, PairGeom pg, int oa, int sa,
             int sb, int64_t chunks_per_split, float2* __restrict__ part)
{
    using G = GemmShape<ROWS>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    typename G::Smem& S = *reinterpret_cast<typename G::Smem*>(smem_raw);

    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int i0 = blockIdx.y * ROWS, j0 = blockIdx.x * TN;
    const int64_t nchunks = (L + KC - 1) / KC;
    const int64_t ch0 = (int64_t)blockIdx.z * chunks_per_split;
    const int nch = (int)(min(nchunks, ch0 + chunks_per_split) - ch0);

    // factors of chunk c (of this block's nch) into tab[c & 1]; a warp's lanes
    // take its 32 samples for one factor
    auto factors = [&](int c) {
        const int64_t lg = (ch0 + c) * KC + (tid & 31);
#pragma unroll
        for (int f0 = 0; f0 < G::FACTORS; f0 += G::THREADS / 32) {
            const int f = f0 + (tid >> 5);
            if (f < G::FACTORS) {
                constexpr int AB = ROWS / 8, B0 = AB + 8, BB = TN / 8;
                const bool isA = f < B0;
                const int q = isA ? f : f - B0;  // factor within its side
                const int nb = isA ? AB : BB;
                float2 v = make_float2(0.f, 0.f);  // samples past L: zero
                if (lg < L) {
                    const int64_t k = isA ? ka[lg] : kb[lg];
                    const int j = q >= nb ? q - nb : 8 * q + (isA ? i0 + oa : j0);
                    // a half-integer offset adds k / 2 (an error of 2^-65 cycles)
                    v = phasor_q(k, j, !isA && q < nb && pg.half ? k >> 1 : 0);
                    if ((isA ? sa : sb) < 0) v.y = -v.y;
                    if (WEIGHTED && isA && q >= nb) v = cmul(v, w[lg]);
                }
                S.tab[c & 1][f][tid & 31] = v;
            }
        }
    };
    // operands of chunk c from its factors
    auto operands = [&](int c) {
        constexpr int AB = ROWS / 8, B0 = AB + 8, BB = TN / 8;
        const int bf = c & 1;
#pragma unroll
        for (int e = tid; e < KC * ROWS; e += G::THREADS) {
            const int l = e / ROWS, i = e % ROWS;
            S.As[bf][l][i] = cmul(S.tab[bf][i >> 3][l], S.tab[bf][AB + (i & 7)][l]);
        }
#pragma unroll
        for (int e = tid; e < KC * TN; e += G::THREADS) {
            const int l = e / TN, i = e % TN;
            S.Bs[bf][l][i] = cmul(S.tab[bf][B0 + (i >> 3)][l], S.tab[bf][B0 + BB + (i & 7)][l]);
        }
    };

    uint64_t accr[4][4], acci[4][4];  // (P_ac, P_ad), (P_bc, P_bd)
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) accr[r][c] = acci[r][c] = 0;  // two FP32 zeros

    if (nch > 0) factors(0);
    __syncthreads();
    if (nch > 0) operands(0);
    if (nch > 1) factors(1);
    __syncthreads();
    const bool form_first = (tid >> 7) & 1;
    for (int c = 0; c < nch; ++c) {
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            if ((ph == 0) == form_first) {
                // the buffers written were last read before the barrier
                if (c + 1 < nch) operands(c + 1);
                if (c + 2 < nch) factors(c + 2);
            } else {
                // rows 2 ty + (0, 1) + ROWS / 2 h, columns 2 tx + (0, 1) + 32 h:
                // 16-byte loads of two neighbours, A's duplicated in registers
                // for the packed multiply-adds
                const float2* As = &S.As[c & 1][0][2 * ty];
                const float2* Bs = &S.Bs[c & 1][0][2 * tx];
#pragma unroll 4
                for (int l = 0; l < KC; ++l) {
                    uint64_t b[4];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(Bs + l * TN + 32 * h);
                        b[2 * h] = v.x;
                        b[2 * h + 1] = v.y;
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 a = *reinterpret_cast<const float4*>(As + l * ROWS + (ROWS / 2) * h);
                        const uint64_t ar0 = dup2(a.x), ai0 = dup2(a.y), ar1 = dup2(a.z), ai1 = dup2(a.w);
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            fma2(accr[2 * h][q], ar0, b[q]);
                            fma2(acci[2 * h][q], ai0, b[q]);
                            fma2(accr[2 * h + 1][q], ar1, b[q]);
                            fma2(acci[2 * h + 1][q], ai1, b[q]);
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
    float2* out = part + (int64_t)blockIdx.z * pg.R * pg.C;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = i0 + 2 * ty + (r & 1) + (ROWS / 2) * (r >> 1);
        if (i >= pg.R) continue;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j = j0 + 2 * tx + (c & 1) + 32 * (c >> 1);
            if (j >= pg.J) continue;
            const float2 ar = unpack2(accr[r][c]), ai = unpack2(acci[r][c]);  // (ac, ad), (bc, bd)
            const int off = 2 * j + pg.half;
            float2* row = out + (int64_t)i * pg.C;
            row[(pg.C2 + off) / 2] = make_float2(ar.x - ai.y, ar.y + ai.x);
            if (off > 0) row[(pg.C2 - off) / 2] = make_float2(ar.x + ai.y, ai.x - ar.y);
        }
    }
}

// out[e] = scale * sum_s part[s][e], fixed summation order: Z threads an
// element sum Z contiguous ranges of the slices, four loads in flight, and the
// first adds the ranges' sums in order (latency-bound: a small image has few
// elements and hundreds of slices).
template <int Z>
__global__ void __launch_bounds__(256) k_reduce_splits(const float2* __restrict__ part, int S, int64_t RC, float scale,
                                                       float2* __restrict__ out)
{
    constexpr int E = 256 / Z;  // elements a block
    __shared__ float2 sums[Z > 1 ? 256 : 1];
    const int ex = threadIdx.x % E, z = threadIdx.x / E;
    for (int64_t e0 = blockIdx.x * (int64_t)E; e0 < RC; e0 += (int64_t)gridDim.x * E) {
        const int64_t e = e0 + ex;
        float2 a = make_float2(0.f, 0.f);
        if (e < RC) {
            const int se = S * (z + 1) / Z;
#pragma unroll 4
            for (int s = S * z / Z; s < se; ++s) {
                const float2 v = part[(int64_t)s * RC + e];
                a.x += v.x;
                a.y += v.y;
            }
        }
        if constexpr (Z > 1) {
            __syncthreads();  // the previous elements' sums are read
            sums[threadIdx.x] = a;
            __syncthreads();
            if (z == 0)
#pragma unroll
                for (int k = 1; k < Z; ++k) {
                    a.x += sums[k * E + ex].x;
                    a.y += sums[k * E + ex].y;
                }
        }
        if (z == 0 && e < RC) out[e] = make_float2(a.x * scale, a.y * scale);
    }
}

// Eight threads an element where there are slices for them.
void launch_reduce_splits(cudaStream_t st, const float2* part, int S, int64_t RC, float scale, float2* out)
{
    const int E = S >= 16 ? 32 : 256;
    int64_t blocks = (RC + E - 1) / E;
    if (blocks > 8 * 152) blocks = 8 * 152;
    if (S >= 16) k_reduce_splits<8><<<(unsigned)blocks, 256, 0, st>>>(part, S, RC, scale, out);
    else k_reduce_splits<1><<<(unsigned)blocks, 256, 0, st>>>(part, S, RC, scale, out);
}

// y = H x.  Z[n][l] = sum_m x[n][m] exp(i2pi kx_l m) as a GEMM (A = image rows,
// B = generated phases), then y_l += sum_n exp(i2pi ky_l n) Z[n][l] in the
// epilogue; the N x L intermediate never leaves registers.  grid.y splits the
// row blocks; partials ypart[split][l].
__global__ void __launch_bounds__(NT, 2)
k_forward(const int64_t* __restrict__ kxq, const int64_t* __restrict__ kyq,
          const float2* __restrict__ x, int N, int64_t L, float2* __restrict__ ypart)
{
    __shared__ float2 As[TM][KC + 1];   // image tile [row][m]
    __shared__ float2 Bs[KC][TN];       // phases [m][l]
    __shared__ float2 off[TN][8];       // exp(i2pi kx_l b), b < 8
    __shared__ float2 base[TN][KC / 8]; // exp(i2pi kx_l (m0 + 8a))
    __shared__ float2 red[16][TN];

    const int tid = threadIdx.x;
    const int tx = tid & 15, ty = tid >> 4;
    const int64_t l0 = (int64_t)blockIdx.x * TN;
    const int nblocks = (N + TM - 1) / TM;

    for (int e = tid; e < TN * 8; e += NT) {
        const int c = e / 8, b = e % 8;
        const int64_t lg = l0 + c;
        off[c][b] = lg < L ? phasor_q(kxq[lg], b) : make_float2(0.f, 0.f);
    }
    float2 yacc = make_float2(0.f, 0.f);  // thread c < TN owns sample l0 + c

    for (int nb = blockIdx.y; nb < nblocks; nb += gridDim.y) {
        const int n0 = nb * TM;
        float2 acc[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.f, 0.f);

        for (int m0 = 0; m0 < N; m0 += KC) {
            __syncthreads();
            for (int e = tid; e < TN * (KC / 8); e += NT) {
                const int c = e / (KC / 8), a = e % (KC / 8);
                const int64_t lg = l0 + c;
                base[c][a] = lg < L ? phasor_q(kxq[lg], m0 + 8 * a) : make_float2(0.f, 0.f);
            }
            for (int e = tid; e < TM * KC; e += NT) {
                const int r = e / KC, k = e % KC;
                const int n = n0 + r, m = m0 + k;
                As[r][k] = (n < N && m < N) ? x[(int64_t)n * N + m] : make_float2(0.f, 0.f);
            }
            __syncthreads();
            for (int e = tid; e < KC * TN; e += NT) {
                const int k = e / TN, c = e % TN;
                Bs[k][c] = cmul(base[c][k >> 3], off[c][k & 7]);
            }
            __syncthreads();
#pragma unroll 4
            for (int k = 0; k < KC; ++k) {
                float2 a[4], b[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) a[r] = As[ty + 16 * r][k];
#pragma unroll
                for (int c = 0; c < 4; ++c) b[c] = Bs[k][tx + 16 * c];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        acc[r][c].x = fmaf(a[r].x, b[c].x, acc[r][c].x);
                        acc[r][c].x = fmaf(-a[r].y, b[c].y, acc[r][c].x);
                        acc[r][c].y = fmaf(a[r].x, b[c].y, acc[r][c].y);
                        acc[r][c].y = fmaf(a[r].y, b[c].x, acc[r][c].y);
                    }
            }
        }
        // epilogue: sum_n exp(i2pi ky_l n) Z[n][l] over this row block
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int64_t lg = l0 + tx + 16 * c;
            float2 sacc = make_float2(0.f, 0.f);
            if (lg < L) {
                const int64_t k = kyq[lg];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int n = n0 + ty + 16 * r;
                    if (n < N) {
                        const float2 e = cmul(phasor_q(k, n), acc[r][c]);
                        sacc.x += e.x;
                        sacc.y += e.y;
                    }
                }
            }
            red[ty][tx + 16 * c] = sacc;
        }
        __syncthreads();
        if (tid < TN) {
            for (int r = 0; r < 16; ++r) {
                yacc.x += red[r][tid].x;
                yacc.y += red[r][tid].y;
            }
        }
    }
    if (tid < TN && l0 + tid < L) ypart[(int64_t)blockIdx.y * L + l0 + tid] = yacc;
}

// Rows of a block of k_phase_gemm: 128 (a quarter fewer operand values formed
// per multiply-add), unless that pads the rows by an eighth more than 64 does.
int gemm_rows(int R)
{
    const int p64 = (R + 63) / 64 * 64, p128 = (R + 127) / 128 * 128;
    return 8 * p128 <= 9 * p64 ? 128 : 64;
}
int64_t gemm_tiles(int R, int J)
{
    const int rows = gemm_rows(R);
    return (int64_t)((R + rows - 1) / rows) * ((J + TN - 1) / TN);
}
int gemm_blocks_per_sm(int R) { return 128 / gemm_rows(R); }

// Sample slices of the contraction: the tuned value of the shape, else those
// whose blocks (tiles x slices) take the fewest chunks one after the other,
// waves x chunks a slice, in up to two waves of resident blocks; the fewest
// slices among equals.  Bounded by the work and by the partial-sum buffer.
int choose_splits(spirec_plan p, int knob, int sms, const PairGeom& pg, int64_t nchunks)
{
    const size_t part_cap_elems = p->kpart_bytes / sizeof(float2);
    const int64_t RC = (int64_t)pg.R * pg.C, tiles = gemm_tiles(pg.R, pg.J);
    const int tuned = tune_lookup(knob, p, sms);
    int64_t S = tuned;
    if (tuned <= 0) {
        const int64_t slots = (int64_t)gemm_blocks_per_sm(pg.R) * sms;
        int64_t best = INT64_MAX;
        S = 1;
        for (int64_t z = 1; z == 1 || (tiles * z <= 2 * slots && z <= nchunks); ++z) {
            const int64_t cost = (tiles * z + slots - 1) / slots * ((nchunks + z - 1) / z);
            if (cost < best && (size_t)(z * RC) <= part_cap_elems) {
                best = cost;
                S = z;
            }
        }
    }
    if (S > nchunks) S = nchunks;
    if (S < 1) S = 1;
    while (S > 1 && (size_t)(S * RC) > part_cap_elems) --S;
    return (int)S;
}

template <int ROWS>
void launch_gemm(cudaStream_t st, const int64_t* ka, const int64_t* kb, const float2* w, int64_t L, const PairGeom& pg,
                 int oa, int sa, int sb, int64_t cps, int S, float2* part)
{
    using G = GemmShape<ROWS>;
    const dim3 grid((pg.J + TN - 1) / TN, (pg.R + ROWS - 1) / ROWS, S);
    if (w)
        k_phase_gemm<true, ROWS><<<grid, G::THREADS, sizeof(typename G::Smem), st>>>(ka, kb, w, L, pg, oa, sa, sb, cps, part);
    else
        k_phase_gemm<false, ROWS><<<grid, G::THREADS, sizeof(typename G::Smem), st>>>(ka, kb, w, L, pg, oa, sa, sb, cps, part);
}

// out[i][c] = scale sum_l A(l,i) B(l,c), as tc_pair_gemm.
int phase_gemm(spirec_plan p, int knob, const int64_t* ka, const int64_t* kb, bool weighted, int oa, int sa, int sb,
               float scale, float2* out)
{
    const PairGeom pg = pair_geom(p, knob);
    const int64_t nchunks = (p->L + KC - 1) / KC;
    const int64_t RC = (int64_t)pg.R * pg.C;
    int sms = 0, rc;
    if ((rc = device_sms(&sms)) != SPIREC_OK) return rc;
    const float2* w = weighted ? p->wpair : nullptr;
    const int S = choose_splits(p, knob, sms, pg, nchunks);
    const int64_t cps = (nchunks + S - 1) / S;
    const int Seff = (int)((nchunks + cps - 1) / cps);
    float2* part = reinterpret_cast<float2*>(p->kpart);
    if (gemm_rows(pg.R) == 128) launch_gemm<128>(p->stream, ka, kb, w, p->L, pg, oa, sa, sb, cps, Seff, part);
    else launch_gemm<64>(p->stream, ka, kb, w, p->L, pg, oa, sa, sb, cps, Seff, part);
    SPIREC_CK(cudaGetLastError());
    launch_reduce_splits(p->stream, part, Seff, RC, scale, out);
    SPIREC_CK(cudaGetLastError());
    p->launches += 2;
    return SPIREC_OK;
}

}  // namespace

int launch_gram(spirec_plan p)
{
    if (p->precision != SPIREC_FP32) return launch_gram_tc(p);
    const int N = p->N;
    // G[u][v+N-1] = (1/N^2) sum_l exp(i2pi kx_l u) exp(i2pi ky_l v)
    return phase_gemm(p, SPIREC_KNOB_GRAM_SPLIT, p->kxq, p->kyq, false, 0, +1, +1,
                      1.0f / ((float)N * (float)N), p->G);
}

int launch_adjoint_prepared(spirec_plan p, float2* x)
{
    if (p->precision != SPIREC_FP32) return launch_adjoint_tc(p, x);
    // x[n][m] = (1/N) sum_l exp(-i2pi ky_l n) * (y_l exp(-i2pi kx_l m))
    return phase_gemm(p, SPIREC_KNOB_ADJOINT_SPLIT, p->kyq, p->kxq, true, 0, -1, -1, 1.0f / (float)p->N, x);
}

int launch_adjoint(spirec_plan p, const float2* y, float2* x)
{
    const int rc = launch_pair_weights(p, y, false);
    return rc != SPIREC_OK ? rc : launch_adjoint_prepared(p, x);
}

int contraction_split(spirec_plan p, int knob, int* value, int* sms_used)
{
    int sms = 0, rc;
    if ((rc = device_sms(&sms)) != SPIREC_OK) return rc;
    if (p->precision != SPIREC_FP32) {
        int64_t P = 0;
        if ((rc = tc_ctas(p, knob, sms, &P)) != SPIREC_OK) return rc;
        *value = (int)P;
        *sms_used = (int)P;  // one CTA per SM (its shared memory)
        return SPIREC_OK;
    }
    const PairGeom pg = pair_geom(p, knob);
    const int64_t nchunks = (p->L + KC - 1) / KC;
    const int S = choose_splits(p, knob, sms, pg, nchunks);
    const int64_t cps = (nchunks + S - 1) / S;
    const int64_t blocks = gemm_tiles(pg.R, pg.J) * ((nchunks + cps - 1) / cps);
    const int per_sm = gemm_blocks_per_sm(pg.R);
    const int64_t used = (blocks + per_sm - 1) / per_sm;
    *value = S;
    *sms_used = (int)(used < sms ? used : sms);
    return SPIREC_OK;
}

// Floats of split-K partials that the FP32 contractions use: at least eight
// slices of G, and one wave of blocks (which a small image cuts into many
// slices).
size_t kpart_floats_simt(int N, int64_t L)
{
    const size_t GC = (size_t)N * (2 * N - 1);
    size_t S = (size_t)gemm_blocks_per_sm(N) * 152 / (size_t)gemm_tiles(N, N);
    const size_t nchunks = (size_t)((L + KC - 1) / KC);
    if (S > nchunks) S = nchunks;
    if (S < 8) S = 8;
    return 2 * S * GC;
}

template <int ROWS>
static int gemm_attributes()
{
    const int bytes = (int)sizeof(typename GemmShape<ROWS>::Smem);
    SPIREC_CK(cudaFuncSetAttribute(k_phase_gemm<true, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    SPIREC_CK(cudaFuncSetAttribute(k_phase_gemm<false, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    return SPIREC_OK;
}

int simt_setup_attributes()
{
    const int rc = gemm_attributes<64>();
    return rc != SPIREC_OK ? rc : gemm_attributes<128>();
}

int launch_forward(spirec_plan p, const float2* x, float2* y)
{
    if (p->precision != SPIREC_FP32) return launch_forward_tc(p, x, y);
    const int64_t lblocks = (p->L + TN - 1) / TN;
    const int nblocks = (p->N + TM - 1) / TM;
    int ns = (int)((4 * 152 + lblocks - 1) / lblocks);
    if (ns > nblocks) ns = nblocks;
    if (ns < 1) ns = 1;
    while (ns > 1 && (size_t)ns * p->L * sizeof(float2) > p->kpart_bytes) --ns;
    float2* part = reinterpret_cast<float2*>(p->kpart);
    dim3 grid((unsigned)lblocks, ns);
    k_forward<<<grid, NT, 0, p->stream>>>(p->kxq, p->kyq, x, p->N, p->L, part);
    SPIREC_CK(cudaGetLastError());
    launch_reduce_splits(p->stream, part, ns, p->L, 1.0f / (float)p->N, y);
    SPIREC_CK(cudaGetLastError());
    p->launches += 2;
    return SPIREC_OK;
}

}  // namespace spirec
