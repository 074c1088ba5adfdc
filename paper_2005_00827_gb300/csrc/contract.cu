// Contraction of the bubble tables with two vertices, all output triples.
//
// With B_f[Q][a][b] from bubble.cu (a = patch of the loop point p, b = patch of
// its partner), the three channels of the one-loop flow (App. A.1,
// Eq. (vertex_flow_general)) become, for k = (a, b) in N^2:
//   pp (Q = k1+k2 = (i,j)):  dV[i,j,l] -= sum_k B_pp[i,j][k] V[i,j,a] * V[a,b,l]
//   cr (Q = k3-k2 = (l,j)):  dV[i,j,l] -= sum_k B_ph[l,j][k] V[b,j,l] * V[i,a,b]
//   d  (Q = k1-k3 = (i,l)):  dV[i,j,l] += sum_k B_ph[i,l][k] {(2V[i,a,l] - V[a,i,l]) V[b,j,a]
//                                                          - V[i,a,l] V[j,b,a]}
// Each channel is a GEMM with the table's rows Q as rows, K = N^2 and N
// columns n (n = l, i, j), whose A operand is a table row times a vertex factor
// (formed while staging into shared memory) and whose B operand is a permuted
// view of V; d is two such GEMMs of the same size.  FP64 and FP32 (SIMT):
//   stage_prep_kernel   the permuted views P[k][n] of cr, d1, d2, the FP32 copy
//                       and the C4v test of the inputs, one launch
//   contract_kernel     the four GEMMs, one launch, into partial rows
//   reduce_kernel       sums the partial rows
//   expand_kernel       sums the channels into out
// A C4v-symmetric (V, Z) tables and contracts one row per orbit of transfer
// pairs (row orbits, symmetry.cu); the expansion permutes the columns.  Which
// form a right-hand side takes may be decided on the device (SymMode), so that
// the call stays asynchronous.
#include <algorithm>

#include "qpfrg_internal.h"

namespace qpfrg {

constexpr int CBK = 16;      // reduction columns b per staged block

// Rows of the table and split of the reduction over a, per form of the RHS.
struct ContractShape {
    int rows, mtiles, splits, a_per;
};

template <typename R>
struct ContractArgs {
    const R *B;                  // bubble tables [f][row][a][b], family stride N^4
    const R *V;                  // stage vertex
    const R *P;                  // permuted views [cr, d1, d2][a][b][n]
    const int *rep;              // compact form: [family][row] transfer pair of a row
    int n_can;                   // compact form: rows of the table (row m >= n_can holds the table row m - n_can)
    double *part;                // [split][job][row][n]
    int N, ntiles, njobs;
    int jobs[4];                 // 0 pp, 1 cr, 2 d first product, 3 d second product
    ContractShape sh[2];         // every row, representative rows
    SymMode sym;
};

// One CTA: rows m0 .. m0 + 16 TM - 1, columns n0 .. n0 + 16 NB - 1, one job and
// one range of a; 256 threads as 16 x 16, TM rows x NB columns each.
//
// What bounds it: GB300 issues 2 FP64 FMAs per clock and SM (64 clocks per warp
// instruction and scheduler), so in FP64 the staging, its index arithmetic and
// the two shared reads per FMA hide behind the FMA pipe, and what counts is the
// number of rows contracted and an even share of the SMs (the split over a).  In FP32
// 12 FMAs per 5 shared reads keep the FMA pipe ahead of shared memory.  The
// next block's table values and factors are loaded while the present one is
// multiplied.  The crossed channel's factor depends on b, not on a: its blocks
// run with b outside and a inside, so the gathered factor is read once per b.
// np48, 16 x 16 points, symmetric vertex: FP64 6232 -> 350 us, FP32 1487 -> 28 us
// (every row, one launch per channel -> representative rows, one launch).
template <typename R, int TM, int NB>
__global__ void __launch_bounds__(256) contract_kernel(const ContractArgs<R> A)
{
    constexpr int BM = 16 * TM, BN = 16 * NB;
    const bool compact = sym_compact(A.sym);
    const ContractShape sh = A.sh[compact ? 1 : 0];
    int id = blockIdx.x;
    const int mt = id % sh.mtiles;
    id /= sh.mtiles;
    const int nt = id % A.ntiles;
    id /= A.ntiles;
    const int ji = id % A.njobs, sp = id / A.njobs;
    if (sp >= sh.splits) return;            // CTAs of the other form's grid
    const int job = A.jobs[ji];
    const int N = A.N, m0 = mt * BM, n0 = nt * BN;
    const long NN = (long)N * N;
    const int a0 = sp * sh.a_per, a1 = min(N, a0 + sh.a_per);
    const int tid = threadIdx.x, tr = tid >> 4, tn = tid & 15;

    __shared__ R As[2][CBK][BM + 4];
    __shared__ R Bs[2][CBK][BN];

    // staged A elements of this thread: rows (tid / 16) + 16 e, column tid % 16
    const int kk = tid & 15;
    const R *Brow[TM];
    const R *frow[TM], *grow[TM];           // factor of (row, x): frow[x fstride] (and grow for d1)
    bool rok[TM];
    // pp: V[i,j,a]; cr: V[b,j,l]; d1: 2V[i,a,l] - V[a,i,l]; d2: -V[i,a,l]
    const long fstride = job == 0 ? 1 : (job == 1 ? NN : N);
#pragma unroll
    for (int e = 0; e < TM; ++e) {
        const int m = m0 + (tid >> 4) + 16 * e;
        rok[e] = m < sh.rows;
        const int mm = rok[e] ? m : 0;
        const int Q = compact ? A.rep[mm + (job == 0 ? 0 : sh.rows)] : mm;
        const int trow = compact && mm >= A.n_can ? mm - A.n_can : mm;
        const int q1 = Q / N, q2 = Q - q1 * N;
        Brow[e] = A.B + (job == 0 ? 0 : NN * NN) + (long)trow * NN;
        frow[e] = A.V + (job == 0 ? (long)Q * N : (job == 1 ? (long)q2 * N + q1 : (long)q1 * NN + q2));
        grow[e] = A.V + (long)q1 * N + q2;   // + a N^2
    }
    const R *Pj = job == 0 ? A.V : A.P + (job - 1) * NN * N;

    R acc[TM][NB];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) acc[i][j] = R(0);

    R an[TM], fn[TM], bn[NB];
    auto load = [&](int a, int b0, bool newfac) {
        const int b = b0 + kk;
        const bool bok = b < N;
#pragma unroll
        for (int e = 0; e < TM; ++e) {
            an[e] = (rok[e] && bok) ? Brow[e][(long)a * N + b] : R(0);
            if (newfac) {
                const int x = job == 1 ? (bok ? b : 0) : a;
                R f = frow[e][x * fstride];
                if (job == 2) f = R(2) * f - grow[e][(long)a * NN];
                else if (job == 3) f = -f;
                fn[e] = f;
            }
        }
#pragma unroll
        for (int e = 0; e < NB; ++e) {
            const int idx = tid + 256 * e, kb = idx / BN, n = n0 + idx % BN;
            bn[e] = (b0 + kb < N && n < N) ? Pj[((long)a * N + b0 + kb) * N + n] : R(0);
        }
    };
    const int nbc = (N + CBK - 1) / CBK, na = a1 - a0;
    const int total = na * nbc;
    int a = a0, b0 = 0;
    if (total > 0) load(a, b0, true);
    for (int t = 0; t < total; ++t) {
        const int s = t & 1;
#pragma unroll
        for (int e = 0; e < TM; ++e) As[s][kk][(tid >> 4) + 16 * e] = an[e] * fn[e];
#pragma unroll
        for (int e = 0; e < NB; ++e) {
            const int idx = tid + 256 * e;
            Bs[s][idx / BN][idx % BN] = bn[e];
        }
        __syncthreads();     // also: every warp is past the block of two trips ago
        bool nf;
        if (job == 1) {      // b outside, a inside
            nf = ++a == a1;
            if (nf) {
                a = a0;
                b0 += CBK;
            }
        } else {
            b0 += CBK;
            nf = b0 >= N;
            if (nf) {
                b0 = 0;
                ++a;
            }
        }
        if (t + 1 < total) load(a, b0, nf);
#pragma unroll
        for (int k = 0; k < CBK; ++k) {
            R av[TM], bv[NB];
#pragma unroll
            for (int i = 0; i < TM; ++i) av[i] = As[s][k][tr * TM + i];
#pragma unroll
            for (int j = 0; j < NB; ++j) bv[j] = Bs[s][k][tn + 16 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < NB; ++j) acc[i][j] += av[i] * bv[j];
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int m = m0 + tr * TM + i;
        if (m >= sh.rows) continue;
        double *dst = A.part + (((long)sp * A.njobs + ji) * sh.rows + m) * N;
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            const int n = n0 + tn + 16 * j;
            if (n < N) dst[n] = (double)acc[i][j];
        }
    }
}

// Channel rows outc[0 pp, 1 cr, 2 d][row][n] = the signed sums of the partial
// rows over splits (and both products of d), in split order, so that the result
// does not depend on the launch.  Compact form: a mirror that leaves the row's pair
// in place takes column n to an equal one up to rounding; both get the sum of the
// lower one, so that the expanded right-hand side is C4v symmetric to the last bit (a
// flow keeps its symmetry, and takes the same form when it is resumed from an image).
// Then out[k1,k2,k3] = scale * (pp + cr + d): pp
// row (k1,k2) column k3, cr row (k3,k2) column k1, d row (k1,k3) column k2.
// Compact form: row Q = g rep at column n is the representative's at g^-1 n.
// Two launches: an expansion that summed the splits itself read each partial
// row once per image (np48 symmetric: 34 us against 4 + 4).
struct ExpandArgs {
    const double *part;
    double *outc;
    const int *rowmap;
    const uint8_t *rstab;
    double *out;
    double scale;
    int N, ns, njobs;
    int first[3], count[3];          // jobs of a channel
    int rows[2], splits[2];
    SymMode sym;
};

// C4v element g on patch j (wedge part, ns shells per wedge, Na wedges)
__device__ __forceinline__ int c4v_patch(int g, int j, int ns, int Na)
{
    const int w = ns == 1 ? j : j / ns, sh = j - w * ns;
    const int off = (g & 3) * (Na >> 2);
    int r = (g & 4) ? off - w : w + off;      // in (-Na, 2 Na)
    r = r >= Na ? r - Na : (r < 0 ? r + Na : r);
    return r * ns + sh;
}

__global__ void __launch_bounds__(128) reduce_kernel(const ExpandArgs A)
{
    const int c = sym_compact(A.sym) ? 1 : 0, ch = blockIdx.y, nj = A.count[ch], ns = A.splits[c];
    if (nj == 0) return;
    const long stride = (long)A.rows[c] * A.N, per = stride * A.njobs;
    const double *src = A.part + A.first[ch] * stride;
    for (long o = blockIdx.x * (long)blockDim.x + threadIdx.x; o < stride; o += (long)gridDim.x * blockDim.x) {
        double v = 0.0;
        long oc = o;
        if (c) {
            const int row = (int)(o / A.N), n = (int)(o - (long)row * A.N), s = __ldg(A.rstab + row);
            if (s) oc = o + min(0, c4v_patch(s, n, A.ns, A.N / A.ns) - n);
        }
        // 16 loads in flight (one after the other they cost 18 us at 32 partial rows)
        for (int j = 0; j < nj; ++j)
            for (int k0 = 0; k0 < ns; k0 += 16) {
                double t[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) t[u] = k0 + u < ns ? __ldg(src + (k0 + u) * per + j * stride + oc) : 0.0;
                // as a tree: an FP64 add waits long for its operands
#pragma unroll
                for (int w = 8; w > 0; w >>= 1)
#pragma unroll
                    for (int u = 0; u < w; ++u) t[u] += t[u + w];
                v += t[0];
            }
        A.outc[ch * stride + o] = ch < 2 ? -v : v;
    }
}

// Block (k2, k1).
__global__ void expand_kernel(const ExpandArgs A)
{
    const bool c = sym_compact(A.sym);
    const int N = A.N, Na = N / A.ns, k1 = blockIdx.y, k2 = blockIdx.x;
    const long stride = (long)A.rows[c ? 1 : 0] * N;
    double *row = A.out + ((long)k1 * N + k2) * N;
    for (int k3 = threadIdx.x; k3 < N; k3 += blockDim.x) {
        double v = 0.0;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
            if (A.count[ch] == 0) continue;
            const int Q = ch == 0 ? k1 * N + k2 : (ch == 1 ? k3 * N + k2 : k1 * N + k3);
            const int n = ch == 0 ? k3 : (ch == 1 ? k1 : k2);
            long o = (long)Q * N + n;
            if (c) {
                const int e = __ldg(A.rowmap + (ch == 0 ? 0 : (long)N * N) + Q);
                o = (long)(e & 0xfffff) * N + c4v_patch(c4v_inverse(e >> 24), n, A.ns, Na);
            }
            v += __ldg(A.outc + ch * stride + o);
        }
        row[k3] = A.scale * v;
    }
}

// ---- stage operands ---------------------------------------------------------
// Job blockIdx.y (all when 0 < gridDim.y; a missing output skips its job): 0
// the C4v test of (V, Z) and the FP32 copy of V; 1, 2, 3 the permuted views
// V[n,a,b], V[b,n,a], V[n,b,a] as [a][b][n].  One warp per row of N values.
//
// The C4v test reduces max|V| and the largest deviation under the two
// generators (rotation by 90 degrees, reflection); any image differs by at most
// three generator steps, so a deviation below a third of the tolerance
// guarantees every image.  A non-finite value sets sym[4] and counts as asymmetric:
// an infinite deviation against the maximum of the finite values.
template <typename IN, typename R>
__global__ void __launch_bounds__(256) stage_prep_kernel(const IN *__restrict__ V, const double *__restrict__ Z, int nz, int N,
                                                         int ns, unsigned long long *sym, float *__restrict__ Vf,
                                                         R *__restrict__ P)
{
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int w0 = blockIdx.x * nw + (threadIdx.x >> 5), ws = gridDim.x * nw;
    const int NN = N * N, job = blockIdx.y;
    if (job > 0) {
        if (!P) return;
        R *dst = P + (long)(job - 1) * NN * N;
        for (int r = w0; r < NN; r += ws) {
            const int a = r / N, b = r - a * N;
            for (int n = lane; n < N; n += 32) {
                const long o = job == 1 ? (long)n * NN + r : (job == 2 ? ((long)b * N + n) * N + a : ((long)n * N + b) * N + a);
                dst[(long)r * N + n] = (R)V[o];
            }
        }
        return;
    }
    if (!sym && !Vf) return;
    __shared__ short ir[256], is[256];       // images under the generators
    for (int x = threadIdx.x; sym && x < N; x += blockDim.x) {
        ir[x] = (short)c4v_apply(1, x, N, ns);
        is[x] = (short)c4v_apply(4, x, N, ns);
    }
    __syncthreads();
    // maxima of magnitudes as integers (the bits of non-negative doubles order like
    // the values, NaN above infinity): two FP64 subtractions per element are left
    // on the FP64 pipe (with FP64 maxima and tests np96 took 23 us)
    unsigned long long m = 0, d = 0;
    const unsigned long long mag = 0x7fffffffffffffffULL, inf = 0x7ff0000000000000ULL;
    bool fin = true;
    for (int r = w0; r < NN; r += ws) {
        const int i = r / N, j = r - i * N;
        const IN *row = V + (long)r * N;
        const IN *rr = nullptr, *rs = nullptr;
        if (sym) {
            rr = V + ((long)ir[i] * N + ir[j]) * N;
            rs = V + ((long)is[i] * N + is[j]) * N;
        }
        for (int l = lane; l < N; l += 32) {
            const IN v = row[l];
            if (Vf) Vf[(long)r * N + l] = (float)v;
            if (!sym) continue;
            const IN e1 = rr[ir[l]] - v, e2 = rs[is[l]] - v;
            const unsigned long long b1 = (unsigned long long)__double_as_longlong((double)e1) & mag;
            const unsigned long long b2 = (unsigned long long)__double_as_longlong((double)e2) & mag;
            const unsigned long long bv = (unsigned long long)__double_as_longlong((double)v) & mag;
            d = max(d, max(b1, b2));
            if (bv < inf) m = max(m, bv);
            else fin = false;
        }
    }
    if (!sym) return;
    if (!fin) d = inf;
    // one atomic a block, and only where it raises the maximum
    auto raise = [&](unsigned long long v, unsigned long long *slot) {
        if (v > *(volatile unsigned long long *)slot) atomicMax(slot, v);
    };
    __shared__ unsigned long long sm[8], sd[8];
    for (int off = 16; off > 0; off >>= 1) {
        m = max(m, __shfl_down_sync(0xffffffffu, m, off));
        d = max(d, __shfl_down_sync(0xffffffffu, d, off));
    }
    if (lane == 0) {
        sm[threadIdx.x >> 5] = m;
        sd[threadIdx.x >> 5] = d;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < nw; ++k) {
            m = max(m, sm[k]);
            d = max(d, sd[k]);
        }
        raise(m, sym);
        raise(d, sym + 1);
    }
    if (!fin) atomicOr(&sym[4], 1ull);
    if (w0 == 0) {
        unsigned long long mz = 0, dz = 0;
        bool zfin = true;
        for (int y = lane; y < nz * N; y += 32) {
            const int x = y % N;
            const double *Zy = Z + (y - x);
            const double z = Zy[x];
            const unsigned long long b1 = (unsigned long long)__double_as_longlong(Zy[ir[x]] - z) & mag;
            const unsigned long long b2 = (unsigned long long)__double_as_longlong(Zy[is[x]] - z) & mag;
            const unsigned long long bz = (unsigned long long)__double_as_longlong(z) & mag;
            dz = max(dz, max(b1, b2));
            if (bz < inf) mz = max(mz, bz);
            else zfin = false;
        }
        if (!zfin) {
            dz = inf;
            atomicOr(&sym[4], 1ull);
        }
        for (int off = 16; off > 0; off >>= 1) {
            mz = max(mz, __shfl_down_sync(0xffffffffu, mz, off));
            dz = max(dz, __shfl_down_sync(0xffffffffu, dz, off));
        }
        if (lane == 0) {
            raise(mz, sym + 2);
            raise(dz, sym + 3);
        }
    }
}

// The C4v test of V and of nz arrays of N weights Z into red (read by
// sym_compact; nz = 0: no test), the FP32 copy
// when Vf is given and, outside the tensor-core precision, the permuted views.
static qpfrg_status launch_prep(qpfrg_ctx *c, const void *V, bool v64, const double *d_Z, int nz, float *Vf, bool operands,
                                unsigned long long *red)
{
    const bool test = nz > 0;
    const int N = c->pb.N, ns = c->pb.n_shell;
    cudaError_t e;
    if (test && (e = cudaMemsetAsync(red, 0, 5 * sizeof(unsigned long long), c->stream)) != cudaSuccess)
        return cuda_fail(c, e, "memset symmetry test");
    unsigned long long *sym = test ? red : nullptr;
    const bool views = operands && c->opt.precision != QPFRG_MIXED_TC;
    const dim3 grid(std::max(1, std::min(div_up((long)N * N, 8), 608)), views ? 4 : 1);
    prof_begin(c);
    if (c->opt.precision == QPFRG_FP64 || !operands)
        stage_prep_kernel<double, double><<<grid, 256, 0, c->stream>>>((const double *)V, d_Z, nz, N, ns, sym, nullptr,
                                                                       views ? (double *)c->d_views : nullptr);
    else if (v64)
        stage_prep_kernel<double, float><<<grid, 256, 0, c->stream>>>((const double *)V, d_Z, nz, N, ns, sym, Vf,
                                                                      views ? (float *)c->d_views : nullptr);
    else
        stage_prep_kernel<float, float><<<grid, 256, 0, c->stream>>>((const float *)V, d_Z, nz, N, ns, sym, nullptr,
                                                                     (float *)c->d_views);
    prof_end(c, K_CONVERT);
    e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "stage_prep_kernel");
}

// Operands of one right-hand side of the given FP64 vertex (qpfrg_rhs, the
// first stage of a step): C4v test of V and nz weight arrays (nz = 0: none),
// FP32 copy in the mixed precisions, permuted views of the SIMT contraction.
qpfrg_status launch_stage_prep(qpfrg_ctx *c, const double *d_V, const double *d_Z, int nz)
{
    return launch_prep(c, d_V, true, d_Z, nz, c->opt.precision == QPFRG_FP64 ? nullptr : c->d_Vf, true, c->d_sym);
}

// The same of a later stage's vertex (FP64, or FP32 in mixed precision).
qpfrg_status launch_stage_views(qpfrg_ctx *c, const void *d_Vin, const double *d_Z, int nz)
{
    if (c->opt.precision == QPFRG_MIXED_TC) return QPFRG_OK;
    return launch_prep(c, d_Vin, c->opt.precision == QPFRG_FP64, d_Z, nz, nullptr, true, c->d_sym);
}

qpfrg_status launch_sym_test(qpfrg_ctx *c, const double *d_V, const double *d_Z, int nz, unsigned long long *red)
{
    return launch_prep(c, d_V, true, d_Z, nz, nullptr, false, red);
}

// Columns per thread: the count (1..3) whose 16-wide tiles pad N least.
static int contract_nb(int N)
{
    int best = 3;
    for (int nb = 3; nb >= 1; --nb)
        if (div_up(N, 16 * nb) * nb < div_up(N, 16 * best) * best) best = nb;
    return best;
}

// Shape of the contraction of `rows` rows: two CTAs per SM where the reduction
// can be split that far (every split costs partial rows to write and sum).
static ContractShape contract_shape(const qpfrg_ctx *c, int rows)
{
    const int N = c->pb.N, tm = c->opt.precision == QPFRG_FP64 ? 2 : 4;
    ContractShape s;
    s.rows = rows;
    s.mtiles = div_up(rows, 16 * tm);
    const long per = 4L * s.mtiles * div_up(N, 16 * contract_nb(N));
    int sp = (int)std::min<long>(N, std::max<long>(1, (2 * 152 + per - 1) / per));
    s.a_per = div_up(N, sp);
    s.splits = div_up(N, s.a_per);
    return s;
}

// Partial rows and permuted views of the SIMT contraction, sized for both forms.
qpfrg_status contract_alloc(qpfrg_ctx *c)
{
    const long N = c->pb.N, n3 = N * N * N;
    const ContractShape all = contract_shape(c, (int)(N * N));
    long n = (long)all.splits * all.rows;
    if (c->rows_ok) {
        const ContractShape rep = contract_shape(c, c->n_rrep);
        n = std::max(n, (long)rep.splits * rep.rows);
    }
    const size_t rsz = c->opt.precision == QPFRG_FP64 ? sizeof(double) : sizeof(float);
    cudaError_t e = cudaMalloc((void **)&c->d_partial, (size_t)n * 4 * N * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void **)&c->d_outc, 3 * n3 * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void **)&c->d_views, 3 * n3 * rsz);
    if (e == cudaSuccess) return QPFRG_OK;
    cudaGetLastError();
    return cuda_fail(c, e, "cudaMalloc(contraction work space)");
}

template <typename R>
static qpfrg_status launch_simt(qpfrg_ctx *c, const R *V, double scale, double *out)
{
    const int N = c->pb.N;
    ContractArgs<R> A{};
    A.B = reinterpret_cast<const R *>(c->d_B);
    A.V = V;
    A.P = reinterpret_cast<const R *>(c->d_views);
    A.rep = c->d_rrep;
    A.n_can = c->n_rcan;
    A.part = c->d_partial;
    A.N = N;
    const int nb = contract_nb(N);
    A.ntiles = div_up(N, 16 * nb);
    const unsigned ch = c->pb.channels;
    if (ch & QPFRG_CH_PP) A.jobs[A.njobs++] = 0;
    if (ch & QPFRG_CH_CR) A.jobs[A.njobs++] = 1;
    if (ch & QPFRG_CH_D) {
        A.jobs[A.njobs++] = 2;
        A.jobs[A.njobs++] = 3;
    }
    A.sh[0] = contract_shape(c, N * N);
    A.sh[1] = c->rows_ok ? contract_shape(c, c->n_rrep) : A.sh[0];
    A.sym = c->rhs_sym;
    const int m = c->rhs_sym.mode;
    const long g0 = (long)A.sh[0].mtiles * A.sh[0].splits, g1 = (long)A.sh[1].mtiles * A.sh[1].splits;
    const long ctas = (m == 0 ? g0 : (m == 1 ? g1 : std::max(g0, g1))) * A.ntiles * A.njobs;
    constexpr int TM = sizeof(R) == 8 ? 2 : 4;
    if (ctas > 0) {
        prof_begin(c);
        if (nb == 1) contract_kernel<R, TM, 1><<<(unsigned)ctas, 256, 0, c->stream>>>(A);
        else if (nb == 2) contract_kernel<R, TM, 2><<<(unsigned)ctas, 256, 0, c->stream>>>(A);
        else contract_kernel<R, TM, 3><<<(unsigned)ctas, 256, 0, c->stream>>>(A);
        prof_end(c, K_CONTRACT_PP);   // one launch for every channel
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(c, e, "contract_kernel");
    }
    ExpandArgs E{};
    E.part = c->d_partial;
    E.outc = c->d_outc;
    E.rowmap = c->d_rowmap;
    E.rstab = c->d_rstab;
    E.out = out;
    E.scale = scale;
    E.N = N;
    E.ns = c->pb.n_shell;
    E.njobs = A.njobs;
    for (int k = 0; k < A.njobs; ++k) {
        const int q = std::min(A.jobs[k], 2);
        if (E.count[q]++ == 0) E.first[q] = k;
    }
    for (int k = 0; k < 2; ++k) {
        E.rows[k] = A.sh[k].rows;
        E.splits[k] = A.sh[k].splits;
    }
    E.sym = c->rhs_sym;
    const long rows = m == 1 ? E.rows[1] : E.rows[0];
    prof_begin(c);
    reduce_kernel<<<dim3((unsigned)std::min(div_up(rows * N, 128), 1216), 3), 128, 0, c->stream>>>(E);
    expand_kernel<<<dim3(N, N), std::min(256, (N + 31) / 32 * 32), 0, c->stream>>>(E);
    prof_end(c, K_ROWS_EXPAND);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "expand_kernel");
}

// Expansion of the representative rows (row orbits, symmetry.cu): with a
// C4v-symmetric state each channel's output is invariant, out(g t) = out(t),
// so row Q = g rep of a channel at column n is the representative's row at
// column g^-1 n.  One thread per output triple (k1, k2, k3) adds the three
// channels' values: pp row (k1, k2) column k3, cr row (k3, k2) column k1,
// d row (k1, k3) column k2 (the row/column roles of the channel GEMMs above).  Columns
// that a mirror of the row exchanges read the lower one (as reduce_kernel).
// Row (k1, k2) of out, threads over k3.
__device__ __forceinline__ void expand_row(const double *__restrict__ outc, const int *__restrict__ rowmap, int nr,
                                           int N, int ns, unsigned channels, double *__restrict__ out, int k1, int k2)
{
    const int Na = N / ns;
    const long ch_stride = (long)nr * N;
    double *row = out + ((long)k1 * N + k2) * N;
    const int e_pp = __ldg(rowmap + k1 * N + k2);
    rowmap += N * N;             // the particle-hole family's
    for (int k3 = threadIdx.x; k3 < N; k3 += blockDim.x) {
        double v = 0.0;
        auto take = [&](int ch, int e, int n) {
            const int m = e & 0xfffff, gi = c4v_inverse(e >> 24), s = (e >> 20) & 15;
            int col = c4v_patch(gi, n, ns, Na);
            if (s) col = min(col, c4v_patch(s, col, ns, Na));
            v += __ldg(outc + ch * ch_stride + (long)m * N + col);
        };
        if (channels & QPFRG_CH_PP) take(0, e_pp, k3);
        if (channels & QPFRG_CH_CR) take(1, __ldg(rowmap + k3 * N + k2), k1);
        if (channels & QPFRG_CH_D) take(2, __ldg(rowmap + k1 * N + k3), k2);
        row[k3] += v;
    }
}

// Block (k2, k1), thread k3.
__global__ void rows_expand_kernel(const double *__restrict__ outc, const int *__restrict__ rowmap, int nr, int N,
                                   int ns, unsigned channels, double *__restrict__ out)
{
    expand_row(outc, rowmap, nr, N, ns, channels, out, blockIdx.y, blockIdx.x);
}

// Runge-Kutta stage (1 .. 4) of the batched flows on the representative rows: their
// state is V[m][n], acc[m][n] of the particle-particle representatives
// Q_m = (x, y), n = k3, and every other element is an image of these.  The three
// channels' values of (x, y, n) give dV; Vr is the FP32 vertex of the next stage.
//
// What bounds it: latency and the gathers of cr and d (L2).  FP64 costs 64 clocks a
// warp instruction: on all N^3 elements of 12 flows at np96 the expansion into dV,
// the stage update and the clearing of dV took 140 + 600 us (1 GB), of which an
// eighth of the elements is needed (sweep of 24 flows with this and
// vertex_expand_batch_kernel: 640 -> 440 ms).
__global__ void rows_rk_batch_kernel(int stage, TcBatch bt, const int *__restrict__ rep, const int *__restrict__ rowmap,
                                     int nr, int N, int ns, unsigned channels, double *const *Vs, double *const *accs,
                                     float *const *Vrs, unsigned long long *red)
{
    const int f = blockIdx.y;
    const double h = bt.h_tab[(long)bt.step * bt.nflows + f];
    if (bt.status[f] != QPFRG_FLOW_RUNNING || h == 0.0) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x, per = nr * N;
    double m = 0.0;
    bool bad = false;
    if (i < per) {
        const double *__restrict__ outc = bt.outc[f];
        double *V = Vs[f], *acc = accs[f];
        const int Na = N / ns, r = i / N, n = i - r * N;
        const int Q = __ldg(rep + r), x = Q / N, y = Q - x * N;
        const int *__restrict__ ph = rowmap + N * N;
        auto take = [&](int ch, int e, int col) {
            return __ldg(outc + (long)ch * per + (long)(e & 0xfffff) * N + c4v_patch(c4v_inverse(e >> 24), col, ns, Na));
        };
        const double v = V[i], a0 = stage > 1 ? acc[i] : 0.0;
        double k = 0.0;
        if (channels & QPFRG_CH_PP) k += __ldg(outc + i);
        if (channels & QPFRG_CH_CR) k += take(1, __ldg(ph + n * N + y), x);
        if (channels & QPFRG_CH_D) k += take(2, __ldg(ph + x * N + n), y);
        if (stage < 4) {
            acc[i] = stage == 1 ? k : a0 + 2.0 * k;
            Vrs[f][i] = (float)(v + (stage == 3 ? h : 0.5 * h) * k);
        } else {
            const double w = v + h / 6.0 * (a0 + k);
            V[i] = w;
            Vrs[f][i] = (float)w;
            bad = !isfinite(w);
            m = bad ? 0.0 : fabs(w);
        }
    }
    if (stage < 4) return;
    for (int off = 16; off > 0; off >>= 1) {
        m = fmax(m, __shfl_down_sync(0xffffffffu, m, off));
        bad = __shfl_down_sync(0xffffffffu, (int)bad, off) || bad;
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&red[2 * f], (unsigned long long)__double_as_longlong(m));
        if (bad) atomicOr(&red[2 * f + 1], 1ull);
    }
}

// The FP32 stage vertex of every running flow from its representative rows, four
// consecutive k3 per thread, and the contraction rows cleared for the next stage.
__global__ void vertex_expand_batch_kernel(TcBatch bt, const int *__restrict__ rowmap, int nr, int N, int ns,
                                           const float *const *Vrs)
{
    const int f = blockIdx.y;
    if (bt.status[f] != QPFRG_FLOW_RUNNING || bt.h_tab[(long)bt.step * bt.nflows + f] == 0.0) return;
    const int t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    double *outc = bt.outc[f];
    for (int i = t; i < 3 * nr * N; i += nt) outc[i] = 0.0;
    const int n4 = N / 4;                 // N is a multiple of 4
    if (t >= N * N * n4) return;
    const int Q = t / n4, k3 = 4 * (t - Q * n4), Na = N / ns;
    const int e = __ldg(rowmap + Q), gi = c4v_inverse(e >> 24);
    const float *__restrict__ row = Vrs[f] + (long)(e & 0xfffff) * N;
    float4 v;
    v.x = row[c4v_patch(gi, k3, ns, Na)];
    v.y = row[c4v_patch(gi, k3 + 1, ns, Na)];
    v.z = row[c4v_patch(gi, k3 + 2, ns, Na)];
    v.w = row[c4v_patch(gi, k3 + 3, ns, Na)];
    *reinterpret_cast<float4 *>(const_cast<float *>(bt.Vf[f]) + (long)Q * N + k3) = v;
}

qpfrg_status launch_rows_rk_batch(qpfrg_ctx *c, int stage, const TcBatch &bt, double *const *V, double *const *acc,
                                  float *const *Vr, unsigned long long *red)
{
    const int N = c->pb.N;
    prof_begin(c);
    rows_rk_batch_kernel<<<dim3(div_up((long)c->n_rrep * N, 256), bt.nflows), 256, 0, c->stream>>>(
        stage, bt, c->d_rrep, c->d_rowmap, c->n_rrep, N, c->pb.n_shell, c->pb.channels, V, acc, Vr, red);
    prof_end(c, stage < 4 ? K_RK_STAGE : K_RK_FINAL);
    prof_begin(c);
    vertex_expand_batch_kernel<<<dim3(div_up((long)N * N * N / 4, 256), bt.nflows), 256, 0, c->stream>>>(
        bt, c->d_rowmap, c->n_rrep, N, c->pb.n_shell, Vr);
    prof_end(c, K_ROWS_EXPAND);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "rows_rk_batch_kernel");
}

qpfrg_status launch_contractions(qpfrg_ctx *c, const void *d_Vin, double scale, double *d_out)
{
    if (c->opt.precision == QPFRG_MIXED_TC) {
        // the weighted tables of this stage, formed into A tiles inside the
        // contraction; representative rows go into compact rows, then expanded
        const unsigned ch = c->pb.channels;
        qpfrg_status s = QPFRG_OK;
        const int N = c->pb.N;
        const bool orbits = c->rhs_sym.mode != 0;
        const long per = orbits ? (long)c->n_rrep * N : 0;
        cudaError_t e = cudaMemsetAsync(d_out, 0, (size_t)N * N * N * sizeof(double), c->stream);
        if (e == cudaSuccess && orbits) e = cudaMemsetAsync(c->d_outc, 0, 3 * per * sizeof(double), c->stream);
        if (e != cudaSuccess) return cuda_fail(c, e, "memset right-hand side");
        if ((ch & QPFRG_CH_PP) && (s = launch_tc_fused(c, 0, -scale, d_out, c->d_outc, K_TC_PP))) return s;
        if ((ch & QPFRG_CH_CR) && (s = launch_tc_fused(c, 1, -scale, d_out, c->d_outc + per, K_TC_CR))) return s;
        if ((ch & QPFRG_CH_D) && (s = launch_tc_fused(c, 2, scale, d_out, c->d_outc + 2 * per, K_TC_D))) return s;
        if (orbits) {
            prof_begin(c);
            rows_expand_kernel<<<dim3(N, N), std::min(256, (N + 31) / 32 * 32), 0, c->stream>>>(
                c->d_outc, c->d_rowmap, c->n_rrep, N, c->pb.n_shell, ch, d_out);
            prof_end(c, K_ROWS_EXPAND);
            e = cudaGetLastError();
            if (e != cudaSuccess) return cuda_fail(c, e, "rows_expand_kernel");
        }
        return QPFRG_OK;
    }
    if (c->opt.precision == QPFRG_FP64)
        return launch_simt<double>(c, reinterpret_cast<const double *>(d_Vin), scale, d_out);
    return launch_simt<float>(c, reinterpret_cast<const float *>(d_Vin), scale, d_out);
}

}  // namespace qpfrg
