// C4v orbits of the loop-kernel rows (wedge and shell modes).
//
// The point group C4v of the square lattice acts on the wedges as
// g = (m, s): w -> s w + m N_a/4 (mod N_a), s = +-1, and leaves the energy
// shells in place (patch j = w n_s + s -> (g w) n_s + s), on the transfers
// Q = (x, y) (Q = k_F(x) +- k_F(y)) as (x, y) -> (g x, g y), and on the fine
// points of a patch as (a, t, r) -> (g a, t, r) for the rotations and
// (g a, n_theta - 1 - t, r) for the reflections.  The dispersion (Eq.
// (free_dispersion_xi)) and the quadrature weights are invariant, and where
// the patch projection is covariant, proj(g k) = g proj(k), the Z-free binned
// loop kernels satisfy
//     B_f[g Q][g a][g b] = B_f[Q][a][b].
// Exchange: the transfer pairs (x, y) and (y, x) have the same momentum
// k_F(x) + k_F(y), and (x, y) and (y', x') the same k_F(x) - k_F(y), x' = x + N_a/2
// the patch opposite to x, so that B_pp[x,y] = B_pp[y,x] and B_ph[x,y] =
// B_ph[y',x'] row by row, columns in place.  The exchange commutes with C4v; the
// orbits below are those of the 16 elements (g, s): first the exchange if s,
// then g.  That halves the loop-kernel evaluations (np96, 32 x 32 points, row
// orbits: 394 -> 229 us a launch).
// So one row per orbit of (Q, a) is evaluated and written to every image,
// its columns permuted by g (the Z weights and vertex factors are applied per
// image).  Covariance is not assumed: check_covariance_kernel compares every
// image row of the partner maps with its representative's row, byte by byte,
// and a row that differs anywhere is evaluated by itself.
//
// When V and Z are C4v symmetric, each channel's output is invariant as well,
// dV_ch(g k1, g k2, g k3) = dV_ch(k1, k2, k3), so the contraction needs one
// output row per orbit of transfer pairs Q only (build_row_orbits:
// representatives, and per pair Q its representative and the g with Q = g
// rep); a pair with a row that breaks covariance is a row of its own.
// contract.cu expands the rows.
#include <algorithm>
#include <cstring>
#include <vector>

#include "qpfrg_internal.h"

namespace qpfrg {

// flag[f][Q N + a] = 1 where the partner-map row (f, Q, a) is not the image of its
// representative's row under g.  rep[f][Q N + a] = representative's Q N + a,
// gof[f][Q N + a] = g with (Q, a) = g, after an exchange perhaps, of the
// representative.
__global__ void check_covariance_kernel(const uint8_t *__restrict__ part, const int *__restrict__ rep,
                                        const uint8_t *__restrict__ gof, uint8_t *__restrict__ flag, int N, int M,
                                        int P, int nt, int nr, int ns)
{
    const int Q = blockIdx.x, f = blockIdx.y;
    const long NN = (long)N * N, fo = (long)f * NN * N;
    __shared__ int bad;
    for (int a = 0; a < N; ++a) {
        const long row = (long)Q * N + a;
        const int r = rep[fo + row];
        if (r == row) continue;                    // uniform over the block
        const int g = gof[fo + row];
        const int Qr = r / N, ar = r - Qr * N;
        const uint8_t *src = part + ((long)f * NN + Qr) * (long)M + (long)ar * P;
        const uint8_t *dst = part + ((long)f * NN + Q) * (long)M + (long)a * P;
        if (threadIdx.x == 0) bad = 0;
        __syncthreads();
        int mine = 0;
        for (int li = threadIdx.x; li < P; li += blockDim.x) {
            const int t = li / nr, s = li - t * nr;
            const int ts = (g & 4) ? nt - 1 - t : t;   // the representative's point mapped onto (t, s)
            const int want = c4v_apply(g, src[part_byte(ts, s, nt, nr)], N, ns);
            if (dst[part_byte(t, s, nt, nr)] != want) mine = 1;
        }
        if (mine) bad = 1;
        __syncthreads();
        if (threadIdx.x == 0) flag[(long)f * NN * N + row] = (uint8_t)bad;
        __syncthreads();
    }
}

// (x, y) exchanged, with the same transfer momentum in family f (0 pp, 1 ph)
static void exchange(int f, int N, int ns, int &x, int &y)
{
    const int u = x;
    x = f == 0 ? y : c4v_apply(2, y, N, ns);
    y = f == 0 ? u : c4v_apply(2, u, N, ns);
}

// Row orbits of the contraction: rowmap[f][Q] = (row | s << 20 | g << 24) with Q = g
// rrep[f][row], s the mirror that leaves the row's pair in place (0: none).  The first n_rcan rows are one pair of each orbit under C4v and
// exchange, the same in both families: the rows of the table, those first whose
// exchanged pair lies in another C4v orbit.  The others
// are these exchanged pairs, in the same order: row n_rcan + i holds the table row
// i.  A pair Q that failed the covariance check (own[Q]: a momentum on a boundary
// between patches or shells, decided by rounding) is a row for itself, so that the
// table rows of the remaining images are exactly the representative's, permuted.
// (The exchanged row of an orbit may be such a pair: it then stands for the other
// images only.)  exch = false: every C4v orbit is a row of the table.
static qpfrg_status build_row_orbits(qpfrg_ctx *c, bool exch, const std::vector<uint8_t> &own)
{
    const int N = c->pb.N, ns = c->pb.n_shell;
    const long NN = (long)N * N;
    std::vector<int> paired, single;
    std::vector<uint8_t> seen(NN, 0);
    for (long Q0 = 0; Q0 < NN; ++Q0) {
        if (seen[Q0]) continue;
        // the orbit of Q0; its row is the smallest pair that passed the check
        // (none did: they are all rows for themselves)
        long can = NN;
        int x = (int)(Q0 / N), y = (int)(Q0 - (long)x * N);
        for (int k = 0; k < (exch ? 2 : 1); ++k) {
            for (int g = 0; g < 8; ++g) {
                const long Q = (long)c4v_apply(g, x, N, ns) * N + c4v_apply(g, y, N, ns);
                seen[Q] = 1;
                if (!own[Q]) can = std::min(can, Q);
            }
            std::swap(x, y);      // exchanges of both families share their C4v orbit
        }
        if (can == NN) continue;
        bool other = exch;        // the exchanged pair lies in another C4v orbit
        x = (int)(can / N);
        y = (int)(can - (long)x * N);
        for (int g = 0; g < 8 && other; ++g)
            other = (long)c4v_apply(g, y, N, ns) * N + c4v_apply(g, x, N, ns) != can;
        (other ? paired : single).push_back((int)can);
    }
    const size_t norb = single.size();
    for (long Q = 0; Q < NN; ++Q)
        if (own[Q]) single.push_back((int)Q);
    const int npar = (int)paired.size(), ncan = npar + (int)single.size(), nr = ncan + npar;
    std::vector<int> reps(2 * (size_t)nr), rowmap(2 * NN);
    for (int f = 0; f < 2; ++f) {
        int *rep = reps.data() + (size_t)f * nr, *map = rowmap.data() + f * NN;
        std::copy(paired.begin(), paired.end(), rep);
        std::copy(single.begin(), single.end(), rep + npar);
        for (int i = 0; i < npar; ++i) {
            int x = paired[i] / N, y = paired[i] - x * N;
            exchange(f, N, ns, x, y);
            rep[ncan + i] = x * N + y;
        }
        for (int m = 0; m < nr; ++m)
            for (int g = 7; g >= 0 && !(m >= npar + (int)norb && m < ncan); --g) {
                const int x = rep[m] / N, y = rep[m] - x * N;
                map[c4v_apply(g, x, N, ns) * N + c4v_apply(g, y, N, ns)] = m | (g << 24);
            }
        for (int m = npar + (int)norb; m < ncan; ++m) map[rep[m]] = m;
    }
    std::vector<uint8_t> stab(nr, 0);      // the same in both families; rows of their own have no images
    for (int m = 0; m < nr; ++m)
        for (int g = 4; g < 8 && (m < npar + (int)norb || m >= ncan); ++g)
            if (c4v_apply(g, reps[m] / N, N, ns) == reps[m] / N && c4v_apply(g, reps[m] % N, N, ns) == reps[m] % N)
                stab[m] = (uint8_t)g;
    for (int &e : rowmap) e |= stab[e & 0xfffff] << 20;
    cudaError_t e;
    if ((e = cudaMalloc((void **)&c->d_rrep, 2 * (size_t)nr * sizeof(int))) != cudaSuccess ||
        (e = cudaMalloc((void **)&c->d_rstab, nr)) != cudaSuccess ||
        (e = cudaMalloc((void **)&c->d_rowmap, 2 * NN * sizeof(int))) != cudaSuccess ||
        (e = cudaMalloc((void **)&c->d_rtask, (2L * N * ((ncan + 7) / 8) + 8) * sizeof(int4))) != cudaSuccess ||
        (c->opt.precision == QPFRG_MIXED_TC &&
         (e = cudaMalloc((void **)&c->d_outc, 3L * nr * N * sizeof(double))) != cudaSuccess))
        return cuda_fail(c, e, "cudaMalloc(row orbits)");
    e = cudaMemcpy(c->d_rrep, reps.data(), reps.size() * sizeof(int), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(c->d_rstab, stab.data(), nr, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(c->d_rowmap, rowmap.data(), 2 * NN * sizeof(int), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(c, e, "upload row orbits");
    c->n_rrep = nr;
    c->n_rcan = ncan;
    c->rtask_qchunk = 0;
    c->loop_evals_rows = 2LL * nr * c->pb.M;
    c->rows_ok = true;
    c->rows_exact = std::count(own.begin(), own.end(), 1) == 0;
    return QPFRG_OK;
}

// ap[g N + j]: the image of patch j under g
static std::vector<int> patch_images(int N, int ns)
{
    std::vector<int> ap(8 * (size_t)N);
    for (int g = 0; g < 8; ++g)
        for (int j = 0; j < N; ++j) ap[(size_t)g * N + j] = c4v_apply(g, j, N, ns);
    return ap;
}

// Representatives (rep, gof as check_covariance_kernel reads them) of every row
// (f, Q, a) under C4v and, where exch[f], the exchange: the image with the
// smallest (a, Q), whose patch lies in the fundamental domain 0..N/8.
static void row_representatives(int N, int ns, const bool (&exch)[2], std::vector<int> &rep, std::vector<uint8_t> &gof)
{
    const long NN = (long)N * N, rows = NN * N;
    const std::vector<int> ap = patch_images(N, ns);
    // per patch the elements that take it to its smallest image
    std::vector<int> amin(N), ng(N), gl(8 * (size_t)N);
    for (int a = 0; a < N; ++a) {
        int m = a;
        for (int g = 0; g < 8; ++g) m = std::min(m, ap[(size_t)g * N + a]);
        amin[a] = m;
        for (int g = 0; g < 8; ++g)
            if (ap[(size_t)g * N + a] == m) gl[8 * (size_t)a + ng[a]++] = g;
    }
    for (int f = 0; f < 2; ++f)
        for (int x = 0; x < N; ++x)
            for (int y = 0; y < N; ++y) {
                int ex = x, ey = y;
                exchange(f, N, ns, ex, ey);
                for (int a = 0; a < N; ++a) {
                    int best = -1, bg = 0;
                    for (int k = 0; k < ng[a]; ++k) {
                        const int g = gl[8 * (size_t)a + k];
                        const int *A = &ap[(size_t)g * N];
                        int Q = A[x] * N + A[y];
                        if (exch[f]) Q = std::min(Q, A[ex] * N + A[ey]);
                        if (best < 0 || Q < best) {
                            best = Q;
                            bg = g;
                        }
                    }
                    const long row = ((long)x * N + y) * N + a;
                    rep[f * rows + row] = (int)((long)best * N + amin[a]);
                    gof[f * rows + row] = (uint8_t)c4v_inverse(bg);    // (Q, a) = g^-1 applied to the representative
                }
            }
}

// flag[f][row] = 1 where a partner-map row is not its representative's image
static qpfrg_status check_rows(qpfrg_ctx *c, const std::vector<int> &rep, const std::vector<uint8_t> &gof,
                               std::vector<uint8_t> &flag)
{
    const size_t n = rep.size();
    const long NN = (long)c->pb.N * c->pb.N;
    int *d_rep = nullptr;
    uint8_t *d_g = nullptr, *d_flag = nullptr;
    cudaError_t e;
    if ((e = cudaMalloc((void **)&d_rep, n * sizeof(int))) == cudaSuccess &&
        (e = cudaMalloc((void **)&d_g, n)) == cudaSuccess && (e = cudaMalloc((void **)&d_flag, n)) == cudaSuccess) {
        e = cudaMemcpyAsync(d_rep, rep.data(), n * sizeof(int), cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d_g, gof.data(), n, cudaMemcpyHostToDevice, c->stream);
        if (e == cudaSuccess) e = cudaMemsetAsync(d_flag, 0, n, c->stream);
        if (e == cudaSuccess) {
            check_covariance_kernel<<<dim3((unsigned)NN, 2), 256, 0, c->stream>>>(
                c->d_part, d_rep, d_g, d_flag, c->pb.N, c->pb.M, c->pb.P, c->pb.n_theta, c->pb.n_r, c->pb.n_shell);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpyAsync(flag.data(), d_flag, n, cudaMemcpyDeviceToHost, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    }
    cudaFree(d_rep);
    cudaFree(d_g);
    cudaFree(d_flag);
    return e == cudaSuccess ? QPFRG_OK : cuda_fail(c, e, "partner-map covariance check");
}

qpfrg_status build_loop_orbits(qpfrg_ctx *c)
{
    c->loop_red = false;
    if ((c->pb.mode != QPFRG_GRID_WEDGE && c->pb.mode != QPFRG_GRID_SHELL) ||
        (c->opt.no_loop_symmetry != 0 && c->opt.no_loop_symmetry != 2))
        return QPFRG_OK;
    const int N = c->pb.N, ns = c->pb.n_shell;
    if ((N / ns) % 4 != 0) return QPFRG_OK;
    const long NN = (long)N * N, rows = NN * N;
    std::vector<int> rep(2 * rows);
    std::vector<uint8_t> gof(2 * rows), flag(2 * rows);
    // Where rows differ, C4v alone may leave fewer of them (opposite Fermi momenta
    // are opposite to rounding only): the grouping with fewer rows to evaluate
    bool exch[2] = {true, true};
    cudaError_t e = cudaSuccess;
    auto differ = [&](const std::vector<uint8_t> &v) { return (long)std::count(v.begin(), v.end(), 1); };
    row_representatives(N, ns, exch, rep, gof);
    qpfrg_status st = check_rows(c, rep, gof, flag);
    const long d16 = st == QPFRG_OK ? differ(flag) : 0;
    if (d16 > 0) {
        std::vector<int> rep8(2 * rows);
        std::vector<uint8_t> gof8(2 * rows), flag8(2 * rows);
        const bool none[2] = {false, false};
        row_representatives(N, ns, none, rep8, gof8);
        st = check_rows(c, rep8, gof8, flag8);
        const long d8 = differ(flag8);
        if (st == QPFRG_OK && (d8 == 0 || d8 + rows / 4 < d16 + rows / 8)) {
            exch[0] = exch[1] = false;
            rep.swap(rep8);
            gof.swap(gof8);
            flag.swap(flag8);
        }
    }
    if (st != QPFRG_OK) return st;

    // representatives per family grouped by patch, each with its images;
    // rows whose partner bytes broke covariance are representatives of themselves
    struct Rep {
        int a, Q, n;
        int2 img[kLoopImages];
    };
    // Collected per patch, so that the rows (144 bytes each) need no sorting, the
    // images read from a table: a context of 96 patches, 69 -> 55 ms.
    std::vector<std::vector<Rep>> reps[2] = {std::vector<std::vector<Rep>>(N), std::vector<std::vector<Rep>>(N)};
    const std::vector<int> ap = patch_images(N, ns);
    long mism = 0, nrep = 0;
    for (int f = 0; f < 2; ++f) {
        const uint8_t *fl = flag.data() + (long)f * rows;
        for (long row = 0; row < rows; ++row) {
            const int Q = (int)(row / N), a = (int)(row - (long)Q * N);
            if (fl[row]) {
                ++mism;
                Rep r{a, Q, 1, {}};
                r.img[0] = make_int2(Q, a);
                reps[f][a].push_back(r);
                continue;
            }
            if (rep[f * rows + row] != row) continue;
            Rep r{a, Q, 0, {}};
            for (int s = 0; s < (exch[f] ? 2 : 1); ++s) {
                int x = Q / N, y = Q - x * N;
                if (s) exchange(f, N, ns, x, y);
                for (int g = 0; g < 8; ++g) {
                    const int *A = &ap[(size_t)g * N];
                    const int Qi = A[x] * N + A[y], ai = A[a];
                    if (fl[(long)Qi * N + ai]) continue;   // evaluated by itself
                    bool dup = false;
                    for (int k = 0; k < r.n; ++k) dup |= r.img[k].x == Qi && (r.img[k].y & 0xffff) == ai;
                    if (!dup) r.img[r.n++] = make_int2(Qi, ai | (g << 16));
                }
            }
            reps[f][a].push_back(r);
        }
        for (const auto &p : reps[f]) nrep += (long)p.size();
    }
    std::vector<int> hQ(nrep), hn(nrep);
    std::vector<int2> himg(kLoopImages * nrep, make_int2(0, 0));
    c->lgroups.clear();
    long k = 0, evals = 0;
    for (int f = 0; f < 2; ++f)
        for (int a = 0; a < N; ++a) {
            const std::vector<Rep> &p = reps[f][a];
            if (p.empty()) continue;
            c->lgroups.push_back({f, a, (int)k, (int)p.size()});
            for (const Rep &r : p) {
                hQ[k] = r.Q;
                hn[k] = r.n;
                for (int m = 0; m < r.n; ++m) himg[kLoopImages * k + m] = r.img[m];
                evals += c->pb.P;
                ++k;
            }
        }
    if ((e = cudaMalloc((void **)&c->d_lrepQ, nrep * sizeof(int))) != cudaSuccess ||
        (e = cudaMalloc((void **)&c->d_lnimg, nrep * sizeof(int))) != cudaSuccess ||
        (e = cudaMalloc((void **)&c->d_limg, kLoopImages * nrep * sizeof(int2))) != cudaSuccess ||
        (e = cudaMalloc((void **)&c->d_ltask, (nrep + 2 * (long)N + 8) * sizeof(int4))) != cudaSuccess)
        return cuda_fail(c, e, "cudaMalloc(loop representatives)");
    e = cudaMemcpy(c->d_lrepQ, hQ.data(), nrep * sizeof(int), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(c->d_lnimg, hn.data(), nrep * sizeof(int), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(c->d_limg, himg.data(), kLoopImages * nrep * sizeof(int2), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(c, e, "upload loop representatives");
    c->n_lrep = nrep;
    c->ltask_qchunk = 0;
    c->loop_evals_red = evals;
    c->loop_mismatch_rows = mism;
    c->loop_red = true;
    if (c->opt.no_loop_symmetry != 0) return QPFRG_OK;
    std::vector<uint8_t> own(NN, 0);
    for (int f = 0; f < 2; ++f)
        for (long row = 0; row < rows; ++row)
            if (flag[f * rows + row]) own[row / N] = 1;
    // row orbits while the pairs of their own leave at least half of the saving
    if (std::count(own.begin(), own.end(), 1) > NN / 2) return QPFRG_OK;
    return build_row_orbits(c, exch[0], own);
}

// Tasks of the reduced loop-kernel launch for a chunk size: (family, patch,
// first representative, count) per CTA; rebuilt when the chunk size changes.
qpfrg_status loop_tasks(qpfrg_ctx *c, int qchunk, int *ntask)
{
    if (c->ltask_qchunk == qchunk) {
        *ntask = c->n_ltask;
        return QPFRG_OK;
    }
    std::vector<int4> t;
    for (const LoopGroup &g : c->lgroups)
        for (int s = 0; s < g.count; s += qchunk) t.push_back(make_int4(g.fam, g.a, g.start + s, std::min(qchunk, g.count - s)));
    if ((long)t.size() > c->n_lrep + 2L * c->pb.N + 8) {
        c->err = "loop-kernel task list overflow";
        return QPFRG_ERR_INVALID;
    }
    cudaError_t e = cudaMemcpyAsync(c->d_ltask, t.data(), t.size() * sizeof(int4), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "upload loop tasks");
    c->ltask_qchunk = qchunk;
    c->n_ltask = (int)t.size();
    *ntask = c->n_ltask;
    return QPFRG_OK;
}

// Tasks of the loop-kernel launch on representative rows: (family, patch,
// first representative, count) per CTA, chunks of qchunk rows (qchunk >= 8).
qpfrg_status row_tasks(qpfrg_ctx *c, int qchunk, int *ntask)
{
    if (c->rtask_qchunk == qchunk) {
        *ntask = c->n_rtask;
        return QPFRG_OK;
    }
    if (qchunk < 8) {
        c->err = "row tasks: chunk below 8 rows";
        return QPFRG_ERR_INVALID;
    }
    std::vector<int4> t;
    for (int f = 0; f < 2; ++f)
        for (int a = 0; a < c->pb.N; ++a)
            for (int s0 = 0; s0 < c->n_rcan; s0 += qchunk) t.push_back(make_int4(f, a, s0, std::min(qchunk, c->n_rcan - s0)));
    cudaError_t e = cudaMemcpyAsync(c->d_rtask, t.data(), t.size() * sizeof(int4), cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(c, e, "upload row tasks");
    c->rtask_qchunk = qchunk;
    c->n_rtask = (int)t.size();
    *ntask = c->n_rtask;
    return QPFRG_OK;
}

}  // namespace qpfrg

extern "C" qpfrg_status qpfrg_sigma_table(qpfrg_t c, size_t *bytes, long long offset, long long count,
                                          unsigned char *h_out)
{
    if (!c) return QPFRG_ERR_INVALID;
    const size_t size = c->d_rtab ? (size_t)c->n_irr * c->pb.N * (size_t)c->pb.M * (size_t)c->pb.P : 0;
    if (bytes) *bytes = size;
    if (!h_out) return QPFRG_OK;
    if (offset < 0 || count < 0 || (size_t)offset + (size_t)count > size) {
        c->err = "qpfrg_sigma_table: range outside the table";
        return QPFRG_ERR_INVALID;
    }
    cudaError_t e = cudaMemcpyAsync(h_out, c->d_rtab + offset, (size_t)count, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return e == cudaSuccess ? QPFRG_OK : qpfrg::cuda_fail(c, e, "qpfrg_sigma_table");
}

// c->rows_compact of the last RHS
static qpfrg_status read_form(qpfrg_ctx *c)
{
    if (c->rhs_sym.mode == 2) {     // the form was decided on the device: read the test
        double r[4];
        cudaError_t e = cudaMemcpyAsync(r, c->d_sym, sizeof(r), cudaMemcpyDeviceToHost, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
        if (e != cudaSuccess) return qpfrg::cuda_fail(c, e, "qpfrg_rhs_work");
        const double tol = c->rhs_sym.tol;
        c->rows_compact = r[1] <= tol * r[0] && r[3] <= tol * r[2];
    }
    return QPFRG_OK;
}

extern "C" qpfrg_status qpfrg_rhs_evaluated(qpfrg_t c, long long *loop_evals, long long *table_rows)
{
    if (!c) return QPFRG_ERR_INVALID;
    const qpfrg_status s = read_form(c);
    if (s != QPFRG_OK) return s;
    const long long NN = (long long)c->pb.N * c->pb.N, rows = c->rows_compact ? c->n_rcan : NN;
    if (table_rows) *table_rows = rows;
    if (loop_evals) *loop_evals = !c->rows_compact && c->loop_red ? c->loop_evals_red : 2 * rows * c->pb.M;
    return QPFRG_OK;
}

extern "C" qpfrg_status qpfrg_rhs_work(qpfrg_t c, long long *loop_evals, long long *loop_evals_full,
                                       long long *rows_unreduced, long long *contraction_rows)
{
    if (!c) return QPFRG_ERR_INVALID;
    const long long full = 2LL * c->pb.N * c->pb.N * c->pb.M;
    const qpfrg_status s = read_form(c);
    if (s != QPFRG_OK) return s;
    if (loop_evals) *loop_evals = c->rows_compact ? c->loop_evals_rows : (c->loop_red ? c->loop_evals_red : full);
    if (loop_evals_full) *loop_evals_full = full;
    if (rows_unreduced) *rows_unreduced = c->loop_red ? c->loop_mismatch_rows : 0;
    if (contraction_rows) *contraction_rows = c->rows_compact ? c->n_rrep : (long long)c->pb.N * c->pb.N;
    return QPFRG_OK;
}
