// Problem-level setup shared by the single-laminate context and the batch:
// decomposition, symbolic analysis with global numbering, local element maps
// and the GenEO coarse space (Section 2.3, Fig. eig).
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "host_parallel.h"
#include "problem.h"

namespace gl {

namespace {

// Coarse columns whose Cholesky pivot of the unit-diagonal-scaled K_0 falls to
// 1e-10 or below (the column lies within an angle of about 1e-5, in the K
// inner product, of the span of the earlier ones) are dropped as dependent:
// this happens when two subdomains coincide (a box grown by the overlap to the
// whole extent of a narrow laminate) or when Xi_j p vanishes.
constexpr double COARSE_DROP_TOL = 1e-10;

std::vector<std::pair<int, int>> split_range(int n, int p) {
    std::vector<std::pair<int, int>> out;
    int q = n / p, r = n % p, s = 0;
    for (int i = 0; i < p; ++i) {
        int size = q + (i < r ? 1 : 0);
        out.push_back({s, s + size});
        s += size;
    }
    return out;
}

void check_err(const Problem &P, const char *what) {
    int h = 0;
    GL_CUDA(cudaMemcpyAsync(&h, P.d_err, sizeof(int), cudaMemcpyDeviceToHost, P.stream));
    GL_CUDA(cudaStreamSynchronize(P.stream));
    if (h) {
        GL_CUDA(cudaMemsetAsync(P.d_err, 0, sizeof(int), P.stream));
        if (h == 2) fail(GL_ERR_TIMEOUT, std::string(what) + ": a tensor-core wait gave up");
        fail(GL_ERR_NOT_SPD, std::string(what) + ": non-positive pivot");
    }
}

// G (n x m, column stride n) [gdof_j[i] - gshift, :] = Y_j[i, :] (or 0)
__global__ void k_scatter_cols(const int64_t *__restrict__ gdof, int64_t off, int64_t n, const double *__restrict__ Y,
                               int64_t yoff, int m, double *__restrict__ G, int64_t N, int64_t gshift, int zero) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n * m; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t a = i / n, r = i % n;
        G[a * N + gdof[off + r] - gshift] = zero ? 0.0 : Y[yoff + a * n + r];
    }
}

// Blocks (l, j) of K0 for the neighbours l = nbr[blockIdx.y] of subdomain j:
// K0[((l - sub0) m + a) + (col0 + b) n0] = sum_i Z_l[i, a] G[gdof_l[i] - gshift, b].
__global__ void __launch_bounds__(256) k_coarse_block(const int *__restrict__ nbr, const int64_t *__restrict__ voff,
                                                      const int64_t *__restrict__ vlen,
                                                      const int64_t *__restrict__ gdof, const double *__restrict__ Z,
                                                      int m, const double *__restrict__ G, int64_t N, int64_t gshift,
                                                      double *__restrict__ K0, int64_t n0, int sub0, int col0) {
    const int a = blockIdx.x / m, b = blockIdx.x % m, l = nbr[blockIdx.y];
    const int64_t n = vlen[l];
    const double *Za = Z + voff[l] * m + a * n, *Gb = G + b * N - gshift;
    const int64_t *gd = gdof + voff[l];
    double v = 0.0;
#pragma unroll 4
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) v += Za[i] * Gb[gd[i]];
    __shared__ double red[256];
    red[threadIdx.x] = v;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) K0[((int64_t)(l - sub0) * m + a) + (int64_t)(col0 + b) * n0] = red[0];
}

}  // namespace

void part_boxes(const MeshHost &m, int px, int py, int pz, int overlap, std::vector<SubBox> &out) {
    auto rx = split_range(m.nx, px), ry = split_range(m.ny, py), rz = split_range(m.nz, pz);
    const int ne[3] = {m.nx, m.ny, m.nz};
    for (int kz = 0; kz < pz; ++kz)
        for (int ky = 0; ky < py; ++ky)
            for (int kx = 0; kx < px; ++kx) {
                SubBox b{};
                std::pair<int, int> core[3] = {rx[kx], ry[ky], rz[kz]};
                for (int d = 0; d < 3; ++d) {
                    int lo = std::max(0, core[d].first - overlap), hi = std::min(ne[d], core[d].second + overlap);
                    b.ebox[2 * d] = lo;
                    b.ebox[2 * d + 1] = hi;
                    b.nbox[2 * d] = 2 * lo;
                    b.nbox[2 * d + 1] = 2 * hi;
                    b.art[2 * d] = lo > 0;
                    b.art[2 * d + 1] = hi < ne[d];
                }
                out.push_back(b);
            }
}

void problem_symbolic(const Problem &P, bool neumann, int leaf_nodes, std::vector<SubSymbolic> &syms) {
    const int nsub = (int)P.boxes.size();
    syms.assign(nsub, SubSymbolic());
    parallel_for(nsub, [&](int j) {
        const Part &pt = P.parts[P.sub_part[j]];
        build_symbolic(*pt.m, P.boxes[j], pt.is_dir, neumann, leaf_nodes, syms[j]);
        for (auto &g : syms[j].gdof) g += pt.dof_off;
        for (auto &e : syms[j].pair_elem) e += (int)pt.elem_off;
    });
}

void problem_local_elems(const Problem &P, int s0, int s1, const FactorPlan &plan, LocalElems &E) {
    std::vector<int64_t> at(s1 - s0 + 1, 0);   // first pair of each subdomain
    for (int j = s0; j < s1; ++j) {
        const int *e = P.boxes[j].ebox;
        at[j - s0 + 1] = at[j - s0] + (int64_t)(e[1] - e[0]) * (e[3] - e[2]) * (e[5] - e[4]);
    }
    std::vector<int> elem(at.back()), sub(at.back()), loc(81 * at.back());
    parallel_for(s1 - s0, [&](int jl) {
        const int j = s0 + jl;
        const Part &pt = P.parts[P.sub_part[j]];
        const MeshHost &m = *pt.m;
        const SubBox &b = P.boxes[j];
        const int nbx = b.nbox[1] - b.nbox[0] + 1, nby = b.nbox[3] - b.nbox[2] + 1, nbz = b.nbox[5] - b.nbox[4] + 1;
        std::vector<int> map((size_t)nbx * nby * nbz * 3, -1);
        const int64_t off = plan.vec_off[jl];
        for (int64_t i = 0; i < plan.vec_len[jl]; ++i) {
            int64_t g = plan.h_gdof[off + i] - pt.dof_off;
            int64_t node = g / 3;
            int comp = (int)(g % 3);
            int x = (int)(node % m.NX), y = (int)((node / m.NX) % m.NY), z = (int)(node / ((int64_t)m.NX * m.NY));
            map[3 * ((size_t)(x - b.nbox[0]) + (size_t)nbx * ((y - b.nbox[2]) + (size_t)nby * (z - b.nbox[4]))) + comp] =
                (int)i;
        }
        int64_t k = at[jl];
        for (int ez = b.ebox[4]; ez < b.ebox[5]; ++ez)
            for (int ey = b.ebox[2]; ey < b.ebox[3]; ++ey)
                for (int ex = b.ebox[0]; ex < b.ebox[1]; ++ex, ++k) {
                    elem[k] = (int)(pt.elem_off + ex + (int64_t)m.nx * (ey + (int64_t)m.ny * ez));
                    sub[k] = jl;
                    int *l = &loc[81 * k];
                    for (int a = 0; a < 27; ++a) {
                        int yg = 2 * ey + (a / 3) % 3;
                        if (m.periodic && yg == m.NY - 1) yg = 0;   // the first-plane partner carries the DOFs
                        int x = 2 * ex + a % 3 - b.nbox[0], y = yg - b.nbox[2], z = 2 * ez + a / 9 - b.nbox[4];
                        for (int cc = 0; cc < 3; ++cc)
                            l[3 * a + cc] = map[3 * ((size_t)x + (size_t)nbx * (y + (size_t)nby * z)) + cc];
                    }
                }
    });
    E.n_pairs = (int64_t)elem.size();
    E.elem.upload(elem, P.stream);
    E.sub.upload(sub, P.stream);
    E.loc.upload(loc, P.stream);
    GL_CUDA(cudaStreamSynchronize(P.stream));
}

std::future<std::vector<SubSymbolic>> neumann_symbolic(const Problem &P, int leaf_nodes) {
    return in_background([&P, leaf_nodes] {
        std::vector<SubSymbolic> syms;
        problem_symbolic(P, true, leaf_nodes, syms);
        return syms;
    });
}

void problem_coarse(const Problem &P, const gl_opts &o, const FactorPlan &PD, std::vector<SubSymbolic> syms,
                    Coarse &out) {
    cudaStream_t s = P.stream;
    const int nev = o.nev;
    const double sigma = o.sigma > 0 ? o.sigma : 1e-3;
    const int nsub = (int)P.boxes.size();
    build_plan(syms, out.PN, s);
    out.PN.s20 = PD.s20;
    P.stamp("Neumann plan");
    FactorPlan &PN = out.PN;
    for (int j = 0; j < nsub; ++j)
        if (PN.vec_len[j] < nev) fail(GL_ERR_INVALID_ARG, "subdomain has fewer DOFs than nev");
    // partition of unity: 1/multiplicity over the Dirichlet (interior) sets, 0 on artificial boundaries
    std::vector<int> mult(P.n_dof, 0);
    for (int64_t g : PD.h_gdof) mult[g] += 1;
    std::vector<double> xi(PN.n_local, 0.0);
    parallel_for(nsub, [&](int j) {
        const Part &pt = P.parts[P.sub_part[j]];
        const MeshHost &m = *pt.m;
        const SubBox &b = P.boxes[j];
        for (int64_t i = 0; i < PN.vec_len[j]; ++i) {
            const int64_t g = PN.h_gdof[PN.vec_off[j] + i];
            const int64_t node = (g - pt.dof_off) / 3;
            int pos[3] = {(int)(node % m.NX), (int)((node / m.NX) % m.NY), (int)(node / ((int64_t)m.NX * m.NY))};
            bool art = false;
            for (int d = 0; d < 3; ++d) {
                if (b.art[2 * d] && pos[d] == b.nbox[2 * d]) art = true;
                if (b.art[2 * d + 1] && pos[d] == b.nbox[2 * d + 1]) art = true;
            }
            if (!art) {
                if (mult[g] == 0) fail(GL_ERR_INVALID_ARG, "a free DOF lies in no subdomain interior (overlap >= 1?)");
                xi[PN.vec_off[j] + i] = 1.0 / mult[g];
            }
        }
    });
    DBuf<double> d_xi;
    d_xi.upload(xi, s);
    // basis columns: room for about four times nev before a restart, and Ritz vectors kept by one
    const int mmax = nev <= 12 ? 64 : KRY_MAX, keep = nev + KRY_B;
    const int64_t nl = PN.n_local;
    out.nev = nev;
    out.n0 = nsub * nev;
    out.Z.alloc(nl * nev);
    out.eig.assign((size_t)nsub * nev, 0.0);
    const int iters = o.eig_iters > 0 ? o.eig_iters : 100;
    // Groups of subdomains: factor of M = A^N + sigma B, B = Xi A^N Xi, and the
    // block Krylov iteration, one group at a time.  Beside the factors a local DOF
    // holds a row of the basis and its two images, of the four blocks and of a
    // restart's copy.
    const int64_t budget = (int64_t)((o.eig_group_bytes > 0 ? o.eig_group_bytes : 4e10) / sizeof(double));
    const int64_t per_dof = 3 * mmax + 4 * KRY_B + keep;
    int j0 = 0, max_its = 0;
    LocalElems E;
    while (j0 < nsub) {
        int j1 = j0;
        int64_t acc = 0;
        for (; j1 < nsub; ++j1) {
            const int64_t need = syms[j1].l_size + per_dof * syms[j1].n;
            if (j1 > j0 && acc + need > budget) break;
            acc += need;
        }
        const int ng = j1 - j0;
        ++out.n_groups;
        // a group of all subdomains is the whole problem's plan
        FactorPlan group;
        if (ng < nsub) {
            build_plan(std::vector<SubSymbolic>(syms.begin() + j0, syms.begin() + j1), group, s);
            group.s20 = PD.s20;
        }
        FactorPlan &PG = ng < nsub ? group : PN;
        PG.ws_budget_bytes = PD.ws_budget_bytes;
        const int64_t goff = PN.vec_off[j0], gl = PG.n_local;
        DBuf<double> LN;
        LN.alloc(PG.l_size);
        const double *xg = d_xi.p + goff;
        numeric_factor<double>(PG, P.C, P.geo, xg, sigma, LN.p, P.d_err, s);
        check_err(P, "GenEO shifted Neumann factorisation");
        P.stamp("Neumann factorisation (group)");
        problem_local_elems(P, j0, j1, PG, E);
        // Block Krylov (Lanczos) method for the largest mu of B p = mu M p, M = A^N + sigma B factored: the basis
        // V grows by the block M^{-1} B V_last, made M-orthonormal against all of V, and T = V^T B V gives the Ritz
        // pairs.  It stops when the residuals |M^{-1} B p - mu p|_M of the kept pairs are below EIG_RESID mu in
        // every subdomain.  About ten steps of eight solves did for nev = 10 on the corner, where a subspace
        // iteration with 20 vectors took 20 steps.
        constexpr double EIG_RESID = 1e-6;
        DBuf<double> V, MV, BV, W, MW, BW, ysc, T, H, G, R, Y, mu;
        DBuf<unsigned long long> worst;
        for (DBuf<double> *v : {&V, &MV, &BV}) v->alloc(gl * mmax);
        for (DBuf<double> *v : {&W, &MW, &BW, &ysc}) v->alloc(gl * KRY_B);
        T.alloc((size_t)ng * mmax * mmax);
        T.zero(s);
        H.alloc((size_t)ng * mmax * KRY_B);
        for (DBuf<double> *v : {&G, &R}) v->alloc((size_t)ng * KRY_B * KRY_B);
        Y.alloc((size_t)ng * KRY_MAX * keep);
        mu.alloc((size_t)ng * keep);
        worst.alloc(1);
        const int64_t ts = (int64_t)mmax * mmax, hs = (int64_t)mmax * KRY_B, ys = (int64_t)KRY_MAX * keep;
        const KryBlocks first{2, {V.p, MV.p}, {W.p, BW.p}}, all{3, {V.p, MV.p, BV.p}, {W.p, MW.p, BW.p}};
        const KryBlocks only_w{1, {V.p}, {W.p}};
        auto gram_block = [&](const double *MWp) {
            G.zero(s);
            kry_gram(PG, W.p, KRY_B, KRY_B, MWp, G.p, KRY_B * KRY_B, KRY_B, s);
        };
        auto apply_B = [&]() {
            BW.zero(s);
            local_K_apply(PG, E, P.C, P.geo, xg, W.p, BW.p, KRY_B, s);
        };
        fill_random(W.p, gl * KRY_B, 0x1707042280000001ull + (uint64_t)j0, s);
        apply_B();
        int it = 0, m = 0, kept = 0, next_check = 0;
        double resid = 0.0;
        for (;;) {
            // the last block's columns of T; W = M^{-1} B W_last (MW holds the sweeps' right-hand side)
            if (m > 0) kry_gram(PG, V.p, mmax, m, BW.p, T.p + (m - KRY_B), ts, mmax, s);
            GL_CUDA(cudaMemcpyAsync(MW.p, BW.p, sizeof(double) * gl * KRY_B, cudaMemcpyDeviceToDevice, s));
            W.zero(s);
            ysc.zero(s);
            factor_solve8(PG, LN.p, MW.p, ysc.p, W.p, P.d_err, s);
            ++it;
            // first pass: M W = B W_last up to the solve's error, so G is good for the residuals and a first scaling
            H.zero(s);
            kry_gram(PG, MV.p, mmax, m, W.p, H.p, hs, KRY_B, s);
            kry_project(PG, first, mmax, m, H.p, hs, KRY_B, s);
            gram_block(BW.p);
            // The Ritz pairs when they are needed: to restart, at the end, and when the residuals should have got
            // there at 10 a step, the fastest they were seen to fall (3 to 10).  A pair costs 1.5 to 2 ms, a step 1 to
            // 6; with 30 a step for the estimate two of six times were in vain.
            const bool last = it > iters && m >= nev;
            if (last || (m >= nev && m + KRY_B > mmax) || (m >= nev + KRY_B / 2 && it >= next_check)) {
                kept = std::min(keep, m);
                kry_ritz(PG, T.p, mmax, m, G.p, nev, kept, Y.p, keep, mu.p, worst.p, s);
                unsigned long long bits = 0;
                GL_CUDA(cudaMemcpyAsync(&bits, worst.p, sizeof(bits), cudaMemcpyDeviceToHost, s));
                check_err(P, "GenEO Rayleigh-Ritz");
                std::memcpy(&resid, &bits, sizeof(resid));
                if (resid <= EIG_RESID || last) break;
                next_check = it + 1 + (int)std::max(0.0, std::min(8.0, std::log10(resid / EIG_RESID)));
            }
            kry_orth(ng, true, G.p, H.p, hs, KRY_B, m, 1e-24, R.p, P.d_err, s);
            kry_scale(PG, only_w, R.p, mmax, -1, s, 0x1707042280000000ull + ((uint64_t)it << 40) + (uint64_t)j0);
            if (m + KRY_B > mmax) {
                // restart from the leading Ritz vectors: V <- V Y, T = diag(mu)
                DBuf<double> tmp;
                tmp.alloc(gl * kept);
                for (DBuf<double> *B : {&V, &MV, &BV}) {
                    kry_combine(PG, B->p, mmax, m, Y.p, ys, keep, kept, tmp.p, kept, s);
                    for (int j = 0; j < ng; ++j)
                        GL_CUDA(cudaMemcpyAsync(B->p + PG.vec_off[j] * mmax, tmp.p + PG.vec_off[j] * kept,
                                                PG.vec_len[j] * kept * sizeof(double), cudaMemcpyDeviceToDevice, s));
                }
                kry_diag(ng, T.p, mmax, mu.p, keep, kept, s);
                m = kept;
                GL_CUDA(cudaStreamSynchronize(s));
            }
            // second pass with the block's own images B W and M W = A^N W + sigma B W: orthonormal to rounding.
            // (Carrying M W along from the first pass lets the solves' errors grow by the ratio of the largest mu,
            // 1 / sigma, to the kept ones.)
            apply_B();
            MW.zero(s);
            axpy(MW.p, sigma, BW.p, gl * KRY_B, s);
            local_K_apply(PG, E, P.C, P.geo, nullptr, W.p, MW.p, KRY_B, s);
            H.zero(s);
            kry_gram(PG, V.p, mmax, m, MW.p, H.p, hs, KRY_B, s);
            kry_project(PG, all, mmax, m, H.p, hs, KRY_B, s);
            gram_block(MW.p);
            kry_orth(ng, false, G.p, H.p, hs, KRY_B, m, 1e-6, R.p, P.d_err, s);
            kry_scale(PG, all, R.p, mmax, m, s);
            m += KRY_B;
        }
        if (std::getenv("GL_VERBOSE"))
            std::fprintf(stderr, "[gl]   group %d-%d: %d block steps, basis %d, largest residual %.2e\n", j0, j1 - 1, it, m,
                         resid);
        std::vector<double> mu_now((size_t)ng * keep);
        GL_CUDA(cudaMemcpyAsync(mu_now.data(), mu.p, mu_now.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
        GL_CUDA(cudaStreamSynchronize(s));
        max_its = std::max(max_its, it);
        for (int j = 0; j < ng; ++j)
            for (int a = 0; a < nev; ++a) out.eig[(size_t)(j0 + j) * nev + a] = 1.0 / mu_now[(size_t)j * keep + a] - sigma;
        // Z columns of these subdomains (whole-problem Neumann layout, nev columns)
        kry_combine(PG, V.p, mmax, m, Y.p, ys, keep, nev, out.Z.p + goff * nev, nev, s);
        GL_CUDA(cudaStreamSynchronize(s));
        P.stamp("GenEO block Krylov (group)");
        j0 = j1;
    }
    out.eig_iters = max_its;
    syms.clear();
    scale_rows(PN, out.Z.p, d_xi.p, nev, s);                        // Z = Xi p
    if (out.n_groups > 1) problem_local_elems(P, 0, nsub, PN, E);
    // K_0 = Z^T K Z per part: Y_j = A^N_j Z_j, then blocks against the overlapping subdomains of the part
    DBuf<double> KZ;
    KZ.alloc(nl * nev);
    KZ.zero(s);
    local_K_apply(PN, E, P.C, P.geo, nullptr, out.Z.p, KZ.p, nev, s);
    out.koff.clear();
    out.kvoff.clear();
    out.n_dropped = 0;
    out.part_dropped.assign(P.parts.size(), 0);
    out.kn.clear();
    int64_t ktot = 0;
    for (const Part &pt : P.parts) {
        int n0p = (pt.sub1 - pt.sub0) * nev;
        out.koff.push_back(ktot);
        out.kvoff.push_back(pt.sub0 * nev);
        out.kn.push_back(n0p);
        ktot += (int64_t)n0p * n0p;
    }
    out.Kinv.alloc(std::max<int64_t>(ktot, 1));
    for (size_t ip = 0; ip < P.parts.size(); ++ip) {
        const Part &pt = P.parts[ip];
        const int n0p = out.kn[ip];
        if (n0p == 0) continue;
        const int64_t Np = pt.m->n_dof;
        DBuf<double> G, K0;
        G.alloc((size_t)Np * nev);
        G.zero(s);
        K0.alloc((size_t)n0p * n0p);
        K0.zero(s);
        // the neighbours of every subdomain (boxes that meet), one launch for all of one's blocks
        std::vector<int> nbr, at(1, 0);
        for (int j = pt.sub0; j < pt.sub1; ++j) {
            for (int l = pt.sub0; l < pt.sub1; ++l) {
                bool overlap = true;
                for (int d = 0; d < 3; ++d)
                    if (P.boxes[l].nbox[2 * d] > P.boxes[j].nbox[2 * d + 1] ||
                        P.boxes[j].nbox[2 * d] > P.boxes[l].nbox[2 * d + 1])
                        overlap = false;
                if (overlap) nbr.push_back(l);
            }
            at.push_back((int)nbr.size());
        }
        DBuf<int> d_nbr;
        d_nbr.upload(nbr, s);
        for (int j = pt.sub0; j < pt.sub1; ++j) {
            const int64_t nj = PN.vec_len[j], oj = PN.vec_off[j];
            const int k = j - pt.sub0;
            k_scatter_cols<<<256, 256, 0, s>>>(PN.d_gdof.p, oj, nj, KZ.p, oj * nev, nev, G.p, Np, pt.dof_off, 0);
            k_coarse_block<<<dim3(nev * nev, at[k + 1] - at[k]), 256, 0, s>>>(
                d_nbr.p + at[k], PN.d_vec_off.p, PN.d_vec_len.p, PN.d_gdof.p, out.Z.p, nev, G.p, Np, pt.dof_off, K0.p,
                n0p, pt.sub0, k * nev);
            k_scatter_cols<<<256, 256, 0, s>>>(PN.d_gdof.p, oj, nj, KZ.p, oj * nev, nev, G.p, Np, pt.dof_off, 1);
            GL_CUDA(cudaGetLastError());
        }
        out.part_dropped[ip] = dense_inverse(K0.p, n0p, out.Kinv.p + out.koff[ip], P.d_err, s, COARSE_DROP_TOL);
        out.n_dropped += out.part_dropped[ip];
        check_err(P, "coarse Cholesky");
    }
    out.d_koff.upload(out.koff, s);
    out.d_kvoff.upload(out.kvoff, s);
    out.d_kn.upload(out.kn, s);
    GL_CUDA(cudaStreamSynchronize(s));
}

void coarse_apply(const Coarse &Cs, const double *r, double *z, double *c1, double *c2, cudaStream_t s) {
    if (Cs.n0 == 0) return;
    coarse_restrict(Cs.PN, Cs.Z.p, Cs.nev, r, c1, s);
    dense_symv_blocks(Cs.Kinv.p, Cs.d_koff.p, Cs.d_kvoff.p, Cs.d_kn.p, (int)Cs.kn.size(), Cs.n0, c1, c2, s);
    coarse_prolong(Cs.PN, Cs.Z.p, Cs.nev, c2, z, s);
}

}  // namespace gl
