// FP64 plans: a step's Tucker sums as phases of grouped mode products.  All
// sums that share an input (every slot, term and component of the group on F)
// advance one mode per phase, so a phase is three launches whatever their
// number: the tensors' digit images, the products, what those leave to FMA chains.
// The k terms of a sum are one contraction in its last mode (concatenated over the terms, the
// split weights eta folded into the matrices).
#include <algorithm>

#include "step64.h"

namespace ds {

using mm::Image;
using mm::Product;
using mm::View;

namespace {
const SplitCoeffs &coeffs(const ds_phi_set *s, int slot)
{
    return s->co[s->scheme == DS_ETD2RKDS ? slot : kSlotEll[slot] - 1];
}

void append(View &v, const double *src, double scale)
{
    v.src[v.ncat] = src;
    v.scale[v.ncat++] = scale;
}

std::vector<long long> view_key(const View &v)
{
    std::vector<long long> k = {v.ncat, v.n, v.I};
    for (int t = 0; t < v.ncat; ++t) {
        long long b;
        static_assert(sizeof(b) == sizeof(double), "");
        __builtin_memcpy(&b, &v.scale[t], sizeof b);
        k.push_back((long long)(uintptr_t)v.src[t]);
        k.push_back(b);
    }
    return k;
}

// Products of terms [i0, i1) of one sum in mode mu; z: the sum's intermediates.
// A term carries `parts` tensors between modes: 1, or 2 for the complex
// scheme (real, imaginary) and the tangent (derivative, value).
void sum_products(const ds_phi_set *s, SumKind kind, const SumOp &op, int i0, int i1, int mu, double *z, int64_t N,
                  std::vector<Product> &out)
{
    const int d = s->d;
    const bool cplx = s->scheme == DS_EXPRK3DS_CPLX, two = cplx || kind == SumKind::tangent;
    const int parts = two ? 2 : 1, nterm = i1 - i0, tr = kind == SumKind::transposed;
    const SplitCoeffs &co = coeffs(s, op.slot);
    const int64_t n = s->n[mu];
    auto tensor = [&](int m, int i, int part) { return z + N * (((m % 2) * nterm + (i - i0)) * parts + part); };
    const bool first = mu == 0, last = mu == d - 1;
    const double w = tr ? kSlotW[op.slot] * s->tau : 1.0;
    Product acc{};
    for (int i = i0; i < i1; ++i) {
        const int64_t o = s->P_off[op.c][op.slot][i][mu];
        const double *P = s->P_dev + o, *D = cplx ? s->Pim_dev + o : kind == SumKind::tangent ? s->dP_dev + o : nullptr;
        // input: one tensor (X or a term's value) or a term's two parts
        View a1 = mm::tensor_view(d, s->n, mu, first ? op.X : tensor(mu - 1, i, 0)), a2 = a1;
        if (two && !first) append(a2, tensor(mu - 1, i, 1), 1.0);
        auto product = [&](const View &A, const View &B, double *dst) {
            Product p{};
            p.A = A;
            p.B = B;
            p.out = dst;
            out.push_back(p);
        };
        auto pair = [&](const double *L0, double s0, const double *L1, double s1) {
            View v = mm::matrix_view(n, L0, tr, s0);
            append(v, L1, s1);
            return v;
        };
        if (!last) {
            const View m1 = mm::matrix_view(n, P, tr);
            if (!two) {
                product(a1, m1, tensor(mu, i, 0));
            } else if (first) {
                // complex: (Pr, Pi); tangent: (dP, P)
                const View m2 = mm::matrix_view(n, D, 0);
                product(a1, cplx ? m1 : m2, tensor(mu, i, 0));
                product(a1, cplx ? m2 : m1, tensor(mu, i, 1));
            } else if (cplx) {
                product(a2, pair(P, 1.0, D, -1.0), tensor(mu, i, 0));
                product(a2, pair(D, 1.0, P, 1.0), tensor(mu, i, 1));
            } else {
                product(a2, pair(P, 1.0, D, 1.0), tensor(mu, i, 0));
                const View v = mm::tensor_view(d, s->n, mu, tensor(mu - 1, i, 1));
                product(v, m1, tensor(mu, i, 1));
            }
            continue;
        }
        // last mode: every term into one contraction
        auto join = [&](const double *src, const double *L, double scale) {
            if (acc.A.ncat == 0) {
                acc.A = mm::tensor_view(d, s->n, mu, src);
                acc.B = mm::matrix_view(n, L, tr, scale);
            } else {
                append(acc.A, src, 1.0);
                append(acc.B, L, scale);
            }
        };
        if (cplx) {
            const double *M = s->Mf_dev + s->Mf_off[op.c][op.slot][i];
            join(a2.src[0], M, 1.0);
            join(a2.src[1], M + n * n, 1.0);
        } else if (kind == SumKind::tangent) {
            join(a2.src[0], P, co.eta[i]);
            join(a2.src[1], D, co.eta[i]);
        } else {
            join(a1.src[0], P, w * co.eta[i]);
        }
    }
    if (last) {
        acc.out = op.out;
        acc.accumulate = op.accumulate || i0 > 0;
        out.push_back(acc);
    }
}

void kron_products(const ds_phi_set *s, const double *X, double *Y, int mu, int transpose, int64_t N,
                   std::vector<Product> &out)
{
    for (int c = 0; c < 2; ++c) {
        Product p{};
        p.A = mm::tensor_view(s->d, s->n, mu, X + c * N);
        p.B = mm::matrix_view(s->n[mu], s->A_dev + s->A_off[c][mu], transpose);
        p.out = Y + c * N;
        p.accumulate = mu > 0;
        out.push_back(p);
    }
}

// ops (of k terms each) that fit the intermediates at once; 0: not even one
int ops_at_once(const Sums64 &e, SumKind kind)
{
    const int t = sum_tensors(e.set, kind);
    return t == 0 ? 1 << 20 : (int)(e.z_tensors / t);
}
}  // namespace

int sum_tensors(const ds_phi_set *s, SumKind kind)
{
    const int parts = s->scheme == DS_EXPRK3DS_CPLX || kind == SumKind::tangent ? 2 : 1;
    return s->k * parts * std::min(s->d - 1, 2);
}

void sums_create(Sums64 &e, const ds_phi_set *s, int64_t N, const std::vector<SumGroup> &groups, double *z,
                 int64_t z_tensors, cudaStream_t st)
{
    e.set = s;
    e.N = N;
    e.z = z;
    e.z_tensors = z_tensors;
    // the phases' matrices and the scratch of the largest phase
    std::vector<View> views;
    std::vector<Image> ims;
    std::vector<size_t> offs;
    size_t bytes = 0, scratch = 0;
    auto phase = [&](std::vector<Product> &ps) {
        const int count = (int)ps.size();
        if (!count || !mm::use_digits(ps[0].A.rows, ps[0].A.n, count)) return;
        scratch = std::max(scratch, mm::scratch_bytes(N, ps[0].A.n, count, ps[0].A.ncat, false));
        for (const Product &p : ps) {
            Image &im = e.images[view_key(p.B)];
            if (im.rb) continue;   // already listed
            im.rb = mm::tile_cols(p.A.rows, (int)p.B.rows, count, mm::slabs_of(p.B.n, p.B.ncat));
            im.slabs = mm::slabs_of(p.B.n, p.B.ncat);
            im.rows = p.B.rows;
            offs.push_back(bytes);
            bytes += mm::image_total(p.B, im.rb);
            views.push_back(p.B);
            ims.push_back(im);
        }
    };
    for (const SumGroup &g : groups) {
        std::vector<SumOp> ops;
        for (int c = 0; c < 2; ++c)
            for (int q : g.slots) ops.push_back({c, q, nullptr, nullptr, false});
        const int at_once = std::max(1, std::min(ops_at_once(e, g.kind), (int)ops.size()));
        for (size_t b = 0; b < ops.size(); b += at_once)
            for (int mu = 0; mu < s->d; ++mu) {
                std::vector<Product> ps;
                for (size_t q = b; q < std::min(ops.size(), b + at_once); ++q)
                    sum_products(s, g.kind, ops[q], 0, s->k, mu, nullptr, N, ps);
                phase(ps);
            }
    }
    if (!s->tridiag[0] || !s->tridiag[1])
        for (int tr = 0; tr < 2; ++tr)
            for (int mu = 0; mu < s->d; ++mu) {
                std::vector<Product> ps;
                kron_products(s, nullptr, nullptr, mu, tr, N, ps);
                phase(ps);
            }
    if (scratch && device_alloc(&e.ctx.ws, scratch) == cudaSuccess) {
        e.ctx.ws_bytes = scratch;
    } else {
        cudaGetLastError();
        e.ctx.ws = nullptr;
    }
    if (views.empty() || device_alloc(&e.mats, bytes) != cudaSuccess) {
        cudaGetLastError();
        e.mats = nullptr;
        e.images.clear();
        return;
    }
    for (size_t q = 0; q < views.size(); ++q) {
        Image &im = ims[q];
        im.place(e.mats + offs[q], 1);
        e.images[view_key(views[q])] = im;
    }
    for (size_t q = 0; q < views.size(); q += mm::kMaxProd)
        mm::launch_split(&views[q], &ims[q], (int)std::min<size_t>(mm::kMaxProd, views.size() - q), nullptr, st);
    cudaStreamSynchronize(st);
}

void sums_destroy(Sums64 &e)
{
    cudaFree(e.ctx.ws);
    cudaFree(e.mats);
    e.ctx.ws = e.mats = nullptr;
    e.images.clear();
}

namespace {
int run_phase(const Sums64 &e, std::vector<Product> &ps, Prof *prof, cudaStream_t st)
{
    for (Product &p : ps) {
        auto it = e.images.find(view_key(p.B));
        if (it != e.images.end()) p.ib = it->second;
    }
    mm::Context c = e.ctx;
    c.prof = prof;
    return mm::run_products(c, ps.data(), (int)ps.size(), st);
}
}  // namespace

int run_sums(const Sums64 &e, SumKind kind, const SumOp *ops, int count, Prof *prof, cudaStream_t st)
{
    const ds_phi_set *s = e.set;
    const int per_op = sum_tensors(s, kind), fit = ops_at_once(e, kind);
    const int at_once = std::max(1, std::min(fit, count));
    const int terms = fit > 0 ? s->k : 1;   // short of memory: term by term
    int launches = 0;
    for (int b = 0; b < count; b += at_once)
        for (int i0 = 0; i0 < s->k; i0 += terms)
            for (int mu = 0; mu < s->d; ++mu) {
                std::vector<Product> ps;
                for (int q = b; q < std::min(count, b + at_once); ++q)
                    sum_products(s, kind, ops[q], i0, std::min(s->k, i0 + terms), mu, e.z + e.N * per_op * (q - b), e.N, ps);
                launches += run_phase(e, ps, prof, st);
            }
    return launches;
}

int run_partial(const Sums64 &e, int c, int slot, int term, int md, const double *X, double *out, Prof *prof, cudaStream_t st)
{
    const ds_phi_set *s = e.set;
    int launches = 0;
    for (int mu = 0; mu < s->d; ++mu) {
        std::vector<Product> ps(1);
        ps[0].A = mm::tensor_view(s->d, s->n, mu, mu ? e.z + e.N * ((mu - 1) % 2) : X);
        ps[0].B = mm::matrix_view(s->n[mu], (mu == md ? s->dP_dev : s->P_dev) + s->P_off[c][slot][term][mu], 0);
        ps[0].out = mu == s->d - 1 ? out : e.z + e.N * (mu % 2);
        launches += run_phase(e, ps, prof, st);
    }
    return launches;
}

int run_kronsum(const Sums64 &e, const double *X, double *Y, int transpose, Prof *prof, cudaStream_t st)
{
    int launches = 0;
    for (int mu = 0; mu < e.set->d; ++mu) {
        std::vector<Product> ps;
        kron_products(e.set, X, Y, mu, transpose, e.N, ps);
        launches += run_phase(e, ps, prof, st);
    }
    return launches;
}

}  // namespace ds
