// Adjoint of the assembly (sta_adjoint): dL/dE, dL/dnu and dL/dx for an upstream gradient dL/dA
// given per CSR entry.
//
// With G_ab = dL/dA restricted to the block of nodes (a, b) of a tetrahedron, g_a the barycentric
// gradients and K = V (lam A + mu B), A[ai][bj] = g_a[i] g_b[j], B[ai][bj] = g_a[j] g_b[i] + d_ij
// g_a.g_b:
//   SA = sum_ab g_a^T G_ab g_b,   SB = sum_ab (g_b^T G_ab g_a + tr(G_ab) g_a.g_b)
//   dL/dE  = V (lam_E SA + mu_E SB),  dL/dnu = V (lam_nu SA + mu_nu SB)
//   dL/dx_c = V [ (lam SA + mu SB) g_c - sum_a (h_a . g_c) g_a ],  h_a = d(lam SA + mu SB)/dg_a
// using dV/dx_c = V g_c and dg_a = -(g_a . dx_c) g_c (barycentric gradients of a P1 tetrahedron).
//
// What bounds it: the FP64 pipe (an SM quadrant issues one FP64 warp instruction per 64 cycles;
// the kernel that worked on the four nodes' 16 blocks kept it 91% busy with 892 instructions a
// tetrahedron, 610 us for 376,000; now 336 us, and 34 us for k_grad_units).  So the algebra is
// arranged for few FP64 operations, about 450:
//  * the blocks (a, b) and (b, a) enter every sum through H = G_ab + G_ba^T only, and H through its
//    symmetric and antisymmetric parts: SA = FS + FA, SB = FS - FA + FT with FS = sum g_a^T S_ab
//    g_b, FA the same over the antisymmetric parts (cross products: 6 operations, not 9) and FT
//    over the traces.  H is the same for every tetrahedron of a node pair (7 on average), so its
//    parts are formed once per pair by a pass over the gradient (k_grad_units), which also turns
//    the 144 scattered 8-byte loads of a tetrahedron into 42 16-byte ones;
//  * g_0 = -(g_1 + g_2 + g_3) is put into the quadratic forms: 6 blocks instead of 10, 3 gradients
//    instead of 4, and dx_0 = -(dx_1 + dx_2 + dx_3).  Node 0 here is the node with the largest
//    gradient (k_elements notes which: the edges' differences start at it as well): the others'
//    gradients are no larger than what they add up to, so nothing cancels.  With a node of small
//    gradient in its place, the far tip of a tetrahedron 100 times as high as wide, and the upstream
//    gradient on that node, the results lost four digits;
//  * the value of a form is half its gradient's product with g; 3 divisions instead of 8.
// No evaluation order is fixed here; every product-sum is an FMA chain.
#include "sta_internal.cuh"

namespace sta {
namespace {

constexpr int GU = 10;  // doubles of a unit's row in the gradient buffer

// Symmetric and antisymmetric parts of every unit's gradient: a diagonal unit's G + G^T
// (00 01 02 11 12 22), a pair unit's S = (H + H^T) / 2 (the same six) and A = (H - H^T) / 2
// (01 02 12), H with the rows of the lower node.  One thread per unit; bound by the loads of the
// blocks' 24-byte row pieces (34 us for 26 M gradient entries: 3.4x its bytes at copy rate).
__global__ void __launch_bounds__(256)
k_grad_units(int64_t nunits, const int4 *__restrict__ bmeta, const int2 *__restrict__ bmirror,
             const double *__restrict__ gval, double *__restrict__ gu) {
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nunits;
         u += (int64_t)gridDim.x * blockDim.x) {
        const int4 bm = bmeta[u];
        const int rs = bm.y >> 1;
        const double *p = gval + bm.x;
        double h[3][3], o[GU];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) h[i][j] = __ldg(p + i * rs + j);
        if (bm.y & 1) {
#pragma unroll
            for (int k = 6; k < GU; ++k) o[k] = 0.0;
            o[0] = h[0][0] + h[0][0];
            o[1] = h[0][1] + h[1][0];
            o[2] = h[0][2] + h[2][0];
            o[3] = h[1][1] + h[1][1];
            o[4] = h[1][2] + h[2][1];
            o[5] = h[2][2] + h[2][2];
        } else {
            const int2 mir = bmirror[u];
            const double *q = gval + mir.x;
            double m[3][3];
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int i = 0; i < 3; ++i) m[j][i] = __ldg(q + j * mir.y + i);
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) h[i][j] += m[j][i];
            o[0] = h[0][0];
            o[1] = 0.5 * (h[0][1] + h[1][0]);
            o[2] = 0.5 * (h[0][2] + h[2][0]);
            o[3] = h[1][1];
            o[4] = 0.5 * (h[1][2] + h[2][1]);
            o[5] = h[2][2];
            o[6] = 0.5 * (h[0][1] - h[1][0]);
            o[7] = 0.5 * (h[0][2] - h[2][0]);
            o[8] = 0.5 * (h[1][2] - h[2][1]);
            o[9] = 0.0;
        }
        double2 *out = reinterpret_cast<double2 *>(gu + GU * u);
#pragma unroll
        for (int k = 0; k < GU / 2; ++k) out[k] = make_double2(o[2 * k], o[2 * k + 1]);
    }
}

struct V3 {
    double x, y, z;
};

__device__ __forceinline__ V3 diff(const double4_32a &a, const double4_32a &b) {
    return {a.x - b.x, a.y - b.y, a.z - b.z};
}
__device__ __forceinline__ V3 cross(const V3 &u, const V3 &v) {
    return {__fma_rn(u.y, v.z, -(u.z * v.y)), __fma_rn(u.z, v.x, -(u.x * v.z)),
            __fma_rn(u.x, v.y, -(u.y * v.x))};
}
__device__ __forceinline__ V3 scaled(const V3 &u, double s) { return {u.x * s, u.y * s, u.z * s}; }
__device__ __forceinline__ double dot_add(const V3 &u, const V3 &v, double s) {
    return __fma_rn(u.z, v.z, __fma_rn(u.y, v.y, __fma_rn(u.x, v.x, s)));
}
__device__ __forceinline__ void axpy(double s, const V3 &v, V3 &y) {
    y.x = __fma_rn(s, v.x, y.x);
    y.y = __fma_rn(s, v.y, y.y);
    y.z = __fma_rn(s, v.z, y.z);
}

struct Sym {  // 00 01 02 11 12 22
    double c[6];
};

template <typename T> __device__ __forceinline__ void swap_if(bool on, T &a, T &b) {
    const T t = on ? b : a;
    b = on ? a : b;
    a = t;
}
__device__ __forceinline__ void swap_if(bool on, V3 &a, V3 &b) {
    swap_if(on, a.x, b.x);
    swap_if(on, a.y, b.y);
    swap_if(on, a.z, b.z);
}

__device__ __forceinline__ double tr(const Sym &s) { return (s.c[0] + s.c[3]) + s.c[5]; }
// y += S g
__device__ __forceinline__ void sym_add(const Sym &s, const V3 &g, V3 &y) {
    y.x = __fma_rn(s.c[2], g.z, __fma_rn(s.c[1], g.y, __fma_rn(s.c[0], g.x, y.x)));
    y.y = __fma_rn(s.c[4], g.z, __fma_rn(s.c[3], g.y, __fma_rn(s.c[1], g.x, y.y)));
    y.z = __fma_rn(s.c[5], g.z, __fma_rn(s.c[4], g.y, __fma_rn(s.c[2], g.x, y.z)));
}
// y += A g for the antisymmetric A with the entries a = (01, 02, 12)
__device__ __forceinline__ void asym_add(const V3 &a, const V3 &g, V3 &y) {
    y.x = __fma_rn(a.y, g.z, __fma_rn(a.x, g.y, y.x));
    y.y = __fma_rn(a.z, g.z, __fma_rn(-a.x, g.x, y.y));
    y.z = __fma_rn(-a.z, g.y, __fma_rn(-a.y, g.x, y.z));
}

__device__ __forceinline__ Sym load_sym(const double *__restrict__ row) {
    const double2 *r = reinterpret_cast<const double2 *>(row);
    const double2 p = __ldg(r), q = __ldg(r + 1), t = __ldg(r + 2);
    return {{p.x, p.y, q.x, q.y, t.x, t.y}};
}
// the antisymmetric entries of a pair row, for the local order of its nodes
__device__ __forceinline__ V3 load_asym(const double *__restrict__ row, bool flip) {
    const double2 *r = reinterpret_cast<const double2 *>(row);
    const double2 p = __ldg(r + 3), q = __ldg(r + 4);
    return flip ? V3{-p.x, -p.y, -q.x} : V3{p.x, p.y, q.x};
}

// One thread per active tetrahedron (inactive ones were zeroed beforehand).
__global__ void __launch_bounds__(128, 3)
k_adjoint(const double4_32a *__restrict__ X, const int4 *__restrict__ tets,
          const double2 *__restrict__ mat, const int32_t *__restrict__ list,
          const unsigned long long *__restrict__ count, const int32_t *__restrict__ tunit,
          const uint8_t *__restrict__ steep, const double *__restrict__ gu, double *__restrict__ dE, double *__restrict__ dnu,
          double *__restrict__ dXe) {
    const int64_t n = (int64_t)*count;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = list[i];
        int4 q = tets[t];
        const double2 em = mat[t];
        int32_t unit[10];  // slots 0..3 diagonal, 4..9 pairs (01) (02) (03) (12) (13) (23)
        {
            const int2 *tu = reinterpret_cast<const int2 *>(tunit + 10 * t);
#pragma unroll
            for (int h = 0; h < 5; ++h) {
                const int2 v = __ldg(tu + h);
                unit[2 * h] = v.x;
                unit[2 * h + 1] = v.y;
            }
        }
        // node k in the place of k ^ z, z the node to eliminate: an even permutation
        const int z = __ldg(steep + t);
        const bool z1 = z & 1, z2 = z & 2;
        swap_if(z1, q.x, q.y);
        swap_if(z1, q.z, q.w);
        swap_if(z1, unit[0], unit[1]);
        swap_if(z1, unit[2], unit[3]);
        swap_if(z1, unit[5], unit[8]);
        swap_if(z1, unit[6], unit[7]);
        swap_if(z2, q.x, q.z);
        swap_if(z2, q.y, q.w);
        swap_if(z2, unit[0], unit[2]);
        swap_if(z2, unit[1], unit[3]);
        swap_if(z2, unit[4], unit[9]);
        swap_if(z2, unit[6], unit[7]);
        const double *row[10];
#pragma unroll
        for (int h = 0; h < 10; ++h) row[h] = gu + GU * (int64_t)unit[h];
        const double4_32a x0 = X[q.x];
        const V3 d1 = diff(X[q.y], x0), d2 = diff(X[q.z], x0), d3 = diff(X[q.w], x0);
        const V3 c1 = cross(d2, d3), c2 = cross(d3, d1), c3 = cross(d1, d2);
        const double det = __fma_rn(d1.z, c1.z, __fma_rn(d1.y, c1.y, d1.x * c1.x));
        const double r = 1.0 / det;
        const V3 g[3] = {scaled(c1, r), scaled(c2, r), scaled(c3, r)};  // of nodes 1, 2, 3
        // u, v, w: gradients of FS, FA, FT with respect to g_1, g_2, g_3
        V3 u[3] = {}, v[3] = {}, w[3] = {};
        {
            // R_a = S_0a - S_00;  S'_aa = S_aa - R_a;  S'_ab = S_ab - R_a - R_b;
            // A'_ab = A_ab + A_0a - A_0b
            const Sym s00 = load_sym(row[0]);  // 2 S_00
            Sym R[3];
            V3 A0[3];
            const int gid[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                R[a] = load_sym(row[4 + a]);
                A0[a] = load_asym(row[4 + a], gid[0] > gid[a + 1]);
#pragma unroll
                for (int k = 0; k < 6; ++k) R[a].c[k] = __fma_rn(-0.5, s00.c[k], R[a].c[k]);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                Sym d = load_sym(row[1 + a]);  // 2 S_aa
#pragma unroll
                for (int k = 0; k < 6; ++k) d.c[k] = __fma_rn(-2.0, R[a].c[k], d.c[k]);
                sym_add(d, g[a], u[a]);
                axpy(tr(d), g[a], w[a]);
#pragma unroll
                for (int b = a + 1; b < 3; ++b) {
                    const double *p = row[6 + a + b];  // (1,2) 7, (1,3) 8, (2,3) 9
                    Sym s = load_sym(p);
                    V3 as = load_asym(p, gid[a + 1] > gid[b + 1]);
#pragma unroll
                    for (int k = 0; k < 6; ++k) s.c[k] = (s.c[k] - R[a].c[k]) - R[b].c[k];
                    as = {(as.x + A0[a].x) - A0[b].x, (as.y + A0[a].y) - A0[b].y,
                          (as.z + A0[a].z) - A0[b].z};
                    sym_add(s, g[b], u[a]);
                    sym_add(s, g[a], u[b]);
                    asym_add(as, g[b], v[a]);
                    asym_add({-as.x, -as.y, -as.z}, g[a], v[b]);
                    const double ts = tr(s);
                    axpy(ts, g[b], w[a]);
                    axpy(ts, g[a], w[b]);
                }
            }
        }
        double fs = 0.0, fa = 0.0, ft = 0.0;  // twice the forms
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            fs = dot_add(g[a], u[a], fs);
            fa = dot_add(g[a], v[a], fa);
            ft = dot_add(g[a], w[a], ft);
        }
        const double E = em.x, nu = em.y, onu = 1.0 + nu, omn = 1.0 - (nu + nu);
        const double inv = 1.0 / (onu * omn), ionu = 1.0 / onu;
        const double lamE = nu * inv, muE = 0.5 * ionu, lam = E * lamE, mu = E * muE;
        const double V = det * (1.0 / 6.0), hV = 0.5 * V;
        const double SA = fs + fa, SB = (fs - fa) + ft;  // twice
        dE[t] = hV * __fma_rn(lamE, SA, muE * SB);
        dnu[t] = hV * __fma_rn(E * __fma_rn(nu + nu, nu, 1.0) * (inv * inv), SA, -(mu * ionu) * SB);
        const double VS = hV * __fma_rn(lam, SA, mu * SB);
        const double ks = V * (lam + mu), ka = V * (lam - mu), kt = V * mu;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            u[a] = scaled(u[a], ks);
            axpy(ka, v[a], u[a]);
            axpy(kt, w[a], u[a]);
        }
        V3 o[4];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o[c + 1] = scaled(g[c], VS);
#pragma unroll
            for (int a = 0; a < 3; ++a) axpy(-dot_add(u[a], g[c], 0.0), g[a], o[c + 1]);
        }
        o[0] = {-((o[1].x + o[2].x) + o[3].x), -((o[1].y + o[2].y) + o[3].y),
                -((o[1].z + o[2].z) + o[3].z)};
        swap_if(z1, o[0], o[1]);
        swap_if(z1, o[2], o[3]);
        swap_if(z2, o[0], o[2]);
        swap_if(z2, o[1], o[3]);
        double2 *out = reinterpret_cast<double2 *>(dXe + 12 * t);
        out[0] = make_double2(o[0].x, o[0].y);
        out[1] = make_double2(o[0].z, o[1].x);
        out[2] = make_double2(o[1].y, o[1].z);
        out[3] = make_double2(o[2].x, o[2].y);
        out[4] = make_double2(o[2].z, o[3].x);
        out[5] = make_double2(o[3].y, o[3].z);
    }
}

// Offset in dXe of every (node, incident tetrahedron) pair's gradient, once per context.
__global__ void k_node_runs(const int32_t *__restrict__ nt_ptr, const int32_t *__restrict__ nt_list,
                            const int4 *__restrict__ tets, int64_t n, int32_t *__restrict__ run) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x)
        for (int32_t e = nt_ptr[v]; e < nt_ptr[v + 1]; ++e) {
            const int4 q = tets[nt_list[e]];
            run[e] = 12 * nt_list[e] + (q.x == v ? 0 : (q.y == v ? 3 : (q.z == v ? 6 : 9)));
        }
}

// dL/dX of each node: fold over its incident tetrahedra in ascending id (deterministic).  One
// thread per component, four loads in flight each, at offsets formed once (a thread per node that
// looked each one up in the tetrahedron: 28 us for 384,000 tetrahedra, this 16 us).
__global__ void k_node_grad(const int32_t *__restrict__ nt_ptr, const int32_t *__restrict__ run,
                            const double *__restrict__ dXe, int64_t n, double *__restrict__ dX) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 3 * n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = i / 3;
        const double *p = dXe + (i - 3 * v);
        const int32_t e1 = nt_ptr[v + 1];
        int32_t e = nt_ptr[v];
        double s = 0.0;
        for (; e + 4 <= e1; e += 4) {
            double d[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) d[k] = __ldg(p + __ldg(run + e + k));
#pragma unroll
            for (int k = 0; k < 4; ++k) s += d[k];
        }
        for (; e < e1; ++e) s += __ldg(p + __ldg(run + e));
        dX[i] = s;
    }
}

int64_t capped(int64_t items, int threads, int64_t most) {
    const int64_t g = (items + threads - 1) / threads;
    return g < 1 ? 1 : (g > most ? most : g);
}

}  // namespace

int launch_adjoint(Ctx *c, const double *gval, double *dE, double *dnu, double *dX,
                   cudaStream_t s) {
    if (!c->dXe) {
        double *buf = nullptr;  // dXe, the units' gradients, the runs: one allocation
        STA_TRY(dev_alloc(c, &buf, 12 * c->T + GU * c->nunits + 2 * c->T));
        c->gunit = buf + 12 * c->T;
        c->nt_run = reinterpret_cast<int32_t *>(c->gunit + GU * c->nunits);
        if (c->n > 0)
            k_node_runs<<<(unsigned)capped(c->n, 256, c->num_sms * 16), 256, 0, s>>>(
                c->nt_ptr, c->nt_list, c->tets, c->n, c->nt_run);
        STA_CUDA_TRY(cudaGetLastError());
        c->dXe = buf;
    }
    if (c->T > 0) {
        STA_TRY(launch_active_list(c, dE, dnu, c->dXe, s));
        k_grad_units<<<(unsigned)capped(c->nunits, 256, c->num_sms * 8), 256, 0, s>>>(
            c->nunits, c->bmeta, c->bmirror, gval, c->gunit);
        k_adjoint<<<(unsigned)capped(c->T, 128, c->num_sms * 3), 128, 0, s>>>(
            c->X, c->tets, c->mat, c->act_list, c->act_count, c->tunit, c->steep, c->gunit, dE, dnu, c->dXe);
    }
    if (c->n > 0)
        k_node_grad<<<(unsigned)capped(3 * c->n, 256, c->num_sms * 8), 256, 0, s>>>(
            c->nt_ptr, c->nt_run, c->dXe, c->n, dX);
    STA_CUDA_TRY(cudaGetLastError());
    return STA_OK;
}

}  // namespace sta
