// Double-floats in packed pairs (tt_df.cuh) against the same operations one at a time,
// bit for bit: the stage sums of step_ray_df on random numbers, and the tabulated
// metric's flow on random states.
// Argument: a table's patch coefficients (tartarus_table_coefficients, raw doubles),
// its nr and nth, r_min, r_max.
// Prints: name, evaluations, evaluations that differ.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "tt_df.cuh"

using namespace tt;

struct Rng {
    unsigned long long s;
    __device__ double uniform(double lo, double hi) {
        unsigned long long z = (s += 0x9E3779B97F4A7C15ull);
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return lo + (hi - lo) * ((double)((z ^ (z >> 31)) >> 11) * 0x1p-53);
    }
    // a double-float of any sign over 12 binary orders, at times zero
    __device__ DF df() {
        const double m = uniform(-1.0, 1.0);
        return uniform(0.0, 1.0) < 0.02 ? DF{0.0f, 0.0f} : df_of(m * exp2(uniform(-6.0, 6.0)));
    }
};

__device__ bool same(float a, float b) { return __float_as_uint(a) == __float_as_uint(b) || (a != a && b != b); }
__device__ bool same(DF a, DF b) { return same(a.hi, b.hi) && same(a.lo, b.lo); }

__global__ void k_sums(int n, unsigned* out) {
    Rng g{(blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 77777ull + 9};
    for (int i = 0; i < n; ++i) {
        DF c[6], x[6], z[6];
        for (int k = 0; k < 6; ++k) {
            c[k] = g.df();
            x[k] = g.df();
            z[k] = g.df();
        }
        const DF y = g.df(), v = g.df();
        const float h = (float)g.uniform(0.01, 30.0);
        // the sums of 1 to 6 flows, and what a step makes of them
        DotAcc a = dot_first(c[0], x[0]), b = dot_first(c[0], z[0]);
        DotAcc2 p = dot_first(df2(c[0]), df2(x[0], z[0]));
        bool ok = true;
        for (int k = 1; k < 6; ++k) {
            const DF ea = dot_end(a), eb = dot_end(b);
            const DF2 ep = dot_end(p);
            const DF sa = df_add(y, df_mul_f(ea, h)), sb = df_add(v, df_mul_f(eb, h));
            const DF2 sp = df_add(df2(y, v), df_mul_f(ep, f2_pack(h, h)));
            const f32x2 err = f2_mul(f2_pack(h, h), ep.hi);
            ok = ok && same(ea, ep.x()) && same(eb, ep.y()) && same(sa, sp.x()) && same(sb, sp.y()) &&
                 same(__fmul_rn(h, ea.hi), f2_x(err)) && same(__fmul_rn(h, eb.hi), f2_y(err));
            a = dot_next(a, c[k], x[k]);
            b = dot_next(b, c[k], z[k]);
            p = dot_next(p, df2(c[k]), df2(x[k], z[k]));
        }
        const DF2 m = df_add(df2(y, v), df_mul_f(df_mul(df2(x[0], z[0]), df2(c[0])), f2_pack(h, h)));
        ok = ok && same(df_add(y, df_mul_f(df_mul(x[0], c[0]), h)), m.x()) &&
             same(df_add(v, df_mul_f(df_mul(z[0], c[0]), h)), m.y());
        atomicAdd(out, 1u);
        if (!ok) atomicAdd(out + 1, 1u);
    }
}

// table_flow_df and table_fields_df one double-float at a time
__device__ void flow_scalar(const ImageDesc& d, const RayDF& R, const StateDF& y, StateDF& f, DF& H) {
    DF F[5], Fr[5], Ft[5];
    const DF idu = DF{d.idu_df.x, d.idu_df.y}, idth = DF{d.idth_df.x, d.idth_df.y};
    const DF tu = df_mul(df_sub(df_log(y.r), DF{d.u0_df.x, d.u0_df.y}), idu), tw = df_mul(y.th, idth);
    const int k = df_cell(tu, d.nr - 2), j = df_cell(tw, d.nth - 2);
    const DF t = df_add_f(tu, -(float)k), w = df_add_f(tw, -(float)j);
    const float2* cell = d.table_df + ((size_t)j * (d.nr - 1) + k) * kTableCoef;
    const DF inv_dur = df_mul(idu, df_rcp(y.r));
    for (int fi = 0; fi < 5; ++fi) {
        const float2* c = cell + 16 * fi;
        DF P[4], Q[4], v, vt;
        for (int i = 0; i < 4; ++i)
            horner_d_df(DF{c[4 * i].x, c[4 * i].y}, DF{c[4 * i + 1].x, c[4 * i + 1].y}, DF{c[4 * i + 2].x, c[4 * i + 2].y},
                        DF{c[4 * i + 3].x, c[4 * i + 3].y}, w, P[i], Q[i]);
        horner_d_df(P[0], P[1], P[2], P[3], t, v, vt);
        const DF vw = df_fma_lazy(df_fma_lazy(df_fma_lazy(Q[3], t, Q[2]), t, Q[1]), t, Q[0]);
        F[fi] = df_norm(v);
        Fr[fi] = df_mul(df_norm(vt), inv_dur);
        Ft[fi] = df_mul(df_norm(vw), idth);
    }
    const DF D = df_sub(df_mul(F[0], F[3]), df_sqr(F[1])), iD = df_rcp(D);
    const DF W = dot_end(dot_next(dot_next(dot_first(F[3], R.ptsq), df_neg(F[1]), R.ptp), F[0], R.pph2));
    const DF WiD = df_mul(W, iD), ith = df_rcp(F[2]), pr2 = df_sqr(y.pr), pthi = df_mul(y.pth, ith);
    const DF H2 = df_add(WiD, df_fma(F[4], pr2, df_mul(y.pth, pthi)));
    H = DF{0.5f * H2.hi, 0.5f * H2.lo};
    const DF pthi2 = df_sqr(pthi);
    auto d2H = [&](const DF* G) {
        const DF dW = dot_end(dot_next(dot_next(dot_first(G[3], R.ptsq), df_neg(G[1]), R.ptp), G[0], R.pph2));
        const DF dD = dot_end(dot_next(dot_next(dot_first(G[0], F[3]), F[0], G[3]),
                                       DF{-2.0f * F[1].hi, -2.0f * F[1].lo}, G[1]));
        const DF s = df_add(df_mul(df_sub(dW, df_mul(WiD, dD)), iD), df_sub(df_mul(G[4], pr2), df_mul(G[2], pthi2)));
        return DF{-0.5f * s.hi, -0.5f * s.lo};
    };
    f = StateDF{df_mul(F[4], y.pr), pthi, d2H(Fr), d2H(Ft)};
}

__global__ void __launch_bounds__(kDfBlock) k_flow(int n, const __grid_constant__ ImageDesc d, unsigned* out) {
    df_sincos_table(s_df_tab);
    df_log_table(s_df_ln);
    __syncthreads();
    Rng g{(blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) * 55555ull + 1};
    for (int i = 0; i < n; ++i) {
        // (a few outside the table in r or theta: cells are clamped)
        const RayDF R = make_ray_df(make_ray_const(d.a, g.uniform(-1.1, -0.9), (i & 7) ? g.uniform(-20.0, 20.0) : 0.0));
        const StateDF y{df_of(exp(g.uniform(0.3, 7.2))), df_of(g.uniform(-0.1, 3.3)), df_of(g.uniform(-2.0, 2.0)),
                        df_of((i & 15) ? g.uniform(-10.0, 10.0) : 0.0)};
        StateDF f;
        DF H;
        flow_scalar(d, R, y, f, H);
        const FlowDF2 o = table_flow_df_call(&d, R, pairs(y));
        const StateDF q = halves(o.f);
        atomicAdd(out, 1u);
        if (!(same(f.r, q.r) && same(f.th, q.th) && same(f.pr, q.pr) && same(f.pth, q.pth) && same(H, o.H)))
            atomicAdd(out + 1, 1u);
    }
}

static float2 split(double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
}

int main(int argc, char** argv) {
    if (argc != 6) return 2;
    ImageDesc d = {};
    d.nr = atoi(argv[2]);
    d.nth = atoi(argv[3]);
    const double r_min = atof(argv[4]), r_max = atof(argv[5]), u0 = std::log(r_min);
    d.kind = 1;
    d.M = 1.0;
    d.u0_df = split(u0);
    d.idu_df = split((d.nr - 1) / (std::log(r_max) - u0));
    d.idth_df = split((d.nth - 1) / M_PI);
    const size_t len = (size_t)(d.nr - 1) * (d.nth - 1) * kTableCoef;
    std::vector<double> coef(len);
    std::vector<float2> pairs_of(len);
    FILE* f = std::fopen(argv[1], "rb");
    if (!f || std::fread(coef.data(), sizeof(double), len, f) != len) return 3;
    std::fclose(f);
    for (size_t i = 0; i < len; ++i) pairs_of[i] = split(coef[i]);
    float2* table;
    unsigned *dev, h[2];
    if (cudaMalloc(&table, len * sizeof(float2)) != cudaSuccess || cudaMalloc(&dev, sizeof h) != cudaSuccess ||
        cudaMemcpy(table, pairs_of.data(), len * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess)
        return 4;
    d.table_df = table;
    for (int k = 0; k < 2; ++k) {
        if (cudaMemset(dev, 0, sizeof h) != cudaSuccess) return 5;
        if (k) k_flow<<<152, kDfBlock>>>(40, d, dev);
        else k_sums<<<304, 128>>>(100, dev);
        if (cudaMemcpy(h, dev, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 6;
        printf("%s %u %u\n", k ? "table_flow" : "sums", h[0], h[1]);
    }
    return 0;
}
