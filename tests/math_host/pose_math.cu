// Host check of the sweep's pose and identity-message math (pv_math.cuh), for
// float and double: reads cases as doubles from stdin, writes results as doubles.
//
//   pose_math <32|64> pose     per case: xi_j (6), xi_i (6) ->
//                              R, t of Exp(xi_i) (12), Log(Exp(xi_i)) (6),
//                              Log(Exp(xi_j)^-1 Exp(xi_i)) (6), Log(Exp(xi_i) Exp(xi_j)) (6)
//   pose_math <32|64> message  per case: W (21, packed), u (6), eta_v (6), r (6), lam (1) ->
//                              Lambda (21), eta (6), C^-1 (21), 1 if every pivot was positive
#include <cstdio>
#include <cstring>

#include "pv_math.cuh"

using namespace pv;

template <typename T>
static bool read(T* x, int n) {
    for (int k = 0; k < n; ++k) {
        double v;
        if (fread(&v, sizeof(v), 1, stdin) != 1) return false;
        x[k] = T(v);
    }
    return true;
}
template <typename T>
static void write(const T* x, int n) {
    for (int k = 0; k < n; ++k) {
        const double v = x[k];
        fwrite(&v, sizeof(v), 1, stdout);
    }
}

template <typename T>
static void poses() {
    T xj[6], xi[6], R[9], t[3], q[4], t2[3], r[6];
    while (read(xj, 6) && read(xi, 6)) {
        se3_exp(xi, R, t);
        write(R, 9);
        write(t, 3);
        se3_exp_q(xi, q, t2);
        se3_log_q(q, t2, r);
        write(r, 6);
        se3_between(xj, q, t2, r);
        write(r, 6);
        se3_update(q, t2, xj, r);
        write(r, 6);
    }
}

template <typename T>
static void messages() {
    T W[21], u[6], ev[6], r[6], lam, L[21], e[6], Ci[21];
    while (read(W, 21) && read(u, 6) && read(ev, 6) && read(r, 6) && read(&lam, 1)) {
        IdMsg<T> m;
        const T ok = identity_msg(W, u, ev, r, lam, m) ? T(1) : T(0);
        for (int a = 0; a < 6; ++a) {
            e[a] = lam * m.he[a];
            for (int b = 0; b <= a; ++b) {
                L[pidx(a, b)] = m.lambda(a, b, lam, lam * lam, T(0));
                Ci[pidx(a, b)] = m.ci(a, b);
            }
        }
        write(L, 21);
        write(e, 6);
        write(Ci, 21);
        write(&ok, 1);
    }
}

int main(int argc, char** argv) {
    if (argc != 3) return 2;
    const bool f32 = !strcmp(argv[1], "32"), pose = !strcmp(argv[2], "pose");
    if (pose)
        f32 ? poses<float>() : poses<double>();
    else
        f32 ? messages<float>() : messages<double>();
    return 0;
}
