// Host run of the pose Log on unit quaternions of either sign (pv_math.cuh): reads
// cases as doubles from stdin, writes results as doubles.
//
//   quat_log <32|64> log      per case: q (4), t (3) -> Log (6)
//   quat_log <32|64> between  per case: xi_j (6), xi_i (6) -> Log(Exp(xi_j)^-1 Exp(xi_i)) (6)
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
static void run(bool log) {
    T a[6], b[6], q[4], t[3], r[6];
    while (log ? read(q, 4) && read(t, 3) : read(a, 6) && read(b, 6)) {
        if (log) {
            se3_log_q(q, t, r);
        } else {
            se3_exp_q(b, q, t);
            se3_between(a, q, t, r);
        }
        for (int k = 0; k < 6; ++k) {
            const double v = r[k];
            fwrite(&v, sizeof(v), 1, stdout);
        }
    }
}

int main(int argc, char** argv) {
    if (argc != 3) return 2;
    const bool log = !strcmp(argv[2], "log");
    !strcmp(argv[1], "32") ? run<float>(log) : run<double>(log);
    return 0;
}
