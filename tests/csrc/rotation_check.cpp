// Compares the fixed-point rotational update (rotation.cuh) with the FP64
// update it stands for, increment by increment: argv = dt kT torque count.
// Prints, per part, the lipids that were left to FP64 and the differing
// increments among the others.
#define ORBC_HD
#include "rotation.cuh"

#include <cstdio>
#include <cstdlib>
#include <random>

using namespace orbc;

int main(int argc, char** argv) {
    if (argc < 5) return 2;
    const double dt = atof(argv[1]), kT = atof(argv[2]), torque = atof(argv[3]);
    const long count = atol(argv[4]);
    const double h = 0.5 * dt, cr = std::exp(-dt), crm1 = std::expm1(-dt);
    const double srn = std::ldexp(std::sqrt((1.0 - cr * cr) * kT), 40) * (3.4641016151377544 * 1.16415321826934814453125e-10);
    const double ca = std::ldexp(0.5 * h, -40), hi8 = std::ldexp(h, 8), u80 = 8.271806125530277e-25;
    const RotK K = rot_constants(0.5 * h, h, crm1, srn);
    std::mt19937_64 g(12345);
    std::normal_distribution<double> nd;
    long left[4] = {0, 0, 0, 0}, differ[4] = {0, 0, 0, 0};
    for (long t = 0; t < count; t++) {
        double n[3], w[3], r = 0, wn = 0;
        long long nq[3], wq[3], Tq[3];
        unsigned zw[3];
        for (double& x : n) { x = nd(g); r += x * x; }
        for (int a = 0; a < 3; a++) { n[a] /= std::sqrt(r); w[a] = std::sqrt(kT) * nd(g); wn += n[a] * w[a]; }
        for (int a = 0; a < 3; a++) {
            nq[a] = llrint(std::ldexp(n[a], 40));
            wq[a] = llrint(std::ldexp(w[a] - wn * n[a], 40));
            Tq[a] = llrint(std::ldexp(torque * nd(g), 32));
            zw[a] = (unsigned)g();
        }
        const Dir d = dir_of(nq);
        const double N[3] = {(double)nq[0], (double)nq[1], (double)nq[2]};
        const double W[3] = {(double)wq[0], (double)wq[1], (double)wq[2]};
        long long want[4][3], got[4][3];
        // kick
        const double T[3] = {(double)Tq[0], (double)Tq[1], (double)Tq[2]};
        const double ut = (T[0] * N[0] + T[1] * N[1] + T[2] * N[2]) * u80;
        for (int a = 0; a < 3; a++) want[0][a] = wq[a] + llrint(hi8 * (T[a] - ut * N[a]));
        // turn
        const double q[3] = {ca * W[0], ca * W[1], ca * W[2]};
        const double aa = q[0] * q[0] + q[1] * q[1] + q[2] * q[2];
        const double k = aa <= 6.103515625e-05 ? std::fma(aa, std::fma(aa, std::fma(-2.0, aa, 2.0), -2.0), 2.0) : 2.0 / (1.0 + aa);
        for (int a = 0; a < 3; a++) {
            const int u = (a + 1) % 3, v = (a + 2) % 3;
            want[1][a] = nq[a] + llrint(k * std::fma(-aa, N[a], q[u] * N[v] - q[v] * N[u]));
        }
        // noise
        double z[3];
        for (int a = 0; a < 3; a++) z[a] = srn * (double)(2 * (long long)(int)(zw[a] ^ 0x80000000u) + 1);
        const double uz = (z[0] * N[0] + z[1] * N[1] + z[2] * N[2]) * u80;
        for (int a = 0; a < 3; a++) want[2][a] = wq[a] + llrint(std::fma(crm1, W[a], z[a] - uz * N[a]));
        // renormalisation of a director off unit length by up to 1e-9 (1e-6 now and then)
        const long long off = t % 64 ? 1000 : 1000000;
        __int128 e = -((__int128)1 << 80);
        for (int a = 0; a < 3; a++) {
            got[3][a] = nq[a] + (long long)(g() % (2 * off + 1)) - off;
            e += (__int128)got[3][a] * got[3][a];
        }
        const double hd = (double)(long long)e * 4.1359030627651384e-25;
        for (int a = 0; a < 3; a++) want[3][a] = got[3][a] - llrint((double)got[3][a] * hd);
        for (int a = 0; a < 3; a++) { got[0][a] = got[2][a] = wq[a]; got[1][a] = nq[a]; }
        const bool ok[4] = {K.ok && rot_kick(got[0], d, Tq, K, 1), K.ok && rot_turn(got[1], d, wq, K),
                            K.ok && rot_noise(got[2], d, zw, K), rot_renorm(got[3])};
        for (int c = 0; c < 4; c++) {
            left[c] += !ok[c];
            for (int a = 0; a < 3 && ok[c]; a++) differ[c] += got[c][a] != want[c][a];
        }
    }
    for (int c = 0; c < 4; c++) printf("%ld %ld\n", left[c], differ[c]);
    return 0;
}
