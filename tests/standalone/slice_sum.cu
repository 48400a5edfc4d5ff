// Standalone check of the FP64 slice sum over FP32 values on values that add exactly and on
// values that do not (zeros, wide ranges, cancellation, subnormals, infinities, NaN): equal to
// the sum formed one value after the other where that sum never rounds, else no further from
// the exact sum than the roundings allow: one per value, 2^-53 of the sum of the magnitudes
// each.  Exits 1 on a difference or error.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
#include "../../paper_2112_15083_gb300/csrc/kernels.cuh"

#define CK(x) do { cudaError_t e = (x); if (e != cudaSuccess) { printf("%s: %s\n", #x, cudaGetErrorString(e)); return 1; } } while (0)

int main() {
    const int nout = 9, nver = 3;
    std::mt19937 g(7);
    std::normal_distribution<float> nd(0.f, 1.f);
    std::uniform_int_distribution<int> e40(-40, 40), pct(0, 99);
    for (int nfree : {0, 3, 4, 6, 10}) {
        const size_t n = size_t(1) << (nout + nfree);
        std::vector<float2> x(n * nver);
        for (size_t i = 0; i < x.size(); i++) {
            const size_t o = i & 511;  // output: its kind of values
            float v[2];
            for (float &y : v) {
                y = nd(g) * 1e-4f;
                switch (o % 10) {
                    case 1: if (pct(g) < 60) y = pct(g) < 50 ? 0.f : -0.f; break;
                    case 2: y = std::ldexp(y, e40(g)); break;
                    case 3: y = (i >> nout) & 1 ? 1.5f : -1.5f; break;
                    case 4: if (pct(g) < 3) y = std::ldexp(y, -60); break;
                    case 5: y = std::ldexp(y, -130); break;
                    case 6: if (pct(g) < 1) y = pct(g) < 50 ? INFINITY : NAN; break;
                    case 7: y = std::ldexp(1.f, -(int)((i >> nout) % 50)); break;
                    case 8: y = std::ldexp(y, 120); break;
                    case 9: y = 0.f; break;
                }
            }
            x[i] = make_float2(v[0], v[1]);
        }
        float2 *dx;
        double2 *dout;
        const void **dptr;
        CK(cudaMalloc(&dx, x.size() * 8));
        CK(cudaMalloc(&dout, 16 << nout));
        CK(cudaMalloc(&dptr, nver * sizeof(void *)));
        CK(cudaMemcpy(dx, x.data(), x.size() * 8, cudaMemcpyHostToDevice));
        const void *hp[nver];
        for (int v = 0; v < nver; v++) hp[v] = dx + v * n;
        CK(cudaMemcpy(dptr, hp, sizeof(hp), cudaMemcpyHostToDevice));
        tnk::slice_sum<float2><<<2, 256>>>((const void *const *)dptr, nver, nfree, nout, dout);
        CK(cudaGetLastError());
        std::vector<double2> out(size_t(1) << nout);
        CK(cudaMemcpy(out.data(), dout, out.size() * 16, cudaMemcpyDeviceToHost));
        for (size_t o = 0; o < out.size(); o++) {
            for (int part = 0; part < 2; part++) {
                const double got = part ? out[o].y : out[o].x;
                double seq = 0, mag = 0, err = 0;  // err: the exact sum minus seq, from two-sums
                bool rounds = false;
                int terms = 0;
                for (int v = 0; v < nver; v++)
                    for (size_t f = 0; f < (size_t(1) << nfree); f++, terms++) {
                        const float2 w = x[v * n + (f << nout) + o];
                        const double y = part ? w.y : w.x, s = seq + y, b = s - seq;
                        const double e = (seq - (s - b)) + (y - b);
                        rounds |= e != 0;
                        err += e;
                        seq = s;
                        mag += std::fabs(y);
                    }
                bool same;
                if (!std::isfinite(seq)) same = std::isnan(seq) ? std::isnan(got) : got == seq;
                else if (!rounds) same = std::memcmp(&got, &seq, 8) == 0;
                else same = std::fabs((got - seq) - err) <= terms * std::ldexp(mag, -53);
                if (!same) {
                    printf("nfree %d output %zu.%d (kind %zu): %.17g, one by one %.17g\n", nfree, o, part, o % 10, got, seq);
                    return 1;
                }
            }
        }
        CK(cudaFree(dx));
        CK(cudaFree(dout));
        CK(cudaFree(dptr));
    }
    printf("ok\n");
    return 0;
}
