// Host build of the reduced-range integer-pipe functions of the flux kernels
// (emu64.cuh), loaded by tests/test_emu64_mid_host.py through ctypes.
// EMU_RCP_ERROR shifts the 24-bit start of the reciprocal by some units.
#include "emu64.cuh"

extern "C" {

// m = a*b, r = 1/a, h = ab/(a+b), q = sqrt(a), p = a+b elementwise with their range flags (bits 0 to 4)
void emu64_mid_host(const double* a, const double* b, double* m, double* r, double* h, double* q, double* p,
                    unsigned char* ok, long long n) {
    for (long long i = 0; i < n; ++i) {
        bool o0 = true, o1 = true, o2 = true, o3 = true, o4 = true;
        m[i] = jfnk::emu::mul_mid(a[i], b[i], o0);
        r[i] = jfnk::emu::recip_mid(a[i], o1);
        h[i] = jfnk::emu::harm_mid(a[i], b[i], o2);
        q[i] = jfnk::emu::sqrt_mid(a[i], o3);
        p[i] = jfnk::emu::add_mid(a[i], b[i], o4);
        ok[i] = (unsigned char)(o0 + 2 * o1 + 4 * o2 + 8 * o3 + 16 * o4);
    }
}
}
