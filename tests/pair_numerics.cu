// The arithmetic helpers of the pair sums over arrays, for
// test_gpu_pair_helpers.py, which compiles this file against the library's
// headers.  Each entry returns the CUDA error code.
#include <cmath>

#include "kernels.cuh"

using namespace sph;

template <class F>
__global__ void k_each(int n, F f) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) f(i);
}
template <class F>
static int each(int n, F f) {
    k_each<<<(n + 255) / 256, 256>>>(n, f);
    return (int)cudaDeviceSynchronize();
}

// Separations of one axis pair by the rule on integers, and by the library.
__device__ static float sep_rule(const Anchor &an, int ax, int ki, int kj, float xi, float xj) {
    int k = ki - kj;
    if (an.periodic[ax]) {
        if (2 * k > an.n[ax]) k -= an.n[ax];
        else if (2 * k < -an.n[ax]) k += an.n[ax];
    }
    return fmaf((float)k, an.A[ax], xi - xj);
}

extern "C" {

int num_frcp(int n, const double *x, double *o) {
    return each(n, [=] __device__(int i) { o[i] = frcp(x[i]); });
}
int num_frsqrt(int n, const double *x, double *o) {
    return each(n, [=] __device__(int i) { o[i] = frsqrt_lean(x[i]); });
}
int num_is_normal(int n, const double *x, int *o) {
    return each(n, [=] __device__(int i) { o[i] = is_normal(x[i]) ? 1 : 0; });
}
int num_qs(int n, const double *q, double *w, double *s) {
    return each(n, [=] __device__(int i) {
        double t;
        qs_ws(q[i], w[i], t);
        s[i] = qs_s(q[i]);
        if (s[i] != t) w[i] = NAN;   // one derivative, by either call
    });
}
// o: by the helper, ref: by the conversion instruction
int num_d2f(int n, const double *x, float *o, float *ref) {
    return each(n, [=] __device__(int i) { o[i] = d2f(x[i]); ref[i] = __double2float_rn(x[i]); });
}
int num_d2f_up(int n, const double *x, float *o, float *ref) {
    return each(n, [=] __device__(int i) { o[i] = d2f_up(x[i]); ref[i] = __double2float_ru(x[i]); });
}
int num_f2d(int n, const float *x, double *o, double *ref) {
    return each(n, [=] __device__(int i) { o[i] = f2d(x[i]); ref[i] = (double)x[i]; });
}
int num_u2d(int n, const uint32_t *x, double *o, double *ref) {
    return each(n, [=] __device__(int i) { o[i] = u2d(x[i]); ref[i] = (double)x[i]; });
}
// a, b: records; out: dx, dy of the rule, of anchor_sep, of Sep2, six a pair
int num_sep(int n, const float4 *a, const float4 *b, double Ax, double Ay, int nx, int ny, int px,
            int py, float *out) {
    Anchor an;
    set_anchor_axis(an, 0, Ax, nx, px != 0);
    set_anchor_axis(an, 1, Ay, ny, py != 0);
    return each(n, [=] __device__(int i) {
        const float4 p = a[i], q = b[i];
        const unsigned gp = __float_as_uint(p.w), gq = __float_as_uint(q.w);
        float *o = out + 6 * (size_t)i;
        o[0] = sep_rule(an, 0, gp & 0xffffu, gq & 0xffffu, p.x, q.x);
        o[1] = sep_rule(an, 1, gp >> 16, gq >> 16, p.y, q.y);
        anchor_sep(an, p, q, o[2], o[3]);
        const F2 d = Sep2(an, p).get(q);
        o[4] = lo(d);
        o[5] = hi(d);
    });
}
}
