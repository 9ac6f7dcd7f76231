// Arithmetic on cell pairs for the step kernels, which are bound by the issue and latency of few
// warps: a packed Laplacian takes about half the instructions.  3D gradient of two shots of
// 150 x 131 x 187 21.75 -> 20.72 ms, DTFT at 400^3 37.5 -> 36.3; 2D saddle gradient of 16 shots of
// 801 x 241 10.34 -> 9.71 ms, forward 10.96 -> 10.58.  Same bits: the sums keep the order and the
// contractions of the scalar code, fma(2 w0, u, w1 s1) first.
#pragma once

namespace esi {
namespace {

// FP32 has packed instructions with the rounding of the scalar ones (a
// pair per issue slot), FP64 goes cell by cell.
template <typename T>
struct Pk;
template <>
struct Pk<float> {
    using t = unsigned long long;
    static constexpr int n = 2;
    static __device__ __forceinline__ t pack(const float *v) {
        t r;
        asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v[0]), "f"(v[1]));
        return r;
    }
    static __device__ __forceinline__ void unpack(t a, float *v) {
        asm("mov.b64 {%0, %1}, %2;" : "=f"(v[0]), "=f"(v[1]) : "l"(a));
    }
    static __device__ __forceinline__ t dup(float a) {
        const float v[2] = {a, a};
        return pack(v);
    }
    static __device__ __forceinline__ t add(t a, t b) {
        t r;
        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
        return r;
    }
    static __device__ __forceinline__ t mul(t a, t b) {
        t r;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
        return r;
    }
    static __device__ __forceinline__ t fma(t a, t b, t c) {
        t r;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
        return r;
    }
    // a - b: the product with -1 is exact
    static __device__ __forceinline__ t sub(t a, t b) { return fma(b, dup(-1.0f), a); }
};
template <>
struct Pk<double> {
    using t = double;
    static constexpr int n = 1;
    static __device__ __forceinline__ t pack(const double *v) { return *v; }
    static __device__ __forceinline__ void unpack(t a, double *v) { *v = a; }
    static __device__ __forceinline__ t dup(double a) { return a; }
    static __device__ __forceinline__ t add(t a, t b) { return a + b; }
    static __device__ __forceinline__ t mul(t a, t b) { return a * b; }
    static __device__ __forceinline__ t fma(t a, t b, t c) { return ::fma(a, b, c); }
    static __device__ __forceinline__ t sub(t a, t b) { return a - b; }
};
// the same, cell by cell
struct PkCell {
    using t = float;
    static constexpr int n = 1;
    static __device__ __forceinline__ t pack(const float *v) { return *v; }
    static __device__ __forceinline__ void unpack(t a, float *v) { *v = a; }
    static __device__ __forceinline__ t dup(float a) { return a; }
    static __device__ __forceinline__ t add(t a, t b) { return a + b; }
    static __device__ __forceinline__ t mul(t a, t b) { return a * b; }
    static __device__ __forceinline__ t fma(t a, t b, t c) { return fmaf(a, b, c); }
};
// the 16 bytes of a row segment
template <typename T, typename P = Pk<T>>
struct alignas(16) Seg {
    static constexpr int n = 16 / (int)sizeof(T) / P::n;
    typename P::t v[n];
};
template <typename T, typename P = Pk<T>>
__device__ __forceinline__ Seg<T, P> ldp(const T *p) {
    return *reinterpret_cast<const Seg<T, P> *>(p);
}

}  // namespace
}  // namespace esi
