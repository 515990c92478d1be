// FP32 sums that are not less accurate for being long.
//
// The dot products of the solve are sums of FP32 products, handed over to FP64 once per
// warp or lane group.  Before that, the products of a thread's layers are added as a tree
// (log2 of their number in depth), and what a thread adds up one after the other carries
// its rounding errors beside it (Knuth's exact two-term sum), so its length costs nothing.
// FP64 in a thread would do the same at 16 cycles of the pipe per warp and addition.
#pragma once

struct Sum2 {
  float s, e;  // sum, and the rounding errors of its additions
};

__host__ __device__ __forceinline__ void sum2_add(Sum2& a, float v) {
  const float t = a.s + v, b = t - a.s;
  a.e += (a.s - (t - b)) + (v - b);
  a.s = t;
}

__host__ __device__ __forceinline__ void sum2_add(Sum2& a, const Sum2& o) {
  sum2_add(a, o.s);
  a.e += o.e;
}

// (an overflow or a NaN stays what it is in s; e is a NaN then)
__host__ __device__ __forceinline__ double sum2_value(const Sum2& a) {
  return a.e - a.e == 0.f ? (double)a.s + (double)a.e : (double)a.s;
}

// t[0] + ... + t[N - 1], in t[0], as a tree
template <int N, typename T, typename F>
__host__ __device__ __forceinline__ void tree_sum(T (&t)[N], F add) {
#pragma unroll
  for (int w = 1; w < N; w *= 2)
#pragma unroll
    for (int k = 0; k + w < N; k += 2 * w) t[k] = add(t[k], t[k + w]);
}

// additions on the way of a term through tree_sum of n
__host__ __device__ constexpr int tree_depth(int n) { return n <= 1 ? 0 : 1 + tree_depth((n + 1) / 2); }
