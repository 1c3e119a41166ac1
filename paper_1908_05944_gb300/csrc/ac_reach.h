// How far a line of equal power reaches inside the grown balls, and whether it
// gets there at all (AC3), from one directed difference. A is the directed
// arithmetic of the precision (ac_local.cu's Ar; the host test has its own).
#pragma once

#if defined(__CUDACC__)
#define AC_REACH_FN __device__ __forceinline__
#else
#define AC_REACH_FN inline
#endif

namespace ac {

template <class R>
struct Reach {
    R lo, up;  // bounds of T - |y|^2, the squared reach: 0 <= lo <= up
    int ac3;   // AC3, |y|^2 <= T: +1 holds, -1 fails, 0 undecided
};

// From S = fl(|y~|^2), |S - |y|^2| <= eS, and T. The sign and the bounds are one
// question and must have one answer: an undecided line has lo = 0, so that no
// simplex over it is taken as decided (k_local leaves those to the exact kernels,
// and nothing else would test them). S + eS < T rounded by itself is not that
// answer: above 2^23 FP32 values are whole numbers, and a triangle whose S + eS
// lies between T - 1 and T was undecided with lo > 0; its tetrahedra were lost.
template <class A, class R>
AC_REACH_FN Reach<R> reach_of(R T, R S, R eS) {
    Reach<R> r;
    const R lo = A::sub_dn(A::sub_dn(T, S), eS), up = A::add_up(A::add_up(T, -S), eS);
    r.ac3 = lo > R(0) ? 1 : up < R(0) ? -1 : 0;
    r.lo = A::max(lo, R(0));
    r.up = A::max(up, R(0));
    return r;
}

}  // namespace ac
