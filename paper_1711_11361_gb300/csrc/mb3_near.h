// mb3_near.h -- the positions along a line whose update reads body data
// (plain C++ too, so that the split can be enumerated on the CPU)
#pragma once
#ifdef __CUDACC__
#define MB3_HD __host__ __device__ __forceinline__
#else
#define MB3_HD inline
#endif

namespace mb3 {

// positions a .. a + len - 1 (modulo a periodic line)
struct Near { int a, len; bool wrap; };

// a line of nal cells whose body region is r0 .. r0 + rn - 1: from two cells
// before it to two after its last face
MB3_HD Near near_span(int r0, int rn, int nal, bool periodic) {
    Near N;
    N.a = r0 - 2;
    N.len = rn > 0 ? rn + 5 : 0;
    N.wrap = periodic;
    if (periodic) {
        // the whole line: from its first cell on, which near_pos needs on a
        // line of one cell (two periods lie between r0 - 2 and r0 there)
        if (N.len >= nal) {
            N.a = 0;
            N.len = nal;
        }
    } else {
        const int e = N.a + N.len < nal ? N.a + N.len : nal;
        if (N.a < 0) N.a = 0;
        N.len = e > N.a ? e - N.a : 0;
    }
    return N;
}
// position m of the line, 0 <= m < nal (r0 lies on the line, so at most one
// period lies between m and N.a)
MB3_HD bool near_pos(const Near &N, int m, int nal) {
    int r = m - N.a;
    if (N.wrap) r += r >= nal ? -nal : r < 0 ? nal : 0;
    return r >= 0 && r < N.len;
}

}  // namespace mb3
