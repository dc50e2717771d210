// rid_pair_loads.cuh -- which weight loads a CTA pair may still have in flight
// when it gives up (k_mlp_tc_pair; plain arithmetic, for host and device).
#pragma once

#ifdef __CUDACC__
#define RID_HD __host__ __device__ __forceinline__
#else
#define RID_HD inline
#endif

// Iteration `it` of the weight stream puts a part of one chunk into stage
// it % ns of either CTA.  Both parts are counted on the even CTA's barrier of
// that stage, whose phase the even CTA arms (one arrival, both parts' bytes)
// when it issues its own part; neither CTA issues an iteration before both
// parts of iteration it - ns have been consumed.
struct PairStageLoads {
    int it;            // the last iteration that put anything into the stage, -1: none
    bool even, odd;    // the parts of it that have been issued
};
// even, odd: iterations whose part that CTA has issued.
RID_HD PairStageLoads pair_stage_loads(int even, int odd, int ns, int s) {
    const int a = even > s ? s + (even - 1 - s) / ns * ns : -1;
    const int b = odd > s ? s + (odd - 1 - s) / ns * ns : -1;
    const int it = a > b ? a : b;
    return PairStageLoads{it, it >= 0 && a == it, it >= 0 && b == it};
}
