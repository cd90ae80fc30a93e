// Reciprocals of densities and radii.
#pragma once

// 1 / x of a density: the hardware reciprocal alone.  __fdividef(1, x) has the
// same bits for every normal x whose reciprocal is normal, but wraps the
// reciprocal in a rescaling for the others (five more instructions each).
__device__ __forceinline__ float rcp1(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// In FP64 the hardware's approximation (some 3e-7 off) and two Newton iterations
// x (1 + e), e = 1 - r x: the second starts 1e-13 off and leaves 1e-26, so that
// the result is the correctly rounded 1 / r (all of 800,000 densities and radii
// tested).  Four FP64 instructions.  One cubic iteration, x (1 + e + e^2), takes
// three, but rounds 3 to 7 arguments in 10,000 the other way (256 x 512: 87.9 us
// per step, 89.3 so).
__device__ __forceinline__ double rcp1(double r)
{
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(r));
    x = __fma_rn(x, __fma_rn(-r, x, 1.0), x);
    return __fma_rn(x, __fma_rn(-r, x, 1.0), x);
}
