// What a served slot does with its sum (deterministic backward), shared by the apply kernels.
#pragma once
#include "robe_internal.h"

namespace robe {

// MODE: 0 - add the sum delta to a dense gradient; 1 - the SGD step fma(-lr, delta, old); 3 - the Adagrad
// step (Duchi, Hazan, Singer): one accumulator m2 of squared gradients per slot; 2 - the Adam step (Kingma
// & Ba, Algorithm 1; the paper trains five of its six models with Adam, Section 5) on the slot and its two
// moment slots, every operation a separate correctly rounded fp32 one.  Returns the slot's new value.
template <int MODE>
__device__ __forceinline__ float slot_step(const AdamState& ad, float lr, float delta, float old, float& m1, float& m2) {
    if (MODE == 0) return __fadd_rn(old, delta);
    if (MODE == 1) return __fmaf_rn(-lr, delta, old);
    if (MODE == 3) {
        m2 = __fadd_rn(m2, __fmul_rn(delta, delta));
        const float den = __fadd_rn(__fsqrt_rn(m2), ad.eps);
        return __fsub_rn(old, __fmul_rn(lr, __fdiv_rn(delta, den)));
    }
    m1 = __fadd_rn(__fmul_rn(ad.beta1, m1), __fmul_rn(__fsub_rn(1.0f, ad.beta1), delta));
    m2 = __fadd_rn(__fmul_rn(ad.beta2, m2), __fmul_rn(__fsub_rn(1.0f, ad.beta2), __fmul_rn(delta, delta)));
    const float den = __fadd_rn(__fsqrt_rn(__fdiv_rn(m2, ad.bias2)), ad.eps);
    return __fsub_rn(old, __fmul_rn(lr, __fdiv_rn(__fdiv_rn(m1, ad.bias1), den)));
}

// The step of slot j with its state in memory; `old` is target[j].  A: anything with mp, target, lr, adam.
template <int MODE, class A>
__device__ __forceinline__ void commit_slot(const A& a, uint32_t j, float delta, float old) {
    if (!ROBE_CHK(j < a.mp.m, ROBE_DBG_ARRAY_SLOT)) return;
    float m1 = 0.0f, m2 = 0.0f;
    if (MODE == 2) m1 = a.adam.m1[j];
    if (MODE >= 2) m2 = a.adam.m2[j];
    a.target[j] = slot_step<MODE>(a.adam, a.lr, delta, old, m1, m2);
    if (MODE == 2) a.adam.m1[j] = m1;
    if (MODE >= 2) a.adam.m2[j] = m2;
}

}  // namespace robe
