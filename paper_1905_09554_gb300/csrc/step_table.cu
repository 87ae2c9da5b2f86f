// Table of the step kernels by (storage, collision).
#include "step_args.h"

namespace lbm {

extern const StepKernels kStep_f64_srt;
extern const StepKernels kStep_f64_mrt;
extern const StepKernels kStep_f64_mrts;
extern const StepKernels kStep_f64_mrtu;
extern const StepKernels kStep_f64_mrtsh;
extern const StepKernels kStep_f32_srt;
extern const StepKernels kStep_f32_mrt;
extern const StepKernels kStep_f32_mrts;
extern const StepKernels kStep_f32_mrtu;
extern const StepKernels kStep_f32_mrtsh;
extern const StepKernels kStep_f16_srt;
extern const StepKernels kStep_f16_mrt;
extern const StepKernels kStep_f16_mrts;
extern const StepKernels kStep_f16_mrtu;
extern const StepKernels kStep_f16_mrtsh;
extern const StepKernels kStep_bf16_srt;
extern const StepKernels kStep_bf16_mrt;
extern const StepKernels kStep_bf16_mrts;
extern const StepKernels kStep_bf16_mrtu;
extern const StepKernels kStep_bf16_mrtsh;
extern const StepKernels kStep_f16l_srt;
extern const StepKernels kStep_f16l_mrt;
extern const StepKernels kStep_f16l_mrts;
extern const StepKernels kStep_f16l_mrtu;
extern const StepKernels kStep_f16l_mrtsh;
extern const StepKernels kStep_bf16l_srt;
extern const StepKernels kStep_bf16l_mrt;
extern const StepKernels kStep_bf16l_mrts;
extern const StepKernels kStep_bf16l_mrtu;
extern const StepKernels kStep_bf16l_mrtsh;

extern const MomentKernels kMoment_f32_srt;
extern const MomentKernels kMoment_f32_mrts;
extern const MomentKernels kMoment_f32_mrtu;
extern const MomentKernels kMoment_f32_mrtsh;
extern const MomentKernels kMoment_f16_srt;
extern const MomentKernels kMoment_f16_mrtu;
extern const MomentKernels kMoment_bf16_srt;
extern const MomentKernels kMoment_bf16_mrtu;
extern const MomentKernels kMoment_f16l_srt;
extern const MomentKernels kMoment_f16l_mrtu;
extern const MomentKernels kMoment_bf16l_srt;
extern const MomentKernels kMoment_bf16l_mrtu;

// 9 or 10 float moments (36 or 40 B) would not be less than 19 16-bit
// populations (38 B): there only the operators with 4.
const MomentKernels* moment_kernels(int storage, int coll) {
    static const MomentKernels* table[6][COLL_COUNT] = {
        {},
        {&kMoment_f32_srt, nullptr, &kMoment_f32_mrts, &kMoment_f32_mrtu, &kMoment_f32_mrtsh},
        {&kMoment_f16_srt, nullptr, nullptr, &kMoment_f16_mrtu, nullptr},
        {&kMoment_bf16_srt, nullptr, nullptr, &kMoment_bf16_mrtu, nullptr},
        {&kMoment_f16l_srt, nullptr, nullptr, &kMoment_f16l_mrtu, nullptr},
        {&kMoment_bf16l_srt, nullptr, nullptr, &kMoment_bf16l_mrtu, nullptr},
    };
    return table[storage][coll];
}

cudaError_t split_step_f64(const SplitLaunch& l, int coll, void* src, void* dst, void* psi);
cudaError_t split_step_f32(const SplitLaunch& l, int coll, void* src, void* dst, void* psi);
cudaError_t split_step_f16(const SplitLaunch& l, int coll, void* src, void* dst, void* psi);
cudaError_t split_step_bf16(const SplitLaunch& l, int coll, void* src, void* dst, void* psi);
cudaError_t split_step_f16l(const SplitLaunch& l, int coll, void* src, void* dst, void* psi);
cudaError_t split_step_bf16l(const SplitLaunch& l, int coll, void* src, void* dst, void* psi);

cudaError_t split_step(const SplitLaunch& l, int storage, int coll, void* src, void* dst, void* psi) {
    static constexpr decltype(&split_step_f64) table[6] = {split_step_f64,  split_step_f32,  split_step_f16,
                                                           split_step_bf16, split_step_f16l, split_step_bf16l};
    return table[storage](l, coll, src, dst, psi);
}

const StepKernels& step_kernels(int storage, int coll) {
    static const StepKernels* table[6][COLL_COUNT] = {
        {&kStep_f64_srt, &kStep_f64_mrt, &kStep_f64_mrts, &kStep_f64_mrtu, &kStep_f64_mrtsh},
        {&kStep_f32_srt, &kStep_f32_mrt, &kStep_f32_mrts, &kStep_f32_mrtu, &kStep_f32_mrtsh},
        {&kStep_f16_srt, &kStep_f16_mrt, &kStep_f16_mrts, &kStep_f16_mrtu, &kStep_f16_mrtsh},
        {&kStep_bf16_srt, &kStep_bf16_mrt, &kStep_bf16_mrts, &kStep_bf16_mrtu, &kStep_bf16_mrtsh},
        {&kStep_f16l_srt, &kStep_f16l_mrt, &kStep_f16l_mrts, &kStep_f16l_mrtu, &kStep_f16l_mrtsh},
        {&kStep_bf16l_srt, &kStep_bf16l_mrt, &kStep_bf16l_mrts, &kStep_bf16l_mrtu, &kStep_bf16l_mrtsh},
    };
    return *table[storage][coll];
}

}  // namespace lbm
