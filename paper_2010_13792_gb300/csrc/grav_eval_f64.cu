// Instantiations of the FP64 force kernel (K4) and of the split reduction (K9).
#include "grav_eval_df.cuh"

namespace grav {

// Open boundaries take the two-part kernel, on tiles of 2 S sources (the FP64
// conversions and carries per tile are its second cost), the other modes the
// FP64 one.
template <int NT, int S, bool POT>
void launch_df(const EvalArgs &a, int grid, cudaStream_t st)
{
    eval_df_kernel<NT, S, POT><<<grid, NT, sizeof(DfSmem<NT, S, POT>), st>>>(a);
}

template <int NT, int S, bool POT>
void launch_df_batched(const EvalArgs &a, const BatchView &b, int grid, cudaStream_t st)
{
    eval_df_batched_kernel<NT, S, POT><<<grid, NT, sizeof(DfSmem<NT, S, POT>), st>>>(a, b);
}

template <typename K>
int occupancy_dynamic(int *b, K k, int threads, size_t bytes)
{
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(b, k, threads, bytes);
}

template <int NT, int S, bool POT>
int occupancy_df(int *b)
{
    return occupancy_dynamic(b, eval_df_kernel<NT, S, POT>, NT, sizeof(DfSmem<NT, S, POT>));
}

template <int NT, int S, bool POT>
int occupancy_df_batched(int *b)
{
    return occupancy_dynamic(b, eval_df_batched_kernel<NT, S, POT>, NT, sizeof(DfSmem<NT, S, POT>));
}

#define GRAV_F64_FN3(DF, FN, NT, S)                                                               \
    {{DF<NT, 2 * S, false>, DF<NT, 2 * S, true>},                                                            \
     {FN<NT, S, false, kModePeriodic>, FN<NT, S, true, kModePeriodic>},                              \
     {FN<NT, S, false, kModeSoft>, FN<NT, S, true, kModeSoft>}}

#define GRAV_F64_FN2(DF, FN, NT, S)                                                               \
    {{DF<NT, 2 * S, false>, DF<NT, 2 * S, true>},                                                            \
     {FN<NT, S, false, kModePeriodic>, FN<NT, S, true, kModePeriodic>}}

#define GRAV_F64_CFG(NT, S)                                                                       \
    {GRAV_F64, NT, 1, S, 4, 0, GRAV_F64_FN3(launch_df, launch_f64, NT, S),                         \
     GRAV_F64_FN3(occupancy_df, occupancy_f64, NT, S),                                             \
     {launch_pack<2 * S, false, true, false, true>, launch_pack<S, false, true, false>,                \
      launch_pack<S, false, true, false>},                                                         \
     GRAV_F64_FN2(launch_df_batched, launch_f64_batched, NT, S),                                   \
     GRAV_F64_FN2(occupancy_df_batched, occupancy_f64_batched, NT, S),                             \
     {launch_pack_batched<2 * S, false, true, false, true>, launch_pack_batched<S, false, true, false>}, \
     false,                                                                                        \
     {launch_df<NT, S, false>, launch_df<NT, S, true>},                                            \
     {occupancy_df<NT, S, false>, occupancy_df<NT, S, true>},                                      \
     launch_pack<S, false, true, false, true>,                                                     \
     {launch_f64<NT, S, false, kModeOpen>, launch_f64<NT, S, true, kModeOpen>},                    \
     {occupancy_f64<NT, S, false, kModeOpen>, occupancy_f64<NT, S, true, kModeOpen>},              \
     launch_pack<S, false, true, false>}

static const EvalConfig kF64Configs[] = {
    GRAV_F64_CFG(128, 128),
    GRAV_F64_CFG(64, 128),
    GRAV_F64_CFG(256, 64),
};

const EvalConfig *f64_configs(int *count)
{
    *count = (int)(sizeof(kF64Configs) / sizeof(kF64Configs[0]));
    return kF64Configs;
}

void launch_reduce(const EvalArgs &a, int32_t BT, bool pot, bool etrace, int64_t n_targets,
                   cudaStream_t st)
{
    const int tpb = pot ? reduce_targets_per_block<true>() : reduce_targets_per_block<false>();
    int sms = 0;
    if (device_sm_count(&sms) != GRAV_OK || sms <= 0) sms = 1;
    const unsigned blocks =
        (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_targets + tpb - 1) / tpb, 16LL * sms));
    if (pot && etrace)
        reduce_partials_kernel<true, true><<<blocks, kReduceThreads, 0, st>>>(a, BT);
    else if (pot)
        reduce_partials_kernel<true, false><<<blocks, kReduceThreads, 0, st>>>(a, BT);
    else if (etrace)
        reduce_partials_kernel<false, true><<<blocks, kReduceThreads, 0, st>>>(a, BT);
    else
        reduce_partials_kernel<false, false><<<blocks, kReduceThreads, 0, st>>>(a, BT);
}

}  // namespace grav
