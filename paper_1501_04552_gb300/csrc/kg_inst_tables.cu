// kg_inst_tables.cu -- the pass-launcher tables of the three FFT precisions, built from
// the per-share functions of kg_inst.cu.
#include "kg_fft.cuh"
#include "kg_inst.h"
#include "../../include/kg.h"

namespace kg {

template <class P>
static int lay_lg_of(int N) {
    return N >= 512 ? LayLg<P, 512>::value : LayLg<P, 256>::value;
}

#define KG_TABLE_COMMON(ns, S, LG)                                                                               \
    &ns::pass_x, &ns::yf, &ns::yi, &ns::zcol, &ns::z_from_f64, &ns::update, &ns::update_parts, &ns::ens_run, \
        &ns::ens_blocks_per_sm, &ns::ens_fill, &ns::x_parts, S, LG, &ns::passc_x, &ns::xc_parts, &ns::yfc, &ns::yic, &ns::zcolc, \
        &ns::zc_from_f64, &ns::updatec, &ns::updatec_parts

const PassLaunch kLaunchF64 = {
    KG_TABLE_COMMON(inst_f64, 16, &lay_lg_of<PrecF64>),
    nullptr, nullptr,   // no fused z pass: the three-kernel form is faster for FP64
    nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,    // set-up and read-out: the FP64 kernels
    nullptr, nullptr, nullptr, nullptr};                     // no fused xy or plane pass
const PassLaunch kLaunchDF = {
    KG_TABLE_COMMON(inst_df, 16, &lay_lg_of<PrecDF>),
    &inst_df::zstep, &inst_df::zstep_parts,
    &inst_df::x_setup, &inst_df::x_readout, &inst_df::z_to_f64,
    &inst_df::xc_setup, &inst_df::xc_readout, &inst_df::zc_to_f64,
    nullptr, nullptr,    // no fused xy pass: the double-float passes are bound by the FMA pipes, not HBM
    &inst_df::plane, &inst_df::plane_parts};
const PassLaunch kLaunchF32 = {
    KG_TABLE_COMMON(inst_f32, 8, &lay_lg_of<PrecF32>),
    &inst_f32::zstep, &inst_f32::zstep_parts,
    nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,    // set-up and read-out stay FP64
    &inst_f32::xy_fused, &inst_f32::xy_parts, nullptr, nullptr};

}  // namespace kg
