// kg_inst.h -- the pass launchers of one precision as plain functions.
//
// Launchers<P> (kg_launch_impl.cuh) instantiates every kernel template of a precision;
// compiled as one unit per precision the double-float share alone took minutes.  So
// kg_inst.cu is compiled once per (precision, share) with KG_PREC_ID and KG_PART set,
// each compile defining the functions of one share in namespace kg::inst_f64,
// kg::inst_df or kg::inst_f32, and kg_inst_tables.cu builds the three PassLaunch
// tables from the declarations below.
#pragma once
#include <type_traits>

#include "kg_launch.h"

#define KG_INST_FN(m) std::remove_pointer_t<decltype(::kg::PassLaunch::m)>

#define KG_INST_DECLARE(ns)                                                            \
    namespace ns {                                                                     \
    KG_INST_FN(pass_x) pass_x;                /* share 0: x pass, x set-up/read-out */ \
    KG_INST_FN(x_parts) x_parts;                                                       \
    KG_INST_FN(x_setup) x_setup;                                                       \
    KG_INST_FN(x_readout) x_readout;                                                   \
    KG_INST_FN(xy_fused) xy_fused;                                                     \
    KG_INST_FN(xy_parts) xy_parts;                                                     \
    KG_INST_FN(plane) plane;                                                           \
    KG_INST_FN(plane_parts) plane_parts;                                               \
    KG_INST_FN(yf) yf;                        /* share 1: column passes */             \
    KG_INST_FN(yi) yi;                                                                 \
    KG_INST_FN(zcol) zcol;                                                             \
    KG_INST_FN(z_from_f64) z_from_f64;                                                 \
    KG_INST_FN(z_to_f64) z_to_f64;                                                     \
    KG_INST_FN(zstep) zstep;                  /* share 2: z pass and update */         \
    KG_INST_FN(zstep_parts) zstep_parts;                                               \
    KG_INST_FN(update) update;                                                         \
    KG_INST_FN(update_parts) update_parts;                                             \
    KG_INST_FN(passc_x) passc_x;              /* share 3: complex field */             \
    KG_INST_FN(xc_parts) xc_parts;                                                     \
    KG_INST_FN(yfc) yfc;                                                               \
    KG_INST_FN(yic) yic;                                                               \
    KG_INST_FN(zcolc) zcolc;                                                           \
    KG_INST_FN(zc_from_f64) zc_from_f64;                                               \
    KG_INST_FN(updatec) updatec;                                                       \
    KG_INST_FN(updatec_parts) updatec_parts;                                           \
    KG_INST_FN(xc_setup) xc_setup;                                                     \
    KG_INST_FN(xc_readout) xc_readout;                                                 \
    KG_INST_FN(zc_to_f64) zc_to_f64;                                                   \
    KG_INST_FN(ens_run) ens_run;              /* share 4: ensemble step */             \
    KG_INST_FN(ens_blocks_per_sm) ens_blocks_per_sm;                                   \
    KG_INST_FN(ens_fill) ens_fill;                                                     \
    }

namespace kg {
KG_INST_DECLARE(inst_f64)
KG_INST_DECLARE(inst_df)
KG_INST_DECLARE(inst_f32)
}  // namespace kg
