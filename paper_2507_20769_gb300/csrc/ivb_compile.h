// ivb_compile.h -- host tape validation and compilation into the device
// program format of ivb_internal.h (implemented in ivb_compile.cpp).
#pragma once
#include <string>
#include <vector>

#include "../../include/ivb.h"
#include "ivb_internal.h"

namespace ivb {

// "" for a valid tape, else the reason it is rejected (ivb_create_problem's IVB_ETAPE cases)
std::string validate_tape(const ivb_tape* t);

// point / tangent sweep, per-output adjoint programs, constants, frame layout
// and operation counts of a validated tape; "" on success
std::string compile_tape(const ivb_tape* t, HostProgram& P, std::vector<Ins>& ins, std::vector<RIns>& rins,
                         std::vector<double>& consts);

// the interpreter's form of the value and reverse programs, entry by entry beside
// `ins` and `rins`, then that of the tangent program, then the value programs of
// the outputs' cones on [c,c], entry by entry again (one unread entry more at the
// end, for the prefetch)
void interpreter_programs(const HostProgram& P, const std::vector<Ins>& ins, const std::vector<RIns>& rins,
                          std::vector<XIns>& xins, std::vector<XRIns>& xrins);

// the point gradients' form of the outputs' programs, entry by entry beside `ins`
// and `rins`: one frame unit per value, x_i at unit i, then G_i, the adjoints and
// the tape of the output; returns the frame units
int point_programs(const HostProgram& P, const std::vector<Ins>& ins, const std::vector<RIns>& rins,
                   std::vector<XIns>& xins, std::vector<XRIns>& xrins);

// variables that the operands of each tangent instruction depend on (bit i: x_i;
// a at 2k, b at 2k + 1), and each output
void tangent_masks(const HostProgram& P, const std::vector<Ins>& ins, std::vector<uint32_t>& masks, uint32_t out_mask[64]);

}  // namespace ivb
