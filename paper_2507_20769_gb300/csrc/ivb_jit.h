// ivb_jit.h -- tape-specialised bounding kernels (generated CUDA C++,
// compiled with NVRTC at problem creation); see ivb_jit.cpp.
//
// Variants of the generated source: compact (the default, option specialize
// = 1) puts the point sweep and each output's adjoint sweeps in __noinline__
// functions and calls the long primitives out of line, which halves the
// compile time at the same speed; specialize = 2 inlines everything. With
// form 1 (the natural interval extension alone) the gradient sweeps are left
// out. Every variant is bit-identical to the interpreter.
#pragma once
#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "ivb_internal.h"
#include "ivb_kparams.h"
#include "ivb_launch.h"

namespace ivb {

// generated kernels: __launch_bounds__(kJitBlockMax, kJitMinBlocks), i.e. at
// most 128 registers per thread; specialize = -1 compiles tapes of at most
// kJitAutoMaxOps interval operations per subdomain as one program (beyond that,
// compile time grows to tens of seconds and the interpreter was within 5 % on
// the configurations measured). In adjoint mode the segmented kernel takes
// over from kSegMinOps on, where it is ahead in calls of every size and compiles in half to a
// tenth of the time. Segmented against compact, 2^20 and 1024 subdomains: 620 operations (16 x 16^4)
// 2.07 ms against 2.77; 209 and four outputs 0.74 ms and 62 us against 0.91 and 83; 171 and one output
// 0.61 ms and 75 us against 0.68 and 78. Below the line large calls still gain 4 to 12 % (122
// operations 0.47 ms against 0.54, 62 0.23 against 0.25) but small ones lose (122 69 us against 67, 39 56
// against 52), so the compact kernel stays there.
constexpr int kJitBlockMax = kCompiledBlockMax, kJitMinBlocks = 2, kJitAutoMaxOps = 1024, kSegMinOps = 128;
// chunks from which a segmented kernel keeps its warps on one chunk (below, the
// autotuner times both). Warps that drift apart stream through the code
// separately, and a sample of uniform subdomains does not show it: 306 chunks 56
// ms with the barriers, 178 without; 27 chunks 8.8 and 8.2 ms on one uniform batch
// (configuration 3), but 37 and 45 ms on 256 uneven nodes; 12 chunks 4.4 and 4.0 ms
constexpr int kSegSyncChunks = 20;
// endpoint operations emulated on the integer pipes by default (ivb_iv.cuh
// policy bits): none. The integer ALU is half busy with the selects and the fixed-point
// primitives, so every policy is slower (2^19 subdomains of configuration 5: 48.9 ms with none, 54.6
// with 1, 62 with 3, 73 with 12; configuration 2, 16 x 16^4: 2.05, 2.36 with 1, 4.0 with 15)
constexpr int kJitDefaultEmulate = 0;

struct JitKernel {
    cudaLibrary_t lib = nullptr;
    cudaKernel_t kern = nullptr;
    int mode = -1;             // KM_FWD_REDUCE or KM_ADJ_REDUCE
    int block_max = 0;         // __launch_bounds__ of the generated kernel
    int emulate = 0;           // emulation policy compiled in
    bool compact = false;      // long primitives called out of line
    int regs = 0, local_bytes = 0, max_threads = 0;
    double compile_seconds = 0.0;
    // segmented kernels (ivb_jit_seg.cpp): per-thread state area in doubles
    // (0 for the other variants), chunks, state loads and stores and
    // recomputed forward operations per subdomain, recomputation policy
    int state_units = 0, chunks = 0, recompute = -1, ilp = 1;
    long long state_loads = 0, state_stores = 0, recomputed = 0;
    // kernels of the segmented variant for 1, 2 and 4 threads per subdomain
    // (index 0, 1, 2; nullptr where not compiled), without and with the
    // warps of a thread group kept on the same chunk by a barrier
    cudaKernel_t kern_t[3] = {nullptr, nullptr, nullptr};
    cudaKernel_t kern_sync[3] = {nullptr, nullptr, nullptr};
};

// Segmented kernels for large tapes (ivb_jit_seg.cpp): the per-subdomain
// program cut into chunk functions of bounded estimated work, values that
// cross chunks in a per-thread state area, reverse chunks recomputing their
// segment's forward values (policy 0: none, stored; 1: the cheap operations
// + - * sqr neg; 2: all), chunks compiled in `units` parallel NVRTC programs
// and linked with nvJitLink.
struct SegPolicy {
    double chunk_cost = 320.0;   // estimated FP64 issue slots per chunk
    int chunk_stmts = 96;        // statements per chunk
    int recompute = 0;           // measured fastest: recomputation adds FP64 work, the state area streams with room to spare
    int units = 16;
    // register budget of every chunk function: 64 lets one block of 32 warps fill
    // an SM (configuration 5, 2^19 subdomains: 48.9 ms; 72 registers and 28 warps 48.8, 80
    // and 24 52.9, 128 and 16 58.9; as two blocks of 16 warps, which stream
    // through the code separately, 64.6; configuration 2 2.05 ms, 128 and 2 x 8 warps 2.68)
    int max_regs = 64;
    // subdomains per thread: 2 interleaved take 58.7 ms on configuration 5 (69.3 with 128
    // registers and half the threads), 2.66 on configuration 2 (3.07)
    int ilp = 1;
    // short interval operations out of line: 0 none, 1 all, 2 products only (a
    // call costs more than the two instructions of a sum: configuration 5 48.9 ms
    // against 51.4 with 1 and 53.9 with 0, configuration 3 7.84 against 8.01 and 8.48)
    int outline = 2;
};
struct SegSource {
    std::string kernel;               // tile loop, Step 1, chunk calls, Step 3 (one kernel per T)
    std::vector<std::string> units;   // the chunk functions
    std::vector<int> ts;              // threads per subdomain with a kernel: ivb_jit_bound (1), _t2, _t4
    int state_units = 0, chunks = 0, ilp = 1;
    long long loads = 0, stores = 0, recomputed = 0;
    std::string error;                // "" unless the program could not be planned
};
SegSource jit_seg_source(const HostProgram& P, const std::vector<Ins>& ins, const std::vector<RIns>& rins,
                         const std::vector<double>& consts, int block_max, int emulate, int form, const SegPolicy& pol);
// compile the units in parallel and link them; "" on success
std::string jit_seg_compile(const SegSource& src, int max_regs, std::vector<char>& cubin, std::string& tables_name,
                            double* seconds, int* registers, int* spill_bytes);

// CUDA C++ of the reduce-mode bounding kernel for this program; form 1 (the
// natural interval extension alone) leaves out the gradient sweeps
std::string jit_source(const HostProgram& P, const std::vector<Ins>& ins, const std::vector<RIns>& rins,
                       const std::vector<double>& consts, int mode, int block_max, int min_blocks, int emulate,
                       bool compact, int form);
// NVRTC for sm_103a; "" on success, else the compiler's message. With
// `registers` / `spill_bytes` non-NULL, ptxas reports them (parsed from its log).
std::string jit_compile(const std::string& src, std::vector<char>& cubin, std::string& tables_name, double* seconds,
                        int* registers, int* spill_bytes);
cudaError_t jit_load(const std::vector<char>& cubin, const std::string& tables_name, JitKernel& K);
// launch / occupancy of the kernel for `tpsub` threads per subdomain (1 for
// every variant but the segmented one)
cudaError_t jit_launch(const JitKernel& K, const KParams& P, int grid, int block, cudaStream_t s, int tpsub = 1,
                       bool sync = false);
int jit_occupancy(const JitKernel& K, int block, int tpsub = 1, bool sync = false);
// index of a threads-per-subdomain value in JitKernel::kern_t (-1 if none)
inline int tpsub_index(int t) { return t == 1 ? 0 : t == 2 ? 1 : t == 4 ? 2 : -1; }
void jit_unload(JitKernel& K);

}  // namespace ivb
