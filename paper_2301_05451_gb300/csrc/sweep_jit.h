// Specialised sweep programs: the register passes of one circuit (in a linear
// frame of the basis index, lin_program.h) written out as straight-line device
// code -- every gate kind, pairing and table row a compile-time constant --,
// compiled at run time for the device in use.
#pragma once

#include <functional>
#include <string>
#include <vector>

#include "lin_program.h"
#include "sweep_tiled.cuh"
#include "tdq_internal.h"

namespace tdq {

// Source of a K2 kernel named `name` for the whole-state program `prog` (one
// tile; grad: with its reverse passes).  nthreads threads per CTA, nparams
// gradient columns.
// fine: with the values' own CTAs (SweepArgs::fine_rows).
std::string k2_specialised_source(const LinProgram& prog, bool grad, int nthreads, int nparams, const char* name,
                                  bool fine = false);

// One circuit of a multi-circuit whole-state kernel.
struct K2Part {
  const LinProgram* prog;
  int P;
};

// Modules of a persistent kernel `name` over several circuits: module 0 is the
// kernel, whose CTAs take (circuit, row) items (int2) from a global counter
// and call circuit c's row function (module c + 1: its specialised program);
// arguments (const MultiCirc*, const int2* items, int n_items, int* next,
// params, inputs, values, gw, grads), every buffer packed by circuit at the
// MultiCirc offsets.  grad: adjoint sweeps.  The modules compile separately
// (relocatable device code) and are linked into one kernel.
std::vector<std::string> k2_multi_modules(const std::vector<K2Part>& parts, bool grad, int nthreads,
                                          const char* name);
// Separates the modules in the one text tdq_multi_source writes: each module
// follows a line kModuleMark + its number.
constexpr const char* kModuleMark = "// ==== tdq module ";

// Source of the K1 kernels of every tile pass p of t (program prog):
// tdq_k1f_<p> (forward; the last one also runs its reverse sweep with
// gradients) and tdq_k1r_<p> (reverse, passes before the last).  only >= 0:
// that pass's kernels alone.
std::string k1_specialised_source(const TiledSweep& t, const LinProgram& prog, int nthreads_r, int only = -1);

// Code to compile: bytes that differ wherever its text does, and the text, written
// out only if no kernel of that key is in the cache (writing it takes longer than
// the rest of a compile that finds its kernels there: 2 ms for the 20-qubit ladder).
struct JitCode {
  std::string key;
  std::function<std::vector<std::string>()> modules;
};
JitCode k2_code(const LinProgram& prog, bool grad, int nthreads, int nparams, const char* name, bool fine);
JitCode k1_code(const TiledSweep& t, const LinProgram& prog, int nthreads_r, int pass);

// Whether the code is compiled already.
bool jit_cached(const JitCode& code);

// Compiles the code (one module) for the current device and returns the kernel
// `name` (a handle usable with cudaLaunchKernel / cudaFuncSetAttribute).  Compiled
// kernels are cached by key for the life of the process.
tdq_status jit_kernel(const JitCode& code, const char* name, const void** kernel);

// Compiles the modules concurrently (NVRTC, relocatable device code, one host
// thread each, every function within maxrreg registers -- the kernel's launch
// bounds, which separately compiled callees cannot see), links them
// (nvJitLink) and returns the kernel `name`; cached by key.
tdq_status jit_link_kernel(const JitCode& code, const char* name, int maxrreg, const void** kernel);

}  // namespace tdq
