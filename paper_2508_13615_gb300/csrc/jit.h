// Segment compiler interface (internal): see jit.cu.
#pragma once
#include <functional>
#include <string>
#include <vector>

#include "lqs_internal.cuh"
#include "tile.cuh"

namespace lqs {

// The arithmetic policy a compiled kernel of policy `aname` runs on: packed
// double-float for ArDF (jit_dev.cuh), the policy itself otherwise.
inline std::string jit_policy(const std::string& aname) {
  return aname == "lqs::ArDF" ? "lqs::jit::ArDFP" : aname;
}

int jit_mode();
// Whether compiled segments may run for an n-qubit state under the current mode.
bool jit_enabled_for(int n);
// CUDA C++ source of a register-tile program (LQS_ERR_UNSUPPORTED for a
// program the generator does not take; the interpreter runs those).
template <class A>
int jit_source(const TileProg<A>& P, int r, std::string& src, std::string& name, std::string& why,
               bool adjoint = false);
// Counts one use of the program's structure and queues it for compilation
// when the mode asks for it (or `force`).
template <class A>
int jit_note(const TileProg<A>& P, int r, int n, bool force, std::vector<void*>& todo);
// Compiles queued structures in parallel.
int jit_compile(const std::vector<void*>& todo);
// After jit_compile: *ok = structures in `todo` that compiled; LQS_ERR_UNSUPPORTED
// (with the first failure's log in *err) when any did not.
int jit_states(const std::vector<void*>& todo, int* ok, std::string* err);
// Launches the compiled kernel of the program if there is one (*launched
// tells); otherwise does nothing and the caller runs the interpreter.  fmt
// (double-float forward segments): bit 0, the state holds hi/lo float pairs
// left by the previous compiled segment of the same call; bit 1, leave
// hi/lo pairs for the next one.  Other kernels ignore it.
template <class A>
int jit_launch(const TileProg<A>& P, int r, SV* sv, double bytes, double flops, const char* prof_name,
               bool* launched, unsigned fmt = 0);
// Compiled adjoint programs: scale[s] multiplies gradient slot s's summed
// partials (double-float sweeps un-apply RY/H in unit-row form, which scales
// psi and lambda by 1/m00 per op until the product is folded back; 1 for the
// other programs), and *gprod gets the product of those m00's.
template <class A>
void jit_adjoint_scales(const TileProg<A>& P, std::vector<double>& scale, double* gprod);
// True when jit_launch would launch the program's compiled kernel now.
template <class A>
bool jit_ready(const TileProg<A>& P, int r, const SV* sv);

// Compiled adjoint: the cache entry of a reverse-sweep program (queued for
// compilation by the caller through jit_compile), its shared-memory size,
// and its launch over psi and lambda writing per-block partial sums
// partial[slot * grid + block].
template <class A>
int jit_adjoint_entry(const TileProg<A>& P, int r, void** entry, std::string* why);
size_t jit_adjoint_smem(int k, int r, size_t amp_bytes);
template <class A>
int jit_adjoint_occupancy(void* entry, const TileProg<A>& P, int r, SV* sv, int* per_sm);
template <class A>
int jit_launch_adjoint(void* entry, const TileProg<A>& P, int r, SV* sv, void* lam, double* partial, unsigned grid,
                       double bytes, double flops, const char* prof_name, unsigned fmt = 0);

// Any generated kernel: the cache entry for structure `key` (the source is
// generated by `gen` only for a new key), its residency, and its launch with
// the CUDA driver's parameter array.
void* jit_entry_generic(const std::string& key,
                        const std::function<bool(std::string& src, std::string& name, std::string& why)>& gen,
                        bool count_use, std::string* why);
int jit_occupancy_generic(void* entry, int dev, size_t smem, int threads, int* per_sm);
// Whether an entry may be used (compiled already) or compiled now under the
// current mode for an n-qubit state (auto: at its second use, 20+ qubits).
bool jit_should_compile(void* entry, int n);
int jit_launch_generic(void* entry, SV* sv, unsigned grid, int threads, size_t smem, void** params,
                       const char* prof_name, double bytes, double flops);

}  // namespace lqs
