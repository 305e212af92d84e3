// Programmatic dependent launch: a kernel of an evaluation starts while its
// predecessor's last blocks still run, does what does not depend on it (its
// launch, its descriptor) and then waits for its results.  An evaluation is a
// chain of 10 to 100 launches, a few microseconds each at small sizes.
//
// Rules that keep the chain ordered: every block of a kernel launched this way
// calls pdl_wait() before it reads or writes anything an earlier kernel touches
// and before it exits, so a kernel never completes before its predecessor; the
// first kernel of a call is launched plainly (full order after whatever the stream
// holds: the wait covers the kernel before, not one that this one overtook).
//
// The data of the chain (states, staged coefficients and tables, partials) change
// while a kernel launched early is already running.  A pointer to them is
// therefore neither __restrict__ nor read through the read-only path (__ldg,
// ld.global.nc): both promise data that stay the same for the kernel's lifetime,
// so the compiler may move such a load above the wait, and the wait does not order
// it.  Plain loads after pdl_wait(), __ldcg or chain_load() are ordered.  Tables of
// the plan and of the Hamiltonian, which no kernel of a chain writes, may be both.
#pragma once

#include <cuda_runtime.h>

namespace vqe {

// Lets the next kernel of the stream start once every block has got here.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Returns when the kernel before has completed and its writes are visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A table that an earlier kernel of the chain staged, kept in L1.  (For the
// diagonal tables of the ansatz passes: as fast as __ldg.)
template <class C>
__device__ __forceinline__ C chain_load(const C *p) { return __ldca(p); }

// Where it pays, by the number of blocks (152 SMs; a gradient in us, plain
// against early launch).  Small grids: the gaps between kernels count (14 qubits,
// 8 blocks: 588 -> 550 FP64).
// Large ones: blocks of the next kernel take the places that the last wave frees
// (22 qubits: 5921 -> 5821, complex64 1327 -> 1215).  In between the
// early blocks double up on some SMs while others stay empty (18 qubits, 128
// blocks: 677 -> 837; 19 qubits, 256 blocks: 905 -> 933).  The lines, a quarter of a
// block and three blocks per SM, lie between those sizes; nothing measured places
// them closer.
// The same holds for a small grid behind a short reduction of a middle one (16
// qubits, general Pauli sum: 128 blocks, their sums, then passes of 32 blocks on the
// 24 SMs left: gradient at depth 2 356 -> 406 us): that reduction is launched plainly.
inline bool pdl_pays(dim3 grid) {
    const unsigned long long blocks = (unsigned long long)grid.x * grid.y;
    return blocks <= 38 || blocks >= 456;
}

template <class... Params, class... Args>
cudaError_t pdl_launch(void (*kern)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                       bool early, Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

}  // namespace vqe
