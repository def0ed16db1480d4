// Overlap of a kernel with the end of the one before it on its stream (launch_chained).
#pragma once

namespace msqoc {

// Waits until every kernel before this one on the stream has finished and its writes are visible.
// What comes ahead of it reads only tables written at the problem's creation, or by copies that
// the kernel before waited for.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's blocks be placed once every block of this one has called it or ended.
// Called near a kernel's end: a block that waits holds its registers and shared memory, which
// other streams could use.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace msqoc
