// regsplit.h -- register shares of a kernel's warpgroups (setmaxnreg).
//
// setmaxnreg.inc takes registers from what its CTA was launched with and
// waits, without a limit, until the CTA's other warpgroups have given enough
// back; .dec and .inc are undefined past the launch's own count in the other
// direction.  So a split is sound only where the launch holds exactly its
// sum.  The compiler picks the launch's count (another version, a register
// cap or a debug build may pick another): the launchers compare it with the
// split before they launch (check_reg_split in common.cuh).
#pragma once

namespace kvk {

struct RegSplit {
  int threads[3], regs[3];  // each role's threads (whole warpgroups) and registers a thread
  constexpr int all_threads() const { return threads[0] + threads[1] + threads[2]; }
  constexpr int sum() const { return threads[0] * regs[0] + threads[1] * regs[1] + threads[2] * regs[2]; }
  // `launch_regs`: registers a thread as compiled; they are allocated in
  // units of 8 a thread
  constexpr bool fits(int launch_regs) const { return (launch_regs + 7) / 8 * 8 * all_threads() == sum(); }
};

// pre-fill attention: workers; MMA and copy warps (640 x 96 launched)
constexpr RegSplit kPfRegs{{512, 128, 0}, {104, 64, 0}};
// evictor: epilogues; dequantising; copy and MMA warps (896 x 72 launched)
constexpr RegSplit kEvictRegs{{512, 256, 128}, {88, 56, 40}};
// decode over quantised latents: softmax; products; expansion (512 x 128 launched)
constexpr RegSplit kMlaQRegs{{128, 128, 256}, {256, 96, 80}};

}  // namespace kvk
