// How a CTA whose roles need different numbers of registers shares out what it got at launch (setmaxnreg).
// Integer arithmetic only: compiles for the device, and by itself as plain C++ (the CPU test does so).
#pragma once

namespace baps {

// `threads` threads, `many_threads` of them raise their share to `many` registers, the others lower theirs to `few`.
struct RegisterSplit { int threads, few, many_threads, many; };

// The pool is what the CTA got at launch, the kernel's registers times its threads.  Raising a share beyond what is left
// in it waits for ever, so a kernel that was compiled to fewer registers must not be launched.
constexpr bool split_fits(const RegisterSplit &s, int regs_at_launch)
{
    return (s.threads - s.many_threads) * s.few + s.many_threads * s.many <= s.threads * regs_at_launch;
}

// attention_tc_kernel and paired_attention_tc_kernel: a warpgroup of producer, MMA issuer and two idle warps, sixteen softmax
// warps; 96 at launch.  attention_d64_kernel: the same with eight; 80 at launch (two CTAs per SM).  All use their pool exactly.
constexpr RegisterSplit kTcSplit = {640, 64, 512, 104};
constexpr RegisterSplit kD64Split = {384, 32, 256, 104};

} // namespace baps
