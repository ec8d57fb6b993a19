// Time stamps of the decode kernel.  Compiled in only with -DCOOPT_TRACE (the separate library
// libcoopt_trace.so); the ordinary library contains none of this.  A stamp is the SM's cycle counter
// written to slot `s` of the CTA's record in a caller-supplied buffer (coopt_trace_set_buffer); two slots
// hold the global nanosecond timer at entry and exit so that the CTAs of a launch can be laid side by side.
#pragma once

#include <stdint.h>

namespace coopt {

enum TraceSlot {         // of the decode kernel, by the first lane of warp 0 unless it says otherwise
  kTrEntry = 0,          // first instruction of the CTA (cycles; every other cycle stamp is read against this one)
  kTrEntryNs,            // global timer at entry
  kTrLine,               // context lengths read and summed up
  kTrFirstCopy,          // the ring's first copies requested
  kTrPrevDone,           // the kernel before has finished
  kTrQuery,              // query operand of the first unit ready
  kTrFirstLanded,        // first block has landed
  kTrStreamed,           // all warps have worked through their blocks
  kTrExit,               // last store issued
  kTrExitNs,             // global timer at exit
  kTrSmId,               // 1 + the SM the CTA ran on
  kTrPrevExitNs,         // what kTrExitNs held at entry: the exit of this CTA's slot in the launch before
  kTrBlocks,             // blocks of warp 0 (a count)
  kTrWarpEnd = 16,       // 16 + w: warp w has worked through its blocks
  kTraceSlots = 32
};
constexpr int kTraceMaxCtas = 1024;

#ifdef COOPT_TRACE
unsigned long long* trace_buffer();      // host: what coopt_trace_set_buffer registered (nullptr = none)
#ifdef __CUDACC__
__device__ __forceinline__ void trace_put(unsigned long long* buf, int slot, unsigned long long v) {
  if (buf != nullptr && blockIdx.x < kTraceMaxCtas && slot < kTraceSlots) buf[blockIdx.x * kTraceSlots + slot] = v;
}
__device__ __forceinline__ unsigned long long trace_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
#define COOPT_TRACE_CYCLES(buf, slot, cond) do { if (cond) ::coopt::trace_put((buf), (slot), static_cast<unsigned long long>(clock64())); } while (0)
#define COOPT_TRACE_NS(buf, slot, cond) do { if (cond) ::coopt::trace_put((buf), (slot), ::coopt::trace_ns()); } while (0)
#define COOPT_TRACE_VALUE(buf, slot, cond, v) do { if (cond) ::coopt::trace_put((buf), (slot), static_cast<unsigned long long>(v)); } while (0)
#endif
#else
#define COOPT_TRACE_CYCLES(buf, slot, cond) do { } while (0)
#define COOPT_TRACE_NS(buf, slot, cond) do { } while (0)
#define COOPT_TRACE_VALUE(buf, slot, cond, v) do { } while (0)
#endif

}  // namespace coopt
