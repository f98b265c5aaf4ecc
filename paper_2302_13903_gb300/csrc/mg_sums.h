// mg_sums.h -- exact sums a thread of the integer legs keeps, and the range check
// of what becomes an integer (host and device, so that they are tested on the
// host).
#pragma once

#ifdef __CUDACC__
#define MG_HD __host__ __device__ __forceinline__
#else
#define MG_HD inline
#endif

namespace mg {

// Sum of 64-bit integers that may pass 2^63, in one register more than a plain
// sum takes: the sum modulo 2^64 and that of the values' bits from 2^44 up.  A
// value lies less than 2^44 above those bits, so the two give the sum exactly
// while fewer than 2^19 values are added and |top| stays below 2^31.
struct SplitSum {
  unsigned long long part = 0;
  int top = 0;
  MG_HD void add(long long v) {
    part += (unsigned long long)v;
    top += (int)(v >> 44);
  }
  // The sum is hi() 2^32 + lo().
  MG_HD long long hi() const { return (long long)top * 4096 + (long long)(rest() >> 32); }
  MG_HD long long lo() const { return (long long)(rest() & 0xffffffffu); }
  MG_HD unsigned long long rest() const { return part - ((unsigned long long)(long long)top << 44); }
};

// Whether a binary64 of these bits is 2^bits or more in magnitude, infinite or
// NaN (integer arithmetic only).
MG_HD bool past_range(unsigned long long u, int bits) {
  return (int)((u >> 52) & 0x7ff) >= 1023 + bits;
}

}  // namespace mg
