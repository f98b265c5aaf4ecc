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

// Sum of squares of integers |r| < 2^63, exactly, as top 2^128 + hi 2^64 + lo: 32-bit
// integer instructions only.  A conversion and a multiply-add per cell on the FP64
// units, 64 clocks of a scheduler each, set the pace of the integer legs otherwise.
struct SquareSum {
  unsigned long long lo = 0, hi = 0;
  unsigned top = 0;
  MG_HD void add(long long r) {
    const unsigned long long a = r < 0 ? 0ull - (unsigned long long)r : (unsigned long long)r;
    const unsigned h = (unsigned)(a >> 32), l = (unsigned)a;
    const unsigned long long ll = (unsigned long long)l * l, hh = (unsigned long long)h * h;
    const unsigned long long m = (unsigned long long)l * h;  // r^2 = hh 2^64 + m 2^33 + ll
    sum(ll, hh);
    sum(m << 33, m >> 31);
  }
  MG_HD double total() const {
    return ((double)top * 0x1p64 + (double)hi) * 0x1p64 + (double)lo;
  }

 private:
  MG_HD void sum(unsigned long long l, unsigned long long h) {
#ifdef __CUDA_ARCH__
    asm("add.cc.u64 %0, %0, %3;\n\taddc.cc.u64 %1, %1, %4;\n\taddc.u32 %2, %2, 0;"
        : "+l"(lo), "+l"(hi), "+r"(top)
        : "l"(l), "l"(h));
#else
    lo += l;
    const unsigned long long c = lo < l, k = hi + h;
    hi = k + c;
    top += (k < h) + (hi < c);
#endif
  }
};

// Whether a binary64 of these bits is 2^bits or more in magnitude, infinite or
// NaN (integer arithmetic only).
MG_HD bool past_range(unsigned long long u, int bits) {
  return (int)((u >> 52) & 0x7ff) >= 1023 + bits;
}

}  // namespace mg
