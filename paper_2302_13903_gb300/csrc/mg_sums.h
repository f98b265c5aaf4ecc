// mg_sums.h -- exact sums that threads of the FP64 path's integer kernels keep, and
// the range check of what becomes an integer (host and device, so that they are
// tested on the host).
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

// Sum of squares of integers |r| < 2^63, exactly, in five 32-bit words: integer
// instructions only.  A conversion and a multiply-add per cell on the FP64
// units, 64 clocks of a scheduler each, set the pace of the integer legs otherwise.
struct SquareSum {
  unsigned w0 = 0, w1 = 0, w2 = 0, w3 = 0, w4 = 0;
  MG_HD void add(long long r) {
    const unsigned long long a = r < 0 ? 0ull - (unsigned long long)r : (unsigned long long)r;
    const unsigned h = (unsigned)(a >> 32), l = (unsigned)a, h2 = 2 * h;  // h < 2^31
#ifdef __CUDA_ARCH__
    asm("mad.lo.cc.u32 %0, %5, %5, %0;\n\tmadc.hi.cc.u32 %1, %5, %5, %1;\n\t"
        "addc.cc.u32 %2, %2, 0;\n\taddc.cc.u32 %3, %3, 0;\n\taddc.u32 %4, %4, 0;"
        : "+r"(w0), "+r"(w1), "+r"(w2), "+r"(w3), "+r"(w4)
        : "r"(l));
    if (h)
      asm("mad.lo.cc.u32 %0, %4, %6, %0;\n\tmadc.hi.cc.u32 %1, %4, %6, %1;\n\t"
        "addc.cc.u32 %2, %2, 0;\n\taddc.u32 %3, %3, 0;\n\t"
        "mad.lo.cc.u32 %1, %5, %5, %1;\n\tmadc.hi.cc.u32 %2, %5, %5, %2;\n\taddc.u32 %3, %3, 0;"
        : "+r"(w1), "+r"(w2), "+r"(w3), "+r"(w4)
        : "r"(l), "r"(h), "r"(h2));
#else
    const unsigned long long ll = (unsigned long long)l * l, hh = (unsigned long long)h * h;
    const unsigned long long m = (unsigned long long)l * h2;
    unsigned long long c = (unsigned long long)w0 + (unsigned)ll;
    w0 = (unsigned)c;
    c = (c >> 32) + w1 + (ll >> 32) + (unsigned)m;
    w1 = (unsigned)c;
    c = (c >> 32) + w2 + (unsigned)hh + (m >> 32);
    w2 = (unsigned)c;
    c = (c >> 32) + w3 + (hh >> 32);
    w3 = (unsigned)c;
    w4 += (unsigned)(c >> 32);
#endif
  }
  MG_HD unsigned long long lo() const { return (unsigned long long)w1 << 32 | w0; }
  MG_HD unsigned long long hi() const { return (unsigned long long)w3 << 32 | w2; }
  MG_HD double total() const {
    return ((double)w4 * 0x1p64 + (double)hi()) * 0x1p64 + (double)lo();
  }
};

// Whether a binary64 of these bits is 2^bits or more in magnitude, infinite or
// NaN (integer arithmetic only).
MG_HD bool past_range(unsigned long long u, int bits) {
  return (int)((u >> 52) & 0x7ff) >= 1023 + bits;
}

}  // namespace mg
