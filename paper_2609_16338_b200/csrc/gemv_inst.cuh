// Every instantiation of the products' launch functions, listed once: gemv.cu declares them extern, gemv_inst.cu defines
// the part it is compiled for (BITCOS_INST = `template` and BITCOS_PART = the part's number there).  The parts only
// spread the compilation over processes.
#ifndef BITCOS_INST
#define BITCOS_INST extern template
#define BITCOS_PART 0
#endif
#define BITCOS_IN(part) (BITCOS_PART == 0 || BITCOS_PART == (part))

namespace bitcos_kernels {

#define BITCOS_SINGLE(FMT, NB, XG, XQ, BL) \
    BITCOS_INST int launch<FMT, NB, XG, XQ, BL>(const Problem &, const Plan &, cudaStream_t, const uint32_t *);
#define BITCOS_MULTI(NB, XQ, XG) BITCOS_INST int launch_multi<NB, XQ, XG>(MultiArgs &, cudaStream_t, const uint32_t *const *, int);
#define BITCOS_GROUPED(FMT, NB, PARTS) BITCOS_INST int launch_grouped<FMT, NB, PARTS>(const Problem &, const Plan &, const GroupedArgs &, int, cudaStream_t);
#define BITCOS_PHASED(NB) BITCOS_INST int launch_phased<NB>(PhasedArgs &, int, const int *, cudaStream_t);

#if BITCOS_IN(1)
BITCOS_SINGLE(kBitcos, 1, false, false, false)
BITCOS_SINGLE(kBitcos, 1, true, false, false)
BITCOS_SINGLE(kBitcos, 1, false, true, false)
BITCOS_PHASED(1)
#endif
#if BITCOS_IN(2)
BITCOS_SINGLE(kBitcos, 2, false, false, false)
BITCOS_SINGLE(kBitcos, 2, true, false, false)
BITCOS_SINGLE(kBitcos, 2, false, true, false)
BITCOS_PHASED(2)
#endif
#if BITCOS_IN(3)
BITCOS_SINGLE(kBitcos, 4, false, false, false)
BITCOS_SINGLE(kBitcos, 4, true, false, false)
BITCOS_SINGLE(kBitcos, 8, false, false, false)
BITCOS_SINGLE(kBitcos, 8, true, false, false)
#endif
#if BITCOS_IN(4)
BITCOS_SINGLE(kBitcos, 4, false, false, true)
BITCOS_SINGLE(kBitcos, 8, false, false, true)
BITCOS_SINGLE(kBitcos, 16, false, false, false)
BITCOS_SINGLE(kBitcos, 16, true, false, false)
BITCOS_MULTI(16, false, false)
BITCOS_MULTI(16, false, true)
#endif
#if BITCOS_IN(5)
BITCOS_MULTI(1, false, false)
BITCOS_MULTI(1, false, true)
BITCOS_MULTI(1, true, false)
BITCOS_MULTI(2, false, false)
#endif
#if BITCOS_IN(6)
BITCOS_MULTI(2, false, true)
BITCOS_MULTI(2, true, false)
BITCOS_MULTI(4, false, false)
BITCOS_MULTI(4, false, true)
BITCOS_MULTI(8, false, false)
BITCOS_MULTI(8, false, true)
#endif
#if BITCOS_IN(7)
BITCOS_SINGLE(kTrit5, 1, false, false, false)
BITCOS_SINGLE(kTrit5, 2, false, false, false)
BITCOS_SINGLE(kTrit5, 4, false, false, false)
BITCOS_SINGLE(kTrit5, 8, false, false, false)
BITCOS_SINGLE(kTrit5, 16, false, false, false)
#endif
#if BITCOS_IN(8)
BITCOS_SINGLE(kBit2, 1, false, false, false)
BITCOS_SINGLE(kBit2, 2, false, false, false)
BITCOS_SINGLE(kBit2, 4, false, false, false)
BITCOS_SINGLE(kBit2, 8, false, false, false)
BITCOS_SINGLE(kBit2, 16, false, false, false)
#endif
#if BITCOS_IN(9)
BITCOS_GROUPED(kBitcos, 1, false)
BITCOS_GROUPED(kBitcos, 2, false)
BITCOS_GROUPED(kBitcos, 4, false)
BITCOS_GROUPED(kBitcos, 8, false)
BITCOS_GROUPED(kBitcos, 8, true)
BITCOS_GROUPED(kBitcos, 16, false)
#endif
#if BITCOS_IN(10)
BITCOS_GROUPED(kTrit5, 1, false)
BITCOS_GROUPED(kTrit5, 2, false)
BITCOS_GROUPED(kTrit5, 4, false)
BITCOS_GROUPED(kTrit5, 8, false)
BITCOS_GROUPED(kTrit5, 16, false)
#endif
#if BITCOS_IN(11)
BITCOS_GROUPED(kBit2, 1, false)
BITCOS_GROUPED(kBit2, 2, false)
BITCOS_GROUPED(kBit2, 4, false)
BITCOS_GROUPED(kBit2, 8, false)
BITCOS_GROUPED(kBit2, 16, false)
#endif

#undef BITCOS_SINGLE
#undef BITCOS_MULTI
#undef BITCOS_GROUPED
#undef BITCOS_PHASED
}  // namespace bitcos_kernels
