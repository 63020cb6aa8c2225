// BN254 scalar field: pass kernels.
#define NTT_FIELD FieldBn254Fr
#define NTT_NS bn254
#define NTT_PART_PASS
#include "ntt_kernels.inl"
