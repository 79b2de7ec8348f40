// Layout of the router image read by the row-tiled decision (k_decide.cu)
// and written by the host (ebd_api.cu).
#pragma once

namespace ebd {
namespace rowimg {

// Matrices, bf16, offsets in 16-byte units.  W [N][K] (row-major in the blob)
// is stored as the mma.sync A fragments of its 16-output x 16-input tiles:
// tile (m16, k16) at ((m16 * K/16 + k16) * 32), one 16-byte unit {a0, a1, a2,
// a3} per lane 4 g + t, two consecutive inputs each.  LBS: rows g, g + 8 of
// the fragment are outputs 16 m + 2 g, 2 g + 1 (a lane's results are two
// neighbouring columns), and lane t's inputs are 32 kb + 8 t + 4 s + {0, 1}
// (a0, a1) and + {2, 3} (a2, a3) for k16 = 2 kb + s, as the activations are
// read, 16 bytes of a row per lane.  LPS: natural order.
constexpr int mat16(int n, int k) { return n * k / 8; }
constexpr int M_ENT2 = 0;
constexpr int M_COMB = M_ENT2 + mat16(64, 64);
constexpr int M_LAYER = M_COMB + mat16(128, 128);
constexpr int ML_QKV = 0;
constexpr int ML_OUT = ML_QKV + mat16(384, 128);
constexpr int ML_FF1 = ML_OUT + mat16(128, 128);
constexpr int ML_FF2 = ML_FF1 + mat16(256, 128);
constexpr int ML_STRIDE = ML_FF2 + mat16(128, 256);
constexpr int M_BLOCK = M_LAYER + 2 * ML_STRIDE;
constexpr int MB_QKV = 0;
constexpr int MB_OUT = MB_QKV + mat16(96, 32);
constexpr int MB_FF1 = MB_OUT + mat16(32, 32);
constexpr int MB_FF2 = MB_FF1 + mat16(64, 32);
constexpr int MB_STRIDE = MB_FF2 + mat16(32, 64);
constexpr int M_TOTAL = M_BLOCK + 2 * MB_STRIDE;

// Vectors, fp32, offsets in floats; the positional table follows at V_POS.
constexpr int V_ENT1W = 0, V_ENT1B = 64, V_ENT2B = 128, V_ENTLNG = 192, V_ENTLNB = 256,
              V_TOKB = 320, V_COMBB = 384, V_LAYER = 512;
constexpr int VL_QKVB = 0, VL_OUTB = 384, VL_LN1G = 512, VL_LN1B = 640, VL_FF1B = 768,
              VL_FF2B = 1024, VL_LN2G = 1152, VL_LN2B = 1280, VL_STRIDE = 1408;
constexpr int V_HEADW = V_LAYER + 2 * VL_STRIDE, V_HEADB = V_HEADW + 128;
constexpr int V_LPS = V_HEADB + 4;
constexpr int V_INT = V_LPS;  // input layer [5][32]
constexpr int V_INB = V_INT + 160, V_INLNG = V_INB + 32, V_INLNB = V_INLNG + 32,
              V_BLOCK = V_INLNB + 32;
constexpr int VB_LN1G = 0, VB_LN1B = 32, VB_QKVB = 64, VB_OUTB = 160, VB_LN2G = 192,
              VB_LN2B = 224, VB_FF1B = 256, VB_FF2B = 320, VB_STRIDE = 352;
constexpr int V_PHEADW = V_BLOCK + 2 * VB_STRIDE, V_PHEADB = V_PHEADW + 32;
constexpr int V_POS = V_PHEADB + 4;  // [gen_len][128]
static_assert(V_POS % 4 == 0 && V_LPS % 4 == 0, "float4 copies");

}  // namespace rowimg
}  // namespace ebd
