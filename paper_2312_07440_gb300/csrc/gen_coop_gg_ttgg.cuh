// ---- generated by gen/coop_gen.py, do not edit ----
// Task words, amplitude combination and colour sum of the warp-per-event g g -> t tbar g g code (qcd_coop.cuh).
#pragma once
#include "helas.cuh"

namespace rw { namespace coop {
constexpr int TW_J2 = 0, N_J2 = 18;
constexpr int TW_DOT = 18, N_DOT = 78;
constexpr int TW_J3 = 96, N_J3 = 48;
constexpr int TW_J3B = 144, N_J3B = 48;
constexpr int TW_J4 = 192, N_J4 = 48;
constexpr int TW_J4B = 240, N_J4B = 48;
constexpr int TW_J4C = 288, N_J4C = 48;
constexpr int TW_J4D = 336, N_J4D = 48;
constexpr int TW_X1 = 384, N_X1 = 28;
constexpr int TW_R3 = 412, N_R3 = 160;
constexpr int TW_Y = 572, N_Y = 120;
constexpr int TW_X2 = 692, N_X2 = 144;
constexpr int N_WORDS = 836;
static __device__ const unsigned TASK_WORDS[N_WORDS] = {
    0x108u, 0x110u, 0x218u, 0x220u, 0x328u, 0x330u, 0x259u, 0x261u, 0x25au, 0x262u, 0x369u, 0x371u,
    0x36au, 0x372u, 0x3abu, 0x3b3u, 0x3acu, 0x3b4u, 0x10u, 0x20u, 0x30u, 0x40u, 0x50u, 0x60u,
    0x31u, 0x41u, 0x32u, 0x42u, 0x51u, 0x61u, 0x52u, 0x62u, 0x53u, 0x63u, 0x54u, 0x64u,
    0x68u, 0x78u, 0x88u, 0x98u, 0x29u, 0x39u, 0x2au, 0x3au, 0xbu, 0xcu, 0x1bu, 0x1cu,
    0xa8u, 0xb8u, 0xc8u, 0xd8u, 0x49u, 0x59u, 0x4au, 0x5au, 0xdu, 0xeu, 0x1du, 0x1eu,
    0xe8u, 0xf8u, 0x108u, 0x118u, 0x4bu, 0x5bu, 0x4cu, 0x5cu, 0x2du, 0x2eu, 0x3du, 0x3eu,
    0xe9u, 0xf9u, 0x109u, 0x119u, 0xeau, 0xfau, 0x10au, 0x11au, 0xabu, 0xbbu, 0xacu, 0xbcu,
    0xcbu, 0xdbu, 0xccu, 0xdcu, 0x6du, 0x6eu, 0x7du, 0x7eu, 0x8du, 0x8eu, 0x9du, 0x9eu,
    0x48300c8u, 0x4838108u, 0x48402d0u, 0x4848310u, 0x3130458u, 0x3138660u, 0x3140498u, 0x31486a0u, 0x6850148u, 0x6858188u, 0x6860350u, 0x6868390u,
    0x3950868u, 0x3958a70u, 0x39608a8u, 0x3968ab0u, 0x7070558u, 0x7078598u, 0x7080760u, 0x70887a0u, 0x59708e8u, 0x5978af0u, 0x5980928u, 0x5988b30u,
    0x7270d59u, 0x7278d99u, 0x7280f61u, 0x7288fa1u, 0x727115au, 0x727919au, 0x7281362u, 0x72893a2u, 0x5b714e9u, 0x5b796f1u, 0x5b81529u, 0x5b89731u,
    0x5b718eau, 0x5b79af2u, 0x5b8192au, 0x5b89b32u, 0x6c54d4bu, 0x6c5cd8bu, 0x6c54f4cu, 0x6c5cf8cu, 0x6c65153u, 0x6c6d193u, 0x6c65354u, 0x6c6d394u,
    0x68908c0u, 0x6c98ce0u, 0x70a0901u, 0x74a8d21u, 0x58900c2u, 0x5c980e3u, 0x60a0502u, 0x64a8523u, 0x98f1140u, 0x9cf9560u, 0xa101181u, 0xa5095a1u,
    0x88f0144u, 0x8cf8165u, 0x9100584u, 0x95085a5u, 0xc9511c2u, 0xcd595e2u, 0xd161203u, 0xd569623u, 0xb9509c4u, 0xbd589e5u, 0xc160e04u, 0xc568e25u,
    0x119b29c6u, 0x11dbade6u, 0x121c2a07u, 0x125cae27u, 0x129d31c8u, 0x12ddb5e8u, 0x131e3209u, 0x135eb629u, 0xf9b19cau, 0xfdb99ebu, 0x101c1e0au, 0x105c9e2bu,
    0x109d21ccu, 0x10dda1edu, 0x111e260cu, 0x115ea62du, 0x119f3946u, 0x11dfbd66u, 0x12204147u, 0x1260c567u, 0x12a13988u, 0x12e1bda8u, 0x13224189u, 0x1362c5a9u,
    0x24e18159u, 0x24f18199u, 0x2501c161u, 0x2511c1a1u, 0x24e2035au, 0x24f2039au, 0x25024362u, 0x251243a2u, 0x36e280e9u, 0x36f2c0f1u, 0x37028129u, 0x3712c131u,
    0x36e302eau, 0x36f342f2u, 0x3703032au, 0x37134332u, 0x18a9854bu, 0x18b9858bu, 0x18a9c74cu, 0x18b9c78cu, 0x18ca0553u, 0x18da0593u, 0x18ca4754u, 0x18da4794u,
    0x3aa3846bu, 0x3ab3c473u, 0x3aa4066cu, 0x3ab44674u, 0x3ac384abu, 0x3ad3c4b3u, 0x3ac406acu, 0x3ad446b4u, 0x1c6a88cdu, 0x1c6acaceu, 0x1c7a890du, 0x1c7acb0eu,
    0x1c8b08d5u, 0x1c8b4ad6u, 0x1c9b0915u, 0x1c9b4b16u, 0x2e6b885du, 0x2e6bca5eu, 0x2e7c0865u, 0x2e7c4a66u, 0x2e8b889du, 0x2e8bca9eu, 0x2e9c08a5u, 0x2e9c4aa6u,
    0x3600u, 0x3640u, 0x3681u, 0x36c1u, 0x3702u, 0x3742u, 0x3783u, 0x37c3u, 0x2808u, 0x2849u, 0x2888u, 0x28c9u,
    0x290au, 0x294bu, 0x298au, 0x29cbu, 0x3a04u, 0x3a44u, 0x3a85u, 0x3ac5u, 0x3b06u, 0x3b46u, 0x3b87u, 0x3bc7u,
    0x1810u, 0x1851u, 0x1892u, 0x18d3u, 0x1910u, 0x1951u, 0x1992u, 0x19d3u, 0x2a0cu, 0x2a4du, 0x2a8cu, 0x2acdu,
    0x2b0eu, 0x2b4fu, 0x2b8eu, 0x2bcfu, 0x1614u, 0x1655u, 0x1696u, 0x16d7u, 0x1714u, 0x1755u, 0x1796u, 0x17d7u,
    0x4a33880u, 0x4a3bca0u, 0x4e44080u, 0x4e4c4a0u, 0x5253881u, 0x525bca1u, 0x5664081u, 0x566c4a1u, 0x79f3840u, 0x7dfbc40u, 0x7a04060u, 0x7e0c460u,
    0x8213841u, 0x861bc41u, 0x8224061u, 0x862c461u, 0x4a32882u, 0x4a3aca2u, 0x4e42883u, 0x4e4aca3u, 0x5253082u, 0x525b4a2u, 0x5663083u, 0x566b4a3u,
    0xa9b2802u, 0xadbac02u, 0xb1c2803u, 0xb5cac03u, 0xa9d3022u, 0xaddb422u, 0xb1e3023u, 0xb5eb423u, 0x79f1844u, 0x7df9845u, 0x7a01c64u, 0x7e09c65u,
    0x8212044u, 0x861a045u, 0x8222464u, 0x862a465u, 0xa9b1804u, 0xadb9805u, 0xb1c1c04u, 0xb5c9c05u, 0xa9d2024u, 0xadda025u, 0xb1e2424u, 0xb5ea425u,
    0x4c69536u, 0x4e695b7u, 0x4c6d638u, 0x4e6d6b9u, 0x507153au, 0x52715bbu, 0x507563cu, 0x52756bdu, 0x3499536u, 0x349d5b7u, 0x3699638u, 0x369d6b9u,
    0x38a153au, 0x38a55bbu, 0x3aa163cu, 0x3aa56bdu, 0x6458f3eu, 0x6658fbfu, 0x685cf40u, 0x6a5cfc1u, 0x6461042u, 0x66610c3u, 0x6865044u, 0x6a650c5u,
    0x2cc8f3eu, 0x2cccfbfu, 0x2ed0f40u, 0x2ed4fc1u, 0x30c9042u, 0x30cd0c3u, 0x32d1044u, 0x32d50c5u, 0x5c88946u, 0x5e8c947u, 0x60889c8u, 0x628c9c9u,
    0x5c90a4au, 0x5e94a4bu, 0x6090accu, 0x6294acdu, 0x44b8946u, 0x46bc947u, 0x44c09c8u, 0x46c49c9u, 0x48b8a4au, 0x4abca4bu, 0x48c0accu, 0x4ac4acdu,
    0x20u, 0x28u, 0x41u, 0x49u, 0x42u, 0x4au, 0x83u, 0x8bu, 0x84u, 0x8cu, 0x105u, 0x10du,
    0x106u, 0x10eu, 0x1d0u, 0x1d8u, 0x1b1u, 0x1b9u, 0x1b2u, 0x1bau, 0x173u, 0x17bu, 0x174u, 0x17cu,
    0xf5u, 0xfdu, 0xf6u, 0xfeu, 0x80u, 0x81u, 0x82u, 0x83u, 0xc0u, 0xc1u, 0xc2u, 0xc3u,
    0x84u, 0x85u, 0x86u, 0x87u, 0xc4u, 0xc5u, 0xc6u, 0xc7u, 0x0u, 0x1u, 0x2u, 0x3u,
    0x40u, 0x41u, 0x42u, 0x43u, 0x4u, 0x5u, 0x6u, 0x7u, 0x44u, 0x45u, 0x46u, 0x47u,
    0x88u, 0x89u, 0x8au, 0x8bu, 0xc8u, 0xc9u, 0xcau, 0xcbu, 0x8cu, 0x8du, 0x8eu, 0x8fu,
    0xccu, 0xcdu, 0xceu, 0xcfu, 0x8u, 0x9u, 0xau, 0xbu, 0x48u, 0x49u, 0x4au, 0x4bu,
    0xcu, 0xdu, 0xeu, 0xfu, 0x4cu, 0x4du, 0x4eu, 0x4fu, 0x90u, 0x91u, 0x92u, 0x93u,
    0xd0u, 0xd1u, 0xd2u, 0xd3u, 0x94u, 0x95u, 0x96u, 0x97u, 0xd4u, 0xd5u, 0xd6u, 0xd7u,
    0x10u, 0x11u, 0x12u, 0x13u, 0x50u, 0x51u, 0x52u, 0x53u, 0x14u, 0x15u, 0x16u, 0x17u,
    0x54u, 0x55u, 0x56u, 0x57u, 0x98u, 0x99u, 0x9au, 0x9bu, 0x9cu, 0x9du, 0x9eu, 0x9fu,
    0xd8u, 0xd9u, 0xdau, 0xdbu, 0xdcu, 0xddu, 0xdeu, 0xdfu, 0xa0u, 0xa1u, 0xa2u, 0xa3u,
    0xa4u, 0xa5u, 0xa6u, 0xa7u, 0xe0u, 0xe1u, 0xe2u, 0xe3u, 0xe4u, 0xe5u, 0xe6u, 0xe7u,
    0x18u, 0x19u, 0x1au, 0x1bu, 0x1cu, 0x1du, 0x1eu, 0x1fu, 0x58u, 0x59u, 0x5au, 0x5bu,
    0x5cu, 0x5du, 0x5eu, 0x5fu, 0x20u, 0x21u, 0x22u, 0x23u, 0x24u, 0x25u, 0x26u, 0x27u,
    0x60u, 0x61u, 0x62u, 0x63u, 0x64u, 0x65u, 0x66u, 0x67u, 0x4eu, 0x4fu, 0x50u, 0x51u,
    0x8eu, 0x8fu, 0x90u, 0x91u, 0x6eu, 0x6fu, 0x70u, 0x71u, 0xaeu, 0xafu, 0xb0u, 0xb1u,
    0xcau, 0xcbu, 0x10au, 0x10bu, 0xccu, 0xcdu, 0x10cu, 0x10du, 0xeau, 0xebu, 0x12au, 0x12bu,
    0xecu, 0xedu, 0x12cu, 0x12du, 0x146u, 0x186u, 0x147u, 0x187u, 0x148u, 0x188u, 0x149u, 0x189u,
    0x166u, 0x1a6u, 0x167u, 0x1a7u, 0x168u, 0x1a8u, 0x169u, 0x1a9u, 0xeu, 0xfu, 0x10u, 0x11u,
    0x2eu, 0x2fu, 0x30u, 0x31u, 0xc4u, 0xc5u, 0x104u, 0x105u, 0xe4u, 0xe5u, 0x124u, 0x125u,
    0x142u, 0x182u, 0x143u, 0x183u, 0x162u, 0x1a2u, 0x163u, 0x1a3u, 0xau, 0xbu, 0xcu, 0xdu,
    0x2au, 0x2bu, 0x2cu, 0x2du, 0x44u, 0x45u, 0x84u, 0x85u, 0x64u, 0x65u, 0xa4u, 0xa5u,
    0x140u, 0x180u, 0x141u, 0x181u, 0x160u, 0x1a0u, 0x161u, 0x1a1u, 0x6u, 0x7u, 0x8u, 0x9u,
    0x26u, 0x27u, 0x28u, 0x29u, 0x42u, 0x43u, 0x82u, 0x83u, 0x62u, 0x63u, 0xa2u, 0xa3u,
    0xc0u, 0x100u, 0xc1u, 0x101u, 0xe0u, 0x120u, 0xe1u, 0x121u, 0x38071u, 0x38172u, 0x3c079u, 0x3c17au,
    0x3a080u, 0x3a190u, 0x3e088u, 0x3e198u, 0x58273u, 0x58374u, 0x5c27bu, 0x5c37cu, 0x5a2a0u, 0x5a3b0u, 0x5e2a8u, 0x5e3b8u,
    0xc8ea5u, 0xc8fa6u, 0xc90b5u, 0xc91b6u, 0xcceadu, 0xccfaeu, 0xcd0bdu, 0xcd1beu, 0xcaec3u, 0xcafd3u, 0xcb0c4u, 0xcb1d4u,
    0xceecbu, 0xcefdbu, 0xcf0ccu, 0xcf1dcu, 0xa8a85u, 0xa8b86u, 0xa8c95u, 0xa8d96u, 0xaca8du, 0xacb8eu, 0xacc9du, 0xacd9eu,
    0xaaac1u, 0xaabd1u, 0xaacc2u, 0xaadd2u, 0xaeac9u, 0xaebd9u, 0xaeccau, 0xaeddau, 0x30010u, 0x30120u, 0x34018u, 0x34128u,
    0x32001u, 0x32102u, 0x36009u, 0x3610au, 0x50230u, 0x50340u, 0x54238u, 0x54348u, 0x52203u, 0x52304u, 0x5620bu, 0x5630cu,
    0xc0e53u, 0xc0f63u, 0xc1054u, 0xc1164u, 0xc4e5bu, 0xc4f6bu, 0xc505cu, 0xc516cu, 0xc2e35u, 0xc2f36u, 0xc3045u, 0xc3146u,
    0xc6e3du, 0xc6f3eu, 0xc704du, 0xc714eu, 0xa0a51u, 0xa0b61u, 0xa0c52u, 0xa0d62u, 0xa4a59u, 0xa4b69u, 0xa4c5au, 0xa4d6au,
    0xa2a15u, 0xa2b16u, 0xa2c25u, 0xa2d26u, 0xa6a1du, 0xa6b1eu, 0xa6c2du, 0xa6d2eu, 0x98475u, 0x98576u, 0x9c47du, 0x9c57eu,
    0x9a4c0u, 0x9a5d0u, 0x9e4c8u, 0x9e5d8u, 0x68683u, 0x68784u, 0x68893u, 0x68994u, 0x6c68bu, 0x6c78cu, 0x6c89bu, 0x6c99cu,
    0x6a6a1u, 0x6a7b1u, 0x6a8a2u, 0x6a9b2u, 0x6e6a9u, 0x6e7b9u, 0x6e8aau, 0x6e9bau, 0x90450u, 0x90560u, 0x94458u, 0x94568u,
    0x92405u, 0x92506u, 0x9640du, 0x9650eu, 0x60631u, 0x60741u, 0x60832u, 0x60942u, 0x64639u, 0x64749u, 0x6483au, 0x6494au,
    0x62613u, 0x62714u, 0x62823u, 0x62924u, 0x6661bu, 0x6671cu, 0x6682bu, 0x6692cu,
};

// (ub gamma v).J(abcd) of every ordering from the six W = (ub gamma v).J(0 pi)
template <class R>
__device__ __forceinline__ void from_w(const cx<R> (&W)[6], cx<R> (&A)[24]) {
  A[0] = W[0];  // (0, 1, 2, 3)
  A[1] = W[1];  // (0, 1, 3, 2)
  A[2] = W[2];  // (0, 2, 1, 3)
  A[3] = W[3];  // (0, 2, 3, 1)
  A[4] = W[4];  // (0, 3, 1, 2)
  A[5] = W[5];  // (0, 3, 2, 1)
  A[6] = -W[0] - W[2] - W[3];  // (1, 0, 2, 3)
  A[7] = -W[1] - W[4] - W[5];  // (1, 0, 3, 2)
  A[8] = W[5] + W[3] + W[2];  // (1, 2, 0, 3)
  A[9] = -W[5];  // (1, 2, 3, 0)
  A[10] = W[3] + W[5] + W[4];  // (1, 3, 0, 2)
  A[11] = -W[3];  // (1, 3, 2, 0)
  A[12] = -W[2] - W[0] - W[1];  // (2, 0, 1, 3)
  A[13] = -W[3] - W[5] - W[4];  // (2, 0, 3, 1)
  A[14] = W[4] + W[1] + W[0];  // (2, 1, 0, 3)
  A[15] = -W[4];  // (2, 1, 3, 0)
  A[16] = W[1] + W[4] + W[5];  // (2, 3, 0, 1)
  A[17] = -W[1];  // (2, 3, 1, 0)
  A[18] = -W[4] - W[1] - W[0];  // (3, 0, 1, 2)
  A[19] = -W[5] - W[3] - W[2];  // (3, 0, 2, 1)
  A[20] = W[2] + W[0] + W[1];  // (3, 1, 0, 2)
  A[21] = -W[2];  // (3, 1, 2, 0)
  A[22] = W[0] + W[2] + W[3];  // (3, 2, 0, 1)
  A[23] = -W[0];  // (3, 2, 1, 0)
}

// phase R3, part 0: left.right products of the stored spinors added to the amplitudes
template <class R, class M>
__device__ __forceinline__ void add_r3_0(const M& m, int lt, int lb, int h1, int h2, int h3, cx<R> (&A)[24]) {
  { const cx<R> d = ts_dot<R>(m.w(0 + 4 * lt + 2 * h1 + h2), m.s(10 + 2 * h3 + lb));
    A[0] = A[0] + d; A[14] = A[14] + d; A[6] = A[6] - d; A[12] = A[12] - d; }
  { const cx<R> d = ts_dot<R>(m.w(8 + 4 * lt + 2 * h1 + h2), m.s(10 + 2 * h3 + lb));
    A[2] = A[2] + d; A[8] = A[8] + d; A[6] = A[6] - d; A[12] = A[12] - d; }
  { const cx<R> d = ts_dot<R>(m.t(10 + 2 * h3 + lt), m.w(16 + 4 * lb + 2 * h1 + h2));
    A[18] = A[18] + d; A[23] = A[23] + d; A[20] = A[20] - d; A[22] = A[22] - d; }
  { const cx<R> d = ts_dot<R>(m.t(10 + 2 * h3 + lt), m.w(24 + 4 * lb + 2 * h1 + h2));
    A[19] = A[19] + d; A[21] = A[21] + d; A[20] = A[20] - d; A[22] = A[22] - d; }
  { const cx<R> d = ts_dot<R>(m.w(32 + 4 * lt + 2 * h1 + h3), m.s(6 + 2 * h2 + lb));
    A[1] = A[1] + d; A[20] = A[20] + d; A[7] = A[7] - d; A[18] = A[18] - d; }
  { const cx<R> d = ts_dot<R>(m.w(40 + 4 * lt + 2 * h1 + h3), m.s(6 + 2 * h2 + lb));
    A[4] = A[4] + d; A[10] = A[10] + d; A[7] = A[7] - d; A[18] = A[18] - d; }
  { const cx<R> d = ts_dot<R>(m.t(6 + 2 * h2 + lt), m.w(48 + 4 * lb + 2 * h1 + h3));
    A[12] = A[12] + d; A[17] = A[17] + d; A[14] = A[14] - d; A[16] = A[16] - d; }
  { const cx<R> d = ts_dot<R>(m.t(6 + 2 * h2 + lt), m.w(56 + 4 * lb + 2 * h1 + h3));
    A[13] = A[13] + d; A[15] = A[15] + d; A[14] = A[14] - d; A[16] = A[16] - d; }
  { const cx<R> d = ts_dot<R>(m.w(64 + 4 * lt + 2 * h2 + h3), m.s(2 + 2 * h1 + lb));
    A[3] = A[3] + d; A[22] = A[22] + d; A[13] = A[13] - d; A[19] = A[19] - d; }
  { const cx<R> d = ts_dot<R>(m.w(72 + 4 * lt + 2 * h2 + h3), m.s(2 + 2 * h1 + lb));
    A[5] = A[5] + d; A[16] = A[16] + d; A[13] = A[13] - d; A[19] = A[19] - d; }
  { const cx<R> d = ts_dot<R>(m.t(2 + 2 * h1 + lt), m.w(80 + 4 * lb + 2 * h2 + h3));
    A[6] = A[6] + d; A[11] = A[11] + d; A[8] = A[8] - d; A[10] = A[10] - d; }
  { const cx<R> d = ts_dot<R>(m.t(2 + 2 * h1 + lt), m.w(88 + 4 * lb + 2 * h2 + h3));
    A[7] = A[7] + d; A[9] = A[9] + d; A[8] = A[8] - d; A[10] = A[10] - d; }
}

// phase R3, part 1: left.right products of the stored spinors added to the amplitudes
template <class R, class M>
__device__ __forceinline__ void add_r3_1(const M& m, int lt, int lb, int h1, int h2, int h3, cx<R> (&A)[24]) {
  { const cx<R> d = ts_dot<R>(m.w(0 + 8 * lt + 4 * h1 + 2 * h2 + h3), m.s(lb));
    A[9] = A[9] + d; A[23] = A[23] + d; A[15] = A[15] - d; A[21] = A[21] - d; }
  { const cx<R> d = ts_dot<R>(m.w(16 + 8 * lt + 4 * h1 + 2 * h2 + h3), m.s(lb));
    A[11] = A[11] + d; A[17] = A[17] + d; A[15] = A[15] - d; A[21] = A[21] - d; }
  { const cx<R> d = ts_dot<R>(m.t(lt), m.w(32 + 8 * lb + 4 * h1 + 2 * h2 + h3));
    A[0] = A[0] + d; A[5] = A[5] + d; A[2] = A[2] - d; A[4] = A[4] - d; }
  { const cx<R> d = ts_dot<R>(m.t(lt), m.w(48 + 8 * lb + 4 * h1 + 2 * h2 + h3));
    A[1] = A[1] + d; A[3] = A[3] + d; A[2] = A[2] - d; A[4] = A[4] - d; }
}

// phase Y, part 0: left.right products of the stored spinors added to the amplitudes
template <class R, class M>
__device__ __forceinline__ void add_y_0(const M& m, int lt, int lb, int h1, int h2, int h3, cx<R> (&A)[24]) {
  { const cx<R> d = ts_dot<R>(m.t(lt), m.w(0 + 8 * lb + 4 * h1 + 2 * h2 + h3));
    A[3] = A[3] + d; A[5] = A[5] - d; }
  { const cx<R> d = ts_dot<R>(m.t(lt), m.w(16 + 8 * lb + 4 * h1 + 2 * h2 + h3));
    A[1] = A[1] + d; A[4] = A[4] - d; }
  { const cx<R> d = ts_dot<R>(m.t(lt), m.w(32 + 8 * lb + 4 * h1 + 2 * h2 + h3));
    A[0] = A[0] + d; A[2] = A[2] - d; }
  { const cx<R> d = ts_dot<R>(m.t(2 + 2 * h1 + lt), m.w(48 + 4 * lb + 2 * h2 + h3));
    A[9] = A[9] + d; A[11] = A[11] - d; }
  { const cx<R> d = ts_dot<R>(m.t(2 + 2 * h1 + lt), m.w(56 + 4 * lb + 2 * h2 + h3));
    A[7] = A[7] + d; A[10] = A[10] - d; }
  { const cx<R> d = ts_dot<R>(m.t(2 + 2 * h1 + lt), m.w(64 + 4 * lb + 2 * h2 + h3));
    A[6] = A[6] + d; A[8] = A[8] - d; }
  { const cx<R> d = ts_dot<R>(m.t(6 + 2 * h2 + lt), m.w(72 + 4 * lb + 2 * h1 + h3));
    A[15] = A[15] + d; A[17] = A[17] - d; }
  { const cx<R> d = ts_dot<R>(m.t(6 + 2 * h2 + lt), m.w(80 + 4 * lb + 2 * h1 + h3));
    A[13] = A[13] + d; A[16] = A[16] - d; }
  { const cx<R> d = ts_dot<R>(m.t(6 + 2 * h2 + lt), m.w(88 + 4 * lb + 2 * h1 + h3));
    A[12] = A[12] + d; A[14] = A[14] - d; }
}

// phase Y, part 1: left.right products of the stored spinors added to the amplitudes
template <class R, class M>
__device__ __forceinline__ void add_y_1(const M& m, int lt, int lb, int h1, int h2, int h3, cx<R> (&A)[24]) {
  { const cx<R> d = ts_dot<R>(m.t(10 + 2 * h3 + lt), m.w(0 + 4 * lb + 2 * h1 + h2));
    A[21] = A[21] + d; A[23] = A[23] - d; }
  { const cx<R> d = ts_dot<R>(m.t(10 + 2 * h3 + lt), m.w(8 + 4 * lb + 2 * h1 + h2));
    A[19] = A[19] + d; A[22] = A[22] - d; }
  { const cx<R> d = ts_dot<R>(m.t(10 + 2 * h3 + lt), m.w(16 + 4 * lb + 2 * h1 + h2));
    A[18] = A[18] + d; A[20] = A[20] - d; }
}

// phase X2, part 0: left.right products of the stored spinors added to the amplitudes
template <class R, class M>
__device__ __forceinline__ void add_x2_0(const M& m, int lt, int lb, int h1, int h2, int h3, cx<R> (&A)[24]) {
  A[0] = ts_mac<R>(m.w(0 + 2 * lt + h1), m.w(64 + 4 * lb + 2 * h2 + h3), A[0]);
  A[1] = ts_mac<R>(m.w(0 + 2 * lt + h1), m.w(72 + 4 * lb + 2 * h2 + h3), A[1]);
  A[6] = ts_mac<R>(m.w(4 + 2 * lt + h1), m.w(64 + 4 * lb + 2 * h2 + h3), A[6]);
  A[7] = ts_mac<R>(m.w(4 + 2 * lt + h1), m.w(72 + 4 * lb + 2 * h2 + h3), A[7]);
  A[16] = ts_mac<R>(m.w(16 + 4 * lt + 2 * h2 + h3), m.w(48 + 2 * lb + h1), A[16]);
  A[17] = ts_mac<R>(m.w(16 + 4 * lt + 2 * h2 + h3), m.w(52 + 2 * lb + h1), A[17]);
  A[22] = ts_mac<R>(m.w(24 + 4 * lt + 2 * h2 + h3), m.w(48 + 2 * lb + h1), A[22]);
  A[23] = ts_mac<R>(m.w(24 + 4 * lt + 2 * h2 + h3), m.w(52 + 2 * lb + h1), A[23]);
  A[2] = ts_mac<R>(m.w(8 + 2 * lt + h2), m.w(80 + 4 * lb + 2 * h1 + h3), A[2]);
  A[3] = ts_mac<R>(m.w(8 + 2 * lt + h2), m.w(88 + 4 * lb + 2 * h1 + h3), A[3]);
  A[12] = ts_mac<R>(m.w(12 + 2 * lt + h2), m.w(80 + 4 * lb + 2 * h1 + h3), A[12]);
  A[13] = ts_mac<R>(m.w(12 + 2 * lt + h2), m.w(88 + 4 * lb + 2 * h1 + h3), A[13]);
  A[10] = ts_mac<R>(m.w(32 + 4 * lt + 2 * h1 + h3), m.w(56 + 2 * lb + h2), A[10]);
  A[11] = ts_mac<R>(m.w(32 + 4 * lt + 2 * h1 + h3), m.w(60 + 2 * lb + h2), A[11]);
  A[20] = ts_mac<R>(m.w(40 + 4 * lt + 2 * h1 + h3), m.w(56 + 2 * lb + h2), A[20]);
  A[21] = ts_mac<R>(m.w(40 + 4 * lt + 2 * h1 + h3), m.w(60 + 2 * lb + h2), A[21]);
}

// phase X2, part 1: left.right products of the stored spinors added to the amplitudes
template <class R, class M>
__device__ __forceinline__ void add_x2_1(const M& m, int lt, int lb, int h1, int h2, int h3, cx<R> (&A)[24]) {
  A[4] = ts_mac<R>(m.w(0 + 2 * lt + h3), m.w(32 + 4 * lb + 2 * h1 + h2), A[4]);
  A[5] = ts_mac<R>(m.w(0 + 2 * lt + h3), m.w(40 + 4 * lb + 2 * h1 + h2), A[5]);
  A[18] = ts_mac<R>(m.w(4 + 2 * lt + h3), m.w(32 + 4 * lb + 2 * h1 + h2), A[18]);
  A[19] = ts_mac<R>(m.w(4 + 2 * lt + h3), m.w(40 + 4 * lb + 2 * h1 + h2), A[19]);
  A[8] = ts_mac<R>(m.w(8 + 4 * lt + 2 * h1 + h2), m.w(24 + 2 * lb + h3), A[8]);
  A[9] = ts_mac<R>(m.w(8 + 4 * lt + 2 * h1 + h2), m.w(28 + 2 * lb + h3), A[9]);
  A[14] = ts_mac<R>(m.w(16 + 4 * lt + 2 * h1 + h2), m.w(24 + 2 * lb + h3), A[14]);
  A[15] = ts_mac<R>(m.w(16 + 4 * lt + 2 * h1 + h2), m.w(28 + 2 * lb + h3), A[15]);
}

// sum_st Cint_st Re(A_s^* A_t)
template <class R>
__device__ __forceinline__ R colour_sum(const cx<R> (&A)[24]) {
  R acc[4] = {R(0), R(0), R(0), R(0)};
  const cx<R> b0_0_000 = A[0] + A[6], b0_0_100 = A[0] - A[6];
  const cx<R> b0_0_001 = A[23] + A[22], b0_0_101 = A[23] - A[22];
  const cx<R> b0_0_010 = A[1] + A[7], b0_0_110 = A[1] - A[7];
  const cx<R> b0_0_011 = A[17] + A[16], b0_0_111 = A[17] - A[16];
  const cx<R> b0_1_000 = b0_0_000 + b0_0_010, b0_1_010 = b0_0_000 - b0_0_010;
  const cx<R> b0_1_100 = b0_0_100 + b0_0_110, b0_1_110 = b0_0_100 - b0_0_110;
  const cx<R> b0_1_001 = b0_0_001 + b0_0_011, b0_1_011 = b0_0_001 - b0_0_011;
  const cx<R> b0_1_101 = b0_0_101 + b0_0_111, b0_1_111 = b0_0_101 - b0_0_111;
  const cx<R> b0_2_000 = b0_1_000 + b0_1_001, b0_2_001 = b0_1_000 - b0_1_001;
  const cx<R> b0_2_010 = b0_1_010 + b0_1_011, b0_2_011 = b0_1_010 - b0_1_011;
  const cx<R> b0_2_100 = b0_1_100 + b0_1_101, b0_2_101 = b0_1_100 - b0_1_101;
  const cx<R> b0_2_110 = b0_1_110 + b0_1_111, b0_2_111 = b0_1_110 - b0_1_111;
  const cx<R> b2_0_000 = A[2] + A[8], b2_0_100 = A[2] - A[8];
  const cx<R> b2_0_001 = A[21] + A[19], b2_0_101 = A[21] - A[19];
  const cx<R> b2_0_010 = A[4] + A[10], b2_0_110 = A[4] - A[10];
  const cx<R> b2_0_011 = A[15] + A[13], b2_0_111 = A[15] - A[13];
  const cx<R> b2_1_000 = b2_0_000 + b2_0_010, b2_1_010 = b2_0_000 - b2_0_010;
  const cx<R> b2_1_100 = b2_0_100 + b2_0_110, b2_1_110 = b2_0_100 - b2_0_110;
  const cx<R> b2_1_001 = b2_0_001 + b2_0_011, b2_1_011 = b2_0_001 - b2_0_011;
  const cx<R> b2_1_101 = b2_0_101 + b2_0_111, b2_1_111 = b2_0_101 - b2_0_111;
  const cx<R> b2_2_000 = b2_1_000 + b2_1_001, b2_2_001 = b2_1_000 - b2_1_001;
  const cx<R> b2_2_010 = b2_1_010 + b2_1_011, b2_2_011 = b2_1_010 - b2_1_011;
  const cx<R> b2_2_100 = b2_1_100 + b2_1_101, b2_2_101 = b2_1_100 - b2_1_101;
  const cx<R> b2_2_110 = b2_1_110 + b2_1_111, b2_2_111 = b2_1_110 - b2_1_111;
  const cx<R> b3_0_00 = A[3] + A[9], b3_0_10 = A[3] - A[9];
  const cx<R> b3_0_01 = A[5] + A[11], b3_0_11 = A[5] - A[11];
  const cx<R> b3_1_00 = b3_0_00 + b3_0_01, b3_1_01 = b3_0_00 - b3_0_01;
  const cx<R> b3_1_10 = b3_0_10 + b3_0_11, b3_1_11 = b3_0_10 - b3_0_11;
  const cx<R> b12_0_00 = A[12] + A[14], b12_0_10 = A[12] - A[14];
  const cx<R> b12_0_01 = A[18] + A[20], b12_0_11 = A[18] - A[20];
  const cx<R> b12_1_00 = b12_0_00 + b12_0_01, b12_1_01 = b12_0_00 - b12_0_01;
  const cx<R> b12_1_10 = b12_0_10 + b12_0_11, b12_1_11 = b12_0_10 - b12_0_11;
  {  // characters (1, 1, 1)
    const R r0 = fmadd(R(154.0 / 559.0), b12_1_00.r, fmadd(R(154.0 / 559.0), b3_1_00.r, fmadd(R(-8.0 / 559.0), b2_2_000.r, b0_2_000.r))), i0 = fmadd(R(154.0 / 559.0), b12_1_00.i, fmadd(R(154.0 / 559.0), b3_1_00.i, fmadd(R(-8.0 / 559.0), b2_2_000.i, b0_2_000.i)));
    acc[0] = fmadd(R(559.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[0]);
    const R r1 = fmadd(R(-8.0 / 995.0), b12_1_00.r, fmadd(R(-8.0 / 995.0), b3_1_00.r, b2_2_000.r)), i1 = fmadd(R(-8.0 / 995.0), b12_1_00.i, fmadd(R(-8.0 / 995.0), b3_1_00.i, b2_2_000.i));
    acc[0] = fmadd(R(402975.0 / 4472.0), fmadd(r1, r1, i1 * i1), acc[0]);
    const R r2 = fmadd(R(137.0 / 1132.0), b12_1_00.r, b3_1_00.r), i2 = fmadd(R(137.0 / 1132.0), b12_1_00.i, b3_1_00.i);
    acc[0] = fmadd(R(22923.0 / 199.0), fmadd(r2, r2, i2 * i2), acc[0]);
    const R r3 = b12_1_00.r, i3 = b12_1_00.i;
    acc[0] = fmadd(R(513945.0 / 4528.0), fmadd(r3, r3, i3 * i3), acc[0]);
  }
  {  // characters (1, 1, -1)
    const R r0 = fmadd(R(-2.0 / 5.0), b2_2_001.r, b0_2_001.r), i0 = fmadd(R(-2.0 / 5.0), b2_2_001.i, b0_2_001.i);
    acc[1] = fmadd(R(225.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[1]);
    const R r1 = b2_2_001.r, i1 = b2_2_001.i;
    acc[1] = fmadd(R(729.0 / 8.0), fmadd(r1, r1, i1 * i1), acc[1]);
  }
  {  // characters (1, -1, 1)
    const R r0 = b0_2_010.r, i0 = b0_2_010.i;
    acc[2] = fmadd(R(405.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[2]);
    const R r1 = b2_2_010.r, i1 = b2_2_010.i;
    acc[2] = fmadd(R(405.0 / 8.0), fmadd(r1, r1, i1 * i1), acc[2]);
  }
  {  // characters (1, -1, -1)
    const R r0 = fmadd(R(22.0 / 67.0), b12_1_01.r, fmadd(R(-14.0 / 67.0), b3_1_01.r, fmadd(R(-14.0 / 67.0), b2_2_011.r, b0_2_011.r))), i0 = fmadd(R(22.0 / 67.0), b12_1_01.i, fmadd(R(-14.0 / 67.0), b3_1_01.i, fmadd(R(-14.0 / 67.0), b2_2_011.i, b0_2_011.i)));
    acc[3] = fmadd(R(603.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[3]);
    const R r1 = fmadd(R(-260.0 / 671.0), b12_1_01.r, fmadd(R(-468.0 / 671.0), b3_1_01.r, b2_2_011.r)), i1 = fmadd(R(-260.0 / 671.0), b12_1_01.i, fmadd(R(-468.0 / 671.0), b3_1_01.i, b2_2_011.i));
    acc[3] = fmadd(R(30195.0 / 536.0), fmadd(r1, r1, i1 * i1), acc[3]);
    const R r2 = fmadd(R(-19.0 / 100.0), b12_1_01.r, b3_1_01.r), i2 = fmadd(R(-19.0 / 100.0), b12_1_01.i, b3_1_01.i);
    acc[3] = fmadd(R(91125.0 / 671.0), fmadd(r2, r2, i2 * i2), acc[3]);
    const R r3 = b12_1_01.r, i3 = b12_1_01.i;
    acc[3] = fmadd(R(6561.0 / 80.0), fmadd(r3, r3, i3 * i3), acc[3]);
  }
  {  // characters (-1, 1, 1)
    const R r0 = b0_2_100.r, i0 = b0_2_100.i;
    acc[0] = fmadd(R(405.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[0]);
    const R r1 = b2_2_100.r, i1 = b2_2_100.i;
    acc[0] = fmadd(R(405.0 / 8.0), fmadd(r1, r1, i1 * i1), acc[0]);
  }
  {  // characters (-1, 1, -1)
    const R r0 = fmadd(R(-14.0 / 67.0), b12_1_10.r, fmadd(R(22.0 / 67.0), b3_1_10.r, fmadd(R(-14.0 / 67.0), b2_2_101.r, b0_2_101.r))), i0 = fmadd(R(-14.0 / 67.0), b12_1_10.i, fmadd(R(22.0 / 67.0), b3_1_10.i, fmadd(R(-14.0 / 67.0), b2_2_101.i, b0_2_101.i)));
    acc[1] = fmadd(R(603.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[1]);
    const R r1 = fmadd(R(-468.0 / 671.0), b12_1_10.r, fmadd(R(-260.0 / 671.0), b3_1_10.r, b2_2_101.r)), i1 = fmadd(R(-468.0 / 671.0), b12_1_10.i, fmadd(R(-260.0 / 671.0), b3_1_10.i, b2_2_101.i));
    acc[1] = fmadd(R(30195.0 / 536.0), fmadd(r1, r1, i1 * i1), acc[1]);
    const R r2 = fmadd(R(-19.0 / 64.0), b12_1_10.r, b3_1_10.r), i2 = fmadd(R(-19.0 / 64.0), b12_1_10.i, b3_1_10.i);
    acc[1] = fmadd(R(58320.0 / 671.0), fmadd(r2, r2, i2 * i2), acc[1]);
    const R r3 = b12_1_10.r, i3 = b12_1_10.i;
    acc[1] = fmadd(R(32805.0 / 256.0), fmadd(r3, r3, i3 * i3), acc[1]);
  }
  {  // characters (-1, -1, 1)
    const R r0 = fmadd(R(-2.0 / 7.0), b12_1_11.r, fmadd(R(-2.0 / 7.0), b3_1_11.r, b0_2_110.r)), i0 = fmadd(R(-2.0 / 7.0), b12_1_11.i, fmadd(R(-2.0 / 7.0), b3_1_11.i, b0_2_110.i));
    acc[2] = fmadd(R(567.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[2]);
    const R r1 = b2_2_110.r, i1 = b2_2_110.i;
    acc[2] = fmadd(R(405.0 / 8.0), fmadd(r1, r1, i1 * i1), acc[2]);
    const R r2 = fmadd(R(1.0 / 8.0), b12_1_11.r, b3_1_11.r), i2 = fmadd(R(1.0 / 8.0), b12_1_11.i, b3_1_11.i);
    acc[2] = fmadd(R(810.0 / 7.0), fmadd(r2, r2, i2 * i2), acc[2]);
    const R r3 = b12_1_11.r, i3 = b12_1_11.i;
    acc[2] = fmadd(R(3645.0 / 32.0), fmadd(r3, r3, i3 * i3), acc[2]);
  }
  {  // characters (-1, -1, -1)
    const R r0 = fmadd(R(-2.0 / 9.0), b2_2_111.r, b0_2_111.r), i0 = fmadd(R(-2.0 / 9.0), b2_2_111.i, b0_2_111.i);
    acc[3] = fmadd(R(729.0 / 8.0), fmadd(r0, r0, i0 * i0), acc[3]);
    const R r1 = b2_2_111.r, i1 = b2_2_111.i;
    acc[3] = fmadd(R(405.0 / 8.0), fmadd(r1, r1, i1 * i1), acc[3]);
  }
  return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}
}}  // namespace
