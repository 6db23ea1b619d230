// The launch shape of the particle push (pic.cu): plain constants and rules.
#pragma once

namespace hyb {

// 8^3 tiles hold thousands of particles, 4^3 tiles a few hundred: smaller CTAs
// there leave fewer lanes idle in a species' last pass and fewer warps waiting
constexpr int push_threads(int T) { return T == 8 ? 256 : 128; }

// CTAs per SM by shared memory (8^3: 73 KB linear, 114 KB quadratic shape; 4^3: 25 and 42 KB) and registers
constexpr int push_ctas(int T, int order) { return T == 8 ? (order == 1 ? 3 : 2) : (order == 1 ? 6 : 5); }

// CTAs per tile.  A small grid has fewer tiles than the chip holds CTAs (sms x
// push_ctas), and one CTA's walk through its tile then decides: its tiles are split
// over clusters of up to 4 CTAs while all of them are resident at once.  Every CTA
// stages the tile's fields and clears a frame, so what fills the chip is left whole.
// `tiles` counts the tiles of every context that steps at the same time (a batch).
// One step, us, for 1 / 2 / 3 / 4 CTAs a tile on 152 SMs (* this rule's choice):
//   8^3 linear (456 resident)     80 tiles 153 / 122 / 104 / 104*   144 tiles 137 / 117 / 114* / 139
//                                216 tiles 167 / 141* / 173 / 164
//   8^3 quadratic (304)           80 tiles 263 / 214 / 179* / 203   144 tiles 248 / 217* / 281 / 238
//                                216 tiles 342* / 358 / 386 / 337
//   4^3 linear (912)             144 tiles 63 / 58 / 56 / 54*       216 tiles 68 / 65 / 63 / 62*
//                                343 tiles 74 / 70* / 84 / 84       512 tiles 83* / 94 / 99 / 108
//   4^3 quadratic (760)          216 tiles 114 / 105 / 99* / 112    343 tiles 141 / 137* / 143 / 134
//                                512 tiles 177* / 200 / 203 / 193
//   batches of 64-tile 8^3 runs  2 runs 144 / 124 / 124* / 136      4 runs 192* / 208 / 204 / 209
//                                8 runs 335* / 347 / 362 / 367      16 runs 896* / 951 / 1019 / 1023
constexpr int push_split(int T, int order, long long tiles, int sms) {
    const long long fit = tiles > 0 ? (long long)sms * push_ctas(T, order) / tiles : 1;
    return fit < 1 ? 1 : (fit > 4 ? 4 : (int)fit);
}

// warps of the largest push a context of so many tiles launches (in a batch it is no larger)
constexpr long long push_warps(int T, int order, long long tiles, int sms) {
    return tiles * push_split(T, order, tiles, sms) * (push_threads(T) / 32);
}

}  // namespace hyb
