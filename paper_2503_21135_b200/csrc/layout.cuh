// Where a logical code lives inside a packed atom (16 rows x 128 k of one bit-width), and the
// power-of-two scale the activations carry so that codes can be used where they lie.
//
// The layout is "fragment native" for mma.sync m16n8k16 with the weights as the A operand: lane
// (gid = lane/4, tid4 = lane%4) of a warp owns rows gid and gid+8 of the atom and, in MMA step
// s (k in [16s, 16s+16)), the four consecutive k = 16s + 4*tid4 + {0,1,2,3}.  A-fragment register
// ri = rowhalf + 2*h holds (row gid + 8*rowhalf, k = 16s + 4*tid4 + 2*h + {0,1}) as an fp16 pair.
//
// A code is NOT shifted down to bit 0 before use.  A field of width b at bit offset o (o + b <= 10)
// of a 16-bit half, masked in place, is the fp16 SUBNORMAL q * 2^(o-24); the matching activation is
// stored pre-multiplied by 2^(bias - o), so the product is q * x * 2^(bias-24) whatever o is, and one
// AND per register pair (plus one shift per 32-bit word to bring the upper fields below bit 10)
// replaces shift + mask + or.  The offset o of a k must not depend on the row (the B fragment is
// shared by all rows), so the two row halves live in different words:
//
//   2-bit: atom = [32 lanes x 16 B]; word jh*2 + rowhalf (jh = s/4, the 64-k half chunk);
//          field phi = 2*(s%4) + h at bits [2phi, 2phi+2) (even k) and +16 (odd k);
//          phi <= 4 used in place (o = 2phi), phi >= 5 after >> 10 (o = 2phi - 10).
//   3-bit: three words per row half hold the sixteen fields of a lane: W0 and W1 (jh = 0, 1; [32 lanes x 16 B], word
//          jh*2 + rowhalf) and W2 ([32 lanes x 8 B], word = rowhalf), each with four whole fields at bits 0, 4, 8 and 12 of its
//          16-bit halves and single bits at 3, 7, 11 and 15.  o = 2(phi % 4).
//          phi = 0, 2 at bits 0, 4 of W(jh), in place; phi = 1, 3 at bits 8, 12 after >> 6; phi = 4, 6 of jh = 0 at bits 0, 4
//          of W2, in place, of jh = 1 at bits 8, 12 after >> 8.  phi = 5, 7 (o = 2, 6) are spread over single bits that lie
//          four apart as the fields do, so one shift of a word serves both: bit 0 of the code at bits 11, 15 of W(jh) (>> 9),
//          bit 1 at 3, 7 of W(jh), in place, bit 2 in W2 at 3, 7 (jh = 0) or, after >> 8, 11, 15 (jh = 1), << 1.  54 logical
//          instructions an atom and lane (32 of them the masks that every width has); a 2-bit and a 1-bit plane take 76:
//          1, 12, 24, 32 and 100 tokens of a layer with two 3-bit experts of eight (4096 x 14336, mean of eight routers) 65,
//          167, 187, 201 and 261 us a pass, as planes 68, 170, 188, 206 and 269.  Fields packed three bits apart (o = 0, 3, 6;
//          46 instructions) take 63, 165, 184, 199 and 255, but the tensor cores align the products of an MMA by the operands'
//          exponents, and with o = 0 in three steps of four instead of two a sum over 14336 hidden activations from 0.02 to 2
//          is twice as far from its value in 64 bits (2-norm 2.7e-5 -> 5.0e-5).
//   4-bit: atom = 2 planes (= half chunks) x [32 lanes x 16 B]; word rowhalf*2 + (s%4)/2;
//          nibble phi = 2*(s%2) + h at bits [4phi, 4phi+4) (even k) and +16 (odd k);
//          phi <= 1 in place (o = 4phi), phi >= 2 after >> 8 (o = 4phi - 8): o = 4h.
//   8-bit: atom = 4 planes x [32 lanes x 16 B]; plane s/2, word 2*(s%2) + h; byte 2*rowhalf + odd
//          (expanded with one byte permute per pair; o = 0).
//   6-bit: low four bits stored exactly as a 4-bit atom (1024 B, o = 4h), then a 2-bit plane [32 lanes x 16 B] with
//          the high two bits, word jh*2 + rowhalf as in a 2-bit atom.  The high bits of step s4 = s%4, pair h must
//          land on bits [o+4, o+6) = 4 + 4h (even k; +16 odd k) of a copy of that word: the copies are the word
//          itself (s4 = 0), the word >> 2 (s4 = 1), the word with the bytes of each half swapped (s4 = 2) and that
//          one >> 2 (s4 = 3), so the field is stored at bit (4 + 4h + {0, 2, 8, 10}[s4]) % 16 of its half.  The
//          eight fields of a half tile its sixteen bits exactly.
#pragma once
#include <stdint.h>

namespace dyn {

struct CodeLoc {
    int byte_off;  // byte offset of the 32-bit word inside the atom
    int shift;     // bit position of the field inside that word
    int width;     // field width
    int lo;        // bit of the code that the field begins with
};

// Number of parts that the code of input index kk lies in.
__host__ __device__ inline int code_parts(int bits, int kk) {
    return bits == 6 ? 2 : (bits == 3 && (kk & 0x22) == 0x22 ? 3 : 1);
}

// r: row in atom (0..15), kk: k in chunk (0..127).  For 6-bit, part 0 = low four bits, part 1 = high two bits; for 3-bit,
// part = the bit of a code that is spread over three words.
__host__ __device__ inline CodeLoc code_loc(int bits, int r, int kk, int part) {
    const int gid = r & 7, rowhalf = r >> 3;
    const int s = kk >> 4, kq = kk & 15;
    const int tid4 = kq >> 2, h = (kq >> 1) & 1, odd = kq & 1;
    const int lane = gid * 4 + tid4;
    const int jh = s >> 2, s4 = s & 3;
    CodeLoc L;
    L.lo = 0;
    if (bits == 6 && part == 1) {  // 6-bit, high two bits
        const int rot = (s4 & 1) * 2 + (s4 >> 1) * 8;
        L.byte_off = 1024 + lane * 16 + (jh * 2 + rowhalf) * 4;
        L.shift = ((4 + 4 * h + rot) & 15) + 16 * odd;
        L.width = 2;
        L.lo = 4;
    } else if (bits == 4 || bits == 6) {
        const int phi = 2 * (s4 & 1) + h;
        L.byte_off = jh * 512 + lane * 16 + (rowhalf * 2 + (s4 >> 1)) * 4;
        L.shift = 4 * phi + 16 * odd;
        L.width = 4;
    } else if (bits == 8) {
        L.byte_off = (s >> 1) * 512 + lane * 16 + (2 * (s & 1) + h) * 4;
        L.shift = 8 * (2 * rowhalf + odd);
        L.width = 8;
    } else if (bits == 2) {
        const int phi = 2 * s4 + h;
        L.byte_off = lane * 16 + (jh * 2 + rowhalf) * 4;
        L.shift = 2 * phi + 16 * odd;
        L.width = 2;
    } else {  // 3-bit
        const int phi = 2 * s4 + h;
        const bool spread = (phi & 5) == 5;
        const int w = (spread ? part < 2 : phi < 4) ? jh : 2;
        L.byte_off = (w == 2 ? 512 + lane * 8 : lane * 16 + 8 * w) + rowhalf * 4;
        L.shift = 16 * odd + 4 * (phi >> 1 & 1) +
                  (spread ? 3 + 8 * (part == 2 ? jh : 1 - part) : 8 * (phi < 4 ? phi & 1 : jh));
        L.width = spread ? 1 : 3;
        L.lo = spread ? part : 0;
    }
    return L;
}

// Activations feeding a matrix packed at `bits` are stored multiplied by 2^x_scale_exp(bits, k):
// bias - o(k), with o the in-place bit offset of the code of input index k (periodic in k mod 64).
__host__ __device__ inline int x_scale_bias(int bits) {
    return bits == 2 ? 4 : (bits == 3 ? 3 : ((bits == 4 || bits == 6) ? 2 : 0));
}
__host__ __device__ inline int x_scale_exp(int bits, int k) {
    const int s4 = (k >> 4) & 3, h = (k >> 1) & 1;
    const int phi = 2 * s4 + h;
    int o = 0;
    if (bits == 2) o = phi <= 4 ? 2 * phi : 2 * phi - 10;
    else if (bits == 3) o = 2 * (phi & 3);
    else if (bits == 4 || bits == 6) o = 4 * h;
    return x_scale_bias(bits) - o;
}

}  // namespace dyn
