// Node shapes with exactly unrolled tensor kernels (tensor_fixed.cu). Plain
// C++, also compiled by the host tests.
#pragma once

namespace ckks {

// Terms of the children, largest first (c = 0: two children).
struct TensorShape {
    int a, b, c;
};

// Two children of 4..7 terms except 6 and 4 (children of 5 and 3 inputs: no
// tree within the depth rule has that node for k <= 16), three of 4 or 5 terms;
// then the small shapes (every child at most 3 terms). A shape's code is its
// position.
constexpr TensorShape kTensorShapes[] = {
    {4, 4, 0}, {5, 4, 0}, {5, 5, 0}, {6, 5, 0}, {6, 6, 0}, {7, 4, 0}, {7, 5, 0}, {7, 6, 0}, {7, 7, 0},
    {4, 4, 4}, {5, 4, 4}, {5, 5, 4}, {5, 5, 5},
    {2, 2, 0}, {3, 3, 0}, {2, 2, 2}, {3, 3, 2},
};
constexpr int kTensorShapeCount = sizeof(kTensorShapes) / sizeof(kTensorShapes[0]);
// First small shape: those only in contexts whose products run on limbs
// (limbs30).
constexpr int kTensorSmallCode = 13;

// Code of a node of m children with a >= b (>= c) terms, -1 when no kernel is
// compiled for exactly these terms.
inline int tensor_fixed_code(int m, int a, int b, int c) {
    if (m < 2 || m > 3) return -1;
    if (m == 2) c = 0;
    else if (c < 1) return -1;
    for (int i = 0; i < kTensorShapeCount; ++i)
        if (kTensorShapes[i].a == a && kTensorShapes[i].b == b && kTensorShapes[i].c == c) return i;
    return -1;
}

}  // namespace ckks
