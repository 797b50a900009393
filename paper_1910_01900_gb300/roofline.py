"""Algorithmic work of the operator apply, for roofline accounting.

flops_alg follows the count of the even-odd 1D kernels (Section 4 cites the
even-odd decomposition): one sweep over n^2 lines costs
n^2 (2 (ceil(n/2)^2 + floor(n/2)^2) + 2n) flops and a cell does 12 sweeps;
each interior face, per side and per direction (evaluation and integration)
costs one normal-derivative pass n^2 * 2n plus 4 face sweeps of
n (2 (ceil^2 + floor^2) + 2n) each, about 3 faces per cell with both sides
counted; pointwise 18 flops per cell point and 12 per face point per side;
curved faces add 2 tangential-derivative sweeps per side and direction.  The
evaluation pass gets the forward half, the integration pass the backward half
plus the pointwise work.

Axis-aligned cells take one pass of six line products (csrc/dg_box.cuh), all of
it booked as the integration pass: per line and direction the n x (n + 4)
flux product (even-odd, 2 (hc (hc + 2) + h (h + 2)) + 2n), two end derivatives
(2n each) and 12 for the ends' coefficients, and the mass product
(2 (hc^2 + h^2) + 2n), hc = ceil(n/2), h = floor(n/2).  (Degrees 1 and 2 take
five mass products instead of three, for their rounding; the count is the
smaller number.)

bytes_alg: read u and write v (2 words per DoF); curved cells add the stored
geometry of the paper's scheme (J^-T and JxW per cell point, n^T J^-T and the
area element per face point and side).
"""


def flops_alg(k, curved):
    """(eval, integrate) algorithmic flops per DoF of one operator apply."""
    n = k + 1
    h, hc = n // 2, (n + 1) // 2
    line = 2 * (hc * hc + h * h) + 2 * n
    if not curved:
        flux = 2 * (hc * (hc + 2) + h * (h + 2)) + 2 * n
        return 0.0, 3 * (flux + 2 * 2 * n + 12 + line) / n
    sweep = n * n * line
    face_sweep = n * line
    n3 = n ** 3
    per_side = n * n * 2 * n + 6 * face_sweep
    cell_half = 6 * sweep
    face_half = 3 * 2 * per_side
    point = 18 * n3 + 3 * 2 * 12 * n * n
    return (cell_half + face_half) / n3, (cell_half + face_half + point) / n3


def bytes_alg(k, curved, word):
    """Algorithmic bytes per DoF of one apply (word = 8 for FP64, 4 for FP32)."""
    n = k + 1
    b = 2 * word
    if curved:
        b += 10 * word                                   # J^-T (9) + JxW per cell point
        b += 3 * n * n * 2 * 4 * word / n ** 3           # per face point and side: n^T J^-T (3) + dA
    return b
