"""What the accuracy tests of the FP32 tensor-core kernels ask, and an emulation of their
arithmetic in 64 bits that shows on a CPU what the question can tell apart."""
import numpy as np

# A chunk of at most 16 steps truncates its accumulator by less than 2^-23 of the sum so
# far at each, on average half of that; a few more roundings of 2^-24 add the orders and
# the chunks up.  The products left out are below 2^-24 of |x w| and of random sign.
# Without the third order the error is about 2^-18.
NORMWISE = 20 * 2.0 ** -24


def rel2(a, ref) -> float:
    """Relative error in the 2-norm."""
    a, ref = np.asarray(a, dtype=np.float64), np.asarray(ref, dtype=np.float64)
    return float(np.linalg.norm((a - ref).ravel()) / np.linalg.norm(ref.ravel()))


def bf16(v):
    """v rounded to BF16 (to nearest even), as FP32."""
    u = np.ascontiguousarray(v, dtype=np.float32).view(np.uint32)
    u = (u + np.uint32(0x7FFF) + ((u >> np.uint32(16)) & np.uint32(1))) & np.uint32(0xFFFF0000)
    return u.view(np.float32)


def split3(v):
    """v = v1 + v2 + v3 exactly, each a BF16 value."""
    v1 = bf16(v)
    v2 = bf16(v - v1)
    v3 = v - v1 - v2
    assert np.array_equal(v3, bf16(v3))
    return v1, v2, v3


def six_products(op, a, b, orders=3):
    """The bilinear `op` of a and b by the products that the kernels keep (the first
    `orders` orders of them), without their rounding."""
    pa, pb = split3(a), split3(b)
    return sum(op(pa[i], pb[o - i]) for o in range(orders) for i in range(o + 1))


def layer(rng, shape, positive=False):
    """Image, bank and gradient with full 24-bit significands."""
    H, W, D, N, fh, fw = shape
    def draw(*s):
        v = rng.uniform(2.0 ** -6, 1.0, s).astype(np.float32)
        return v if positive else v * rng.choice(np.array([-1, 1], np.float32), s)
    return draw(H, W, D), draw(N, fh, fw, D), draw(H - fh + 1, W - fw + 1, N)


FORWARD = [((20, 37, 1, 5, 3, 4), "f32tc:nt=16,r=1,gc=8,jt=4,ru=2"),
           ((33, 40, 4, 4, 8, 8), "f32tc:nt=32,r=8,gc=8,jt=8,ru=4"),
           ((30, 47, 8, 16, 9, 9), "f32tc:nt=64,r=4,gc=8,jt=5,ru=2"),
           ((17, 140, 12, 40, 5, 3), "f32tc:nt=48,r=1,gc=16,jt=3,ru=3"),
           ((23, 26, 16, 64, 7, 7), "f32tc:nt=64,r=1,gc=16,jt=7,ru=2"),
           ((15, 300, 32, 90, 3, 5), "f32tc:nt=48,r=1,gc=32,jt=5,ru=1"),
           ((16, 21, 33, 17, 5, 11), "f32tc:nt=32,r=1,gc=16,jt=6,ru=1"),
           ((24, 29, 64, 160, 1, 1), "f32tc:nt=80,r=1,gc=32,jt=1,ru=1")]
GRADIENT = [((20, 23, 16, 64, 7, 7), "f32tc:nt=64,r=4,gc=32,jt=7,ru=1"),
            ((19, 26, 12, 40, 5, 3), "f32tc:nt=48,r=3,gc=8,jt=3,ru=4"),
            ((24, 31, 5, 7, 3, 4), "f32tc:nt=16,r=1,gc=8,jt=4,ru=2"),
            ((17, 40, 33, 3, 2, 5), "f32tc:nt=48,r=1,gc=8,jt=3,ru=1")]
BANK = [(30, 41, 16, 64, 7, 7), (19, 26, 12, 40, 5, 3), (24, 31, 4, 8, 3, 4), (17, 40, 24, 132, 2, 5),
        (25, 29, 32, 68, 4, 13), (21, 60, 4, 36, 2, 19), (9, 11, 20, 4, 3, 1)]
