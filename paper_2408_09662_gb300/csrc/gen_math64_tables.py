"""Constants of csrc/math64.cuh, from their definitions (mpmath, 60 digits).

    python gen_math64_tables.py > table.txt

Prints the exp constants and its 256-entry table (2^((j - 1/16)/256) in units
of 2^-61) and the sin/cos polynomials (see fit()).  Everything here is derived
from the functions' mathematical definitions.
"""
import mpmath as mp

mp.mp.prec = 400


def hexs(v, n=16):
    return "0x%0*xull" % (n, v)


def exp_constants():
    c = mp.log(2) / 256                       # one table step
    cfix = int(mp.nint(c * mp.mpf(2) ** 90))  # units of 2^-90
    neg = (1 << 96) - cfix                    # -c modulo 2^96
    k0 = int(mp.nint((mp.mpf(0x4B400000) + mp.mpf(1) / 16) * cfix / 2 ** 32)) % (1 << 64)
    print("// exp: -ln2/256 in units of 2^-90 (96-bit two's complement), and the offset")
    print("n0 0x%08xu n1 0x%08xu n2 0x%08xu  k0 %s" % (neg & 0xffffffff, neg >> 32 & 0xffffffff, neg >> 64, hexs(k0)))
    print("scale 256/ln2 = %s" % float(256 / mp.log(2)).hex())
    tab = [int(mp.nint(mp.mpf(2) ** ((mp.mpf(j) - mp.mpf(1) / 16) / 256) * mp.mpf(2) ** 61)) for j in range(256)]
    for i in range(0, 256, 4):
        print("  " + ", ".join(hexs(t) for t in tab[i:i + 4]) + ",")


def fit(f, deg, hi):
    """Polynomial of degree deg in z interpolating f at the Chebyshev nodes of [0, hi]."""
    n = deg + 1
    xs = [hi / 2 + hi / 2 * mp.cos(mp.pi * (2 * i + 1) / (2 * n)) for i in range(n)]
    A = mp.matrix(n, n)
    b = mp.matrix(n, 1)
    for i, x in enumerate(xs):
        for j in range(n):
            A[i, j] = x ** j
        b[i] = f(x)
    co = mp.lu_solve(A, b)
    err = max(abs(sum(co[j] * x ** j for j in range(n)) - f(x)) for x in [hi * k / 400 for k in range(1, 401)])
    return [co[j] for j in range(n)], err


def sincos_constants():
    hi = mp.mpf("0.685")                      # r^2 <= 0.67 with the quadrant estimate's slack
    def fs(z):                                # (1 - sin(r)/r)/z
        r = mp.sqrt(z)
        return (1 - mp.sin(r) / r) / z if z > 0 else mp.mpf(1) / 6
    def fc(z):                                # (1 - cos r)/z
        return (1 - mp.cos(mp.sqrt(z))) / z if z > 0 else mp.mpf(1) / 2
    p = int(mp.nint(mp.pi / 2 * mp.mpf(2) ** 95))
    print("// pi/2 in units of 2^-95: p0 0x%08xu p1 0x%08xu p2 0x%08xu" % (p & 0xffffffff, p >> 32 & 0xffffffff, p >> 64))
    for name, f in (("sin", fs), ("cos", fc)):
        co, err = fit(f, 6, hi)
        print("// %s: fit error %s" % (name, mp.nstr(err, 4)))
        for n, c in enumerate(co):
            v = c * (-1) ** n * mp.mpf(64) ** n          # c1 - z(c2 - z(...)) with y = z/64
            if n < 5:
                print("  a%d %s   // %s" % (n + 1, hexs(int(mp.nint(v * mp.mpf(2) ** 61))), mp.nstr(v, 8)))
            else:
                print("  a%d 0x%08xu   // %s" % (n + 1, int(mp.nint(v * mp.mpf(2) ** 29)), mp.nstr(v, 8)))


if __name__ == "__main__":
    exp_constants()
    sincos_constants()
