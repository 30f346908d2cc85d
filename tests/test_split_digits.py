"""The digit tables of the split-product kernels (csrc/dg_split.cuh, dg_adj_split.cu):
bounds on the sums that the tensor cores form.

A table entry is cut into six signed ten-bit digits relative to its table's largest
exponent, an operand's digits are at most 512 in magnitude, and level L sums the digit
products i + j = L over the contraction.  Float32 holds such a sum exactly below 2^24
whatever the operand's digits are, if 512 sum_k sum_{j <= L} |e_j(k)| is below it for
every output.  Levels 0 and 1 have to be exact for any operand (a unit of theirs is
2^-18 and 2^-28 of the largest product); levels 2 and 3 of the projection may pass it from p = 4
and 3 on, where the digits of an operand and a table column line up.  The bounds are
pinned here so that another rule or degree does not pass them unnoticed.
"""
import numpy as np
import pytest

DIGITS, LIMIT = 6, 2 ** 24
CASES = [(1, 0), (2, 0), (3, 0), (3, 3), (4, 0), (5, 0)]


@pytest.fixture(scope="module")
def dgmod():
    from paper_1601_07944_gb300 import _build, dg
    _build.build()
    dg.load()
    return dg


def tables(dgmod, oracle_mod, p, ne, rule):
    """name -> [output, input] for every contraction."""
    r, s, w, phi = dgmod.volume_rule(p, rule)
    _, dr, ds = oracle_mod.dubiner(p, r, s)
    h = dgmod.host_tables(p, ne or p + 1)
    face = h["phi_face"].reshape(-1, phi.shape[1])
    lift = (h["edge_w"][None, :, None] * h["phi_face"]).reshape(face.shape)
    Dr, Ds = w[:, None] * dr, w[:, None] * ds
    return {"interpolation": phi, "projection": np.concatenate([Dr, Ds, lift]).T, "traces": face,
            "adjoint r": Dr, "adjoint s": Ds, "adjoint lift": lift, "adjoint interpolation": phi.T,
            "adjoint traces": face.T}


def digits(b):
    """|digit j| of every entry, [DIGITS, output, input]."""
    e = int(np.frexp(np.abs(b).max())[1])
    bias = 512 * sum(1 << (10 * k) for k in range(DIGITS))
    t = [[int(round(float(np.ldexp(x, 59 - e)))) + bias for x in row] for row in b]
    out = np.zeros((DIGITS,) + b.shape, dtype=np.int64)
    for j in range(DIGITS):
        for o, row in enumerate(t):
            for k, u in enumerate(row):
                v = u >> (10 * (DIGITS - 1 - j))
                out[j, o, k] = abs((v if j == 0 else v & 1023) - 512)
    assert out.max() <= 512
    return out


@pytest.mark.parametrize("rule", ["collapsed", "symmetric"])
@pytest.mark.parametrize("p,ne", CASES)
def test_level_sums_are_exact(dgmod, oracle_mod, p, ne, rule):
    for name, b in tables(dgmod, oracle_mod, p, ne, rule).items():
        if name.startswith("adjoint") and p > 3:
            continue                                   # the adjoint's split kernels end at p = 3
        # the range of exponents that the kernels' results are put together in
        assert 2.0 ** -5 <= np.abs(b).max() < 2.0 ** 8, name
        bound = 512 * np.cumsum(digits(b).sum(axis=2), axis=0).max(axis=1)
        assert bound[0] < LIMIT and bound[1] < LIMIT, (name, bound[:2] / LIMIT)
        assert bound[2] < (2 * LIMIT if p >= 4 and name == "projection" else LIMIT), (name, bound[2] / LIMIT)
        assert bound[3] < LIMIT or (p >= 3 and name == "projection"), (name, bound[3] / LIMIT)
        # the largest partial sums still fit the 64-bit recombination
        assert bound[5] < 2 ** 31
