"""Row scales and tile layouts of the complex128 tensor-core pass: rows whose exponents spread by
exactly what the short cut of the digit split covers and by one more, zero, subnormal and very
large rows, over target layouts (low, high, right below the contiguous part of a tile), against
extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 14
TARGETS = [(0, 5, 6, 9),        # one among the bank bits
           (0, 1, 7, 12),       # two among the bank bits
           (9, 10, 12, 13),     # four high targets
           (8, 9, 11, 13),      # three high, one right below the contiguous part
           (7, 8, 10, 12),      # two high targets
           (8, 9, 10, 12)]      # two right below the contiguous part


def _groups(targets):
    """index[g, c]: the index of member c of group g."""
    free = [b for b in range(N) if b not in targets]
    g = np.arange(1 << len(free))
    base = sum((((g >> i) & 1) << b) for i, b in enumerate(free))
    c = np.arange(16)
    off = sum((((c >> i) & 1) << b) for i, b in enumerate(targets))
    return base[:, None] + off[None, :]


@pytest.mark.parametrize("rows", ["near", "edge", "mixed"])
@pytest.mark.parametrize("targets", TARGETS)
def test_row_scales(gpu, targets, rows):
    import torch
    sv = gpu
    rng = np.random.default_rng(7)
    idx = _groups(targets)
    ng = idx.shape[0]

    def comp():                                  # magnitudes in [1, 2)
        return rng.uniform(1.0, 2.0, (ng, 16)) * rng.choice([-1.0, 1.0], (ng, 16))

    re, im = comp(), comp()
    kind = {"near": np.zeros(ng, int), "edge": rng.integers(0, 2, ng) + 1, "mixed": rng.integers(0, 8, ng)}[rows]
    spread = np.select([kind == 0, kind == 1, kind == 2, kind == 3], [31, 31, 32, 60], 0)
    small = rng.integers(0, 16, ng)
    re[np.arange(ng), small] *= np.exp2(-spread)
    im[kind == 4] = 0.0
    re[kind == 4] = 0.0
    re[(kind == 5)[:, None] & (rng.random((ng, 16)) < 0.5)] = 0.0
    scale = np.select([kind == 6, kind == 7], [2.0 ** -1040, 2.0 ** 1015], 1.0)[:, None]
    re, im = re * scale, im * scale
    psi = np.empty(1 << N, np.complex128)
    psi[idx] = re + 1j * im
    u = (rng.uniform(-1, 1, (16, 16)) + 1j * rng.uniform(-1, 1, (16, 16))) / 4

    s = sv.sv_alloc(N, 1, stream=torch.cuda.current_stream())
    sv.sv_set_state(s, psi)
    sv.sv_apply_gate(s, targets, u)
    got = sv.sv_get_state(s)[idx]
    s.free()

    ul, al = u.astype(np.clongdouble), psi[idx].astype(np.clongdouble)
    want = al @ ul.T
    # a row of components up to M and entries up to R: rounding both to the grid 32 (2^-53 + 2^-53)
    # M R, the dropped levels 5 x 32 x 4 x 2^-54 (1 + 2^-8) M R and what follows them, the rounding of
    # level 5 in its accumulator 12 x 4 x 2^-52 M R, the final rounding 32 x 2^-53 M R: below 2^-44 M R.
    # The grid's exponent field is at least 1, so M counts as at least 2^-1022.
    m = np.maximum(np.abs(al.real), np.abs(al.imag)).max(axis=1, keepdims=True)
    m = np.maximum(m, np.longdouble(2.0 ** -1022))
    r = max(np.abs(u.real).max(), np.abs(u.imag).max())
    bound = np.longdouble(2.0 ** -44) * m * r + np.longdouble(2.0 ** -1074)
    assert np.all(np.abs(got.real - want.real) <= bound)
    assert np.all(np.abs(got.imag - want.imag) <= bound)
