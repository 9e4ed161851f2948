"""The gate operand that the tensor-core kernels expand from their parameters: entries at the
edges of the fixed-point grid (+-1, +-i, powers of two, tiny and zero entries), scaled
matrices, every kernel variant, against the product in FP64 on the host."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _edge_matrix(d, scale, seed):
    rng = np.random.default_rng(seed)
    u = rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))
    u /= np.max(np.abs([u.real, u.imag]))
    u[0, 0], u[0, 1], u[1, 0], u[1, 1] = 1.0, -1j, 1j, -1.0
    u[2, 2], u[3, 3], u[2, 3] = 0.5 - 2.0 ** -27, 2.0 ** -26 + 0.25j, 2.0 ** -60
    u[d - 1, : d // 2] = 0.0
    return u * scale


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("n,targets,scale", [
    (11, (0, 1, 2, 3), 1.0), (12, (0, 1, 2, 3, 4), 1.0), (12, (5, 6, 8, 9, 11), 2.0 ** 20),
    (13, (4, 9, 10, 11, 12), 2.0 ** -20), (14, (0, 2, 7, 13), 1.0), (15, (3, 11, 12, 14), 2.0 ** 7),
    (15, (6, 7), 1.0),
])
def test_operand_entries_at_grid_edges(gpu, svlib, dtype, n, targets, scale):
    sv = svlib
    k = len(targets)
    if dtype == "c128" and k == 5:
        targets, k = targets[:4], 4
    u = _edge_matrix(1 << k, scale, n)
    rng = np.random.default_rng(99 + n)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi = (psi / np.linalg.norm(psi)).astype(np.complex64 if dtype == "c64" else np.complex128)
    s = sv.sv_alloc(n, sv.SV_C64 if dtype == "c64" else sv.SV_C128)
    sv.sv_set_policy(s, sv.SV_POLICY_DENSE_ONLY)
    sv.sv_set_state(s, psi)
    sv.sv_apply_gate(s, targets, u)
    got = sv.sv_get_state(s)
    s.free()
    idx = np.arange(1 << n)
    loc = sum(((idx >> t) & 1) << j for j, t in enumerate(targets))
    base = idx & ~sum(1 << t for t in targets)
    ref = np.zeros(1 << n, dtype=np.complex128)
    for c in range(1 << k):
        src = base | sum(((c >> j) & 1) << t for j, t in enumerate(targets))
        ref += u[loc, c] * psi[src].astype(np.complex128)
    amax = float(np.max(np.abs([psi.real, psi.imag])))
    # complex64: each of the 2^(k+1) real products of an output is formed to 2^-23 of
    # (largest amplitude) x (largest entry) -- both grids may be twice their largest value;
    # complex128: 2^-46 of the grids' product in all, and an ulp
    tol = (2.0 ** (k + 1 - 23) if dtype == "c64" else 2.0 ** -44 + 2.0 ** -50) * amax * scale
    assert np.max(np.abs([(got - ref).real, (got - ref).imag])) < tol
