"""sv_topk at the widths where its selection changes (outcomes, sub-chunks, chunks, groups of
chunks, wider chunks), with planted outcomes, ties across every chunk boundary, NaN and zero
states: the exact (p descending, index ascending) list."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _planted(n, rng):
    """Indices: chunk edges, runs of neighbours, random ones; few distinct values, so that most
    are ties and the 64th place is one."""
    N = 1 << n
    idx = {0, N - 1, N // 2, N // 2 - 1}
    for step in (16, 64, 1024, 4096, 65536):
        idx |= {i for i in (step, step - 1, N - step, N - step - 1) if 0 <= i < N}
    base = int(rng.integers(0, N))
    idx |= {(base + j) % N for j in range(40)}
    idx |= {int(i) for i in rng.integers(0, N, 60)}
    idx = np.array(sorted(idx), dtype=np.int64)
    return idx, rng.choice(np.array([0.5, 0.25, 0.125, 0.0625]), size=idx.size)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("n", [1, 5, 6, 7, 10, 12, 13, 16, 17, 22, 23, 24, 29, 30, 31])
def test_topk_planted(gpu, dtype, n):
    sv = gpu
    import torch
    if n > 29 and dtype == 1:
        pytest.skip("the same widths of chunk as complex64")
    rng = np.random.default_rng(40 + n)
    buf = torch.full((1 << n, 2), 1e-6, device="cuda", dtype=torch.float32 if dtype == 0 else torch.float64)
    idx, amp = _planted(n, rng)
    at = torch.from_numpy(idx).cuda()
    buf[at, 0] = torch.from_numpy(amp).cuda().to(buf.dtype)
    buf[at, 1] = 0.0
    torch.cuda.synchronize()
    s = sv.sv_alloc(n, dtype, dev_buf=torch.empty(1 << n, device="cuda", dtype=torch.complex64 if dtype == 0
                                                  else torch.complex128))
    sv.sv_set_state(s, buf)
    gi, gp = sv.sv_topk(s, 64)
    s.free()
    low = float(np.float32(1e-6) ** 2 * 2) if dtype == 0 else 2e-12
    order = np.lexsort((idx, -amp))
    want_i, want_p = idx[order], amp[order] ** 2
    if want_i.size < 64:                                # the rest in index order
        rest = np.setdiff1d(np.arange(min(1 << n, 4096)), idx)[:64 - want_i.size]
        want_i = np.concatenate([want_i, rest])
        want_p = np.concatenate([want_p, np.full(rest.size, low)])
    m = min(64, 1 << n)
    assert np.array_equal(gi.astype(np.int64), want_i[:m])
    assert np.allclose(gp, want_p[:m], rtol=1e-6, atol=0.0)
    del buf
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [12, 14, 18])
def test_topk_uniform_zero_and_nan(gpu, n):
    sv = gpu
    for dtype in (0, 1):
        s = sv.sv_alloc(n, dtype)
        sv.sv_set_zero(s)
        gi, gp = sv.sv_topk(s, 64)
        assert np.array_equal(gi, np.arange(64)) and not gp.any()
        psi = np.full(1 << n, 0.5, dtype=np.complex64 if dtype == 0 else np.complex128)
        psi[5] = np.nan
        sv.sv_set_state(s, psi)
        gi, gp = sv.sv_topk(s, 64)
        if dtype == 0:                                  # not listed
            assert np.array_equal(gi, np.setdiff1d(np.arange(65), [5])) and np.all(gp == 0.25)
        else:                                           # first
            assert gi[0] == 5 and np.array_equal(gi[1:], np.setdiff1d(np.arange(64), [5]))
        s.free()
