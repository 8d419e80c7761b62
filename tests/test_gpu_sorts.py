"""The re-binning's sorts, which a box chooses by its marker count: one
launch of a thread-block cluster (16 or 8 blocks) up to 2^18 markers, radix
passes of three launches each and two for the bins above.  Both against a
stable sort of the same keys: order, tile ranges, home tiles and flags, with
one, three and five passes; then a box on either side of the line against the
FP64 oracle (bounds as in test_gpu_coupling)."""
import ctypes as C

import numpy as np
import pytest

import synth
from oracle import coupling as OC
from tests.gpu_helpers import make_pair, require_cuda

pytestmark = pytest.mark.gpu

LINE = 1 << 18
# the library's internal launchers (C++ names)
CLUSTER = "_ZN3lbc19launch_sort_clusterExiPKjS1_PjS2_S2_S2_iPiS3_S2_PKiS3_S3_P11CUstream_sti"
RADIX = "_ZN3lbc11launch_sortExiPKjS1_PjS2_S2_S2_PiPKiP11CUstream_st"
BINS = "_ZN3lbc11launch_binsEixPKjS1_PiS2_PjPKiS2_S2_P11CUstream_st"
I, L, P = C.c_int, C.c_longlong, C.c_void_p


def _rebin(form, keys, idx, ntiles, bits, need):
    """ka, va, tile begins and ends, home, (changed, brick count) after the
    re-binning of `keys`, written into the b buffers as the drift does."""
    import torch
    from paper_1406_2211_gb300 import lbc
    lib = lbc.library()
    M = len(keys)
    i32 = dict(dtype=torch.int32, device="cuda")
    ka, va, home = (torch.full((M,), -7, **i32) for _ in range(3))
    kb = torch.as_tensor(keys.astype(np.int32), device="cuda")
    vb = torch.as_tensor(idx.astype(np.int32), device="cuda")
    tb, te = torch.full((ntiles,), -7, **i32), torch.full((ntiles,), -7, **i32)
    hist = torch.zeros(256 * ((M + 2047) // 2048) + 256, **i32)
    words = torch.tensor([need, 0, 5], **i32)          # need, changed, brick count
    p = [P(t.data_ptr()) for t in (ka, va, kb, vb, tb, te, home, hist)]
    w = [P(words.data_ptr() + 4 * k) for k in range(3)]
    s = P(torch.cuda.current_stream().cuda_stream)
    if form == "radix":
        f = getattr(lib, RADIX)
        f.restype, f.argtypes = None, [L, I] + [P] * 9
        f(M, bits, p[2], p[3], p[0], p[1], p[2], p[3], p[7], w[0], s)
        f = getattr(lib, BINS)
        f.restype, f.argtypes = None, [I, L] + [P] * 9
        f(ntiles, M, p[0], p[1], p[4], p[5], p[6], w[0], w[1], w[2], s)
    else:
        f = getattr(lib, CLUSTER)
        f.restype, f.argtypes = None, [L, I] + [P] * 6 + [I] + [P] * 7 + [I]
        f(M, bits, p[2], p[3], p[0], p[1], p[2], p[3], ntiles, p[4], p[5], p[6], w[0], w[1],
          w[2], s, form)
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in (ka, va, tb, te, home, words)]


@pytest.mark.parametrize("form", ["radix", 0, 8])
@pytest.mark.parametrize("M", [1, 1023, 8193, 33333, LINE, LINE + 1])
@pytest.mark.parametrize("ntiles,bits", [(2, 1), (200, 8), (5000, 13), ((1 << 24) + 3, 25)])
def test_sorts_match_a_stable_sort(form, M, ntiles, bits):
    require_cuda()
    rng = np.random.default_rng(M + bits)
    keys = rng.integers(0, ntiles, M)
    keys[: M // 3] = keys[0]                           # a long run of one key
    keys[-1] = ntiles - 1
    idx = rng.permutation(M)
    ka, va, tb, te, home, words = _rebin(form, keys, idx, ntiles, bits, 1)
    order = np.argsort(keys, kind="stable")
    np.testing.assert_array_equal(ka, keys[order])
    np.testing.assert_array_equal(va, idx[order])
    count = np.bincount(keys, minlength=ntiles)
    end = np.cumsum(count)
    np.testing.assert_array_equal(tb, np.where(count == 0, 0, end - count))
    np.testing.assert_array_equal(te, np.where(count == 0, 0, end))
    want = np.empty(M, dtype=np.int64)
    want[idx] = keys
    np.testing.assert_array_equal(home, want)
    assert list(words) == [1, 1, 0]


@pytest.mark.parametrize("form", ["radix", 0, 8])
def test_sorts_that_are_not_needed_write_nothing(form):
    require_cuda()
    rng = np.random.default_rng(1)
    out = _rebin(form, rng.integers(0, 200, 9000), rng.permutation(9000), 200, 8, 0)
    assert all((a == -7).all() for a in out[:5])
    assert list(out[5]) == [0, 0, 5]


@pytest.mark.parametrize("M", [LINE, LINE + 1])
def test_boxes_on_either_side_of_the_line_match_oracle(M):
    require_cuda()
    shape = (60, 64, 68)
    nz, ny, nx = shape
    rng = np.random.default_rng(9)
    pos = rng.uniform(0.0, 1.0, (M, 3)) * [nx, ny, nz]
    parts = dict(pos=pos, vel=0.2 * rng.standard_normal((M, 3)), mass=2.0)
    fbar0 = synth.random_populations(shape, seed=2, amp=1e-3)
    box, sm = make_pair(shape, fbar0, tau=0.8, storage="f64", kind="fc", order=2,
                        stencil="trilinear", gamma=0.2, parts=parts)
    for nsteps in (1, 2, 3):                           # single steps and graph replays
        box.step(nsteps)
        for _ in range(nsteps):
            sm.step()
    p, v, fh = box.get_particles()
    assert np.abs(OC.min_image(p - sm.parts.pos, shape, False)).max() < 1e-11
    assert np.abs(v - sm.parts.vel).max() < 1e-11
    assert np.abs(fh - sm.last_Fh).max() < 1e-11
    assert box.check() == 0
    moved = np.floor(p / 4.0) != np.floor(OC.wrap_positions(pos, shape, False) / 4.0)
    assert moved.any(axis=1).sum() > 1000              # re-binned markers
    box.close()
