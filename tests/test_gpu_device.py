"""GPU: device functions by themselves (device_probe.cu, built here with nvcc)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1109_0286_gb300 import _build  # noqa: E402


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("probe") / "probe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_probe.cu")
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    lib.probe_reduce.argtypes = [ctypes.c_int] * 5 + [ctypes.c_void_p] * 5
    lib.probe_normals.argtypes = [ctypes.c_void_p] * 2 + [ctypes.c_int] + [ctypes.c_void_p] * 2
    return lib


TYPES = {"fp32": 0, "mixed": 1, "fp64": 2}


@pytest.mark.parametrize("power", [0, 99, (0, 99)])
@pytest.mark.parametrize("ncta,nthr,seg,shares", [
    (1, 8, 8, 1), (5, 24, 8, 1), (16, 32, 16, 1), (16, 32, 32, 1), (3, 96, 96, 1), (3, 96, 96, 3),
    (2, 256, 64, 1), (2, 256, 64, 2), (2, 256, 256, 1), (2, 256, 256, 4), (2, 192, 192, 2),
    (1, 512, 128, 1), (1, 512, 512, 1), (1, 512, 512, 8)])
@pytest.mark.parametrize("mode", ["fp32", "mixed", "fp64"])
def test_sums_are_as_close_as_in_64_bits(probe, mode, ncta, nthr, seg, shares, power):
    """Thread sums of 44 bits whose totals fit 53 bits: FP64 additions give the
    exact sum in every order, and so must the reduction.  With a power, 28 bits
    times 2^99, in all warps or every other one: no thread sum exceeds FP32's
    range, but the partials of a CTA do."""
    n = ncta * nthr
    rng = np.random.default_rng(nthr + seg)
    v = rng.integers(2 ** 43, 2 ** 44, n)
    if power == (0, 99):
        big = (np.arange(n) // 32) % 2 == 1
        if not big.any():
            pytest.skip("one warp")
        v, e = np.where(big, v >> 16, 0), np.where(big, 99, 0)
    else:
        v, e = (v if power == 0 else v >> 16), np.full(n, power)
    if mode == "fp64":
        e = np.zeros(n, int)
    v = v * np.where(rng.random(n) < 0.25, -1, 1)
    hi = v.astype(np.float32)
    lo = (v - hi.astype(np.int64)).astype(np.float64)
    exact = sum(int(a) << int(b) for a, b in zip(v, e))
    assert abs(exact) < 2 ** (53 + int(e.max()))
    total = np.abs(np.ldexp(v.astype(np.float64), e)).sum()
    dev = lambda a: torch.from_numpy(np.ldexp(a.astype(np.float64), e)).cuda()   # noqa: E731
    h, l = dev(hi), dev(lo)
    assert float(h.abs().max()) < 3.4e38
    assert power == 0 or mode == "fp64" or n < 64 or total > 3.4e38
    partial = torch.zeros(n // seg + 32, dtype=torch.float64, device="cuda")
    state = torch.zeros(probe.probe_state_bytes(), dtype=torch.uint8, device="cuda")
    for _ in range(2):   # the second run finds the ticket reset
        assert probe.probe_reduce(TYPES[mode], ncta, nthr, seg, shares, h.data_ptr(), l.data_ptr(),
                                  partial.data_ptr(), state.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream) == 0
        o = probe.probe_bb_offset()
        bb = state.cpu()[o:o + 8].view(torch.float64).item()
        assert bb == float(exact)


def test_normals_at_the_edges(probe):
    """Box-Muller on the tables against extended precision: smallest and largest
    uniforms, both sides of every power of two, every interval of the logarithm
    and every sector of the angle, and random words.  Bound: half an ulp each for
    the argument's two additions and the root (2^-52 of the radius in all, with the
    halving of the root), 2^-53 for the unit vector and 2^-53 for the product:
    2^-51 of the radius."""
    rng = np.random.default_rng(5)
    u1, u2 = [0, 1, 2, 2 ** 52 - 1, 2 ** 52 - 2], [0, 1, 2 ** 52 - 1]   # u = (k + 1/2) 2^-52
    for p in range(52):
        u1 += [2 ** p - 1, 2 ** p, 2 ** p + 1]
    for i in range(256):
        for p in (51, 50, 40, 8):   # first value of interval i at that power of two
            k = 2 ** p + (i << p >> 8)
            u1 += [k - 1, k, k + 1]
        k = i << 44
        u2 += [abs(k - 1), k, k + 1, k + 2 ** 43 - 1, k + 2 ** 43, k + 2 ** 43 + 1]
    u1, u2 = np.array(u1, np.int64), np.array(u2, np.int64)
    n = 60000
    a = np.concatenate([u1, rng.integers(0, 2 ** 52, n)])
    b = np.concatenate([rng.choice(u2, u1.size), rng.integers(0, 2 ** 52, n)])
    a = np.concatenate([a, rng.integers(0, 2 ** 52, u2.size)])
    b = np.concatenate([b, u2])
    assert a.min() >= 0 and max(a.max(), b.max()) < 2 ** 52
    low = rng.integers(0, 64, (a.size, 4))   # the six bits of a word that are not used
    words = np.stack([a >> 26, a & (2 ** 26 - 1), b >> 26, b & (2 ** 26 - 1)], 1) << 6 | low
    dw = torch.from_numpy(words.astype(np.uint32).view(np.int32)).cuda()
    tab = torch.empty(probe.probe_noise_entries(), dtype=torch.float64, device="cuda")
    out = torch.empty((a.size, 2), dtype=torch.float64, device="cuda")
    assert probe.probe_normals(tab.data_ptr(), dw.data_ptr(), a.size, out.data_ptr(),
                               torch.cuda.current_stream().cuda_stream) == 0
    L = np.longdouble
    assert np.finfo(L).nmant >= 63
    v = lambda k: (k.astype(L) + L(0.5)) / L(2 ** 52)   # noqa: E731
    rad = np.sqrt(L(-2) * np.where(a < 2 ** 51, np.log(v(a)), np.log1p(v(a) - L(1))))
    th = L(2) * np.arccos(L(-1)) * v(b)
    err = np.abs(out.cpu().numpy().astype(L) - np.stack([rad * np.cos(th), rad * np.sin(th)], 1))
    assert np.max(err / rad[:, None]) <= 2.0 ** -51
