"""State that a scan leaves for the next one: both species' codecs on two streams,
then steps on the same handle; scans whose blocks overlapped on one state, or that
waited in vain for a tile, after which the next one is right all the same."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from oracle import codec
from tests.helpers import lib_codes_from_oracle, oracle_codes_from_lib, records
from tests.test_gpu_kick import _check, _pm, _species

pytestmark = pytest.mark.gpu

ST_TIMEOUT = 8
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_species_on_two_streams_then_steps():
    n, counts = 256, (60001, 140001)
    rng = np.random.default_rng(5)
    codes = [_species(rng, n, counts[s], 2.0, 16) for s in range(2)]
    pm = _pm(n, counts, 16)
    dev = [lib_codes_from_oracle(c) for c in codes]
    want = [codec.decompress(c, n) for c in codes]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(8):
        got, back = [None, None], [None, None]
        for s, st in enumerate(streams):
            with torch.cuda.stream(st):
                got[s] = pm.decompress(s, dev[s])
                back[s] = pm.compress(s, *got[s])
        torch.cuda.synchronize()
        pm.check()
        for s in range(2):
            for g, w in zip(got[s], want[s]):
                assert torch.equal(g.cpu(), torch.from_numpy(w))
            # (v_max is taken anew, from bin centres, so only cells and positions come back as they were)
            b = oracle_codes_from_lib(back[s], n // 4, 16)
            np.testing.assert_array_equal(b.cnt, codes[s].cnt)
            np.testing.assert_array_equal(records(b)[:, :4], records(codes[s])[:, :4])
    for _ in range(3):
        _check(pm, codes, n, 16)


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1611_01545_gb300 import build as b
    so = str(tmp_path_factory.mktemp("probe") / "scan_probe.so")
    subprocess.run([b.nvcc(), *b.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared",
                    "-cudart", "static", "-I", b.INCLUDE, "-I", b.CSRC, "-o", so,
                    os.path.join(ROOT, "tests", "scan_probe.cu")], check=True)
    lib = ctypes.CDLL(so)
    lib.scan_probe_state.restype = ctypes.c_longlong
    lib.scan_probe_state.argtypes = [ctypes.c_longlong]
    lib.scan_probe.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_longlong] * 2 + [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.c_int,
                                                                                                   ctypes.c_longlong]
    return lib


# one tile, two with a remainder, and more tiles than a warp looks back over at once
@pytest.mark.parametrize("ncell", [700, 4095, 90000])
def test_scans_that_overlapped_spoil_no_later_one(probe, ncell):
    g = torch.Generator(device="cuda").manual_seed(ncell)
    cnt = torch.randint(0, 200, (ncell,), generator=g, device="cuda", dtype=torch.uint8)
    want = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), cnt.long().cumsum(0)])
    vmax = torch.ones(1, device="cuda")
    none = torch.zeros(4, dtype=torch.int32, device="cuda")
    state = torch.zeros(probe.scan_probe_state(ncell) // 8, dtype=torch.int64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()

    def scan(launches, skip=0, limit=0):
        off = torch.full((ncell + 1,), -1, dtype=torch.int64, device="cuda")
        status.zero_()
        torch.cuda.synchronize()
        rc = probe.scan_probe(cnt.data_ptr(), vmax.data_ptr(), none.data_ptr(), none.data_ptr(), ncell, int(want[-1]),
                              off.data_ptr(), state.data_ptr(), status.data_ptr(), launches, skip, limit)
        assert rc == 0
        return off, int(status)

    for launches in (1, 2, 3, 2):
        for _ in range(20):
            scan(launches, limit=2000000)      # of those that overlap only the end is asked for
        off, bad = scan(1)
        assert bad == 0
        assert torch.equal(off, want)
    # a first tile that publishes nothing: the others give up after 0.1 ms and say so
    if ncell > 2048:
        assert scan(1, skip=1, limit=200000)[1] & ST_TIMEOUT
        off, bad = scan(1)
        assert bad == 0
        assert torch.equal(off, want)
