"""CPU-side checks of the C interface: the library loads and exports what include/sgs.h declares."""
import ctypes
import os
import re
import subprocess
import sys

import pytest

import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200 import workload as wl
from paper_2306_17266_b200.binding import EXPORTS

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "sgs.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(sgs_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported():
    L = sgs.lib()
    names = declared_functions()
    assert len(names) >= 17
    for n in names:
        assert hasattr(L, n), n
    assert sorted(EXPORTS) == names


def test_split_pointwise_layers_use_the_whole_held_box():
    # persistent execution: whatever the team, the tiles of a layer cover its filters and together take every whole group of 16 filters
    # that the weight buffer holds (hit_ratio and hbm_weight_bytes count the box for every team)
    fn = sgs.lib().sgs_debug_pointwise_tiles
    nt, bn, held = ctypes.c_int(), ctypes.c_int(), (ctypes.c_int * 128)()
    for pixels in (1, 4, 49, 128, 129, 256, 1024, 12544):
        for filters in (8, 16, 24, 40, 120, 256, 264, 960, 1024):
            for team in (1, 2, 4, 8, 16):
                for rows in (0, 16, 48, 256):
                    assert fn(pixels, filters, team, rows, ctypes.byref(nt), ctypes.byref(bn), held, 128) == 0
                    n, b = nt.value, bn.value
                    assert b % 16 == 0 and 16 <= b <= 256 and (n - 1) * b < filters <= n * b
                    got = list(held[:n])
                    assert all(h % 16 == 0 and 0 <= h <= b for h in got)
                    assert sum(got) == min(rows, filters) // 16 * 16, (pixels, filters, team, rows, got)
                    assert all(h == b for h in got[:max(sum(h > 0 for h in got) - 1, 0)])  # a prefix of the layer
    assert fn(0, 16, 1, 0, ctypes.byref(nt), ctypes.byref(bn), held, 128) != 0
    assert fn(49, 16, 3, 0, ctypes.byref(nt), ctypes.byref(bn), held, 128) != 0


def test_struct_sizes_match_the_header():
    # sizes implied by the header's field lists (LP64)
    assert ctypes.sizeof(wl.SubnetCfg) == 4 * (8 + 9 + 64 + 64)
    assert ctypes.sizeof(wl.ArchDesc) == 4 * (2 + 8 + 8 + 3)
    assert ctypes.sizeof(sgs.StreamOpts) == 48  # 2 ints, size_t, 7 ints (padded to 8 bytes)
    assert ctypes.sizeof(sgs.StreamStats) == 8 + 11 * 8 + 8 + 16
    assert ctypes.sizeof(sgs.ConvDesc) == 18 * 4
    assert ctypes.sizeof(sgs.CacheStats) == 8 + 7 * 8 + 4 * 4


def test_null_arguments_are_rejected_without_a_gpu():
    L = sgs.lib()
    assert L.sgs_supernet_load(None, None, 0, 1, 0, None) == sgs.binding.SGS_EINVAL
    assert L.sgs_subnet_validate(None, None) == sgs.binding.SGS_EINVAL
    assert L.sgs_num_layers(None) == 0
    assert L.sgs_last_error(None) == b"null handle"
    assert L.sgs_conv2d_sliced(None, None, None, None, None, None, None, None) == sgs.binding.SGS_EINVAL


@pytest.mark.parametrize("dtype", [sgs.SGS_F32, sgs.SGS_BF16])
@pytest.mark.parametrize("impl", [0, 1, 2])
@pytest.mark.parametrize("N,H,C,k", [(1 << 16, 1 << 8, 4, 1), ((1 << 15) + 1, 1 << 8, 8, 3), (2 ** 31 - 128, 1, 8, 1), (1, 4, 1 << 26, 7)])
def test_convolutions_beyond_32_bit_indexes_are_refused(N, H, C, k, impl, dtype):
    # output pixels or reduction steps from 2^31 - 128 on: refused before any device is touched
    d = sgs.ConvDesc(N=N, H=H, W=H, C=C, K=8, Kmax=8, Cmax=C, R=k, k=k, stride=1, act=0, dtype=dtype, impl=impl)
    p = 1 << 20  # (never read)
    assert sgs.lib().sgs_conv2d_sliced(ctypes.byref(d), p, p, p, p, None, p, None) == sgs.binding.SGS_EUNSUPPORTED


def test_a_failed_host_allocation_is_a_status_without_a_gpu():
    # 65535 members: 8 MB of records that the call cannot have, because the process may not grow
    program = """
import ctypes, resource
import paper_2306_17266_b200 as sgs
from paper_2306_17266_b200.binding import AuxArgs, AuxDesc
n = 65535
L, descs, args = sgs.lib(), (AuxDesc * n)(), (AuxArgs * n)()
assert L.sgs_aux_op(1, descs, args, 0, None) == sgs.binding.SGS_EINVAL
with open("/proc/self/statm") as f:
    size = int(f.read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (size, resource.RLIM_INFINITY))
st = L.sgs_aux_op(n, descs, args, 0, None)
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
print("status", st)
"""
    r = subprocess.run([sys.executable, "-c", program], capture_output=True, text=True, cwd=ROOT, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-1000:])
    assert r.stdout.split() == ["status", str(sgs.binding.SGS_ENOMEM)]
