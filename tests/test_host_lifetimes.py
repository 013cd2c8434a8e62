"""Host memory that a copy to the device may still have to read (no GPU: the
library runs on tests/fake_cudart.c, whose copies from pageable memory are done
at the next synchronisation, as late as CUDA allows).  Whatever a call copies
from memory of its own must stand unchanged until then, and a call that returns,
with an error too, must leave no such copy behind."""

import os
import subprocess
import sys

import pytest

from paper_1501_02565_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))

PRELUDE = """
import ctypes, sys
sys.path.insert(0, {root!r})
from paper_1501_02565_gb300 import native
lib = native.load()
fake = ctypes.CDLL({fake!r})
fake.fake_name.restype = ctypes.c_char_p
names = lambda: [fake.fake_name(i).decode() for i in range(fake.fake_launches())]
memory = [(ctypes.c_char * (64 << 20))() for _ in range(4)]
def buf(i):
    return ctypes.c_void_p((ctypes.addressof(memory[i]) + 255) // 256 * 256)
def handle():
    h = ctypes.c_void_p()
    assert lib.epic_interp_create(ctypes.byref(h), 0, None) == 0
    fake.fake_reset()
    return h
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    build.build()
    fake = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    nvcc = build._nvcc()
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I", include, "-I", "/usr/local/cuda/include",
                    "-o", fake, os.path.join(HERE, "fake_cudart.c")], check=True)

    def child(code):
        # (freed and fresh memory is filled; nothing is given back to the system)
        env = dict(os.environ, LD_PRELOAD=fake, MALLOC_PERTURB_="85", MALLOC_TRIM_THRESHOLD_="1000000000")
        p = subprocess.run([sys.executable, "-c", PRELUDE.format(root=os.path.dirname(HERE), fake=fake) + code],
                           env=env, capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, p.stdout + p.stderr

    return child


def test_exact_table_stands_until_it_is_read(run):
    run("""
h = handle()
rc = lib.epic_exact_interp(h, buf(0), buf(1), 70, 130, 40, 8, 1.0, 0, buf(2), None, None, None)
assert rc == 0, rc
assert "single_kernel" in " ".join(names()), names()
assert fake.fake_pending() == 0
assert fake.fake_stale() == 0, "the cap map's table was freed before its copy"
""")


@pytest.mark.parametrize("failing", ["prepare", "dt_kernel", "single_kernel"])
def test_exact_error_leaves_no_copy(run, failing):
    run(f"""
h = handle()
call = lambda: lib.epic_exact_interp(h, buf(0), buf(1), 70, 130, 40, 8, 1.0, 0, buf(2), None, None, None)
assert call() == 0
# the last launch of that kernel fails
at = max(i for i, n in enumerate(names()) if {failing!r} in n)
fake.fake_reset()
fake.fake_fail_launch(at, 701)
assert call() != 0
assert fake.fake_pending() == 0 and fake.fake_stale() == 0
""")


@pytest.mark.parametrize("failing", [0, 1, 2])
def test_no_alloc_error_leaves_no_copy(run, failing):
    run(f"""
fake.fake_fail_launch({failing}, 701)
rc = lib.epic_geodesic_labels_noalloc(buf(0), buf(1), 70, 130, 40, buf(2), buf(3), None)
assert rc == native.EPIC_ERR_CUDA, rc
assert fake.fake_pending() == 0, "a copy from the call's stack is still to be done"
""")
