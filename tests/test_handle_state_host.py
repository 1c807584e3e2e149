"""CPU tests of a handle's host-side state: which key kernel a call takes after builds that succeed and builds that fail half way.  The C
API's object file is linked with launchers and a CUDA runtime that only note what was called, one of which can be told to fail."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2503_24358_b200 import build as sq_build

FAKES = r"""
#include <stdlib.h>
#include <string.h>
static char failing[64], launched[256];
void fake_fail(const char *name) { strcpy(failing, name); }
const char *fake_launched(void) { static char out[256]; strcpy(out, launched); launched[0] = 0; return out; }
static int launch(const char *name)
{
    if (!strcmp(name, failing)) return 5;
    if (launched[0]) strcat(launched, " ");
    strcat(launched, name);
    return 0;
}
static unsigned word;
int fake_capturing = 0;
int cudaMalloc(void **p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return *p ? 0 : 2; }
int cudaFree(void *p) { free(p); return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaGetSymbolAddress(void **p, const void *s) { *p = &word; return 0; }
int cudaStreamIsCapturing(void *st, int *status) { *status = fake_capturing; return 0; }
const char *cudaGetErrorName(int e) { return "error"; }
const char *cudaGetErrorString(int e) { return "error"; }
void **__cudaRegisterFatBinary(void *p) { static void *h; return &h; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    os.makedirs(sq_build.OBJ_DIR, exist_ok=True)
    obj = sq_build._compile("api.cu", False)
    where = tmp_path_factory.mktemp("fake")
    names = [ln.split()[-1] for ln in subprocess.run(["nm", "-u", obj], capture_output=True, text=True, check=True).stdout.splitlines()]
    src = FAKES
    for n in names:
        m = re.match(r"_Z(\d+)(squat_\w+)", n)
        if m:
            name = m.group(2)[:int(m.group(1))]
            src += 'int %s(void) { return launch("%s"); }\n' % (n, name.replace("squat_launch_", ""))
        elif re.match(r"(__)?cuda", n) and not re.search(r"\b%s\(" % n, FAKES):
            src += "int %s(void) { return 0; }\n" % n
    (where / "fakes.c").write_text(src)
    out = str(where / "libapi.so")
    subprocess.run(["gcc", "-w", "-fPIC", "-c", str(where / "fakes.c"), "-o", str(where / "fakes.o")], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", obj, str(where / "fakes.o"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.fake_launched.restype = ctypes.c_char_p
    return lib


class Handle:
    """One KV head; q, k and the outputs are never touched."""

    def __init__(self, lib):
        self.lib, self.h = lib, ctypes.c_void_p()
        lib.fake_fail(b"")
        assert lib.squat_subspace_create(1, 128, ctypes.byref(self.h)) == 0
        raw = np.zeros(4096 + 16, dtype=np.uint8)
        self.raw, self.p = raw, ctypes.c_void_p((raw.ctypes.data + 15) // 16 * 16)

    def build(self, how, rank, block, fail=b""):
        L, ll, dbl = self.lib, ctypes.c_longlong, ctypes.c_double
        L.fake_fail(fail)
        tail = (rank, dbl(1e-3), block)
        power = (self.p, ll(0), 2)
        if how == "svd":
            rc = L.squat_build_subspace(self.h, self.p, 1, 1, 256, ll(256 * 128), ll(128), *tail, None)
        elif how == "svd-gram":
            rc = L.squat_build_subspace_from_gram(self.h, self.p, *tail, None)
        elif how == "power":
            rc = L.squat_build_subspace_power(self.h, self.p, 1, 1, 256, ll(256 * 128), ll(128), *tail, *power, None)
        else:
            rc = L.squat_build_subspace_power_from_gram(self.h, self.p, *tail, *power, None)
        L.fake_fail(b"")
        L.fake_launched()
        return rc

    def key_kernel(self):
        ll = ctypes.c_longlong
        assert self.lib.squat_quantize_keys(self.h, self.p, 1, 1, 1, 32, 128, ll(0), ll(0), ll(128), 2, 32, self.p, self.p, self.p, ll(0), ll(0), None) == 0
        return self.lib.fake_launched().decode()

    def close(self):
        self.lib.squat_subspace_destroy(self.h)


@pytest.mark.parametrize("how", ["svd", "svd-gram", "power", "power-gram"])
def test_key_kernel_follows_the_build(lib, how):
    h = Handle(lib)
    assert h.key_kernel() == "quant_keys"                        # W = 0
    for block, want in ((64, "quant_keys_block"), (32, "quant_keys_block"), (16, "quant_keys"), (64, "quant_keys_block"), (1, "quant_keys")):
        assert h.build(how, 32, block) == 0
        assert h.key_kernel() == want
    assert h.build(how, 0, 64) == 0                              # no subspace: W = 0 on the dense form
    assert h.key_kernel() == "quant_keys"
    assert h.build(how, 4, 1) == 0
    assert h.key_kernel() == ("quant_keys_lowrank" if how.startswith("svd") else "quant_keys")
    h.close()


STEPS = {"svd": ("gram", "eig", "lowrank_tables", "assemble"), "svd-gram": ("eig", "lowrank_tables", "assemble"),
         "power": ("gram", "power", "assemble"), "power-gram": ("power", "assemble")}


@pytest.mark.parametrize("before", [(32, 1), (4, 1), (32, 64)])
@pytest.mark.parametrize("how,fail,after", [(how, fail, after) for how, steps in STEPS.items() for fail in steps for after in ((32, 64), (4, 1), (32, 1))
                                            if fail != "lowrank_tables" or after == (4, 1)])
def test_a_build_that_fails_half_way_leaves_the_dense_form(lib, how, fail, after, before):
    """The image is then the previous one or a part of the next: only the dense kernels read any image as it is."""
    h = Handle(lib)
    assert h.build(how, *before) == 0
    assert h.build(how, *after, fail=fail.encode()) != 0
    assert h.key_kernel() == "quant_keys"
    h.close()


def test_a_captured_call_with_block_updates_holds_the_dense_form_too(lib):
    h = Handle(lib)
    capturing = ctypes.c_int.in_dll(lib, "fake_capturing")
    for block, want in ((64, "quant_keys_block quant_keys"), (1, "quant_keys")):
        assert h.build("svd", 32, block) == 0
        capturing.value = 1
        assert h.key_kernel() == want
        capturing.value = 0
        assert h.key_kernel() == want.split()[0]
    h.close()
