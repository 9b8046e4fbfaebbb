"""Which x-chunks the FWI gradient's passes may time (csrc/fd_grad_chunks.h,
compiled here for the host): the options' chunk alone where they name one, the
step kernel's alone with tuning off, else that one and candidates of 1 to N_x
planes, each once."""
import ctypes
import shutil
import subprocess

import pytest

from paper_1912_00695_gb300 import build

SRC = """#include "fd_grad_chunks.h"
extern "C" int chunks(int Nx, long long tiles, int sms, int forced, int untimed, int tune, int *out) {
    const std::vector<int> v = fdgb::grad_chunks(Nx, tiles, sms, forced, untimed, tune != 0);
    for (size_t i = 0; i < v.size(); ++i) out[i] = v[i];
    return int(v.size());
}
"""


@pytest.fixture(scope="module")
def chunks(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("chunks")
    (d / "c.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{build.CSRC}",
                    str(d / "c.cpp"), "-o", str(d / "c.so")], check=True)
    fn = ctypes.CDLL(str(d / "c.so")).chunks
    fn.argtypes = [ctypes.c_int, ctypes.c_longlong] + [ctypes.c_int] * 4 + [ctypes.POINTER(ctypes.c_int)]

    def call(Nx, tiles, sms=152, forced=0, untimed=17, tune=True):
        out = (ctypes.c_int * 32)()
        return list(out[:fn(Nx, tiles, sms, forced, untimed, int(tune), out)])

    return call


@pytest.mark.parametrize("forced,want", [(1, 1), (9, 9), (200, 200), (500, 200)])
def test_the_options_chunk_is_the_only_one(chunks, forced, want):
    assert chunks(200, 91, forced=forced) == [want]
    assert chunks(200, 91, forced=forced, tune=False) == [want]


def test_nothing_is_timed_with_tuning_off(chunks):
    assert chunks(200, 91, tune=False) == [17]


@pytest.mark.parametrize("Nx", [1, 7, 12, 56, 200, 65535])
@pytest.mark.parametrize("tiles", [1, 91, 5000, 4096 * 2048])
def test_candidates(chunks, Nx, tiles):
    v = chunks(Nx, tiles, untimed=min(17, Nx))
    assert v[0] == min(17, Nx) and len(v) >= 2
    assert all(1 <= c <= Nx for c in v) and len(set(v[1:])) == len(v) - 1
