"""A pass whose launch fails leaves the results of the pass before it in place. The failure is made on the host: a preloaded library stands
in for the launcher of one-row passes and, when told to, returns an error instead of calling it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <dlfcn.h>
#include <stddef.h>
#define NAME "_ZN3asd14launch_pass_m1ERKNS_10PassParamsEimP11CUstream_st"
static int failing = 0;
extern "C" void set_failing(int v) { failing = v; }
extern "C" int launch(const void* p, int grid, size_t smem, void* stream) __asm__(NAME);
extern "C" int launch(const void* p, int grid, size_t smem, void* stream) {
    if (failing) return 701;  // cudaErrorLaunchOutOfResources
    static auto real = (int (*)(const void*, int, size_t, void*))dlsym(dlopen(LIBASD, RTLD_NOLOAD | RTLD_LAZY), NAME);
    return real(p, grid, smem, stream);
}
"""

PROGRAM = r"""
import ctypes, sys
import numpy as np
import synth
import paper_2410_01028_b200 as asd
fake = ctypes.CDLL(sys.argv[1])
dec = asd.Decoder(synth.TINY, max_seq=64, max_draft=8)
dec.load_weights_host(synth.make_model(synth.TINY, seed=0))
dec.set_debug(True)
dec.prefill([1, 2, 3])
for temperature in (0.7, 0.0):  # logits of a sampled pass stay on the device, those of a greedy one are on the host as well
    dec.set_sampling(temperature, 1)
    dec.decode_step(4)
    want, cosines = dec.get_last_logits(), dec.get_last_cosines()
    dec.set_sampling(0.0)
    fake.set_failing(1)
    try:
        dec.decode_step(5)
        sys.exit("the launch did not fail")
    except asd.AsdError as e:
        assert e.code == -5, e.code
    fake.set_failing(0)
    np.testing.assert_array_equal(dec.get_last_logits(), want)
    np.testing.assert_array_equal(dec.get_last_cosines()[0], cosines[0])
dec.decode_step(5)  # and the decoder goes on
assert not np.array_equal(dec.get_last_logits(), want)
"""


def test_results_of_the_pass_before_survive_a_failed_launch(tmp_path):
    lib = os.path.join(ROOT, "paper_2410_01028_b200", "libasd.so")
    (tmp_path / "fake.cpp").write_text(FAKE)
    (tmp_path / "program.py").write_text(PROGRAM)
    fake = str(tmp_path / "fake.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", '-DLIBASD="%s"' % lib, "-o", fake, str(tmp_path / "fake.cpp"), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, str(tmp_path / "program.py"), fake], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
