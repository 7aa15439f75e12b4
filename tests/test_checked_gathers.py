"""The bounds-checked build tests the addresses that the library ships with: the gathers of the
brick kernel form them the same way in both builds, and only the tap loaders and the
checks themselves know of AC_CHECKED.  On the GPU: the check of a shared-memory address at
every byte around an array, and gathers of voxel types and sample counts that the other
checked cases leave out, in bounds and the same in both builds."""
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_gathers_do_not_depend_on_the_checked_build():
    text = open(os.path.join(ROOT, "paper_1804_06304_gb300", "csrc", "ac_evolve.cuh")).read()
    loaders = text[text.index("template <typename T> struct SmemLoad"):text.index("template <typename T> struct GlobalLoad")]
    loaders += text[text.index("template <typename T> struct GlobalLoad"):].split("\n};")[0]
    assert text.count("AC_CHECKED") == loaders.count("AC_CHECKED") == 2


@pytest.mark.gpu
def test_address_check(tmp_path):
    from paper_1804_06304_gb300 import build
    exe = str(tmp_path / "checked_lds")
    subprocess.run([build.NVCC, *build.ARCH, "-O1", "-std=c++17", "-DAC_CHECKED", "-I" + build.INCLUDE, "-o", exe,
                    os.path.join(HERE, "_checked_lds_ref.cu")], check=True, capture_output=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split() == ["0"]


def _states():
    from paper_1804_06304_gb300 import ac
    rng = np.random.default_rng(8)
    out = {}
    for ndim, dims in ((3, (70, 61, 33)), (2, (150, 131))):
        for dtype in (np.uint8, np.uint16, np.float16, np.float32):
            V = ac.ac_create_volume((rng.random(dims[::-1]) * 200).astype(dtype))
            for N, kw in ((75, {}), (130, dict(compensated=0)), (64, dict(sampling=1))):
                C = ac.ac_seed(V, stride=5.0)
                ac.ac_evolve(C, ac.default_params(ndim, 4.0, 100.0, N=N, T=3, seed=6, **kw))
                out[f"{ndim}{np.dtype(dtype).name}{N}"] = ac.ac_get_state(C)
    return out


@pytest.mark.gpu
def test_other_gathers_stay_in_bounds(tmp_path):
    out = tmp_path / "checked.npz"
    r = subprocess.run([sys.executable, "-m", "tests.test_checked_gathers", str(out)], cwd=ROOT,
                       env=dict(os.environ, AC_BUILD="checked"), capture_output=True, text=True, timeout=1800)
    assert r.returncode == 0, r.stderr[-3000:]   # a bounds report raises at the child's first synchronizing call
    checked, normal = np.load(out), _states()
    assert sorted(checked.files) == sorted(normal)
    for k, v in normal.items():
        np.testing.assert_allclose(checked[k], v, rtol=1e-3, atol=1e-3, err_msg=k)


if __name__ == "__main__":
    np.savez(sys.argv[1], **_states())
