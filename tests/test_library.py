"""CPU-side checks of the native library: it builds for sm_103a, loads, and exports the C ABI."""
import ctypes
import os
import re
import subprocess

import paper_1805_08831_gb300 as dt
from paper_1805_08831_gb300.build import CSRC


def test_library_exports_every_declared_symbol():
    L = dt.lib()
    names = dt.exported_names()
    assert "dt_create" in names and "dt_insert" in names and "dt_get_tets" in names
    for name in names:
        assert hasattr(L, name), name


def test_strerror_and_argument_checks_need_no_gpu():
    L = dt.lib()
    assert L.dt_strerror(dt.DT_EDEGENERATE).decode().startswith("fewer than four")
    assert L.dt_create(None, None) == dt.DT_EINVAL
    cfg = dt.Config()
    cfg.reserved[0] = 1
    h = ctypes.c_void_p()
    assert L.dt_create(ctypes.byref(h), ctypes.byref(cfg)) == dt.DT_EINVAL
    assert L.dt_insert(None, None, 0) == dt.DT_EINVAL
    assert L.dt_get_stats(None, None) == dt.DT_EINVAL
    assert L.dt_eval_predicates(7, None, None, None, 0, None) == dt.DT_EINVAL
    L.dt_destroy(None)


def test_a_value_kept_per_device_is_made_on_each(tmp_path):
    """Kernel attributes belong to a device: a second device gets its own, once."""
    src = tmp_path / "per_device.cpp"
    src.write_text('''
#include "per_device.h"
int main() {
  static dtg::PerDevice kept;
  int made[70] = {};
  for (int turn = 0; turn < 3; ++turn)
    for (int dev = 0; dev < 70; ++dev)
      if (kept.get(dev, [&] { ++made[dev]; return dev % 3; }) != dev % 3) return 1;
  for (int dev = 0; dev < 70; ++dev)
    if (made[dev] != (dev < dtg::PerDevice::kDevices ? 1 : 3)) return 2;
  return kept.get(-1, [] { return 5; }) == 5 ? 0 : 3;
}
''')
    exe = str(tmp_path / "per_device")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", exe])
    assert subprocess.run([exe]).returncode == 0


def test_kernel_attributes_are_not_kept_per_process():
    """A function-local static that is not a PerDevice holds the first device's answer for all."""
    for name in os.listdir(CSRC):
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        for line in text.splitlines():
            if re.match(r"\s+static (const )?(int|bool|unsigned|uint32_t|auto)\b.*=", line) and "constexpr" not in line:
                raise AssertionError(f"{name}: {line.strip()}")
