"""Set-up that belongs to a device (csrc/device_once.h): each device needs it once, whatever other devices had it,
and a device beyond those remembered needs it every time.  flagnet.cu sets its gradient kernel's
shared-memory limit (80 KB, above the default 48) through it, so that a second GPU of a process gets it too."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2304_09724_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "device_once.h"
int main() {
  shweno::DeviceOnce o;
  const int devs[] = {0, 1, 0, 63, 1, 63, 64, 64};
  for (int dev : devs) {
    std::printf("%d", o.needed(dev) ? 1 : 0);
    o.done(dev);
  }
}
"""


def test_each_device_once(tmp_path):
    src, exe = tmp_path / "once.cpp", str(tmp_path / "once")
    src.write_text(PROGRAM)
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", exe])
    assert subprocess.check_output([exe], text=True) == "11010011"


def test_no_process_wide_flag_for_a_device_limit():
    """No source keeps "already set" for a device attribute in one flag for all devices."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            assert "static bool" not in open(os.path.join(CSRC, name)).read(), name
