"""CPU check of the reductions' pool of mapped host memory (csrc/slots.h): at
most 64 slots of one page, given back and taken again, and a page that a device
reset has ended is replaced instead of written to."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_slots(tmp_path):
    exe = str(tmp_path / "slots")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I" + os.path.join(ROOT, "paper_1803_07822_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "slots_check.cpp"), "-o", exe, "-pthread"])
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
