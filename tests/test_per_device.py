"""Kernel attributes hold for one device: the set-up runs once on each device of the
process, not once in the process."""
import ctypes

import numpy as np


def test_set_up_once_on_each_device():
    from paper_1810_01319_gb300 import build
    hc = ctypes.CDLL(build.build_hostcheck())
    devices = np.array([0, 0, 3, 1, 3, 70, 0, 70, 1], np.int32)
    calls = np.zeros(71, np.int32)
    hc.cello_hc_once_per_device(ctypes.c_void_p(devices.ctypes.data), len(devices), ctypes.c_void_p(calls.ctypes.data))
    assert list(np.flatnonzero(calls)) == [0, 1, 3, 70] and calls.max() == 1


def test_no_set_up_is_once_per_process():
    """Every function attribute is set from a set-up that runs per device."""
    import pathlib
    from paper_1810_01319_gb300 import build
    for f in pathlib.Path(build.CSRC).iterdir():
        assert "once_flag" not in f.read_text(), f.name
