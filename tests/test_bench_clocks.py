"""The benchmark's clock record against a stand-in for NVML: only what is sampled inside the timed region counts, however short it is."""
import ctypes
import time

import bench


class FakeNvml:
    def __init__(self, known=True):
        self.known, self.mhz, self.why = known, 345, 0x1           # idle

    def nvmlInit_v2(self):
        return 0

    def nvmlDeviceGetHandleByUUID(self, uuid, dev):
        assert uuid.startswith(b"GPU-")
        return 0 if self.known else 6

    def nvmlDeviceGetClockInfo(self, dev, kind, out):
        ctypes.cast(out, ctypes.POINTER(ctypes.c_uint))[0] = self.mhz
        return 0

    def nvmlDeviceGetMaxClockInfo(self, dev, kind, out):
        ctypes.cast(out, ctypes.POINTER(ctypes.c_uint))[0] = 1965
        return 0

    def nvmlDeviceGetCurrentClocksThrottleReasons(self, dev, out):
        ctypes.cast(out, ctypes.POINTER(ctypes.c_ulonglong))[0] = self.why
        return 0


def test_a_region_of_a_few_milliseconds_has_its_samples():
    nvml = FakeNvml()
    s = bench.ClockSampler("0-1-2", nvml)
    s.start()
    time.sleep(0.03)
    nvml.mhz, nvml.why = 1900, 0x4 | 0x40
    time.sleep(0.01)                                              # (a sample may be under way)
    s.begin()
    time.sleep(0.016)
    assert s.stop() == {"sm_mhz": 1900.0, "sm_max_mhz": 1965.0, "reasons": ["hw_thermal_slowdown", "sw_power_cap"]}


def test_without_the_device_there_is_no_record():
    s = bench.ClockSampler("0-1-2", FakeNvml(known=False))
    s.start()
    s.begin()
    assert s.stop() == {"sm_mhz": None, "sm_max_mhz": None, "reasons": []}
