"""What the binding passes on, without a GPU: a stand-in for the library records the arguments."""
import numpy as np

from paper_2507_14959_b200 import binding


class Recorder:
    def __init__(self):
        self.calls = {}

    def __getattr__(self, name):
        def call(*args):
            self.calls[name] = args
            return binding.PM_OK
        return call


def model():
    m = object.__new__(binding.Model)
    m.lib, m.handle = Recorder(), 1
    return m


def test_buffers_may_be_arrays_or_tensors():
    """Frames and scores are device addresses with a first dimension: torch tensors, or arrays over memory the device can reach
    (pinned or managed)."""
    import torch
    off, ids = np.array([0, 1, 2, 2], np.int32), np.array([4, 0], np.int32)
    for make in (lambda s: np.zeros(s, np.float32), lambda s: torch.zeros(s)):
        frames, scores, words = make((3, 3, 16, 16)), make((3, 5)), make((3, 1))
        m = model()
        m.forward(frames, off, ids, scores, None, stream=0)
        m.forward_device_sets(frames, off, ids, scores, None, stream=0)
        m.forward_branched(frames, off, ids, 1, scores, None, stream=0)
        m.select(scores, 0.5, False, False, words, None, None, torch.zeros(4, dtype=torch.int32), torch.zeros(9, dtype=torch.int32), stream=0)
        for name in ("pm_forward", "pm_forward_device_sets", "pm_forward_branched"):
            args = m.lib.calls[name]
            assert args[1] == binding._ptr(frames) and args[2] == 3 and args[3] == off.ctypes.data, name
        assert m.lib.calls["pm_select"][1:3] == (binding._ptr(scores), 3)
        m.handle = None


def test_set_lists_of_other_types_and_strides_are_converted():
    frames, scores = np.zeros((2, 3, 16, 16), np.float32), np.zeros((2, 5), np.float32)
    m = model()
    seen = []
    m.lib.pm_forward = lambda h, f, n, off, ids, *rest: seen.append(
        (list(np.ctypeslib.as_array((binding.C.c_int32 * 3).from_address(off))), list(np.ctypeslib.as_array((binding.C.c_int32 * 2).from_address(ids))))) or 0
    read_only = np.array([0, 1, 2], np.int32)
    read_only.flags.writeable = False
    for off, ids in ((np.array([0, 1, 2], np.int64), np.array([3, 4], np.int64)), (np.array([0, 9, 1, 9, 2], np.int32)[::2], np.array([3, 4], ">i4")),
                     (read_only, np.array([3, 4], np.int32))):
        m.forward(frames, off, ids, scores, None, stream=0)
    assert seen == [([0, 1, 2], [3, 4])] * 3
    m.handle = None
