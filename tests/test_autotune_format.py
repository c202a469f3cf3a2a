"""Stored tile choices and what their codes meant when they were measured: an entry of the format before code 1
became the rule by size (a bare list) is measured anew, a current one is applied. CPU, with a stand-in for the
library."""
import ctypes as C
import json

from paper_1712_08743_gb300 import autotune


class FakeLib:
    def __init__(self):
        self.tuned, self.applied = 0, 0

    def helm_autotune(self, handle, nrhs, omega, arr):
        self.tuned += 1
        arr[5] = 4
        return 0

    def helm_set_tiles(self, handle, arr):
        self.applied += 1
        return 0


class FakeModel:
    def __init__(self, lib):
        self.lib, self.nx, self.nz, self.handle = lib, 441, 241, C.c_void_p()


def test_choices_of_other_shapes_are_measured_anew(tmp_path):
    path = tmp_path / "tiles.json"
    key = autotune.cache_key(441, 241, 8)
    old = [1] * autotune.NTILES
    path.write_text(json.dumps({key: old, "other": old}))
    lib = FakeLib()
    got = autotune.autotune(FakeModel(lib), 8, 30.0, str(path))
    assert (lib.tuned, lib.applied) == (1, 0) and got[5] == 4
    assert autotune.load_cache(str(path))["other"] == old
    assert autotune.autotune(FakeModel(lib), 8, 30.0, str(path)) == got
    assert (lib.tuned, lib.applied) == (1, 1)
