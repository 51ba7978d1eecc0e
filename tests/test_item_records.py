"""The records of a mixed batch as the library reads them: dicts, Item structures and structures derived from Item."""
import ctypes

from paper_1107_5578_gb300 import cwo


class Tagged(cwo.Item):
    _fields_ = [("tag", ctypes.c_double)]


def test_every_form_gives_the_same_record():
    plain = cwo.Item(0.1, 532e-9, 8e-6, 6e-6, cwo.FRESNEL_CONV, 4)
    tagged = Tagged(0.1, 532e-9, 8e-6, 6e-6, cwo.FRESNEL_CONV, 4, 7.0)
    as_dict = {"z": 0.1, "wavelength": 532e-9, "dx": 8e-6, "dy": 6e-6, "type": cwo.FRESNEL_CONV, "flags": 4}
    got = cwo.item_records([tagged, as_dict, plain, tagged, as_dict])
    assert len(got) == 5
    assert all(bytes(r) == bytes(plain) for r in got)
