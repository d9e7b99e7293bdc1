"""The binding's own state, without a GPU."""
import ctypes

import paper_2512_11280_b200 as adasd
from paper_2512_11280_b200 import binding


class FakeTensor:
    def __init__(self, address):
        self.address = address

    def data_ptr(self):
        return self.address


FIELDS = [n for n, _ in adasd.RoundRecord._fields_]


def record(base):
    return {n: FakeTensor(base + 16 * i) for i, n in enumerate(FIELDS)}


def addresses(ref):
    r = ctypes.cast(ref, ctypes.POINTER(adasd.RoundRecord)).contents
    return [getattr(r, n) for n in FIELDS]


def test_a_call_gets_its_own_record_whatever_another_thread_does_between_two_statements():
    """Two threads that call one Context: whenever the binding stores what it keeps of a call's record, another
    call with another record runs whole.  Each call still gets the addresses of its own record, then and later."""
    a, b = record(1 << 20), record(1 << 30)
    want = {id(r): [t.address for t in r.values()] for r in (a, b)}

    class Interleaved(binding.Context):
        armed = False

        def __setattr__(self, name, value):
            object.__setattr__(self, name, value)
            if self.armed:
                self.armed = False
                assert addresses(self._record_ref(b)) == want[id(b)]

    ctx = Interleaved.__new__(Interleaved)
    ctx.handle = None
    for name in ("_rec", "_rec_key"):
        object.__setattr__(ctx, name, None)
    assert ctx._record_ref(None) is None
    for _ in range(3):
        object.__setattr__(ctx, "armed", True)
        assert addresses(ctx._record_ref(a)) == want[id(a)]
        object.__setattr__(ctx, "armed", False)
        assert addresses(ctx._record_ref(a)) == want[id(a)]
        assert addresses(ctx._record_ref(b)) == want[id(b)]
    a["H_t"] = None
    assert addresses(ctx._record_ref(a))[FIELDS.index("H_t")] is None
