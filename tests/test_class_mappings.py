"""make_classes on mappings other than a dict: a field left out is 0, whatever the
mapping would make up for it, and the caller's mapping is left as it was."""
import collections
import types

from paper_1102_1343_gb300 import make_classes, synth


def test_mappings_with_defaults_of_their_own():
    full = synth.nominal_class()
    part = {k: v for k, v in full.items() if k not in ("st", "chaparral")}
    want = bytes(make_classes([dict(part, st=0.0, chaparral=0)]))

    class Upper(dict):
        def __missing__(self, key):
            return 7.0

    filled = collections.defaultdict(lambda: 3.0, part)
    for c in (part, filled, Upper(part), collections.ChainMap(part), types.MappingProxyType(part)):
        assert bytes(make_classes([c])) == want
    assert dict(filled) == part
