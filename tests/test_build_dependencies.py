"""An object is compiled again when a header it includes has changed."""
import re

from paper_2609_22755_b200 import build


def test_every_included_header_is_a_dependency():
    known = {h.resolve() for h in build.headers_of_library()}
    for src in [*build.CSRC.glob("*.c*"), *build.CSRC.glob("*.h")]:
        for name in re.findall(r'#include "([^"]+)"', src.read_text()):
            assert (src.parent / name).resolve() in known, (src.name, name)
