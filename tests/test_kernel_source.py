"""CPU-side checks of the kernel source: rules that the compiler does not enforce and that no output shows when they are broken."""
import os
import re

from paper_2410_23208_b200 import build

KERNELS = os.path.join(build.HERE, "csrc", "k2d_kernels.cuh")


def _source():
    """the kernel source without its comments"""
    text = re.sub(r"/\*.*?\*/", "", open(KERNELS).read(), flags=re.S)
    return re.sub(r"//[^\n]*", "", text)


def _arguments(text, call):
    """(position, argument text) of every call of the function"""
    for m in re.finditer(r"\b%s\(" % re.escape(call), text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield m.start(), text[m.end():i - 1]


def _without_calls(text, name):
    """the text without the calls name<...>(...), arguments included"""
    out, at = [], 0
    for m in re.finditer(r"\b%s<\w+>\(" % re.escape(name), text):
        if m.start() < at:
            continue
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        out.append(text[at:m.start()])
        at = i
    return "".join(out) + text[at:]


def _base(expression):
    """the pointer an address expression starts from"""
    inner = re.sub(r"reinterpret_cast<[^>]*>\(", "", expression)
    return re.match(r"[\s(]*([A-Za-z_][\w.]*)", inner).group(1)


def test_read_only_cache_loads_read_nothing_but_the_level_pool():
    # A load through the read-only cache (__ldg) is defined only for words that nobody writes while the kernel is on the
    # device, and a kernel launched ahead of its turn is on the device while the kernel in front of it still writes.  The
    # level pool, written once by the host, is the only input that qualifies.
    text = _source()

    def in_pool(name, at):
        if name in ("levels", "prm.levels"):
            return True
        if "." in name:
            return False
        # the definition in force: the last one before the use, a variable's or a level record handed in as a parameter
        found = list(re.finditer(r"\*\s*%s( = [^;]*;|\s*[,)])" % re.escape(name), text[:at]))
        assert found, name
        d = found[-1]
        return name == "lv" if not d.group(1).startswith(" =") else in_pool(_base(d.group(1)[3:]), d.start())

    calls = list(_arguments(text, "__ldg"))
    assert len(calls) > 10
    for at, argument in calls:
        assert in_pool(_base(argument), at), f"__ldg({argument}) does not read the level pool"
    assert not re.search(r"ld\.global\.nc|__restrict__", text)


def test_every_body_index_goes_through_the_index_check():
    # the body fields of a contact pair's word ("ab": alone, in an array of a lane's words or in a record), of a survivor code, of
    # a joint's or thruster's word and of the dense reward's shapes; the checked build replaces an index out of range, a raw
    # field would be used as it is.  An action binding is no index here: it is compared with the number of channels.
    text = _without_calls(_source(), "ck_idx")
    raw = re.findall(r"[^;{}]*\b(?:ab(?:\[i\])?|code|jab|jw0|tp|gb)(?: >> \d+\))? & (?:15|31|255)u?\b[^;{}]*;", text)
    assert not [r for r in raw if "bind = " not in r], raw
    assert len(re.findall(r"ck_idx<CK_BODY>", _source())) > 30


def test_every_level_id_goes_through_the_index_check():
    text = _without_calls(_source(), "ck_idx")
    text = re.sub(r"enum \{ META_STEP[^}]*\}", "", text)
    text = re.sub(r"\w+\[SC::META \+ META_LEVEL\] = [^;]*;", "", text)                # stores
    text = re.sub(r"min\(__ldcg\(st \+ SC::ST_META \+ META_LEVEL\), [^;]*;", "", text)      # limited in every build
    assert not re.findall(r"[^;{}]*META_LEVEL[^;{}]*;", text)
