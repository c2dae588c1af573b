"""Host replay of the asynchronous copies of the strip kernel (strip_walk; no
GPU): which copy each iteration issues, into which slot, in which group, and
which groups its wait leaves in flight.  Every value an iteration reads -- rows of
populations, force rows of every level, the residual snapshot of a checked launch
-- must have been copied to the slot it is read from by a group that the
iteration's wait covers, and no copy may be issued to a slot whose last copy can
still be in flight.  The expressions are read from the kernel's source."""
import os
import re

import pytest

from conftest import ROOT

SRC = open(os.path.join(ROOT, "paper_2208_14870_gb300", "csrc", "lbm_kernels.cuh")).read()
WALK = SRC[SRC.index("void strip_walk("):SRC.index("k_strip(const StepParams")]


def _value(expr, **env):
    """A C++ integer expression of names, arithmetic and ?: (a nested one last, in brackets)."""
    expr = re.sub(r"st_(\w+)<[^>]*>\(\)", r"st_\1", expr).strip()
    m = re.match(r"([^?]*)\?([^:]*):(.*)$", expr)
    if not m:
        return eval(expr, {}, env)
    test, yes, no = (t.strip() for t in m.groups())
    if "?" in no:
        no = no[1:-1]
    return _value(yes if _value(test, **env) else no, **env)


def _function(name):
    return re.search(r"constexpr int st_%s\(\) \{\s*return ([^;]+);" % name, SRC).group(1)


def _constants(S, T):
    env = dict(S=S, T=T, S_F32=1, S_F16S=2, kWvD=int(re.search(r"constexpr int kWvD = (\d+);", SRC).group(1)))
    for name in ("lag", "la", "halo", "ring"):
        env["st_" + name] = _value(_function(name), **env)
    env.update(LAG=env["st_lag"], LA=env["st_la"], H=env["st_halo"], R=env["st_ring"])
    env["SN"] = _value(_function("snaps"), **env)
    env["OFF"] = _value(re.search(r"\bOFF = ([^;]+);", WALK).group(1), **env)
    env["AHEAD"] = _value(re.search(r"\bAHEAD = ([^;]+);", WALK).group(1), **env)
    return env


class Slots:
    """Copies to a ring of slots: what each holds, and by which group."""

    def __init__(self):
        self.held = {}

    def copy(self, slot, what, group, done):
        assert slot not in self.held or self.held[slot][1] <= done, "slot %d: its last copy may be in flight" % slot
        self.held[slot] = (what, group)

    def read(self, slot, what, done):
        assert self.held.get(slot, (None, 0))[0] == what, "slot %d holds %s, not %s" % (slot, self.held.get(slot), what)
        assert self.held[slot][1] <= done, "the copy of %s may be in flight" % (what,)


def _replay(S, T, check, rows):
    c = _constants(S, T)
    wait = _value(re.search(r'cp\.async\.wait_group %0;" ::"n"\((\w+)\)', WALK).group(1), **c)
    lead = _value(re.search(r"snp \+ \(\(i \+ (\w+)\) & ", WALK).group(1), **c)
    put = _value(re.search(r"snp \+ \(\(i \+ \w+\) & (.+?)\) \* 1024;", WALK).group(1), **c)
    got = re.findall(r"lds_pairs\(snp \+ \(i & (.+?)\) \* 1024", WALK)
    assert len(got) == 2 and _value(got[0], **c) == _value(got[1], **c) == put
    nit, H, mask = rows + 2 * c["H"], c["H"], put
    pops, force, snap = Slots(), Slots(), Slots()
    group = 0                      # groups committed
    done = 0                       # groups known to have landed

    def copy_row(r):
        pops.copy(r & (c["kWvD"] - 1), r, group + 1, done)
        force.copy(r & (c["R"] - 1), r, group + 1, done)

    for r in range(c["AHEAD"]):
        copy_row(r)
        group += 1
    for i in range(nit):
        if check and i + lead >= 2 * H and i + lead < nit:
            snap.copy((i + lead) & mask, i + lead, group + 1, done)
        copy_row(i + c["AHEAD"])
        group += 1
        done = max(done, group - wait)
        for r in ((i, i + 1, i + 2) if S == 1 else (i,)):
            pops.read(r & (c["kWvD"] - 1), r, done)
        for j in range(1, T + 1):
            if i < 2 * (j - 1 + c["LAG"]):
                break
            r = i + c["OFF"] - c["LAG"] - (j - 1)
            force.read(r & (c["R"] - 1), r, done)
        if check and i >= 2 * H:
            snap.read(i & mask, i, done)


# every launch the library makes: FP32 (1) two to six steps, checked four and
# five; FP16S (2) three and four, checked four
@pytest.mark.parametrize("S,T,check", [(1, T, False) for T in range(2, 7)] + [(1, 4, True), (1, 5, True), (2, 3, False),
                                                                            (2, 4, False), (2, 4, True)])
@pytest.mark.parametrize("rows", [1, 2, 3, 40])
def test_reads_wait_for_their_copies(S, T, check, rows):
    _replay(S, T, check, rows)
