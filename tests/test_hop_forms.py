"""A launcher refuses, before anything is launched, a form that it does not have (no GPU needed).

The hopping kernels exist for some pairs of mode and precision only, and some of
those with natural output only: a call outside them used to launch nothing, read
fields of another layout or write through a null pointer.  A small program linked
with the library makes such calls and says which were refused.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROBE = r"""
#include <cstdio>
#include "lq_kernels.h"
using namespace lq;

static Geom geom(int l)
{
    Geom g{};
    for (int mu = 0; mu < 4; mu++) g.L[mu] = l;
    g.Lxh = l / 2;
    g.V = (long long)l * l * l * l;
    g.Vh = g.V / 2;
    g.stride = (g.Vh + 63) / 64 * 64;
    g.tbc = -1;
    return g;
}

int main()
{
    Counters ctr{};
    char a, b, n;
    auto refused = [&](const char *name, int l, auto call) {
        Exec e{geom(l), nullptr, &ctr, nullptr};
        const long long before = ctr.launches;
        bool r = false;
        try {
            call(e);
        } catch (const Refused &) {
            r = true;
        }
        std::printf("%s %d %s\n", name, l, r && ctr.launches == before ? "refused" : "launched");
    };
    for (int l : {8, 16, 20}) {   // 2048, 32768 and 80000 sites a parity: either side of every switch
        for (int mode = HOP_K1; mode <= HOP_RECON_RES; mode++)
            for (int prec : {P32, P16}) {
                if (hop_form(mode, prec)) continue;
                refused("hop", l, [&](const Exec &e) {
                    HopCall c{};
                    c.mode = mode;
                    c.prec = prec;
                    c.in = c.in2 = c.b = &a;
                    c.out = c.out2 = &b;
                    hop(e, c);
                });
            }
        auto form = [&](const char *name, int mode, int prec, void *out, void *nat, bool in32, bool out32, int nrhs) {
            refused(name, l, [&](const Exec &e) {
                HopCall c{};
                c.mode = mode;
                c.prec = prec;
                c.in = c.in2 = c.b = &a;
                c.out = out;
                c.nat = nat;
                c.in32 = in32;
                c.out32 = out32;
                c.nrhs = nrhs;
                hop(e, c);
            });
        };
        form("bf16_k2_without_natural", HOP_K2, P16, &b, nullptr, false, false, 1);
        form("bf16_k1_two_fields", HOP_K1, P16, &b, nullptr, false, false, 2);
        form("full_without_natural", HOP_FULL, P32, &b, nullptr, false, false, 1);
        form("k1_natural", HOP_K1, PDF, &b, &n, false, false, 1);
        form("k2_no_output", HOP_K2, PDF, nullptr, nullptr, false, false, 1);
        form("k2_natural_two_fields", HOP_K2, P64, nullptr, &n, false, false, 2);
        form("recon_f64_in32", HOP_RECON, P64, nullptr, &n, true, false, 1);
        form("recon_in32_internal", HOP_RECON, PDF, &b, nullptr, true, false, 1);
        form("prep_f64_out32", HOP_PREP, P64, &b, nullptr, false, true, 1);
        form("prep_out32_two_fields", HOP_PREP, PDF, &b, nullptr, false, true, 2);
        form("unknown_mode", 8, PDF, &b, nullptr, false, false, 1);
        form("unknown_precision", HOP_K1, 4, &b, nullptr, false, false, 1);
        refused("export_half_bf16", l, [&](const Exec &e) { export_half(e, P16, &a, &b); });
        refused("export_full_bf16", l, [&](const Exec &e) { export_full(e, P16, &a, &a, &b); });
        refused("import_full_bf16", l, [&](const Exec &e) { import_full(e, P16, &a, &b, &b); });
        refused("gamma5_bf16", l, [&](const Exec &e) { gamma5(e, P16, &a, &b); });
        refused("clover_mul_bf16", l, [&](const Exec &e) { clover_mul(e, P16, &a, &a, &b); });
        refused("convert_two_f64", l, [&](const Exec &e) { convert(e, P64, &a, P32, &b, 2); });
        refused("convert_two_bf16", l, [&](const Exec &e) { convert(e, P32, &a, P16, &b, 2); });
    }
    // FP32 ends of the df64 hops exist on the larger lattices alone
    refused("recon_in32_small", 8, [&](const Exec &e) {
        HopCall c{};
        c.mode = HOP_RECON;
        c.prec = PDF;
        c.in = c.in2 = &a;
        c.nat = &n;
        c.in32 = true;
        hop(e, c);
    });
    // what the operators, the smoother and the solves ask for
    struct Used {
        int mode, prec;
        bool nat, in32, out32;
        int nrhs, l;
    };
    const Used used[] = {
        {HOP_K1, P64, false, false, false, 1, 8},  {HOP_K2, P64, true, false, false, 1, 20},
        {HOP_K2, P64, false, false, false, 1, 8},  {HOP_RICH, P64, false, false, false, 1, 8},
        {HOP_K1, P32, false, false, false, 1, 20}, {HOP_K2, P32, false, false, false, 1, 20},
        {HOP_K2, P32, true, false, false, 1, 8},   {HOP_RICH, P32, false, false, false, 1, 8},
        {HOP_FULL, P32, true, false, false, 1, 8}, {HOP_FULL, PDF, true, false, false, 1, 20},
        {HOP_K1, PDF, false, false, false, 12, 8}, {HOP_K2, PDF, false, false, false, 12, 8},
        {HOP_PREP, PDF, false, false, false, 12, 16}, {HOP_PREP, PDF, false, false, true, 1, 16},
        {HOP_RECON, PDF, false, false, false, 1, 8}, {HOP_RECON, PDF, true, true, false, 1, 16},
        {HOP_RES, PDF, false, false, false, 12, 8}, {HOP_RECON_RES, P64, false, false, false, 1, 8},
        {HOP_K1, P16, false, false, false, 1, 8},  {HOP_K2, P16, true, false, false, 1, 8},
        {HOP_RICH, P16, false, false, false, 1, 20}};
    for (const Used &u : used) {
        HopCall c{};
        c.mode = u.mode;
        c.prec = u.prec;
        c.in = c.in2 = c.b = &a;
        c.out = u.nat ? nullptr : &b;
        c.nat = u.nat ? &n : nullptr;
        c.in32 = u.in32;
        c.out32 = u.out32;
        c.nrhs = u.nrhs;
        if (const char *why = hop_refused(geom(u.l), c)) std::printf("used %d %d %s\n", u.mode, u.prec, why);
    }
    return 0;
}
"""


def test_forms_that_do_not_exist_are_refused(tmp_path):
    from paper_2407_08092_gb300 import build
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not available")
    lib = build.build()
    src = tmp_path / "probe.cu"
    src.write_text(PROBE)
    exe = tmp_path / "probe"
    r = subprocess.run([cc, *build.ARCH, "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, str(src), "-o", str(exe),
                        lib, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120,
                       env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))   # no device, whatever gets through
    assert r.returncode == 0, r.stderr
    lines = r.stdout.splitlines()
    assert len(lines) > 60
    assert not [x for x in lines if not x.endswith(" refused")]
