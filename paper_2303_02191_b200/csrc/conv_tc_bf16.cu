// The tensor path's kernel forms for bf16 data (see conv_tc_forms.cuh).
#include "conv_tc_forms.cuh"

namespace {
const FormTable& forms() {
    static const FormTable t = make_forms<__nv_bfloat16>();
    return t;
}
}  // namespace

void* rtoss_tc_form_bf16(int form, bool shared) { return find_form(form, shared); }
int rtoss_tc_prepare_forms_bf16() { return prepare_forms(); }
