/* An NVTX injection library that prints the name of every range pushed: a stand-in
 * for a timeline profiler (loaded through NVTX_INJECTION64_PATH). */
#include <nvtx3/nvToolsExt.h>
#include <stdio.h>

static int push(const char *name) {
    fprintf(stderr, "range %s\n", name);
    return 0;
}

int InitializeInjectionNvtx2(NvtxGetExportTableFunc_t get) {
    const NvtxExportTableCallbacks *t = (const NvtxExportTableCallbacks *)get(NVTX_ETID_CALLBACKS);
    NvtxFunctionTable table;
    unsigned int n;
    if (!t || !t->GetModuleFunctionTable(NVTX_CB_MODULE_CORE, &table, &n)) return 0;
    *table[NVTX_CBID_CORE_RangePushA] = (NvtxFunctionPointer)push;
    return 1;
}
